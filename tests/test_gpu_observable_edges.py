"""Observables of states and fields that hold infinities, NaN and signed zeros."""
import numpy as np
import pytest

from paper_2508_18202_gb300 import sclbm as S
from paper_2508_18202_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def ensemble(nx, ny, nz, boxes=(), **over):
    wl = dict(domains=[dict(nx=nx, ny=ny, nz=nz, boxes=list(boxes), bc=W.URBAN_BC, quad_level=3)], tau0=0.56,
              c_smag=0.14, u_ref=0.05, alpha=0.25, angle_deg=5.0, H_ref=0.0, inputs=[W.SPEED], lo=[-0.1], hi=[0.1],
              quad_rule=W.GL, ramp_steps=4, precision=W.FP32_SHIFT, gpc_degree=2)
    wl.update(over)
    return S.Ensemble(S.make_config(wl))


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan, 3e38])
def test_qcriterion_of_an_axis_without_fluid_neighbours(O, value):
    """The derivative along such an axis is zero whatever the cell's own
    velocity: a cell enclosed on all sides has Q = 0, and one enclosed along x
    alone has the Q of its other neighbours (half a unit of a float and 2^-40
    of the terms)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nx, ny, nz = 11, 9, 7
    boxes = [[3, 2, 2, 4, 5, 5], [5, 2, 2, 6, 5, 5], [4, 2, 2, 5, 3, 5], [4, 4, 2, 5, 5, 5], [4, 3, 2, 5, 4, 3],
             [4, 3, 4, 5, 4, 5], [7, 4, 3, 8, 7, 5], [9, 4, 3, 10, 7, 5]]
    ens = ensemble(nx, ny, nz, boxes)
    flags = S.sc_lbm_geometry(ens.cfg, 0)
    cell = lambda x, y, z: x + nx * (y + ny * z)
    closed, corridor = cell(4, 3, 3), cell(8, 5, 3)
    assert not flags[closed] and not flags[corridor] and flags[corridor - 1] and flags[corridor + 1]
    u = np.random.RandomState(2).uniform(-1.0, 1.0, (3, nx * ny * nz)).astype(np.float32)
    u[:, closed] = u[:, corridor] = value
    q = ens.qcriterion(0, torch.from_numpy(u).cuda()).cpu().numpy()
    with np.errstate(over="ignore", invalid="ignore"):
        want = O.qcriterion(u, flags, nx, ny, nz, W.URBAN_BC)
    assert q[closed] == 0.0 and want[closed] == 0.0
    assert np.isfinite(want[corridor])
    assert abs(q[corridor] - want[corridor]) <= abs(want[corridor]) * 2.0 ** -24 + 36.0 * 2.0 ** -40
    ens.close()
