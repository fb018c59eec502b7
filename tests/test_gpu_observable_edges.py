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


C_LAT = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0),
                  (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1),
                  (0, -1, -1), (0, 1, -1), (0, -1, 1)])


def test_velocity_is_the_rounded_quotient():
    """The exported velocity is momentum over density rounded once, bit for bit,
    on random populations and on those of a zero of either sign, of an infinite
    momentum at a finite density, and of a quotient beyond the float range."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nx, ny, nz = 19, 7, 5
    n, pitch, hdr = nx * ny * nz, 768, 48
    ens = ensemble(nx, ny, nz)
    buf = np.zeros(S.sc_lbm_state_size(ens.h), np.uint8)
    S.sc_lbm_save(ens.h, buf)
    g = buf[hdr:].view(np.float32)[19 * pitch:2 * 19 * pitch].reshape(19, pitch)   # node 1, level 0: natural order
    rng = np.random.RandomState(4)
    g[:, :n] = rng.uniform(-0.02, 0.02, (19, n))
    g[:, :40] *= np.float32(1e-12)
    for axis in range(3):
        for sign in (1, -1):
            c = 100 + 2 * axis + (sign < 0)
            g[:, c] = np.where(C_LAT[:, axis] * sign > 0, np.float32(-0.0), np.float32(0.0))
    g[:, 110:118] = 0.0
    for k, (p, m) in enumerate([(1, 2), (2, 1), (3, 4), (5, 6)]):
        g[p, 110 + k], g[m, 110 + k] = 3e38, -3e38                # infinite momentum, density 1
        g[p, 114 + k], g[m, 114 + k] = 1e32, -1e32                # 2e32 over a density of 2^-24
        g[18, 114 + k] = np.float32(2.0 ** -24 - 1.0)             # (added last, after the two cancel)
    with np.errstate(over="ignore"):
        m0, j = g[0, :n].copy(), [np.zeros(n, np.float32) for _ in range(3)]
        for a in range(3):
            j[a] = g[1 + 2 * a, :n].copy()
        for i in range(1, 19):
            m0 = m0 + g[i, :n]
            for a in range(3):
                if C_LAT[i, a] and i > 1 + 2 * a:
                    j[a] = j[a] + np.float32(C_LAT[i, a]) * g[i, :n]
        rho = np.float32(1.0) + m0
        want = np.stack([j[a] / rho for a in range(3)])
    assert np.all(rho > 0) and np.isinf(want[0, 110]) and np.isinf(want[0, 114])
    assert np.signbit(want[0, 100]) and want[0, 100] == 0 and np.signbit(want[2, 104])
    h = 1469598103934665603
    for byte in buf[hdr:].tobytes():
        h = ((h ^ byte) * 1099511628211) & ((1 << 64) - 1)
    buf[24:32] = np.frombuffer(np.uint64(h).tobytes(), np.uint8)
    S.sc_lbm_load(ens.h, buf)
    got = ens.velocity(0, 1).cpu().numpy()
    fluid = S.sc_lbm_geometry(ens.cfg, 0) == 0
    assert fluid.all()
    assert np.array_equal(got.view(np.int32), want.astype(np.float32).view(np.int32))
    ens.close()
