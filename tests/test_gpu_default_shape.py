"""A handle at its default launch shape against one with a given shape."""
import numpy as np
import pytest

from paper_2508_18202_gb300 import sclbm as S
from paper_2508_18202_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size", [(45, 21, 14), (33, 65, 7), (64, 48, 33), (96, 97, 40)])
@pytest.mark.parametrize("precision", [W.FP32_SHIFT, W.FP16_STORE])
@pytest.mark.parametrize("series", [False, True])
def test_default_shape_is_bitwise_the_given_one(size, precision, series):
    """Each class of the default rule (graphs of eight levels, short and long
    slabs), rows and layers that are no multiple of its blocks, steps in
    chunks that start at odd levels and leave remainders of a graph; a level's
    cells are independent, so the populations are the same bits."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nx, ny, nz = size
    wl = dict(domains=[dict(nx=nx, ny=ny, nz=nz, boxes=[[8, 4, 0, 13, 10, 6]], bc=W.URBAN_BC, quad_level=3)],
              tau0=0.52, c_smag=0.14, u_ref=0.05, alpha=0.25, angle_deg=5.0, H_ref=0.0, inputs=[W.SPEED], lo=[-0.1],
              hi=[0.1], quad_rule=W.GL, ramp_steps=5, precision=precision, gpc_degree=2)
    got = []
    for given in (False, True):
        ens = S.Ensemble(S.make_config(wl))
        if given:
            S.sc_lbm_set_tuning(ens.h, 64, 2, 8, tile_order=1)
        if series:
            ens.set_inflow_series([1.0, 1.2, 0.9], [0.0, 15.0, -10.0], 16, 4)
        for n in (1, 8, 7, 16, 9, 25):
            ens.step(n)
        got.append(ens.populations(0, 1).cpu().numpy())
        ens.sync()
        ens.close()
    assert np.array_equal(got[0], got[1])
