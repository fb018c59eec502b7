"""Every class of the default launch shape, by its size and collision."""
import numpy as np
import pytest

from paper_2508_18202_gb300 import sclbm as S
from paper_2508_18202_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# size, nodes per input of two inputs, the class of each collision: block, slab, mode
CLASSES = [((33, 17, 13), 3, (32, 1, 1, S.SC_EXEC_GRAPH), (32, 1, 1, S.SC_EXEC_GRAPH)),
           ((45, 39, 21), 3, (32, 2, 2, S.SC_EXEC_LAUNCH), (32, 2, 2, S.SC_EXEC_LAUNCH)),
           ((65, 129, 31), 5, (32, 2, 4, S.SC_EXEC_LAUNCH), (32, 4, 8, S.SC_EXEC_LAUNCH)),
           ((98, 67, 33), 5, (32, 2, 4, S.SC_EXEC_LAUNCH), (32, 4, 8, S.SC_EXEC_LAUNCH))]


@pytest.mark.parametrize("size,level,bgk,rr", CLASSES)
@pytest.mark.parametrize("collision", [W.BGK, W.RR], ids=["bgk", "rr"])
@pytest.mark.parametrize("precision", [W.FP32_SHIFT, W.BF16_STORE], ids=["fp32", "bf16"])
def test_class_and_its_bits(size, level, bgk, rr, collision, precision):
    """The default is the class of the size and collision, and gives the bits
    of a given shape, on widths, heights and depths that are no multiple of
    its blocks and slabs (even and odd widths: the 16-bit even level pairs
    cells on even ones)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nx, ny, nz = size
    wl = dict(domains=[dict(nx=nx, ny=ny, nz=nz, boxes=[[8, 4, 0, 13, 10, 6], [20, 9, 0, 24, 15, 9]], bc=W.URBAN_BC,
                            quad_level=level)],
              tau0=0.52, c_smag=0.14, u_ref=0.05, alpha=0.25, angle_deg=5.0, H_ref=0.0, inputs=[W.SPEED, W.ALPHA],
              lo=[-0.1, 0.15], hi=[0.1, 0.35], quad_rule=W.GL, ramp_steps=3, precision=precision, gpc_degree=-1,
              collision=collision)
    got = []
    for given in (False, True):
        ens = S.Ensemble(S.make_config(wl))
        if given:
            S.sc_lbm_set_tuning(ens.h, 64, 2, 8, tile_order=1)
        else:
            t = S.sc_lbm_get_tuning(ens.h)
            want = rr if collision == W.RR else bgk
            assert (t["block_x"], t["block_y"], t["slab_z"], t["exec_mode"]) == want
        for n in (1, 14, 6):
            ens.step(n)
        got.append([ens.populations(0, j).cpu().numpy() for j in (0, level * level - 1)])
        ens.close()
    assert np.array_equal(got[0], got[1])
