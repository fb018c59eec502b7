"""FP64 path: several uneven domains in one launch against the oracle."""
import numpy as np
import pytest

from helpers import oracle_nodes, oracle_run_node
from paper_2508_18202_gb300 import sclbm as S
from paper_2508_18202_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("collision", [W.BGK, W.RR], ids=["bgk", "rr"])
@pytest.mark.parametrize("listed", [(True, False, True), (False, True, False), (True, True, True)])
def test_uneven_domains_match_oracle(O, collision, listed):
    """Three domains of 5, 13 and 1 nodes whose cells are no multiple of a
    block's 128, with and without listed cells (an outflow face has them,
    velocity faces all round have none) in first, middle and last place: every
    domain's first and last node at an odd and an even level, 1e-13 (a
    population is below 0.4, and each of 28 levels rounds it a few times)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    bc = [W.URBAN_BC if some else [W.VEL, W.VEL, W.VEL, W.VEL, W.BB, W.FS] for some in listed]
    doms = [dict(nx=37, ny=18, nz=11, seed=1, n_buildings=2, fp=(4, 6), h=(3, 7), bc=bc[0], quad_level=2),
            dict(nx=29, ny=23, nz=14, seed=2, n_buildings=3, fp=(3, 5), h=(3, 9), bc=bc[1], quad_level=3),
            dict(nx=52, ny=11, nz=9, seed=3, n_buildings=1, fp=(3, 4), h=(2, 4), bc=bc[2], quad_level=1)]
    assert all(d["nx"] * d["ny"] * d["nz"] % 128 for d in doms)
    wl = dict(W.URBAN_BATCHED, domains=doms, ramp_steps=5, tau0=0.56, precision=W.FP64_PLAIN, collision=collision,
              angle_deg=12.0)
    ens = S.Ensemble(S.make_config(wl))
    for steps, level in ((27, 27), (1, 28)):
        ens.step(steps)
        for d in range(3):
            _, a = oracle_nodes(O, wl, d)
            assert len(a) == ens.n_nodes[d]
            for j in sorted({0, len(a) - 1}):
                _, flags, f = oracle_run_node(O, wl, d, j, level)
                got = ens.populations(d, j).cpu().numpy()
                fl = np.asarray(flags) == 0
                assert np.max(np.abs(got[:, fl] - f[:, fl])) < 1e-13
    ens.close()
