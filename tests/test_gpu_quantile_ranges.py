"""Quantiles of the gPC surrogate on inputs that the FP32 selection does not
carry."""
import numpy as np
import pytest

from paper_2508_18202_gb300 import sclbm as S
from paper_2508_18202_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    S.lib()
    return torch.device("cuda")


def ensemble(**over):
    wl = dict(domains=[dict(nx=16, ny=16, nz=8, boxes=[], bc=W.URBAN_BC, quad_level=3)], tau0=0.56, c_smag=0.14,
              u_ref=0.05, alpha=0.25, angle_deg=5.0, H_ref=0.0, inputs=[W.SPEED], lo=[0.0], hi=[0.1],
              quad_rule=W.GH, ramp_steps=4, precision=W.FP32_SHIFT, gpc_degree=2)
    wl.update(over)
    return S.Ensemble(S.make_config(wl))


@pytest.mark.parametrize("n_cells", [3, 305, 1301])
def test_basis_beyond_the_float_range(cuda, n_cells):
    """A far sample whose second-order basis value (x^2 - 1) / sqrt(2) is above
    the largest float, where a cell's second coefficient is zero: the surrogate
    is c0 + c1 x, each value two operations away from numpy's (4 units)."""
    ens = ensemble()
    n = 16 * 16 * 8
    rng = np.random.RandomState(n_cells)
    coef = np.zeros((3, n))
    coef[0] = 1.0 + rng.rand(n)
    coef[1] = 1e-3 * (1.0 + rng.rand(n))
    coef[:, ::5] = 0.0
    samples = rng.uniform(-2.0, 2.0, (101, 1))
    samples[50] = 1e20
    samples[7] = -3e21
    cells = rng.permutation(n)[:n_cells].astype(np.int32)
    q = [0.0, 0.025, 0.5, 0.975, 1.0]
    got = ens.gpc_quantiles(0, torch.from_numpy(coef).cuda(), cells, samples, q).cpu().numpy()
    y = np.sort(coef[0, cells] + samples * coef[1, cells], axis=0)
    ranks = [max(int(np.ceil(v * 101)), 1) - 1 for v in q]
    assert np.all(np.abs(got - y[ranks]) <= 4 * 2.0 ** -52 * np.abs(y[ranks]))
    ens.close()
