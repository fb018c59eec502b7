"""Observable kernels on the GPU at the sizes and values where they can go
wrong, against FP64 restatements."""
import numpy as np
import pytest

from paper_2508_18202_gb300 import sclbm as S
from paper_2508_18202_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

VEL, OUT, BB, FS, PER = W.VEL, W.OUT, W.BB, W.FS, W.PER


@pytest.fixture(scope="module")
def cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    S.lib()
    return torch.device("cuda")


def ensemble(nx, ny, nz, bc, boxes=(), **over):
    wl = dict(domains=[dict(nx=nx, ny=ny, nz=nz, boxes=list(boxes), bc=bc, quad_level=3)], tau0=0.56, c_smag=0.14,
              u_ref=0.05, alpha=0.25, angle_deg=5.0, H_ref=0.0, inputs=[W.SPEED], lo=[-0.1], hi=[0.1],
              quad_rule=W.GL, ramp_steps=4, precision=W.FP32_SHIFT, gpc_degree=2)
    wl.update(over)
    return S.Ensemble(S.make_config(wl))


@pytest.mark.parametrize("scale", [1e-35, 1e-15, 1.0, 1e15, 1e25, 2e38])
@pytest.mark.parametrize("periodic", [False, True])
def test_qcriterion_over_the_float_range(O, cuda, periodic, scale):
    """Float-pair products against FP64: Q within half a unit of a float plus
    2^-40 of the sum of the terms' magnitudes (each of the 6 products and
    their sum is carried to about 2^-46); fields whose products leave the
    float range overflow or vanish as the FP64 value does in a float."""
    nx, ny, nz = 19, 7, 5
    bc = [PER] * 6 if periodic else [VEL, OUT, VEL, VEL, BB, FS]
    ens = ensemble(nx, ny, nz, bc, [[4, 2, 0, 8, 5, 3]])
    flags = S.sc_lbm_geometry(ens.cfg, 0)
    rng = np.random.RandomState(3)
    with np.errstate(over="ignore"):
        u = (rng.uniform(-1, 1, (3, nx * ny * nz)) * scale).astype(np.float32)
        u[:, rng.rand(nx * ny * nz) < 0.2] = 0.0
        q = ens.qcriterion(0, torch.from_numpy(u).cuda()).cpu().numpy().astype(np.float64)
        want = O.qcriterion(u, flags, nx, ny, nz, bc)
        as_float = want.astype(np.float32).astype(np.float64)
    terms = 9 * (2.0 * np.abs(u.astype(np.float64)).max()) ** 2
    finite = np.isfinite(as_float)
    assert np.array_equal(finite, np.isfinite(q)) and np.array_equal(q[~finite], as_float[~finite])
    tol = np.abs(want[finite]) * 2.0 ** -24 + terms * 2.0 ** -40 + 2e-45
    assert np.all(np.abs(q[finite] - want[finite]) <= tol)
    assert np.all(q[flags != 0] == 0)
    ens.close()


@pytest.mark.parametrize("n_cells", [1, 300, 303, 1300])
@pytest.mark.parametrize("n_samples", [1, 2, 31, 1000, 4099, 8192])
def test_quantiles_equal_the_sorted_surrogate(cuda, n_cells, n_samples):
    """The selected order statistics are those of the whole sorted surrogate:
    every group size (cells per block, last group ragged), sample counts off
    the vector width, repeated samples, flat, zero, tiny and huge cells.  The
    surrogate here sums in another order, so values agree to the rounding of
    its P terms: P 2^-52 of the sum of their magnitudes."""
    ens = ensemble(16, 16, 8, [VEL, OUT, VEL, VEL, BB, FS], gpc_degree=3, inputs=[W.SPEED, W.ANGLE], lo=[0.0, 0.0],
                   hi=[0.1, 6.0], quad_rule=W.GH)
    n, P = 16 * 16 * 8, 10
    rng = np.random.RandomState(n_samples + n_cells)
    coef = rng.standard_normal((P, n)) * (0.02 * 0.4 ** np.arange(P))[:, None]
    coef[:, ::7] = 0.0                      # solid cells
    coef[1:, 1::11] = 0.0                   # constant in the inputs
    coef[1:, 2::13] *= 1e-13                # flat to FP32
    coef[:, 3::17] *= 1e-60
    coef[:, 4::19] *= 1e60
    coef[0, 5::23] = -1.0
    samples = rng.standard_normal((n_samples, 2))
    samples[n_samples // 2:] = samples[: n_samples - n_samples // 2]   # each sample twice or more
    samples[: n_samples // 3] = samples[0]
    cells = rng.permutation(n)[:n_cells].astype(np.int32)
    q = [0.0, 0.025, 0.5, 0.75, 1.0]
    got = ens.gpc_quantiles(0, torch.from_numpy(coef).cuda(), cells, samples, q).cpu().numpy()
    phi = np.empty((n_samples, P))
    he = [np.polynomial.hermite_e.hermeval(samples, [0] * k + [1]) / np.sqrt([1.0, 1.0, 2.0, 6.0][k]) for k in range(4)]
    k = 0
    for total in range(4):
        for a in range(total, -1, -1):
            phi[:, k] = he[a][:, 0] * he[total - a][:, 1]
            k += 1
    y = np.sort(phi @ coef[:, cells], axis=0)
    ranks = [min(max(int(np.ceil(v * n_samples)), 1), n_samples) - 1 for v in q]
    tol = 64 * 2.0 ** -52 * (np.abs(phi) @ np.abs(coef[:, cells])).max(axis=0)
    assert np.all(np.abs(got - y[ranks]) <= tol)
    ens.close()
