"""The adjoint's workspace: its states, and nothing beyond them."""
import numpy as np
import pytest

from paper_2508_18202_gb300 import sclbm as S
from paper_2508_18202_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bc", [W.URBAN_BC, [W.VEL, W.OUT, W.PER, W.PER, W.FS, W.FS]])
def test_states_and_bounds(bc):
    """K checkpoints, L - 1 further states of a segment and two forward and two
    adjoint buffers; whatever the workspace held before, every count of
    checkpoints gives the same loss and gradient (1e-12: the order of the FP64
    atomics), and the bytes after the workspace stay as they were."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    wl = dict(domains=[dict(nx=37, ny=19, nz=13, boxes=[[6, 3, 0, 10, 8, 5], [33, 9, 0, 37, 13, 6]], bc=bc,
                            quad_level=1)],
              tau0=0.6, c_smag=0.0, u_ref=0.05, alpha=0.25, angle_deg=5.0, H_ref=0.0, inputs=[W.SPEED], lo=[-0.1],
              hi=[0.1], quad_rule=W.GL, ramp_steps=4, precision=W.FP32_SHIFT, gpc_degree=-1)
    ens = S.Ensemble(S.make_config(wl))
    state = 4 * 19 * ((37 * 19 * 13 + 255) // 256 * 256)
    probes, target, steps = [[25, 3, 3], [30, 12, 8]], np.full((2, 3), 0.03), 23
    want = None
    for snapshots in (0, 1, 2, 5, 12, 23):
        K = snapshots or 5
        L = -(-steps // K)
        K = -(-steps // L)
        nbytes = S.sc_lbm_adjoint_workspace_size(ens.h, 0, steps, snapshots, 2)
        assert nbytes // state == K + (L - 1) + 4
        for fill in (0x00, 0x7f, 0xff):
            ws = torch.full((nbytes + 4096,), fill, dtype=torch.uint8, device="cuda")
            torch.cuda.synchronize()
            J, g, _ = S.sc_lbm_adjoint(ens.h, 0, 0, probes, target, steps, snapshots, ws.data_ptr(), nbytes)
            assert bool((ws[nbytes:] == fill).all())
            if want is None:
                want = J, g
            assert J == want[0] and np.allclose(g, want[1], rtol=1e-12, atol=0)
    ens.close()
