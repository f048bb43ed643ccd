"""The FP32 coarse stencil with one thread block per site (32 dofs per site,
up to 8 right-hand sides) and its fused minimal-residual dots, through the MR
smoother of level 1 on 256 coarse sites, against the oracle.

Tolerance 1e-5 per operator (storage rounding 6e-8 times the operator's norm
amplification, as for the other FP32 operators); each of the 3 steps takes one
operator application and an alpha from FP32 products summed exactly, so 3e-5."""
import numpy as np
import pytest

from oracle import smoother as osm
from paper_2509_11424_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip('torch')
if not torch.cuda.is_available():
    pytest.skip('needs a CUDA GPU', allow_module_level=True)

from gpu_util import Setup, dev, host, rel  # noqa: E402


@pytest.fixture(scope='module')
def s():
    s = Setup((8, 8, 8, 8), [(2, 2, 2, 2), (2, 2, 2, 2)], [16, 4], eps=0.4, m0=-0.2, gseed=41,
              solver=dict(coarse_smoother_steps=3))
    yield s
    s.close()


@pytest.mark.parametrize('nrhs', [1, 2, 3, 4, 7, 8, 9])
def test_mr_steps(s, nrhs):
    M = s.M
    A = s.hier.matrix(1).tocsr()
    b = synth.complex_normal((nrhs, A.shape[0]), 42).astype(np.complex64)
    b[nrhs - 1] *= 1e-20  # right-hand sides of very different size
    out = torch.empty((nrhs, A.shape[0]), dtype=torch.complex64, device='cuda')
    M.mgmlmc_apply(s.ctx, M.OP_SMOOTH, 1, M.FP32, dev(b, torch.complex64), out, nrhs)
    got = host(out).astype(np.complex128)
    for r in range(nrhs):
        assert rel(got[r], osm.mr_smooth(A, b[r].astype(np.complex128), 3)) < 3e-5


def test_zero_right_hand_side(s):
    M = s.M
    n = M.mgmlmc_level_info(s.ctx, 1)[2]
    b = synth.complex_normal((2, n), 43)
    b[1] = 0.0
    out = torch.full((2, n), float('nan'), dtype=torch.complex64, device='cuda')
    M.mgmlmc_apply(s.ctx, M.OP_SMOOTH, 1, M.FP32, dev(b, torch.complex64), out, 2)
    got = host(out)
    assert np.isfinite(got[0]).all() and not got[1].any()
