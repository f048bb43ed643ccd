"""The minimal-residual dots of the one-block-per-site FP32 stencil on site
counts that are no multiple of the 256 partial sums added at a time (162 and
324 sites), through the MR smoother of level 1, against the oracle.  Bound: as
for 256 sites, 1e-5 per operator and step, three steps."""
import numpy as np
import pytest

from oracle import smoother as osm
from paper_2509_11424_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip('torch')
if not torch.cuda.is_available():
    pytest.skip('needs a CUDA GPU', allow_module_level=True)

from gpu_util import Setup, dev, host, rel  # noqa: E402


@pytest.mark.parametrize('dims', [(6, 6, 6, 12), (12, 6, 6, 12)])
def test_mr_steps(dims):
    s = Setup(dims, [(2, 2, 2, 2), (3, 3, 3, 3)], [16, 2], eps=0.4, m0=-0.2, gseed=44,
              solver=dict(coarse_smoother_steps=3))
    M = s.M
    try:
        A = s.hier.matrix(1).tocsr()
        for nrhs in (1, 3, 8):
            b = synth.complex_normal((nrhs, A.shape[0]), 45).astype(np.complex64)
            out = torch.empty((nrhs, A.shape[0]), dtype=torch.complex64, device='cuda')
            M.mgmlmc_apply(s.ctx, M.OP_SMOOTH, 1, M.FP32, dev(b, torch.complex64), out, nrhs)
            got = host(out).astype(np.complex128)
            for r in range(nrhs):
                assert rel(got[r], osm.mr_smooth(A, b[r].astype(np.complex128), 3)) < 3e-5
    finally:
        s.close()
