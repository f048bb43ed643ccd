"""The coarsest level's dense inverse at unknowns around the sizes its kernels
step in: 2, 30, a block of 256 columns and one more pair, and just above the
1024 threads of a pivot search.  With partial pivoting the residual is a few
n eps times the growth of |A||A^-1|; with condition numbers below 1e3 here
1e-10 has two digits in hand at n = 1056."""
import numpy as np
import pytest

from oracle import dirac
from paper_2509_11424_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip('torch')
if not torch.cuda.is_available():
    pytest.skip('needs a CUDA GPU', allow_module_level=True)

from gpu_util import Setup, dev, host  # noqa: E402


@pytest.mark.parametrize('dims,block,ntv', [((2, 2, 2, 2), (2, 2, 2, 2), 1), ((2, 2, 6, 2), (2, 2, 2, 2), 5),
                                            ((2, 2, 2, 4), (2, 2, 2, 2), 64), ((2, 2, 6, 2), (2, 2, 2, 2), 43),
                                            ((4, 4, 4, 6), (2, 2, 2, 2), 22)])
def test_direct_solve(dims, block, ntv):
    s = Setup(dims, [block], [ntv], eps=0.4, m0=0.2, gseed=52)
    try:
        A = s.hier.A[1]
        cd = tuple(d // b for d, b in zip(dims, block))
        D = dirac.stencil_matrix(A, cd)
        n = D.shape[0]
        assert np.linalg.cond(D.toarray() if hasattr(D, 'toarray') else D) < 1e3
        b = synth.complex_normal((2, n), 53)
        x = torch.empty((2, n), dtype=torch.complex128, device='cuda')
        s.M.mgmlmc_apply(s.ctx, s.M.OP_SOLVE, 1, s.M.FP64, dev(b), x, 2)
        xs = host(x)
        for r in range(2):
            assert np.linalg.norm(b[r] - D @ xs[r]) <= 1e-10 * np.linalg.norm(b[r])
    finally:
        s.close()
