"""Mixed-precision solves, whose FP32 Krylov vectors are streamed in tiles of
1024 entries, at sizes where tiles and groups of 4 and 8 basis vectors end
raggedly.  The solutions have the true relative residual the solver promises,
measured with the oracle's operator: 1.5 times tol = 1e-12, as in the other
solve tests; the iterations of a solve show that the FP32 cycles themselves
are sound: at most twice those of the FP64 solve with the same restart and one
cycle per refinement more (inner target 1e-6: two refinements reach 1e-12)."""
import numpy as np
import pytest

from oracle import dirac
from paper_2509_11424_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip('torch')
if not torch.cuda.is_available():
    pytest.skip('needs a CUDA GPU', allow_module_level=True)

from gpu_util import Setup, dev, host  # noqa: E402


# n = 12 V entries: 3 x 1024, 6912 = 6 x 1024 + 768, 768; restarts below, at and
# above the groups
@pytest.mark.parametrize('dims,block,restart', [((4, 4, 4, 4), (2, 2, 2, 2), 9), ((6, 4, 4, 6), (3, 2, 2, 3), 4),
                                                ((2, 4, 2, 4), (1, 2, 2, 2), 2), ((4, 4, 4, 4), (2, 2, 2, 2), 20)])
def test_mixed_solve(dims, block, restart):
    its = {}
    for prec in ('FP64', 'FP32'):
        s = Setup(dims, [block], [4], eps=0.4, m0=-0.1, gseed=31, oracle=False,
                  solver=dict(restart=restart, precision=0 if prec == 'FP64' else 1))
        M = s.M
        try:
            D = dirac.wilson_matrix(s.U, -0.1, dims)
            n = D.shape[0]
            b = synth.complex_normal((3, n), 32)
            b[1] *= 2.0 ** -20
            b[2, : n // 2] *= 2.0 ** -10
            x = torch.empty((3, n), dtype=torch.complex128, device='cuda')
            M.mgmlmc_apply(s.ctx, M.OP_SOLVE, 0, M.FP64, dev(b), x, 3)
            xs = host(x)
            for r in range(3):
                assert np.linalg.norm(b[r] - D @ xs[r]) <= 1.5e-12 * np.linalg.norm(b[r])
            its[prec] = M.mgmlmc_last_solve_stats(s.ctx)[0]
        finally:
            s.close()
    assert its['FP32'] <= 2 * its['FP64'] + 2 * restart
