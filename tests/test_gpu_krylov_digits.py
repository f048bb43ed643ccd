"""FP64 solves, whose Krylov basis is kept as fixed-point digits, at sizes
where the tiles of 1024 entries and the groups of 4 and 8 basis vectors end
raggedly, and with right-hand sides of very different size in one block.

The solutions have the true relative residual the solver promises, measured
with the oracle's operator: 1.5 times tol = 1e-12, as in the other solve
tests."""
import numpy as np
import pytest

from oracle import dirac
from paper_2509_11424_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip('torch')
if not torch.cuda.is_available():
    pytest.skip('needs a CUDA GPU', allow_module_level=True)

from gpu_util import Setup, dev, host  # noqa: E402


# 12 V entries: 3 x 1024, 6912 = 6 x 1024 + 768, 768; restarts below, at and
# above the groups
@pytest.mark.parametrize('dims,block,restart', [((4, 4, 4, 4), (2, 2, 2, 2), 9), ((6, 4, 4, 6), (3, 2, 2, 3), 4),
                                                ((2, 4, 2, 4), (1, 2, 2, 2), 1), ((4, 4, 4, 4), (2, 2, 2, 2), 20)])
def test_fp64_solve(dims, block, restart):
    s = Setup(dims, [block], [4], eps=0.4, m0=-0.1, gseed=31, oracle=False, solver=dict(restart=restart))
    M = s.M
    try:
        D = dirac.wilson_matrix(s.U, -0.1, dims)
        n = D.shape[0]
        b = synth.complex_normal((3, n), 32)
        b[1] *= 2.0 ** -300
        b[2, : n // 2] *= 2.0 ** -60
        x = torch.empty((3, n), dtype=torch.complex128, device='cuda')
        M.mgmlmc_apply(s.ctx, M.OP_SOLVE, 0, M.FP64, dev(b), x, 3)
        xs = host(x)
        for r in range(3):
            assert np.linalg.norm(b[r] - D @ xs[r]) <= 1.5e-12 * np.linalg.norm(b[r])
    finally:
        s.close()


def test_rough_setup_vectors():
    """The set-up's unpreconditioned GMRES (basis and update both from digits)
    against the oracle-side argmin over the Krylov space."""
    dims, iters = (4, 4, 4, 4), 11
    s = Setup(dims, [(2, 2, 2, 2)], [2], eps=0.4, m0=-0.1, gseed=33, oracle=False)
    M = s.M
    ctx = M.mgmlmc_create(dims, torch.cuda.current_stream())
    try:
        M.mgmlmc_set_gauge(ctx, s.U)
        M.mgmlmc_set_mass(ctx, -0.1)
        M.mgmlmc_build_hierarchy(ctx, M.mg_params([(2, 2, 2, 2)], [2], setup_rounds=1, setup_iters=iters, seed=9))
        tv = M.mgmlmc_get_test_vectors(ctx, 0)
        D = dirac.wilson_matrix(s.U, -0.1, dims)
        from oracle import noise as onz
        for k in range(2):
            v = onz.z4_vector(D.shape[0], 9, k, 96)
            K = [v / np.linalg.norm(v)]
            for _ in range(iters - 1):
                K.append(D @ K[-1])
                K[-1] /= np.linalg.norm(K[-1])
            Q, _ = np.linalg.qr(np.array(K).T)
            w = Q @ np.linalg.lstsq(D @ Q, v, rcond=None)[0]
            w /= np.linalg.norm(w)
            # the power basis loses about its condition number, ~1e5 after 11
            # steps of an operator of condition number ~10: 1e-9
            assert np.abs(tv[k] - w).max() < 1e-9
    finally:
        M.mgmlmc_destroy(ctx)
        s.close()
