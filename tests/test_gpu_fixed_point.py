"""The FP64 kernels that run in fixed point on the integer pipe
(csrc/fixed.cuh) against the oracle.

Tolerance: a sum of products keeps its operands to 2^-57 of the largest entry
of a vector group and 2^-58 of an operator row's largest entry (2^-61 of its
1-norm), and drops terms below 2^-60 of the product of the two scales; summed
over K <= 2 x 9 x 256 real products this is below K 2^-57 = 3.2e-14 of |row|_1
max|x|, and typically the square root of K of it.  Asserted: 1e-13 of
|row|_1 max|x| per entry for the worst case, 1e-14 norm-wise.
"""
import numpy as np
import pytest

from oracle import dirac
from paper_2509_11424_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip('torch')
if not torch.cuda.is_available():
    pytest.skip('needs a CUDA GPU', allow_module_level=True)

from gpu_util import Setup, dev, host  # noqa: E402


# dofs per site 2 N_tv: below, at and above the 32- and 64-row tiles, not
# multiples of them, and wide ones; right-hand sides around the 1/2/4/8 passes
@pytest.mark.parametrize('ntv,nrhs', [(1, 3), (5, 1), (16, 2), (16, 9), (17, 5), (32, 8), (33, 4), (50, 1), (72, 5)])
def test_coarse_stencil_fp64(ntv, nrhs):
    s = Setup((4, 6, 4, 4), [(2, 3, 2, 2)], [ntv], eps=0.4, m0=-0.2, gseed=61)
    M = s.M
    try:
        A = s.hier.matrix(1).tocsr()
        n1 = A.shape[0]
        x = synth.complex_normal((nrhs, n1), 62)
        # sites of very different size: the scale is chosen per site and right-hand side
        x *= 2.0 ** np.repeat(np.random.default_rng(63).integers(-40, 40, n1 // (2 * ntv)), 2 * ntv)
        y = torch.empty((nrhs, n1), dtype=torch.complex128, device='cuda')
        M.mgmlmc_apply(s.ctx, M.OP_D, 1, M.FP64, dev(x), y, nrhs)
        got = host(y)
        one = np.asarray(abs(A.real).sum(1) + abs(A.imag).sum(1)).ravel()
        pattern = (abs(A) > 0).astype(float)
        for r in range(nrhs):
            want = A @ x[r]
            top = pattern.multiply(np.maximum(abs(x[r].real), abs(x[r].imag))[None, :]).max(1).toarray().ravel()
            assert np.all(np.abs(got[r] - want) <= 1e-13 * one * top)
            assert np.linalg.norm(got[r] - want) < 1e-14 * np.linalg.norm(want) * np.sqrt(18 * ntv)
    finally:
        s.close()


def test_coarse_stencil_fp64_special_values():
    """Inf and NaN reach exactly the right-hand side and the sites that touch
    them; subnormal, huge and zero vectors keep their values."""
    s = Setup((6, 6, 6, 6), [(2, 2, 2, 2)], [4], eps=0.4, m0=-0.2, gseed=64)
    M = s.M
    try:
        A = s.hier.matrix(1).tocsr()
        n1 = A.shape[0]
        x = synth.complex_normal((6, n1), 65)
        x[1, 3] = np.nan
        x[2, 5] = np.inf
        x[3] *= 2.0 ** -1040
        x[4] *= 2.0 ** 1010
        x[5] = 0.0
        y = torch.empty((6, n1), dtype=torch.complex128, device='cuda')
        M.mgmlmc_apply(s.ctx, M.OP_D, 1, M.FP64, dev(x), y, 6)
        got = host(y)
        with np.errstate(all='ignore'):
            near = lambda j: (abs(A[:, [j // 8 * 8 + k for k in range(8)]]).sum(1) > 0).A1 \
                if hasattr(A, 'A1') else np.asarray(abs(A[:, [j // 8 * 8 + k for k in range(8)]]).sum(1)).ravel() > 0
            for r, j in ((1, 3), (2, 5)):
                hit = near(j)
                assert not np.isfinite(got[r][hit]).any()
                clean = x[r].copy()
                clean[j] = 0.0
                assert np.abs(got[r] - A @ clean)[~hit].max() < 1e-13
            # the products of subnormal entries are exact to their last bit (2^-1074) times the row's length
            assert np.abs(got[3] - A @ x[3]).max() <= 2.0 ** -1074 * 200
            big = (A @ (x[4] * 2.0 ** -1010))
            assert np.abs(got[4] * 2.0 ** -1010 - big).max() < 1e-13
            assert not got[5].any()
    finally:
        s.close()


def _wilson(dims, U, x, m0):
    from gpu_util import require_lib
    M = require_lib()
    ctx = M.mgmlmc_create(dims, torch.cuda.current_stream())
    try:
        M.mgmlmc_set_gauge(ctx, U)
        M.mgmlmc_set_mass(ctx, m0)
        xd = dev(x)
        yd = torch.full_like(xd, float('nan'))
        M.mgmlmc_apply(ctx, M.OP_D, 0, M.FP64, xd, yd, x.shape[0])
        return host(yd)
    finally:
        M.mgmlmc_destroy(ctx)


# sites: fewer than a tile of 32, no multiple of the 64 of a block, extents of
# 2 and 3, more right-hand sides than one converted group on small lattices
# (2^18 sites / V) never are, so the group of 4 is crossed with a larger one
@pytest.mark.parametrize('dims,nrhs', [((2, 2, 2, 2), 1), ((3, 2, 2, 5), 3), ((5, 4, 3, 7), 2), ((8, 4, 2, 6), 5),
                                       ((28, 28, 28, 28), 5)])
def test_wilson_fp64_fixed_point(dims, nrhs):
    """Sites of very different size (each is kept in units of its own largest
    entry): entry by entry within 2e-15 of the largest entry among the site
    and its neighbours (7 bits of a 61-bit unit summed over 8 hops is far
    less; the FP64 diagonal term rounds at 2^-53 x 4)."""
    V = dirac.volume(dims)
    U = synth.gauge_field(dims, 0.4, 71)
    x = synth.complex_normal((nrhs, V, 12), 72)
    x *= 2.0 ** np.random.default_rng(73).integers(-30, 30, (nrhs, V, 1))
    got = _wilson(dims, U, x.reshape(nrhs, -1), -0.3).reshape(nrhs, V, 12)
    top = np.abs(x).max(2).reshape(nrhs, *dims[::-1])
    near = np.max([np.roll(top, k, a) for a in range(1, 5) for k in (-1, 0, 1)], 0).reshape(nrhs, V)
    for r in range(nrhs):
        want = dirac.apply_wilson(U, x[r].reshape(-1), -0.3, dims).reshape(V, 12)
        assert np.all(np.abs(got[r] - want).max(1) <= 4e-15 * near[r])


def test_wilson_fp64_special_values():
    """Inf / NaN stay with the sites that touch them; subnormal, huge and zero
    vectors keep their values; links of very different size take the FP64
    kernel."""
    dims = (4, 6, 4, 4)
    V = dirac.volume(dims)
    U = synth.gauge_field(dims, 0.4, 74)
    x = synth.complex_normal((6, V * 12), 75)
    x[1, 7] = np.nan
    x[2, 30] = np.inf
    x[3] *= 2.0 ** -1040
    x[4] *= 2.0 ** 1010
    x[5] = 0.0
    got = _wilson(dims, U, x, -0.3)
    with np.errstate(all='ignore'):
        for r, j in ((1, 7), (2, 30)):
            hit = ~np.isfinite(got[r]).reshape(V, 12).all(1)
            c = x[r].copy()
            c[j] = 0.0
            e = np.zeros_like(c)
            e[j] = 1.0
            touched = np.abs(dirac.apply_wilson(U, e, -0.3, dims)).reshape(V, 12).max(1) > 0
            assert np.array_equal(hit, touched)
            want = dirac.apply_wilson(U, c, -0.3, dims)
            assert np.abs(got[r] - want).reshape(V, 12)[~touched].max() < 1e-14
        assert np.abs(got[3] - dirac.apply_wilson(U, x[3], -0.3, dims)).max() <= 2.0 ** -1074 * 64
        want = dirac.apply_wilson(U, x[4] * 2.0 ** -1010, -0.3, dims)
        assert np.abs(got[4] * 2.0 ** -1010 - want).max() < 1e-13
        assert not got[5].any()
    U2 = U.copy()
    U2[:9] *= 1e-9
    y = _wilson(dims, U2, x[:1], -0.3)
    assert np.abs(y[0] - dirac.apply_wilson(U2, x[0], -0.3, dims)).max() < 1e-13
