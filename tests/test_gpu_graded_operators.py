"""FP64 operators (fixed point on the integer pipe) on vectors whose entries
differ much in size beside one another: inside one spinor, inside one coarse
site, from one site to the next.  Each entry of the result within FP64's bound
for its own sum of products, K 2^-53 of sum |a||x| over its K products."""
import numpy as np
import pytest

from oracle import dirac
from paper_2509_11424_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip('torch')
if not torch.cuda.is_available():
    pytest.skip('needs a CUDA GPU', allow_module_level=True)

from gpu_util import Setup, dev, host, require_lib  # noqa: E402


def _unit(dims):
    U = np.zeros((dirac.volume(dims), 4, 3, 3), dtype=complex)
    U[:] = np.eye(3)
    return U.reshape(-1)


# one colour 2^60 below the others, one spin component, entries at random, one
# site far above the others (a point source), exact zeros in a colour
def _fields(V, rng):
    x = rng.standard_normal((5, V, 4, 3)) + 1j * rng.standard_normal((5, V, 4, 3))
    x[0, :, :, 1] *= 2.0 ** -60
    x[1, :, 2] *= 2.0 ** -45
    x[2] *= 2.0 ** -rng.integers(0, 101, (V, 4, 3))
    x[3] *= 2.0 ** -50
    x[3, V // 2] *= 2.0 ** 50
    x[4, :, :, 0] = 0.0
    x[4, :, 0] *= 2.0 ** -30
    return x


def _moduli(U, x, m0, dims):
    """sum |a||x| over the products of D: the diagonal and, for every hop, (1 +-
    gamma) U (hop by hop: where an extent is 2 the two hops of a direction end
    at the same site and part of their matrices cancels)."""
    shape = dims[::-1]
    a = abs(x).reshape(*shape, 4, 3)
    u = abs(U).reshape(*shape, 4, 3, 3)
    out = (4.0 + m0) * a
    for mu in range(4):
        ax, other = 3 - mu, [3, 2, 1, 0] if mu < 2 else [2, 3, 0, 1]  # gamma_mu exchanges the chiralities
        f, b = np.roll(a, -1, ax), np.roll(a, 1, ax)
        w = np.einsum('...ab,...sb->...sa', u[..., mu, :, :], f) + \
            np.einsum('...ba,...sb->...sa', np.roll(u[..., mu, :, :], 1, ax), b)
        out += 0.5 * (w + w[..., other, :])
    return out.reshape(-1)


# unit links do not mix colours; the others mix every entry
@pytest.mark.parametrize('dims', [(4, 4, 4, 4), (3, 2, 5, 4)])
@pytest.mark.parametrize('links', ['unit', 'random'])
def test_wilson(dims, links):
    """Each entry sums the diagonal and 8 hops of (1 +- gamma) U, 2 x 3 complex
    products each: 100 real products; 100 2^-53 of the sum of their moduli."""
    M = require_lib()
    V = dirac.volume(dims)
    U = _unit(dims) if links == 'unit' else np.ascontiguousarray(synth.gauge_field(dims, 0.4, 71)).reshape(-1)
    x = _fields(V, np.random.default_rng(72)).reshape(5, V * 12)
    ctx = M.mgmlmc_create(dims, torch.cuda.current_stream())
    try:
        M.mgmlmc_set_gauge(ctx, U)
        M.mgmlmc_set_mass(ctx, -0.3)
        xd = dev(x)
        y = torch.empty_like(xd)
        M.mgmlmc_apply(ctx, M.OP_D, 0, M.FP64, xd, y, 5)
        got = host(y)
    finally:
        M.mgmlmc_destroy(ctx)
    D = dirac.wilson_matrix(U, -0.3, dims).tocsr()
    Dl = D.toarray().astype(np.clongdouble)
    for r in range(5):
        want = Dl @ x[r].astype(np.clongdouble)
        assert np.all(abs(got[r] - want) <= 100 * 2.0 ** -53 * _moduli(U, x[r], -0.3, dims))


def _check_coarse(M, ctx, lat, m, kinds, nrhs):
    """OP_D of level 1 on multiples of each of `kinds`: 9 m complex products an
    entry, 4 real ones each, of the blocks that the library holds."""
    V = int(np.prod(lat))
    blocks = np.zeros(2 * V * 9 * m * m)
    M.mgmlmc_get_coarse_op(ctx, 1, blocks)
    blocks = blocks.view(complex).reshape(V, 9, m, m).astype(np.clongdouble)
    for kind in kinds:
        y = torch.empty((nrhs, V * m), dtype=torch.complex128, device='cuda')
        M.mgmlmc_apply(ctx, M.OP_D, 1, M.FP64, dev(np.stack([kind * 2.0 ** k for k in range(nrhs)])), y, nrhs)
        got = host(y)
        f = kind.reshape(*lat[::-1], m).astype(np.clongdouble)
        want, top = 0, 0
        for d in range(9):
            nb = f if d == 0 else np.roll(f, -1 if d % 2 else 1, 3 - (d - 1) // 2)
            nb = nb.reshape(V, 1, m)
            want = want + (blocks[:, d] * nb).sum(-1)
            top = top + (abs(blocks[:, d]) * abs(nb)).sum(-1)
        for r in range(nrhs):
            assert np.all(abs(got[r] - 2.0 ** r * want.ravel()) <= 36 * m * 2.0 ** -53 * 2.0 ** r * top.ravel())


# rows below and above a tile of 32, right-hand sides in groups of 1, 2 and 4
@pytest.mark.parametrize('ntv,nrhs', [(3, 1), (16, 2), (17, 5)])
def test_coarse_stencil(ntv, nrhs):
    """Vectors of graded entries, of one entry per site (columns of the
    operator), of one site far above the others."""
    s = Setup((4, 6, 4, 4), [(2, 3, 2, 2)], [ntv], eps=0.4, m0=-0.2, gseed=61, oracle=False)
    try:
        m = 2 * ntv
        n1, rng = 16 * m, np.random.default_rng(73)
        kinds = np.zeros((3, n1), dtype=complex)
        kinds[0] = (rng.standard_normal(n1) + 1j * rng.standard_normal(n1)) * 2.0 ** -rng.integers(0, 101, n1)
        kinds[1, np.arange(16) * m + rng.integers(0, m, 16)] = 2.0 ** -rng.integers(0, 61, 16)
        kinds[2] = rng.standard_normal(n1) * 2.0 ** -70
        kinds[2, 5 * m:5 * m + 2] = 1.0
        _check_coarse(s.M, s.ctx, (2, 2, 2, 2), m, kinds, nrhs)
    finally:
        s.close()


@pytest.mark.parametrize('nrhs', [1, 3])
def test_coarse_stencil_decoupled(nrhs):
    """Unit links and test vectors of one colour each: the operator does not mix
    them, so a row meets only the entries of its own colour, here 2^-60 and
    2^-30 of the others'."""
    M = require_lib()
    dims = (4, 4, 4, 6)
    V = dirac.volume(dims)
    tv = np.zeros((3, V, 4, 3), dtype=complex)
    rng = np.random.default_rng(74)
    for k in range(3):
        tv[k, :, :, k] = rng.standard_normal((V, 4)) + 1j * rng.standard_normal((V, 4))
    ctx = M.mgmlmc_create(dims, torch.cuda.current_stream())
    try:
        M.mgmlmc_set_gauge(ctx, _unit(dims))
        M.mgmlmc_set_mass(ctx, -0.3)
        M.mgmlmc_set_test_vectors(ctx, 0, tv.reshape(3, -1).copy(), 3, 12 * V)
        M.mgmlmc_build_hierarchy(ctx, M.mg_params([(2, 2, 2, 2)], [3], setup_rounds=0))
        lat = (2, 2, 2, 3)
        x = rng.standard_normal((24, 2, 3)) + 1j * rng.standard_normal((24, 2, 3))
        x[..., 1] *= 2.0 ** -60
        x[..., 2] *= 2.0 ** -30
        _check_coarse(M, ctx, lat, 6, [x.reshape(-1)], nrhs)
    finally:
        M.mgmlmc_destroy(ctx)
