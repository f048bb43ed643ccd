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
