"""Dot products and updates (csrc/kernels_blas.cu) called directly, on inputs
that tell how a sum is carried."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip('torch')
if not torch.cuda.is_available():
    pytest.skip('needs a CUDA GPU', allow_module_level=True)

from kernel_lib import kernels, ptr  # noqa: E402


def _out(n):
    return torch.zeros(n, dtype=torch.complex128, device='cuda')


# 12 entries of 32^4 sites, 24^3 x 48 and one past a step of a block
@pytest.mark.parametrize('n', [12 * 32 ** 4, 12 * 24 ** 3 * 48, 12 * 32 ** 4 + 2])
def test_fp32_chain(n):
    """A thread of an FP32 dot product adds at most 16 entries in FP32 up to n
    = 2^24.  Of every 12 x 1024 consecutive entries the first 1024 are 1 and
    the rest just below the size, 2^-11, whose square a sum of four ones no
    longer takes in: the more of them follow in one thread, the more is lost.
    16 entries are 32 products, each rounded by 2^-24 of the sum: 31 2^-24 of
    the sum at most."""
    L = kernels()
    a = torch.full((n,), complex(2.0 ** -11.01, 2.0 ** -11.01), dtype=torch.complex64, device='cuda')
    a[(torch.arange(n, device='cuda') % 12288) < 1024] = 1.0
    want = float((a.real.double() ** 2 + a.imag.double() ** 2).sum())
    bound = 31 * 2.0 ** -24 * want
    out = _out(4)
    assert L.k_dot(1, ptr(a), ptr(a), n, 1, ptr(out)) == 0
    assert abs(complex(out[0]) - want) <= bound
    assert L.k_dot_qr(1, ptr(a), ptr(a), n, 1, ptr(out), ptr(out[1:])) == 0
    assert abs(complex(out[0]) - want) <= bound and abs(complex(out[1]) - want) <= bound
    V = torch.stack([a, 1j * a])
    assert L.k_multi_dot(1, ptr(V), n, 2, ptr(a), n, 1, ptr(out)) == 0
    assert abs(complex(out[0]) - want) <= bound and abs(complex(out[1]) + 1j * want) <= bound


def test_fp32_infinite_sums():
    """A sum that leaves the range of FP32, or takes in an infinite entry, is
    infinite; only sums of both signs and of NaN are NaN."""
    L = kernels()
    n = 5000
    a = torch.ones(n, dtype=torch.complex64, device='cuda')
    out = _out(4)
    for bad, j in ((1e30, 17), (float('inf'), 4321)):
        q = a.clone()
        q[j] = bad
        assert L.k_dot_qr(1, ptr(q), ptr(q), n, 1, ptr(out), ptr(out[1:])) == 0
        assert out[1].real == float('inf')
        w = q.clone()
        h = _out(1)
        assert L.k_multi_axpy(1, ptr(a), n, 1, ptr(w), n, 1, ptr(h), 1.0, ptr(out)) == 0
        assert out[0].real == float('inf')
    x, y = a.clone(), a.clone()
    x[3], y[3] = 1e30, -1e30
    assert L.k_dot(1, ptr(x), ptr(y), n, 1, ptr(out)) == 0
    assert out[0].real == float('-inf') and out[0].imag == 0.0
    x[4], y[4] = 1e30, 1e30  # the same warp, another thread
    x[7], y[7] = 1e30, 1e30
    assert L.k_dot(1, ptr(x), ptr(y), n, 1, ptr(out)) == 0
    assert torch.isnan(out[0].real)


@pytest.mark.parametrize('nrhs', [1, 4, 7])
def test_site_stencil_infinite_sums(nrhs):
    V = 300
    x = torch.ones(nrhs, V, 32, dtype=torch.complex64, device='cuda')
    x[0, 299, 5] = 1e30
    y, qx, qq = torch.empty_like(x), _out(nrhs), _out(nrhs)
    assert kernels().k_site_dots(ptr(x), ptr(y), 2.0, V, nrhs, ptr(qx), ptr(qq)) == 0
    assert qx[0].real == float('inf') and qq[0].real == float('inf')
    for r in range(1, nrhs):
        assert qx[r] == 2.0 * 32 * V and qq[r] == 4.0 * 32 * V


def _exact(x, y):
    """sum conj(x) y and sum |x||y| over the last axis, in long double."""
    x, y = x.cpu().numpy().astype(np.clongdouble), y.cpu().numpy().astype(np.clongdouble)
    return (x.conj() * y).sum(-1), (abs(x) * abs(y)).sum(-1)


def _graded(seed, *shape):
    """x of entries 1 .. 2^-100, y small where x is large: all products about 2^-100."""
    r = np.random.default_rng(seed)
    e = r.integers(0, 101, shape)
    cn = lambda: r.standard_normal(shape) + 1j * r.standard_normal(shape)  # noqa: E731
    to = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    return to(cn() * 2.0 ** -e), to(cn() * 2.0 ** (e - 100.0))


# n below and above a step of a block (1024), a warp's group ending raggedly;
# vectors read one, up to four and up to eight at a time
@pytest.mark.parametrize('n,k', [(1, 1), (100, 2), (1025, 5), (3000, 1), (3000, 3), (3000, 9)])
def test_fp64_graded_dots(n, k):
    """Vectors whose large entries meet only small ones of the other, equal
    ones, and ones with zeros: each sum of n <= 3000 complex products within
    FP64's bound for it, (256 + 3 steps and blocks) 2^-53 of sum |x||y|, taken
    as 2^-44."""
    L = kernels()
    x, y = _graded(91, 2, n)
    g = torch.Generator(device='cuda').manual_seed(92)
    V = torch.randn(k, 2, n, dtype=torch.complex128, device='cuda', generator=g)
    V[k // 2] = x
    V[0, :, n // 3:] = 0.0
    h = _out(2 * k)
    assert L.k_multi_dot(0, ptr(V), 2 * n, k, ptr(y), n, 2, ptr(h)) == 0
    got = h.cpu().numpy().reshape(2, k).T
    want, top = _exact(V, y[None])
    assert np.all(abs(got - want) <= 2.0 ** -44 * top)
    qq = _out(2)
    assert L.k_dot_qr(0, ptr(x), ptr(y), n, 2, ptr(h), ptr(qq)) == 0
    want, top = _exact(x, y)
    assert np.all(abs(h[:2].cpu().numpy() - want) <= 2.0 ** -44 * top)
    assert np.all(abs(qq.cpu().numpy() - _exact(x, x)[0]) <= 2.0 ** -44 * _exact(x, x)[1])
    assert L.k_dot(0, ptr(x), ptr(y), n, 2, ptr(h)) == 0
    assert np.all(abs(h[:2].cpu().numpy() - want) <= 2.0 ** -44 * top)


def test_fp64_infinite_sums():
    L = kernels()
    n = 2000
    x = torch.ones(n, dtype=torch.complex128, device='cuda')
    y = x.clone()
    y[1500] = float('inf')
    h, qq = _out(1), _out(1)
    assert L.k_dot_qr(0, ptr(y), ptr(y), n, 1, ptr(h), ptr(qq)) == 0
    assert qq[0].real == float('inf')
    assert L.k_dot(0, ptr(x), ptr(y), n, 1, ptr(h)) == 0
    assert h[0].real == float('inf')
    y[3] = complex(float('nan'), 0.0)
    assert L.k_dot(0, ptr(x), ptr(y), n, 1, ptr(h)) == 0
    assert torch.isnan(h[0].real)


# one vector and up to two groups of eight, n below and above the 512 entries of a block
@pytest.mark.parametrize('n,k', [(1, 1), (100, 3), (700, 8), (1300, 11)])
def test_fp64_graded_update(n, k):
    """w -= V h with entries of very different size beside one another: each
    entry within 2^-44 of its own sum of products (2^(8 - 53) of its largest
    product, or the rounding of FP64 sums)."""
    r = np.random.default_rng(93)
    cn = lambda *s: r.standard_normal(s) + 1j * r.standard_normal(s)  # noqa: E731
    V = cn(k, 2, n) * 2.0 ** -r.integers(0, 101, (1, 2, n))
    V[:, :, ::7] = 0.0
    h, w = cn(2, k), cn(2, n) * 2.0 ** -r.integers(60, 101, (2, n))
    to = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    wd, Vd, hd = to(w), to(V), to(h)
    assert kernels().k_multi_axpy(0, ptr(Vd), 2 * n, k, ptr(wd), n, 2, ptr(hd), -1.0, None) == 0
    P = V.astype(np.clongdouble) * h.T[:, :, None]
    assert np.all(abs(wd.cpu().numpy() - (w - P.sum(0))) <= 2.0 ** -44 * (abs(P).sum(0) + abs(w)))


# below and above a tile of 1024 entries, one group and two groups of eight vectors
@pytest.mark.parametrize('n,k', [(700, 3), (2500, 8), (2500, 13)])
@pytest.mark.parametrize('basis', [False, True])
def test_fp64_update_zeros(n, k, basis):
    """Right-hand sides all of whose coefficients are zero (one that has
    converged), groups of them, and vectors that are zero over a whole tile:
    the update is exact where there is nothing to add and as accurate as ever
    beside it, with 2^-48 of the largest product for the entries' digits."""
    r = np.random.default_rng(94)
    cn = lambda *s: r.standard_normal(s) + 1j * r.standard_normal(s)  # noqa: E731
    V, h, w = cn(k, 3, n), cn(3, k), cn(3, n)
    h[0] = 0.0
    h[1, :8] = 0.0
    V[:, 2, :1024] = 0.0
    to = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    wd, Vd, hd, nrm = to(w), to(V), to(h), _out(3)
    L = kernels()
    if basis:
        assert L.k_basis(ptr(Vd), k, ptr(wd), n, 3, ptr(hd), -1.0, ptr(nrm)) == 0
    else:
        assert L.k_multi_axpy(0, ptr(Vd), 3 * n, k, ptr(wd), n, 3, ptr(hd), -1.0, ptr(nrm)) == 0
    got = wd.cpu().numpy()
    P = V.astype(np.clongdouble) * h.T[:, :, None]
    want = w - P.sum(0)
    assert np.array_equal(got[0], w[0]) and np.array_equal(got[2, :1024], w[2, :1024])
    assert np.all(abs(got - want) <= 2.0 ** -48 * (abs(P).max((0, 2))[:, None] + abs(w)))
    assert np.allclose(nrm.cpu().numpy().real, (abs(got) ** 2).sum(1), rtol=1e-14, atol=0.0)


# below and above a tile of 1024 entries, groups of up to eight vectors
@pytest.mark.parametrize('n,k', [(1, 1), (700, 3), (2500, 8), (2500, 13)])
def test_fp64_graded_basis(n, k):
    """A Krylov basis whose vectors hold entries of very different size beside
    one another (every third one), zeros, and equally scaled entries, dotted
    with graded vectors and subtracted from them: dots within FP64's bound (as
    above), entries of an update within 2^-44 of their own sum of products."""
    L = kernels()
    r = np.random.default_rng(95)
    cn = lambda *s: r.standard_normal(s) + 1j * r.standard_normal(s)  # noqa: E731
    to = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    x, y = _graded(96, 2, n)
    V = cn(k, 2, n)
    V[::3] = x.cpu().numpy() * 2.0 ** r.integers(-3, 3, (len(V[::3]), 1, 1))
    V[k // 2, 0] *= 2.0 ** -700
    V[:, :, ::5] = 0.0
    Vd, h = to(V), _out(2 * k)
    assert L.k_basis(ptr(Vd), k, ptr(y), n, 2, ptr(h), 0.0, None) == 0
    want, top = _exact(Vd, y[None])
    assert np.all(abs(h.cpu().numpy().reshape(2, k).T - want) <= 2.0 ** -44 * top)
    c, w = cn(2, k), cn(2, n) * 2.0 ** -r.integers(60, 101, (2, n))
    c[1, 1:] = 0.0
    w[1] *= 2.0 ** -40
    wd, cd, nrm = to(w), to(c), _out(2)
    assert L.k_basis(ptr(Vd), k, ptr(wd), n, 2, ptr(cd), -1.0, ptr(nrm)) == 0
    got = wd.cpu().numpy()
    P = V.astype(np.clongdouble) * c.T[:, :, None]
    assert np.all(abs(got - (w - P.sum(0))) <= 2.0 ** -44 * (abs(P).sum(0) + abs(w)))
    assert np.allclose(nrm.cpu().numpy().real, (abs(got) ** 2).sum(1), rtol=1e-14, atol=0.0)
