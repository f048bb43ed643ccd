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
