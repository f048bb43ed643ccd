"""The FP32 weight gradient (csrc/kernels_learned.cu) called directly."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip('torch')
if not torch.cuda.is_available():
    pytest.skip('needs a CUDA GPU', allow_module_level=True)

from kernel_lib import kernels, ptr  # noqa: E402


# 4096 sites per block above 2^18 sites: full blocks, a short last one
@pytest.mark.parametrize('dims,cout', [((24, 24, 24, 24), 1), ((24, 22, 24, 22), 2)])
def test_fp32_chain(dims, cout):
    """A thread adds at most 16 sites in FP32.  Of every 4096 consecutive sites
    the first 128 hold 1 and the rest just below 2^-12, whose square a sum of
    1 no longer takes in: with all of a block's sites of a thread in one sum 31
    of them are lost, with 16 sites 15.  15 roundings by 2^-24 of the sum at
    most; one spin and colour component, so the other terms are exact zeros."""
    V = int(np.prod(dims))
    a = torch.zeros(1, 6, V, 2, dtype=torch.complex64, device='cuda')  # structure-of-arrays
    a[0, 0, :, 0] = 2.0 ** -12.01
    a[0, 0, torch.arange(V, device='cuda') % 4096 < 128, 0] = 1.0
    gin = a.repeat(cout, 1, 1, 1).contiguous()
    U = torch.zeros(36 * V, dtype=torch.complex64, device='cuda')
    out = torch.zeros(9, cout, 1, 16, dtype=torch.complex128, device='cuda')
    d = (ctypes.c_int * 4)(*dims)
    assert kernels().k_wgrad_f32(ptr(gin), ptr(a), ptr(U), d, 1, cout, 1, ptr(out)) == 0
    got = out.cpu().numpy()
    want = float((a[0, 0, :, 0].real.double() ** 2).sum())
    assert np.abs(got[0, :, 0, 0] - want).max() <= 15 * 2.0 ** -24 * want
    got[0, :, 0, 0] = 0.0
    assert not got.any()
