"""FP32 calls on buffers aligned to one complex number (8 bytes) only: the same
bits as on buffers aligned to 16 bytes, whose kernels move 16 bytes at a time."""
import numpy as np
import pytest

from paper_2509_11424_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip('torch')
if not torch.cuda.is_available():
    pytest.skip('needs a CUDA GPU', allow_module_level=True)

from gpu_util import Setup, host  # noqa: E402


def _at(offset, x):
    """x in a buffer that starts `offset` complex numbers behind an aligned address."""
    buf = torch.zeros(x.size + 2, dtype=torch.complex64, device='cuda')
    v = buf[offset:offset + x.size]
    v.copy_(torch.from_numpy(x.reshape(-1)))
    assert v.data_ptr() % 16 == 8 * offset
    return v


# smoothing of a right-hand side in the internal order (read where it lies) by
# SAP on 2^4 and on 4^4 blocks and by minimal-residual steps, on the fine and
# on a coarse level
@pytest.mark.parametrize('dims,smoother,level', [((4, 4, 4, 4), 'SMOOTHER_SAP', 0), ((8, 8, 8, 8), 'SMOOTHER_SAP', 0),
                                                 ((4, 4, 4, 4), 'SMOOTHER_MR', 0), ((4, 4, 4, 4), 'SMOOTHER_MR', 1)])
def test_smooth(dims, smoother, level):
    s = Setup(dims, [(2, 2, 2, 2)], [4], eps=0.4, m0=0.1, oracle=False)
    M = s.M
    try:
        M.mgmlmc_set_solver(s.ctx, smoother=getattr(M, smoother), smoother_steps=2, sap_iters=3)
        n = M.mgmlmc_level_info(s.ctx, level)[2]
        x = synth.complex_normal((2, n), 81).astype(np.complex64)
        outs = []
        for off in (0, 1):
            y = torch.empty(x.size, dtype=torch.complex64, device='cuda')
            M.mgmlmc_apply(s.ctx, M.OP_SMOOTH | (M.LAYOUT_INTERNAL if level == 0 else 0), level, M.FP32, _at(off, x), y, 2)
            outs.append(host(y))
        assert np.array_equal(outs[0], outs[1])
    finally:
        s.close()
