"""FP32 operator calls on small lattices in the caller's order: one launch from
the second call on, the same bits as the first call's reorderings around the
tuned kernel; buffers aligned to one complex number keep the reorderings."""
import numpy as np
import pytest

from paper_2509_11424_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip('torch')
if not torch.cuda.is_available():
    pytest.skip('needs a CUDA GPU', allow_module_level=True)

from gpu_util import host, require_lib  # noqa: E402


# odd and thin lattices, a last block of 64 sites that is not full; sites times
# right-hand sides at 2^15 and above it, where every call reorders
@pytest.mark.parametrize('dims,nrhs', [((3, 5, 2, 7), 1), ((2, 2, 2, 2), 3), ((8, 4, 4, 5), 6), ((16, 8, 16, 8), 2),
                                       ((16, 8, 16, 8), 3)])
def test_repeated_calls(dims, nrhs):
    M = require_lib()
    n = 12 * int(np.prod(dims))
    ctx = M.mgmlmc_create(dims, torch.cuda.current_stream())
    try:
        M.mgmlmc_set_gauge(ctx, synth.gauge_field(dims, 0.4, 91))
        M.mgmlmc_set_mass(ctx, -0.2)
        x = torch.from_numpy(synth.complex_normal(nrhs * n, 92).astype(np.complex64)).cuda()
        outs = []
        for off in (0, 0, 1, 0):
            a, b = (torch.zeros(nrhs * n + 2, dtype=torch.complex64, device='cuda')[off:off + nrhs * n] for _ in 'ab')
            a.copy_(x)
            M.mgmlmc_apply(ctx, M.OP_D, 0, M.FP32, a, b, nrhs)
            outs.append(host(b))
        for o in outs[1:]:
            assert np.array_equal(o, outs[0])
    finally:
        M.mgmlmc_destroy(ctx)
