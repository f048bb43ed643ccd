"""The first FP64 operator call of a context on a small lattice finds its
workspace: no device memory is allocated in it, whatever the number of
right-hand sides."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip('torch')
if not torch.cuda.is_available():
    pytest.skip('needs a CUDA GPU', allow_module_level=True)

from gpu_util import require_lib  # noqa: E402


@pytest.mark.parametrize('L,nrhs', [(8, 1), (8, 40), (16, 6)])
def test_fp64_operator_allocates_nothing(L, nrhs):
    M = require_lib()
    ctx = M.mgmlmc_create((L,) * 4, torch.cuda.current_stream())
    try:
        M.mgmlmc_gen_gauge(ctx, 0.4, 3)
        M.mgmlmc_set_mass(ctx, -0.2)
        x = torch.ones(nrhs, 12 * L ** 4, dtype=torch.complex128, device='cuda')
        y = torch.empty_like(x)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        M.mgmlmc_apply(ctx, M.OP_D, 0, M.FP64, x, y, nrhs)
        torch.cuda.synchronize()
        assert torch.cuda.mem_get_info()[0] == free
    finally:
        M.mgmlmc_destroy(ctx)
