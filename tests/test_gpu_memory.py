"""Calls where the memory runs out (injected: the next allocations fail) give
back what only makes them faster and go on without it: the FP64 Wilson operator
in its FP64 kernel (to 1e-14), the FP32 coarse operator in the pipelined one
(the same bits)."""
import numpy as np
import pytest

from paper_2509_11424_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip('torch')
if not torch.cuda.is_available():
    pytest.skip('needs a CUDA GPU', allow_module_level=True)

from gpu_util import Setup, dev, host, rel, require_lib  # noqa: E402
from kernel_lib import kernels  # noqa: E402


@pytest.fixture
def fail():
    L = kernels()
    yield L.k_alloc_failures
    L.k_alloc_failures(0, 0)


def _apply(M, ctx, op, level, prec, x):
    y = torch.empty_like(x)
    M.mgmlmc_apply(ctx, op, level, prec, x, y, x.shape[0])
    return host(y)


def test_given_back(fail):
    s = Setup((16, 8, 16, 16), [(4, 2, 4, 4)], [16], eps=0.4, m0=0.1, oracle=False)  # 256 coarse sites of 32 dofs
    M = s.M
    try:
        n = 12 * 16 ** 3 * 8
        x = dev(synth.complex_normal((3, n), 61))
        xc = dev(synth.complex_normal((2, 256 * 32), 62), torch.complex64)
        y, yc = _apply(M, s.ctx, M.OP_D, 0, M.FP64, x), _apply(M, s.ctx, M.OP_D, 1, M.FP32, xc)
        sm = _apply(M, s.ctx, M.OP_SMOOTH, 1, M.FP32, xc)
        M.mgmlmc_release_workspaces(s.ctx)
        fail(1, 1 << 20)
        z = _apply(M, s.ctx, M.OP_SMOOTH, 0, M.FP32, x.to(torch.complex64))
        assert np.isfinite(z).all()
        assert rel(_apply(M, s.ctx, M.OP_D, 0, M.FP64, x), y) < 1e-14
        assert np.array_equal(_apply(M, s.ctx, M.OP_D, 1, M.FP32, xc), yc)
        assert rel(_apply(M, s.ctx, M.OP_SMOOTH, 1, M.FP32, xc), sm) < 1e-5  # dots in another order
        M.mgmlmc_set_gauge(s.ctx, s.U)
        assert np.array_equal(_apply(M, s.ctx, M.OP_D, 0, M.FP64, x), y)
    finally:
        s.close()


@pytest.mark.parametrize('refused', [1, 2, 100])
def test_smaller_groups(fail, refused):
    """No memory for the digits of all right-hand sides: half or a quarter of
    them at a time (the same bits), or the FP64 kernel."""
    M = require_lib()
    dims = (8, 4, 6, 8)
    ctx = M.mgmlmc_create(dims, torch.cuda.current_stream())
    try:
        M.mgmlmc_set_gauge(ctx, synth.gauge_field(dims, 0.4, 63))
        M.mgmlmc_set_mass(ctx, -0.2)
        x = dev(synth.complex_normal((7, 12 * 8 * 4 * 6 * 8), 64))
        y = _apply(M, ctx, M.OP_D, 0, M.FP64, x)
        M.mgmlmc_release_workspaces(ctx)
        fail(refused, 0)
        z = _apply(M, ctx, M.OP_D, 0, M.FP64, x)
        assert rel(z, y) < 1e-14 if refused == 100 else np.array_equal(z, y)
        assert np.array_equal(_apply(M, ctx, M.OP_D, 0, M.FP64, x), z)
    finally:
        M.mgmlmc_destroy(ctx)


def test_no_memory_for_link_digits(fail):
    """A context that cannot hold the link digits is created all the same (120
    sites: their 4 tiles of 32 are the only allocation of this size before the
    workspace's)."""
    M = require_lib()
    dims = (3, 2, 5, 4)
    U, x = synth.gauge_field(dims, 0.4, 65), dev(synth.complex_normal((2, 1440), 66))
    out = []
    for n in (0, 1):
        fail(n, 70000)
        ctx = M.mgmlmc_create(dims, torch.cuda.current_stream())
        fail(n, 70000)
        try:
            M.mgmlmc_set_gauge(ctx, U)
            M.mgmlmc_set_mass(ctx, -0.2)
            out.append(_apply(M, ctx, M.OP_D, 0, M.FP64, x))
        finally:
            M.mgmlmc_destroy(ctx)
    assert rel(out[1], out[0]) < 1e-14
