"""FP32 SAP on blocks of 2^4 sites (one half warp per block and right-hand
side) against the oracle, on lattices whose block count times right-hand sides
does not fill the last thread block.

Tolerance 1e-4, derived where the other FP32 smoother tests state it (block
minimal-residual steps with alpha from FP32 block sums)."""
import numpy as np
import pytest

from oracle import dirac, smoother as osm
from paper_2509_11424_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip('torch')
if not torch.cuda.is_available():
    pytest.skip('needs a CUDA GPU', allow_module_level=True)

from gpu_util import dev, host, rel, require_lib  # noqa: E402


@pytest.mark.parametrize('dims,nrhs,sweeps', [((4, 4, 4, 4), 1, 1), ((12, 4, 4, 4), 3, 2), ((4, 4, 12, 8), 2, 1)])
def test_small_blocks(dims, nrhs, sweeps):
    M = require_lib()
    U = synth.gauge_field(dims, 0.4, 51)
    n = dirac.volume(dims) * 12
    ctx = M.mgmlmc_create(dims, torch.cuda.current_stream())
    try:
        M.mgmlmc_set_gauge(ctx, U)
        M.mgmlmc_set_mass(ctx, 0.1)
        M.mgmlmc_set_solver(ctx, smoother=M.SMOOTHER_SAP, smoother_steps=sweeps, sap_iters=4)
        b = synth.complex_normal((nrhs, n), 52)
        out = torch.empty((nrhs, n), dtype=torch.complex64, device='cuda')
        M.mgmlmc_apply(ctx, M.OP_SMOOTH, 0, M.FP32, dev(b, torch.complex64), out, nrhs)
        got = host(out).astype(np.complex128)
        D = dirac.wilson_matrix(U, 0.1, dims)
        for r in range(nrhs):
            want = osm.sap_smooth(D, dims, (2, 2, 2, 2), b[r].astype(np.complex64).astype(np.complex128),
                                  sweeps=sweeps, iters=4)
            assert rel(got[r], want) < 1e-4
    finally:
        M.mgmlmc_destroy(ctx)


@pytest.mark.parametrize('dims,nrhs', [((4, 4, 4, 4), 1), ((12, 4, 4, 12), 3)])
def test_small_blocks_match_general_kernel(dims, nrhs):
    """Variant 2 runs the general block kernel on these blocks as on any other:
    the same sums in the same order, the same bits."""
    M = require_lib()
    n = dirac.volume(dims) * 12
    ctx = M.mgmlmc_create(dims, torch.cuda.current_stream())
    try:
        M.mgmlmc_set_gauge(ctx, synth.gauge_field(dims, 0.4, 53))
        M.mgmlmc_set_mass(ctx, 0.1)
        M.mgmlmc_set_solver(ctx, smoother=M.SMOOTHER_SAP, smoother_steps=2, sap_iters=3)
        b = dev(synth.complex_normal((nrhs, n), 54), torch.complex64)
        outs = []
        for v in range(M.mgmlmc_kernel_variants(M.VARIANT_SAP_FP32)):
            M.mgmlmc_set_kernel_variant(ctx, M.VARIANT_SAP_FP32, v)
            out = torch.empty_like(b)
            M.mgmlmc_apply(ctx, M.OP_SMOOTH, 0, M.FP32, b, out, nrhs)
            outs.append(host(out))
        assert np.array_equal(outs[0], outs[1]) and np.array_equal(outs[0], outs[2])
    finally:
        M.mgmlmc_destroy(ctx)
