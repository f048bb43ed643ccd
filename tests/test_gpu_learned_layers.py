"""The network's forward pass and loss gradient at channel counts around the
ways a layer is split (1, 2, groups of 4, 16 inputs staged at a time, the
largest) on lattices whose sites do not fill the last block of 128.  FP32:
two sums of up to 9 x 32 x 4 terms and a transport, eps sqrt(N / 2) each, four
standard deviations for the worst entry: 3e-6, bound 1e-5; FP64: 1e-12 and, for
the gradient's longer sums, 1e-10, as in the other tests of the network."""
import numpy as np
import pytest

from oracle import dirac, learned as oln
from paper_2509_11424_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip('torch')
if not torch.cuda.is_available():
    pytest.skip('needs a CUDA GPU', allow_module_level=True)

from gpu_util import dev, host, rel, require_lib  # noqa: E402

M = require_lib()


@pytest.mark.parametrize('dims,C', [((2, 4, 2, 4), 1), ((3, 2, 4, 6), 2), ((2, 2, 6, 2), 5), ((3, 4, 2, 6), 17),
                                    ((2, 4, 2, 2), 32)])
def test_layers(dims, C):
    U = synth.gauge_field(dims, 0.4, 61)
    ctx = M.mgmlmc_create(dims, torch.cuda.current_stream())
    try:
        M.mgmlmc_set_gauge(ctx, U)
        M.mgmlmc_set_mass(ctx, 0.2)
        M.mgmlmc_learned_init(ctx, C, 7)
        shapes = [(9, C, 1, 4, 4), (9, C, C, 4, 4), (9, 1, C, 4, 4)]
        Ws = [0.3 * synth.complex_normal(s, 62 + i) for i, s in enumerate(shapes)]
        M.mgmlmc_learned_weights(ctx, np.concatenate([w.reshape(-1) for w in Ws]).view(np.float64).copy(), 1)
        n = dirac.volume(dims) * 12
        r = synth.complex_normal((3, n), 65)
        for prec, ct, tol in ((0, torch.complex128, 1e-12), (1, torch.complex64, 1e-5)):
            out = torch.empty((3, n), dtype=ct, device='cuda')
            M.mgmlmc_apply(ctx, M.OP_NET, 0, prec, dev(r, ct), out, 3)
            got = host(out)
            for b in range(3):
                assert rel(got[b], oln.network_forward(Ws, r[b], U, dims)[-1][0]) < tol
        grad = np.zeros(2 * M.mgmlmc_learned_size(ctx))
        M.mgmlmc_learned_loss_grad(ctx, dev(r[:1]), 1, grad)
        D = lambda v: dirac.apply_wilson(U, v, 0.2, dims)
        DH = lambda v: dirac.apply_gamma5(D(dirac.apply_gamma5(v)))
        _, g = oln.loss_and_grads(Ws, r[0], U, dims, D, DH)
        assert rel(grad.view(np.complex128), np.concatenate([w.reshape(-1) for w in g])) < 1e-10
    finally:
        M.mgmlmc_destroy(ctx)
