"""A cycle whose smoother is the network is refused while there is none, also
with no smoothing steps."""
import pytest

from paper_2509_11424_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip('torch')
if not torch.cuda.is_available():
    pytest.skip('needs a CUDA GPU', allow_module_level=True)

from gpu_util import Setup, dev  # noqa: E402


@pytest.mark.parametrize('steps', [0, 1])
def test_no_network(steps):
    s = Setup((4, 4, 4, 4), [(2, 2, 2, 2)], [4], m0=0.1, oracle=False)
    M = s.M
    try:
        M.mgmlmc_set_solver(s.ctx, smoother=M.SMOOTHER_NET, smoother_steps=steps)
        b = dev(synth.complex_normal((1, 12 * 256), 3))
        with pytest.raises(Exception, match='network is not initialised'):
            M.mgmlmc_apply(s.ctx, M.OP_SOLVE, 0, M.FP64, b, torch.empty_like(b), 1)
    finally:
        s.close()
