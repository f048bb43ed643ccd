"""The coarse operator of the set-up against the oracle's Galerkin product at
aggregates whose faces are ragged: odd and unit block extents, coarse extents
of 1 (no hop leaves the aggregate), 2 (both hops reach the same neighbour) and
3, one and two coarse levels.  Bound: that of the other coarse-operator
tests (FP64 sums of at most a few thousand terms)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip('torch')
if not torch.cuda.is_available():
    pytest.skip('needs a CUDA GPU', allow_module_level=True)

from gpu_util import Setup, rel  # noqa: E402


@pytest.mark.parametrize('dims,blocks,ntvs', [
    ((4, 6, 2, 3), [(4, 2, 1, 3)], [3]), ((3, 3, 6, 2), [(3, 1, 2, 2)], [5]), ((2, 2, 2, 2), [(1, 1, 1, 1)], [2]),
    ((4, 4, 4, 8), [(2, 2, 2, 2), (1, 2, 2, 4)], [4, 3])])
def test_coarse_operator(dims, blocks, ntvs):
    s = Setup(dims, blocks, ntvs, eps=0.4, m0=-0.1, gseed=51)
    try:
        for l in range(1, len(blocks) + 1):
            A = s.hier.A[l]
            out = np.zeros(A.size, dtype=np.complex128)
            s.M.mgmlmc_get_coarse_op(s.ctx, l, out)
            assert rel(out.reshape(A.shape), A) < 1e-12
    finally:
        s.close()
