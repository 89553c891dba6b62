"""Coarse CG over FP32's range: the recursion is homogeneous in the source, so a
source scaled by 1e-24 or 1e20 converges as one of order 1 does, on the small grids
(one cluster launch an iteration) and beyond them.  Its |r|^2 are squares of FP32
entries, which leave FP32's range.  Tolerance: 1e-5 plus 2e-6 for the FP32 recursion
of a well-conditioned operator."""
import numpy as np
import pytest

from paper_1402_2585_gb300 import F32, F64, Hdcg
from tests.gpu_util import apply_stencil, from_gpu, random_stencil, to_gpu, torch_or_skip

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cd,n,nrhs", [((3, 3, 1, 2), 8, 3), ((4, 4, 4, 8), 24, 16)])
def test_coarse_cg_does_not_depend_on_the_scale(cd, n, nrhs):
    torch = torch_or_skip()
    vc = int(np.prod(cd))
    rng = np.random.default_rng(n)
    A, nb, stored = random_stencil(cd, n, rng)
    h = Hdcg(tuple(4 * d for d in cd), 2, stream=torch.cuda.current_stream().cuda_stream)
    h.set_subspace((4, 4, 4, 4), torch.from_numpy(rng.standard_normal((n, vc * 128, 2, 4, 3, 2))).cuda(), F32)
    h.set_coarse(A.astype(np.complex128), prec=F32)
    b = rng.standard_normal((nrhs, vc, n)) + 1j * rng.standard_normal((nrhs, vc, n))
    its = []
    for scale in (1.0, 1e-24, 1e20):
        x = torch.zeros((nrhs, vc, n, 2), dtype=torch.float64, device="cuda")
        its.append(h.coarse_solve(to_gpu(scale * b, F64), x, nrhs, 1e-5, maxiter=200))
        r = b - apply_stencil(A, nb, stored, from_gpu(x) / scale)
        assert (np.linalg.norm(r, axis=(1, 2)) < 1.2e-5 * np.linalg.norm(b, axis=(1, 2))).all()
    assert max(its) - min(its) <= 1
    h.close()
