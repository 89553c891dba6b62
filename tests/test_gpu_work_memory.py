"""The coarse solvers do not read work memory that they have not written: after a
solve that left NaN in every work vector (a NaN source), the level-1 A-DEF2 solve
and the A-DEF1 solve still meet the dense solution."""
import numpy as np
import pytest

from paper_1402_2585_gb300 import F32, F64, Hdcg, HdcgError
from tests.gpu_util import from_gpu, rel, to_gpu, torch_or_skip

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("method", ["level2", "deflation"])
@pytest.mark.parametrize("nrhs", [1, 3])
def test_coarse_solves_after_a_nan_source(method, nrhs):
    torch = torch_or_skip()
    dims, n, vc = (8, 8, 8, 8), 4, 16
    rng = np.random.default_rng(5)
    z = rng.standard_normal((vc, n, n)) + 1j * rng.standard_normal((vc, n, n))
    D = 0.2 * (z + z.conj().transpose(0, 2, 1)) + 4 * np.eye(n)      # Hermitian, dominated by its diagonal
    A = np.zeros((vc, 81, n, n), dtype=np.complex128)
    A[:, 40] = D
    phi = rng.standard_normal((n, 2048, 4, 4, 3, 2))
    b = rng.standard_normal((nrhs, vc, n)) + 1j * rng.standard_normal((nrhs, vc, n))
    h = Hdcg(dims, 4, stream=torch.cuda.current_stream().cuda_stream)
    h.set_subspace((4, 4, 4, 4), torch.from_numpy(phi).cuda(), F32)
    h.set_coarse(A, prec=F32)
    if method == "level2":
        h.build_subspace((2, 2, 1, 1), 2, F32, inv_steps=1, inv_tol=1e-4, seed=3, level=2)
        h.build_coarse(F32, level=2)
    else:
        h.build_coarse_deflation(4, inv_steps=1, tol=1e-4, seed=3)
    x = torch.zeros((nrhs, vc, n, 2), dtype=torch.float64, device="cuda")
    h.coarse_solve(to_gpu(b, F64), x, nrhs, 1e-6)
    want = np.einsum("ajk,rak->raj", np.linalg.inv(D), b)
    assert rel(from_gpu(x), want) < 1e-5      # condition number below 4, tolerance 1e-6
    try:
        h.coarse_solve(torch.full_like(x, float("nan")), torch.empty_like(x), nrhs, 1e-6, maxiter=4)
    except HdcgError:
        pass                                   # the level-1 solve reports the breakdown
    x.zero_()
    h.coarse_solve(to_gpu(b, F64), x, nrhs, 1e-6)
    assert rel(from_gpu(x), want) < 1e-5
    h.close()
