"""Coarse CG on the tensor-core operator: small grids (couplings split over CTAs, the
rest of an iteration in one cluster launch) up to its limit and one size beyond, odd
site counts, padded and unpadded right-hand sides, one right-hand side already
converged.  The residual is recomputed in numpy: tolerance 1e-5 plus 2e-6 for the
FP32 recursion of a well-conditioned operator (spectrum within [0.4, 1.6])."""
import numpy as np
import pytest

from paper_1402_2585_gb300 import F16, F32, F64, Hdcg
from tests.gpu_util import from_gpu, to_gpu, torch_or_skip

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,cd,n,nrhs", [
    (F32, (1, 1, 1, 3), 5, 1), (F32, (2, 1, 2, 2), 24, 2), (F16, (3, 1, 3, 3), 8, 5), (F32, (3, 3, 3, 3), 64, 16),
    (F32, (4, 4, 4, 4), 32, 16), (F16, (4, 4, 4, 4), 24, 1), (F32, (4, 4, 4, 4), 24, 4), (F32, (4, 4, 4, 4), 40, 16)])
def test_coarse_cg_residual(prec, cd, n, nrhs):
    torch = torch_or_skip()
    dims = tuple(4 * d for d in cd)
    vc = int(np.prod(cd))
    rng = np.random.default_rng(vc * n)
    site, xs, r = np.arange(vc), [], np.arange(vc)
    for L in cd:
        xs.append(r % L)
        r = r // L
    nb = np.zeros((vc, 81), dtype=int)
    stored, mate = [], []
    for l in range(81):
        d = [l // 3 ** mu % 3 - 1 for mu in range(4)]
        idx, mul, m = 0, 1, 0
        for mu, L in enumerate(cd):
            idx = idx + (xs[mu] + d[mu]) % L * mul
            mul *= L
            m += 3 ** mu * ((d[mu] if L == 2 else -d[mu]) + 1)
        nb[:, l] = idx
        mate.append(m)
        stored.append(all(L >= 3 or (q >= 0 if L == 2 else q == 0) for q, L in zip(d, cd)))
    k = sum(stored)
    A = np.zeros((vc, 81, n, n), dtype=np.complex64)
    for l in range(81):
        if not stored[l] or mate[l] < l:
            continue
        z = (rng.standard_normal((vc, n, n)) + 1j * rng.standard_normal((vc, n, n))) * (0.1 / np.sqrt(2 * n * k))
        if mate[l] == l:
            z = 0.5 * (z + z[nb[:, l]].conj().transpose(0, 2, 1))
        A[:, l] = z
        if mate[l] != l:
            A[nb[:, l], mate[l]] = z.conj().transpose(0, 2, 1)
    A[:, 40] += np.eye(n)
    if prec == F16:
        A = (A.real.astype(np.float16).astype(np.float32) + 1j * A.imag.astype(np.float16).astype(np.float32)).astype(np.complex64)
    h = Hdcg(dims, 2, stream=torch.cuda.current_stream().cuda_stream)
    h.set_subspace((4, 4, 4, 4), torch.from_numpy(rng.standard_normal((n, vc * 128, 2, 4, 3, 2))).cuda(), prec)
    h.set_coarse(A.astype(np.complex128), prec=prec)
    b = rng.standard_normal((nrhs, vc, n)) + 1j * rng.standard_normal((nrhs, vc, n))
    if nrhs > 1:
        b[1] = 0.0
    x = torch.zeros((nrhs, vc, n, 2), dtype=torch.float64, device="cuda")
    its = h.coarse_solve(to_gpu(b, F64), x, nrhs, 1e-5, maxiter=200)
    assert 1 <= its < 60
    xn = from_gpu(x)
    y = np.zeros_like(b)
    for l in range(81):
        if stored[l]:
            y += np.einsum("ajk,rak->raj", A[:, l].astype(np.complex128), xn[:, nb[:, l]])
    for q in range(nrhs):
        if not b[q].any():
            assert not xn[q].any()
        else:
            assert np.linalg.norm(b[q] - y[q]) < 1.2e-5 * np.linalg.norm(b[q])
    h.close()
