"""The Chebyshev polynomial of Q_trunc against its recurrence in numpy, at the
edges of the kernel's tiles: odd Nvec (8-byte rows), one to sixteen right-hand
sides (one, four and eight per pass), orders with no, one and several products,
aliased and full offsets.  Bar: relative L2 1e-5, as for the other FP32 coarse
operators."""
import numpy as np
import pytest

from paper_1402_2585_gb300 import F32, F64, Hdcg
from tests.gpu_util import from_gpu, rel, to_gpu, torch_or_skip

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nrhs,order", [(1, 1, 5), (5, 4, 1), (6, 3, 2), (33, 9, 3), (40, 16, 8), (64, 8, 4), (63, 5, 3)])
def test_chebyshev_of_qtrunc(n, nrhs, order):
    torch = torch_or_skip()
    cd = (2, 3, 1, 3) if n % 2 else (3, 2, 3, 1)
    dims = tuple(4 * d for d in cd)
    vc = int(np.prod(cd))
    rng = np.random.default_rng(100 + n)
    A = 0.1 / np.sqrt(n) * (rng.standard_normal((vc, 81, n, n)) + 1j * rng.standard_normal((vc, 81, n, n)))
    A[:, 40] += np.eye(n)
    h = Hdcg(dims, 2, stream=torch.cuda.current_stream().cuda_stream)
    h.set_subspace((4, 4, 4, 4), torch.from_numpy(rng.standard_normal((n, vc * 128, 2, 4, 3, 2))).cuda(), F32)
    h.set_coarse(A, prec=F32)
    lo, hi, shift = 0.2, 2.0, 0.05
    h.set_coarse_preconditioner(order, lo, hi, shift)
    x = rng.standard_normal((nrhs, vc, n)) + 1j * rng.standard_normal((nrhs, vc, n))

    keep = []
    for l in range(81):
        d = [l // 3 ** mu % 3 - 1 for mu in range(4)]
        if sum(abs(q) for q in d) <= 1 and all(L >= 3 or (q >= 0 if L == 2 else q == 0) for q, L in zip(d, cd)):
            keep.append((l, d))
    site = np.arange(vc)
    xs, r = [], site
    for L in cd:
        xs.append(r % L)
        r = r // L

    def Q(v):
        y = shift * v
        for l, d in keep:
            nb, mul = 0, 1
            for mu, L in enumerate(cd):
                nb = nb + (xs[mu] + d[mu]) % L * mul
                mul *= L
            y = y + np.einsum("ajk,rak->raj", A[:, l], v[:, nb])
        return y

    th, de = 0.5 * (hi + lo), 0.5 * (hi - lo)
    y, s, d, rho = np.zeros_like(x), x.copy(), x / th, de / th
    for k in range(order):
        y = y + d
        s = s - Q(d)
        new = 1 / (2 * th / de - rho)
        d, rho = new * rho * d + 2 * new / de * s, new
    out = torch.empty((nrhs, vc, n, 2), dtype=torch.float64, device="cuda")
    h.coarse_precondition(to_gpu(x, F64), out, nrhs)
    assert rel(from_gpu(out), y) < 1e-5
    h.close()
