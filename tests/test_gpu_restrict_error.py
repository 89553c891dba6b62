"""The restriction's sums do not drift: a field along a subspace vector makes every
product of a block's sum positive, so rounding towards zero would show as an error
proportional to the number of terms.  Bar 2e-7: the block's sum is rounded to FP32
three times (granule, thread, result: 2^-24 each)."""
import numpy as np
import pytest

from paper_1402_2585_gb300 import F16, F32, Hdcg
from tests.gpu_util import from_gpu, rel, to_gpu, torch_or_skip

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,vprec", [(F16, F16), (F16, F32), (F32, F32)])
@pytest.mark.parametrize("Ls", [4, 16])
def test_restriction_of_a_field_along_the_subspace(prec, vprec, Ls):
    torch = torch_or_skip()
    dims, n = (8, 4, 4, 8), 5
    n4 = int(np.prod(dims)) // 2
    rng = np.random.default_rng(Ls)
    h = Hdcg(dims, Ls, stream=torch.cuda.current_stream().cuda_stream)
    h.set_subspace((4, 4, 4, 4), torch.from_numpy(rng.standard_normal((n, n4, Ls, 4, 3, 2))).cuda(), prec)
    phi = np.zeros((n, n4, Ls, 4, 3), dtype=np.complex128)
    h.get_subspace(phi)
    lex = 2 * np.arange(n4)
    x = [None, lex // dims[0] % dims[1], lex // (dims[0] * dims[1]) % dims[2], lex // (dims[0] * dims[1] * dims[2])]
    x[0] = lex % dims[0] + (1 + x[1] + x[2] + x[3]) % 2
    blk = np.zeros(n4, dtype=int)
    for q, L in zip(reversed(x), reversed(dims)):
        blk = blk * (L // 4) + q // 4
    v = to_gpu(64.0 * phi[0], vprec)
    c = torch.empty((blk.max() + 1, n, 2), dtype=torch.float64, device="cuda")
    h.restrict(v, vprec, c)
    want = np.zeros((blk.max() + 1, n), dtype=np.complex128)
    np.add.at(want, blk, np.einsum("nisac,isac->in", phi.conj(), from_gpu(v)))
    assert rel(from_gpu(c), want) < 2e-7
    h.close()
