"""Restriction and prolongation at the edges of their kernels' tiles (16 vectors
per tensor-core tile, 16 or 4 per CUDA-core group) against numpy on the stored
subspace.  Bars: FP32 sums 2e-6 (about 1e4 products per sum), 16-bit output of
the prolongation 5e-4 (its rounding), FP64 1e-12."""
import numpy as np
import pytest

from paper_1402_2585_gb300 import F16, F32, F64, Hdcg
from tests.gpu_util import from_gpu, rel, to_gpu, torch_or_skip

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,vprec", [(F16, F16), (F16, F32), (F32, F16), (F32, F32), (F64, F64)])
@pytest.mark.parametrize("n,Ls,dims", [(1, 2, (4, 4, 4, 8)), (5, 16, (4, 8, 4, 4)), (17, 4, (8, 4, 4, 4)), (33, 8, (4, 4, 8, 4)),
                                       (64, 2, (4, 4, 4, 4))])
def test_restrict_and_prolong_against_numpy(prec, vprec, n, Ls, dims):
    torch = torch_or_skip()
    if prec == F64 and n == 64:
        pytest.skip("the block transform refuses 64 FP64 vectors (shared memory)")
    n4 = int(np.prod(dims)) // 2
    rng = np.random.default_rng(n)
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
    vc = blk.max() + 1
    v = to_gpu(rng.standard_normal((n4, Ls, 4, 3)) + 1j * rng.standard_normal((n4, Ls, 4, 3)), vprec)
    vn = from_gpu(v)
    c = torch.empty((vc, n, 2), dtype=torch.float64, device="cuda")
    h.restrict(v, vprec, c)
    want = np.zeros((vc, n), dtype=np.complex128)
    np.add.at(want, blk, np.einsum("nisac,isac->in", phi.conj(), vn))
    bar = 1e-12 if prec == F64 else 2e-6
    assert rel(from_gpu(c), want) < bar
    out = torch.empty_like(v)
    h.prolong(c, out, vprec)
    back = np.einsum("nisac,in->isac", phi, from_gpu(c)[blk])
    assert rel(from_gpu(out), back) < (5e-4 if vprec == F16 else bar)
    h.close()
