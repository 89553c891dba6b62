"""Expired waits in the tensor-core stencil: with no time allowed, the roles of a
CTA give up at different stages of the ring.  The call reports it, every copy and
MMA already issued is waited for, and the handle's next apply gives the same bits
as one before (several stages, one and two sites per MMA, one and two parts)."""
import numpy as np
import pytest

from paper_1402_2585_gb300 import F16, F32, F64, Hdcg, HdcgError
from tests.gpu_util import random_stencil, to_gpu, torch_or_skip

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,prec", [(8, F16), (24, F32), (40, F32)])
def test_apply_after_an_expired_wait(n, prec):
    torch = torch_or_skip()
    cd, nrhs = (3, 4, 3, 4), 5
    vc = int(np.prod(cd))
    rng = np.random.default_rng(n)
    A, _, _ = random_stencil(cd, n, rng)
    h = Hdcg(tuple(4 * d for d in cd), 2, stream=torch.cuda.current_stream().cuda_stream)
    h.set_subspace((4, 4, 4, 4), torch.from_numpy(rng.standard_normal((n, vc * 128, 2, 4, 3, 2))).cuda(), prec)
    h.set_coarse(A.astype(np.complex128), prec=prec)
    x = to_gpu(rng.standard_normal((nrhs, vc, n)) + 1j * rng.standard_normal((nrhs, vc, n)), F64)
    want, y = torch.empty_like(x), torch.empty_like(x)
    h.coarse_apply_multi(x, want, nrhs)
    for _ in range(3):
        h.set_coarse_tc_wait(0.0)
        with pytest.raises(HdcgError) as e:
            h.coarse_apply_multi(x, y, nrhs)
        assert e.value.code == -6
        h.set_coarse_tc_wait(2.0)
        h.coarse_apply_multi(x, y, nrhs)
        assert torch.equal(y, want)
    with pytest.raises(HdcgError) as e:
        h.set_coarse_tc_wait(-1.0)
    assert e.value.code == -1
    h.close()
