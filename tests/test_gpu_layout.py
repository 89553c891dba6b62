"""Canonical <-> internal field conversions: the granule transposition (16-byte
aligned buffers) against the element-wise path (buffers aligned to one element
only), bit for bit, at field sizes around the transposition's tiles."""
import numpy as np
import pytest

from paper_1402_2585_gb300 import BF16, BF16T, DF64, F16, F32, F64, Hdcg
from tests.gpu_util import to_gpu, torch_or_skip

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [F64, DF64, F32, F16, BF16, BF16T])
@pytest.mark.parametrize("dims,Ls", [((2, 2, 2, 2), 2), ((6, 2, 2, 2), 4), ((2, 2, 4, 4), 8), ((4, 4, 4, 6), 16)])
def test_aligned_and_unaligned_buffers_agree(prec, dims, Ls):
    torch = torch_or_skip()
    n4 = int(np.prod(dims)) // 2
    rng = np.random.default_rng(17)
    f = rng.standard_normal((n4, Ls, 4, 3)) + 1j * rng.standard_normal((n4, Ls, 4, 3))
    f[rng.random(f.shape[:2]) < 0.3] = 0.0                      # whole 5D sites, as of a point source
    if prec in (F64, DF64, F32):
        f *= 2.0 ** rng.integers(-60, 30, f.shape[:2])[..., None, None]
    h = Hdcg(dims, Ls, stream=torch.cuda.current_stream().cuda_stream)
    h.set_dwf(1.8, 1.5, 0.5, 0.01)
    h.set_gauge(torch.from_numpy(np.broadcast_to(np.eye(3, dtype=np.complex128), (2 * n4, 4, 3, 3)).copy()).cuda())
    x = to_gpu(f, prec)

    def shifted(t):
        b = torch.empty(t.numel() + 1, dtype=t.dtype, device=t.device)
        return b[1:].view_as(t).copy_(t)

    want = torch.empty_like(x)
    h.apply_mpc(x, want, prec=prec)
    assert x.data_ptr() % 16 == 0 and want.data_ptr() % 16 == 0
    for a, b in ((shifted(x), torch.empty_like(x)), (x, shifted(x)), (shifted(x), shifted(x))):
        h.apply_mpc(a, b, prec=prec)
        assert torch.equal(b, want)
    assert bool(torch.isfinite(want).all()) and float(want.abs().max()) > 0
