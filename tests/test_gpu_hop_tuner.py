"""What the hop autotuner may choose from: for FP64 storage only the variants that
compute in FP64 (a forced variant 3 is double-float and gives other bits), and anew
for another action.  An untuned H costs four launches per pass and candidate more
than a tuned one."""
import pytest

import synthetic as sy
from paper_1402_2585_gb300 import F32, F64, Hdcg
from tests.gpu_util import to_gpu, torch_or_skip

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,candidates", [(F64, 3), (F32, 4)])
def test_candidates(prec, candidates):
    torch = torch_or_skip()
    dims, Ls = (4, 4, 4, 4), 8
    h = Hdcg(dims, Ls, stream=torch.cuda.current_stream().cuda_stream)
    h.set_gauge(torch.from_numpy(sy.gauge_field(dims, 0.4, 730)).cuda())
    x = to_gpu(sy.gaussian_fermion(dims, Ls, 731), prec)
    y = torch.empty_like(x)

    def launches():
        n = h.launch_count()
        h.apply_mdagm(x, y, prec)
        return h.launch_count() - n

    for b, c in ((1.0, 0.0), (1.5, 0.5)):
        h.set_dwf(1.8, b, c, 0.02)
        first = launches()
        assert first - launches() == 4 * 4 * candidates
    tuned = y.clone()
    h.set_hop_variant(0)
    h.apply_mdagm(x, y, prec)
    assert torch.equal(y, tuned)
    h.close()
