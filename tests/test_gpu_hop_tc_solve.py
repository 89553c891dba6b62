"""The tensor-core hop where a solve uses it: the fused CG step, shifts and batches
with a source that is finished from the start, several sites per warp; and the
batched restriction and prolongation at ragged right-hand-side counts."""
import numpy as np
import pytest

import synthetic as sy
from paper_1402_2585_gb300 import ALG_ADEF2, F16, F32, F64, Hdcg
from tests.gpu_util import from_gpu, rel, to_gpu, torch_or_skip

pytestmark = pytest.mark.gpu


def _handle(torch, dims, Ls, seed):
    h = Hdcg(dims, Ls, stream=torch.cuda.current_stream().cuda_stream)
    h.set_dwf(1.8, 1.5, 0.5, 0.05)
    h.set_gauge(torch.from_numpy(sy.gauge_field(dims, 0.4, seed)).cuda())
    return h


@pytest.mark.parametrize("Ls", [8, 16, 32])
def test_several_sites_per_warp(Ls):
    """8192 4D sites, at most 2432 warps: against the scalar pass.  Both round FP32
    sums to FP16; the sums' own errors flip few of these roundings, so that the
    fields differ by less than one rounding of every entry (2^-11)."""
    torch = torch_or_skip()
    dims = (16, 8, 16, 8)
    h = _handle(torch, dims, Ls, 710)
    x = to_gpu(sy.gaussian_fermion(dims, Ls, 711), F16)
    out = {}
    for variant in (0, -1):
        h.set_hop_variant(variant)
        for dagger in (False, True):
            y = torch.zeros_like(x)
            h.apply_mpc(x, y, dagger=dagger, prec=F16)
            out[variant, dagger] = from_gpu(y)
    for dagger in (False, True):
        assert rel(out[-1, dagger], out[0, dagger]) < 2.0 ** -11
    h.close()


@pytest.mark.parametrize("Ls,nrhs", [(8, 1), (8, 2), (8, 3), (8, 9), (8, 16), (16, 5), (32, 5)])
def test_preconditioned_batch(Ls, nrhs):
    """HDCG with the 16-bit preconditioner: the tensor-core pass needs the scalar
    pass's iterations, a batch those of its sources alone (each within a tenth and
    one), every source meets its tolerance, and a zero source stays zero."""
    torch = torch_or_skip()
    dims, tol = (8, 8, 4, 4), 1e-8
    h = _handle(torch, dims, Ls, 720)
    h.set_hop_variant(0)
    h.build_subspace((4, 4, 4, 4), 6, F16, inv_steps=2, inv_tol=1e-3, inv_maxiter=200, seed=721)
    h.build_coarse(F32)
    b = sy.gaussian_fermions(dims, Ls, 722, nrhs)
    if nrhs > 1:
        b[1] = 0.0
    bt = torch.from_numpy(b).cuda()
    par = Hdcg.default_params(algorithm=ALG_ADEF2, outer_prec=F32, sloppy_prec=F16)
    its = {}
    for variant in (0, -1):
        h.set_hop_variant(variant)
        x = torch.full_like(bt, 7.0)
        st = h.solve(bt, x, tol, par, nrhs)
        assert st.status == 0
        its[variant] = st.iterations
        w = torch.empty_like(bt[0])
        for k in range(nrhs):
            if not b[k].any():
                assert not x[k].abs().max()
                continue
            h.apply_mdagm(x[k].contiguous(), w, F64)
            assert float((bt[k] - w).norm() / bt[k].norm()) < 1.05 * tol
    assert abs(its[-1] - its[0]) <= 1 + its[0] // 10
    alone = []
    for k in range(nrhs):
        if b[k].any():
            x = torch.zeros_like(bt[:1])
            alone.append(h.solve(bt[k:k + 1].contiguous(), x, tol, par, 1).iterations)
    assert abs(its[-1] - max(alone)) <= 1 + max(alone) // 10
    h.close()
