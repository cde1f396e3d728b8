"""The coarse end of the cycle in one launch, by one CTA and in slabs over a cluster, against the same
levels stage by stage: bit for bit.  Slabs of different heights, idle CTAs, a short last slab, thin
domains, each kind of face along z, no or several smoothing steps, cells given and by default."""
import numpy as np
import pytest
import torch

from paper_2403_12179_gb300 import mg

pytestmark = pytest.mark.gpu
F64, MIXED = mg.MG_PREC_F64, mg.MG_PREC_MIXED
CASES = [((32, 32, 32), F64, 0), ((64, 16, 16), F64, 0), ((24, 32, 40), F64, 0), ((48, 48, 48), F64, 0),
         ((16, 16, 64), F64, 0), ((64, 64, 8), F64, 4096), ((32, 32, 32), F64, 4096), ((64, 64, 64), F64, 32768),
         ((32, 32, 32), MIXED, 0), ((64, 64, 64), MIXED, 0), ((64, 64, 64), MIXED, 32768), ((24, 40, 112), MIXED, 0),
         ((32, 48, 72), MIXED, 40000), ((48, 40, 56), F64, 0), ((24, 20, 28), F64, 2000), ((48, 40, 56), MIXED, 4000)]


def _solve(ctx, n, per, prec, cells, nu):
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    f = torch.randn(n[2], n[1], n[0], generator=g, device="cuda", dtype=torch.float64)
    if all(per):
        f -= f.mean()
    ba = mg.mg_box_array_create(ctx, (0, 0, 0), tuple(v - 1 for v in n), n)
    fr, fp = mg.mg_fab_alloc(ctx, ba, 1, 0), mg.mg_fab_alloc(ctx, ba, 1, 1)
    mg.mg_fab_set_val(ctx, fp, 0.0)
    torch.cuda.synchronize()
    mg.mg_fab_copy_from_dense(ctx, fr, f.data_ptr(), False)
    opt = mg.make_options(precision=prec, coarse_cells=cells, fixed_vcycles=3, nu1=nu[0], nu2=nu[1])
    res = mg.mg_solve(ctx, fr, fp, mg.make_bc(per), 1e-10, opt)
    out = torch.empty_like(f)
    mg.mg_fab_copy_to_dense(ctx, fp, out.data_ptr(), False)
    torch.cuda.synchronize()
    return out.cpu().numpy(), res.rel_resid


@pytest.mark.parametrize("n,prec,cells", CASES)
@pytest.mark.parametrize("per", [(1, 1, 1), (0, 0, 0), (1, 0, 1), (0, 1, 0)])
@pytest.mark.parametrize("nu", [(2, 2), (0, 1), (1, 0), (3, 1)])
def test_one_launch_equals_stages(n, prec, cells, per, nu):
    ctx = mg.mg_init(0)
    try:
        got, rg = _solve(ctx, n, per, prec, cells, nu)
        ref, rr = _solve(ctx, n, per, prec, -1, nu)
        assert np.isfinite(got).all() and np.abs(got).max() > 0
        assert got.tobytes() == ref.tobytes() and rg == rr
    finally:
        mg.mg_finalize(ctx)
