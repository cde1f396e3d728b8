"""What solves keep in the context's pool."""
import pytest

from paper_2403_12179_gb300 import mg

pytestmark = pytest.mark.gpu


def _kept(n, box, batch=1, **kw):
    """Pool bytes beyond the caller's fabs after a solve."""
    ctx = mg.mg_init(0)
    try:
        ba = mg.mg_box_array_create(ctx, (0, 0, 0), tuple(v - 1 for v in n), box)
        P = [(mg.mg_fab_alloc(ctx, ba, 1, 0), mg.mg_fab_alloc(ctx, ba, 1, 1)) for _ in range(batch)]
        for r, _ in P:
            mg.mg_fab_set_val(ctx, r, 1.0)
        base = mg.mg_pool_info(ctx)[1]
        bc, opt = mg.make_bc((0, 0, 0)), mg.make_options(fixed_vcycles=2, **kw)
        if batch > 1:
            mg.mg_solve_batch(ctx, [p[0] for p in P], [p[1] for p in P], [bc] * batch, 1e-10, opt)
        else:
            mg.mg_solve(ctx, P[0][0], P[0][1], bc, 1e-10, opt)
        return mg.mg_pool_info(ctx)[1] - base
    finally:
        mg.mg_finalize(ctx)


@pytest.mark.parametrize("n,box,batch", [((128, 128, 128), (32, 32, 32), 1), ((64, 64, 256), (64, 64, 32), 1),
                                         ((96, 80, 112), (48, 48, 48), 1), ((64, 64, 64), (64, 64, 64), 8)])
def test_mixed_levels_take_phi_rhs_and_the_residual(n, box, batch):
    """The FP64 residual, and phi and rhs of every FP32 level (8/7 of the finest): no other field.  (The
    tables allowed for: 1 MB a solve; a field of 4 bytes a cell would be 4.2 MB, 3.4 MB in the third
    case and 1.05 MB in the last, whose tables take half of that.)"""
    cells = n[0] * n[1] * n[2]
    tables = 0.5e6 if batch > 1 else 1e6
    assert _kept(n, box, batch, precision=mg.MG_PREC_MIXED) <= batch * (cells * (8 + 8 * 8 / 7) + tables)
