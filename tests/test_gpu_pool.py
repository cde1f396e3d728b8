"""What solves keep in the context's pool."""
import pytest

from paper_2403_12179_gb300 import mg
from tests import gpu_util as gu

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


@pytest.mark.parametrize("n,box", [((64, 64, 64), (32, 32, 32)), ((32, 32, 32), (32, 32, 32))])
@pytest.mark.parametrize("precision", [mg.MG_PREC_F64, mg.MG_PREC_MIXED])
def test_solve_fits_where_a_batch_of_one_fits(n, box, precision):
    """The tables that only a solve on its own launches from are not kept for members of a batch, and a
    solve goes without the cluster's (at least 4096 cells of 8 bytes here) where the pool has no room:
    the same bits.  (16 KB are left for its other tables, some hundred bytes a level.)"""
    def run(pool, batch):
        ctx = mg.mg_init(0, pool)
        try:
            ba = mg.mg_box_array_create(ctx, (0, 0, 0), tuple(v - 1 for v in n), box)
            r, u = mg.mg_fab_alloc(ctx, ba, 1, 0), mg.mg_fab_alloc(ctx, ba, 1, 1)
            mg.mg_fab_set_val(ctx, r, 1.0)
            bc, opt = mg.make_bc((0, 0, 0)), mg.make_options(fixed_vcycles=3, precision=precision)
            if batch:
                res = mg.mg_solve_batch(ctx, [r], [u], [bc], 1e-10, opt)[0]
            else:
                res = mg.mg_solve(ctx, r, u, bc, 1e-10, opt)
            return mg.mg_pool_info(ctx)[1], res.rel_resid, gu.fab_dense(ctx, u, n[::-1]).tobytes()
        finally:
            mg.mg_finalize(ctx)

    alone, in_batch = run(0, False), run(0, True)
    assert alone[0] >= in_batch[0] + 4096 * 8
    tight = run(in_batch[0] + (16 << 10), False)
    assert tight[1:] == alone[1:] == in_batch[1:]


def test_staged_solve_gives_way():
    """An FP64 solve over ragged boxes keeps phi and rhs on a box of its own.  That memory is given back
    when the caller's next fab needs it, and the solve goes without it (the same bits) until there is
    room again."""
    n, box = (96, 80, 112), (48, 48, 48)
    cells = n[0] * n[1] * n[2]

    def solve(ctx, r, u):
        mg.mg_fab_set_val(ctx, u, 0.0)
        res = mg.mg_solve(ctx, r, u, mg.make_bc((0, 0, 0)), 1e-10, mg.make_options(fixed_vcycles=3))
        return res.rel_resid, gu.fab_dense(ctx, u, n[::-1]).tobytes()

    def fabs(ctx):
        ba = mg.mg_box_array_create(ctx, (0, 0, 0), tuple(v - 1 for v in n), box)
        r, u = mg.mg_fab_alloc(ctx, ba, 1, 0), mg.mg_fab_alloc(ctx, ba, 1, 1)
        mg.mg_fab_set_val(ctx, r, 1.0)
        return ba, r, u

    ctx = mg.mg_init(0)
    try:
        _, r, u = fabs(ctx)
        empty = mg.mg_pool_info(ctx)[1]
        ref = solve(ctx, r, u)
        full = mg.mg_pool_info(ctx)[1]
        assert full - empty >= 2 * 8 * cells  # staged: phi and rhs again
    finally:
        mg.mg_finalize(ctx)
    ctx = mg.mg_init(0, full + 8 * cells // 2)  # room for half a fab more
    try:
        ba, r, u = fabs(ctx)
        assert solve(ctx, r, u) == ref and mg.mg_pool_info(ctx)[1] == full
        other = mg.mg_fab_alloc(ctx, ba, 1, 0)  # takes it
        assert mg.mg_pool_info(ctx)[1] < full
        for _ in range(2):
            assert solve(ctx, r, u) == ref and mg.mg_pool_info(ctx)[1] < full
        mg.mg_fab_free(ctx, other)
        assert solve(ctx, r, u) == ref and mg.mg_pool_info(ctx)[1] >= full
    finally:
        mg.mg_finalize(ctx)


def test_amr_tables_per_ghost():
    """A two-level plan's tables: 104 bytes a coarse/fine ghost (offsets of three fine and nine coarse
    cells and the kept coarse value).  From two plans over one pair of levels, of which the second (other
    options) builds its tables once more; the refluxing table takes 88 bytes a coarse face, and 0.9 MB
    are allowed for the hierarchy and the box tables (at 8 bytes a ghost more, the excess is 0.8 MB)."""
    ctx = mg.mg_init(0)
    try:
        n, m = 64, 128  # refined region: the whole domain but one coarse cell at every face
        ba0 = mg.mg_box_array_create(ctx, (0, 0, 0), (n - 1,) * 3, (n,) * 3)
        ba1 = mg.mg_box_array_create(ctx, (2, 2, 2), (m - 3,) * 3, (m,) * 3)
        f = [mg.mg_fab_alloc(ctx, b, 1, g) for b, g in ((ba0, 0), (ba0, 1), (ba1, 0), (ba1, 1))]
        mg.mg_fab_set_val(ctx, f[0], 1.0)
        mg.mg_fab_set_val(ctx, f[2], 1.0)
        used = mg.mg_pool_info(ctx)[1]
        mg.mg_amr2_solve(ctx, *f, mg.make_bc((0, 0, 0)), 1e-10, mg.make_options(fixed_vcycles=1))
        ghosts, c0, c1 = 6 * (m - 4) ** 2, n ** 3, (m - 4) ** 3
        # work fabs r0, e0 (one ghost), r1; the hierarchy's levels below the finest
        fabs = 8 * (c0 + (n + 2) * (n + 2) ** 2 + c1) + 8 * 2 * c0 / 7 * 1.2
        # one-colour arrays of the finest coarse level
        fabs += 8 * c0
        assert mg.mg_pool_info(ctx)[1] - used <= fabs + 104 * ghosts + 88 * ghosts / 4 + 0.5e6
    finally:
        mg.mg_finalize(ctx)


@pytest.mark.parametrize("box", [(4, 4, 4), (4, 4, 24)])
@pytest.mark.parametrize("dt", [mg.MG_F64, mg.MG_F32])
def test_whole_sweep_keeps_one_table(box, dt):
    """mg_smooth with color 2 keeps one box table (272 bytes a box) besides the fill's tags, on a lattice
    of boxes and off it."""
    ctx = mg.mg_init(0)
    try:
        n = (32, 32, 40)
        ba = mg.mg_box_array_create(ctx, (0, 0, 0), tuple(v - 1 for v in n), box)
        nb = len(mg.mg_box_array_info(ctx, ba)[1])
        f, r = mg.mg_fab_alloc(ctx, ba, 1, 1, dt), mg.mg_fab_alloc(ctx, ba, 1, 0, dt)
        bc = mg.make_bc((0, 0, 0))
        mg.mg_fill_boundary(ctx, f, bc)
        used = mg.mg_pool_info(ctx)[1]
        mg.mg_smooth(ctx, f, r, bc, 0.1, 2)
        assert 0 < mg.mg_pool_info(ctx)[1] - used <= 272 * nb + 256
    finally:
        mg.mg_finalize(ctx)
