"""The whole red + black sweep and the residual + restriction of FP32 levels on regular box grids
(csrc/mg_sweep.cu) against the half-sweeps and the row kernel they stand for: the mixed-precision iterates after two outer iterations are equal bit
for bit, alone (levels of at least 2^14 cells are swept whole) and in batches (levels of at least
2^18 cells together).  The shapes put tile edges everywhere: domains narrower and lower than a
tile, one strip more than a tile, row counts that are no multiple of a tile's, single boxes and
boxes of 4 cells, every kind of faces, a domain away from the origin."""
import numpy as np
import pytest
import torch

from paper_2403_12179_gb300 import mg

pytestmark = pytest.mark.gpu

SHAPES = [((32, 32, 32), (32, 32, 32), (1, 1, 1)), ((32, 32, 32), (4, 8, 16), (0, 0, 0)),
          ((16, 40, 48), (8, 8, 8), (0, 1, 0)), ((136, 24, 16), (136, 24, 16), (0, 1, 1)),
          ((64, 88, 24), (16, 8, 24), (1, 0, 0)), ((40, 56, 72), (8, 8, 8), (1, 0, 1)),
          ((96, 48, 16), (32, 16, 16), (0, 0, 1)), ((160, 32, 40), (32, 32, 8), (0, 0, 0))]


def _problem(ctx, n, box, per, seed, lo=(0, 0, 0)):
    ba = mg.mg_box_array_create(ctx, lo, tuple(lo[d] + n[d] - 1 for d in range(3)), box)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    r = torch.randn(n[2], n[1], n[0], generator=g, device="cuda", dtype=torch.float64)
    if all(per):
        r -= r.mean()
    rhs, phi = mg.mg_fab_alloc(ctx, ba, 1, 0), mg.mg_fab_alloc(ctx, ba, 1, 1)
    torch.cuda.synchronize()
    mg.mg_fab_copy_from_dense(ctx, rhs, r.data_ptr(), False)
    torch.cuda.synchronize()
    return rhs, phi, mg.make_bc(per)


def _dense(ctx, phi, n):
    out = torch.empty(n[2], n[1], n[0], dtype=torch.float64, device="cuda")
    mg.mg_fab_copy_to_dense(ctx, phi, out.data_ptr(), False)
    torch.cuda.synchronize()
    return out.cpu().numpy()


def _opt(smoother, nu1=2, nu2=2):
    return mg.make_options(precision=mg.MG_PREC_MIXED, smoother=smoother, fixed_vcycles=2,
                           nu1=nu1, nu2=nu2)


@pytest.mark.parametrize("n,box,per", SHAPES)
@pytest.mark.parametrize("nu", [(2, 2), (3, 1), (1, 2), (4, 0)])
def test_sweep_equals_half_sweeps(n, box, per, nu):
    ctx = mg.mg_init(0)
    try:
        got = []
        for sm in (mg.MG_SMOOTH_AUTO, mg.MG_SMOOTH_HALF):
            rhs, phi, bc = _problem(ctx, n, box, per, 7, lo=(64, 0, -128))
            mg.mg_solve(ctx, rhs, phi, bc, 1e-10, _opt(sm, *nu))
            got.append(_dense(ctx, phi, n))
        assert np.isfinite(got[0]).all() and np.abs(got[0]).max() > 0
        np.testing.assert_array_equal(got[0].view(np.int64), got[1].view(np.int64))
    finally:
        mg.mg_finalize(ctx)


@pytest.mark.parametrize("nu", [(2, 2), (1, 3)])
def test_batched_sweeps_equal_single_solves(nu):
    """Different shapes in one launch (one tiling, one block size for all), each as alone with
    half-sweeps."""
    ctx = mg.mg_init(0)
    try:
        P = [_problem(ctx, n, box, per, 11 + i) for i, (n, box, per) in enumerate(SHAPES)]
        mg.mg_solve_batch(ctx, [p[0] for p in P], [p[1] for p in P], [p[2] for p in P], 1e-10,
                          _opt(mg.MG_SMOOTH_AUTO, *nu))
        for i, (n, box, per) in enumerate(SHAPES):
            got = _dense(ctx, P[i][1], n)
            rhs, phi, bc = _problem(ctx, n, box, per, 11 + i)
            mg.mg_solve(ctx, rhs, phi, bc, 1e-10, _opt(mg.MG_SMOOTH_HALF, *nu))
            np.testing.assert_array_equal(got.view(np.int64), _dense(ctx, phi, n).view(np.int64))
    finally:
        mg.mg_finalize(ctx)


@pytest.mark.parametrize("n,ragged,even", [((48, 40, 56), (32, 24, 32), (8, 8, 8)), ((96, 48, 32), (40, 48, 24), (32, 16, 16))])
@pytest.mark.parametrize("per", [(0, 0, 0), (1, 1, 1), (0, 1, 0)])
@pytest.mark.parametrize("precision", [mg.MG_PREC_F64, mg.MG_PREC_MIXED])
def test_ragged_boxes_equal_even_ones(n, ragged, even, per, precision):
    """Boxes of several sizes (whose internal levels are laid out as one box) against boxes of one size,
    alone and in a batch: the same iterates bit for bit, with and without direct reads."""
    ctx = mg.mg_init(0)
    try:
        got = []
        for box, direct, batch in ((ragged, 1, False), (ragged, 1, True), (ragged, 0, False), (even, 1, False)):
            rhs, phi, bc = _problem(ctx, n, box, per, 23)
            opt = mg.make_options(precision=precision, fixed_vcycles=2, direct_reads=direct)
            if batch:
                mg.mg_solve_batch(ctx, [rhs], [phi], [bc], 1e-10, opt)
            else:
                mg.mg_solve(ctx, rhs, phi, bc, 1e-10, opt)
            got.append(_dense(ctx, phi, n))
        assert np.abs(got[0]).max() > 0
        for g in got[1:]:
            np.testing.assert_array_equal(got[0].view(np.int64), g.view(np.int64))
    finally:
        mg.mg_finalize(ctx)


@pytest.mark.parametrize("kw", [{"precision": mg.MG_PREC_MIXED}, {"precision": mg.MG_PREC_MIXED, "nu1": 1},
                                {"nu1": 0}, {"nu1": 0, "use_graph": 0}, {}])
def test_calls_after_a_timed_solve(kw):
    """A solve whose finest level has no half-sweep to time (whole sweeps, no pre-smoothing) leaves no
    error behind for the next call."""
    ctx = mg.mg_init(0)
    try:
        ba = mg.mg_box_array_create(ctx, (0, 0, 0), (63, 63, 63), (32, 32, 32))
        fr, fp = mg.mg_fab_alloc(ctx, ba, 1, 0), mg.mg_fab_alloc(ctx, ba, 1, 1)
        mg.mg_fab_set_val(ctx, fr, 1.0)
        mg.mg_fab_set_val(ctx, fp, 0.0)
        bc = mg.make_bc((0, 0, 0))
        mg.mg_sweep_timing(ctx, True)
        res = mg.mg_solve(ctx, fr, fp, bc, 1e-8, mg.make_options(fixed_vcycles=2, **kw))
        mg.mg_fill_boundary(ctx, fp, bc)
        _, count = mg.mg_sweep_timing(ctx, False)
        assert res.status == 0 and res.vcycles == 2
        assert count == (0 if kw.get("nu1") == 0 or kw == {"precision": mg.MG_PREC_MIXED} else 2)
    finally:
        mg.mg_finalize(ctx)
