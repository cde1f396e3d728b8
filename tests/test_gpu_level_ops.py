"""Restriction, prolongation and the max-norm at every lane-group width: rows of a few cells, of whole
and ragged groups, aligned for pair loads and not (ghost widths), one box and many; and the norm of
solves of different sizes in one launch."""
import numpy as np
import pytest

from paper_2403_12179_gb300 import inputs, mg
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu
Z3 = (0, 0, 0)
SHAPES = [((4, 4, 4), (4, 4, 4)), ((24, 8, 4), (6, 4, 4)), ((44, 12, 8), (22, 6, 8)), ((64, 16, 8), (64, 8, 4)),
          ((132, 4, 8), (132, 4, 4)), ((288, 8, 8), (144, 8, 8))]

SOLVES = [((24, 8, 8), (12, 8, 8)), ((64, 16, 8), (64, 8, 8)), ((144, 16, 16), (144, 16, 16)),
          ((48, 16, 16), (16, 16, 16)), ((8, 8, 8), (8, 8, 8)), ((40, 8, 8), (8, 8, 8)), ((96, 16, 16), (32, 16, 8))]


@pytest.fixture(scope="module")
def gctx():
    ctx = mg.mg_init(0)
    yield ctx
    mg.mg_finalize(ctx)


def _boxes(ctx, n, mb):
    ba = mg.mg_box_array_create(ctx, Z3, tuple(v - 1 for v in n), mb)
    return ba, mg.mg_box_array_info(ctx, ba)[1]


@pytest.mark.parametrize("n,mb", SHAPES)
@pytest.mark.parametrize("g", [0, 1, 2, 3])
def test_restrict_and_prolong(gctx, orc, n, mb, g):
    ba, boxes = _boxes(gctx, n, mb)
    lev = orc.hierarchy(Z3, tuple(v - 1 for v in n), boxes)
    cba = mg.mg_hierarchy_level(gctx, ba, 1)
    cboxes = mg.mg_box_array_info(gctx, cba)[1]
    r = inputs.rng(7)
    fine = [r.standard_normal(f.shape) for f in orc.new_field(boxes, g)]
    coarse = [r.standard_normal(f.shape) for f in orc.new_field(cboxes, 1)]
    ff, fc = gu.to_fab(gctx, ba, fine, g), gu.to_fab(gctx, cba, coarse, 1)
    mg.mg_restrict(gctx, ff, fc)
    for a, c in zip(gu.from_fab(gctx, fc, len(cboxes)), orc.restrict(lev[0], fine, g, lev[1], 1)):
        assert np.array_equal(gu.valid(a, 1), gu.valid(c, 1))
    mg.mg_prolong_add(gctx, gu.to_fab(gctx, cba, coarse, 1), ff)
    ref = orc.prolong_add(lev[1], coarse, 1, lev[0], fine, g)
    for a, p in zip(gu.from_fab(gctx, ff, len(boxes)), ref):
        assert np.array_equal(gu.valid(a, g), gu.valid(p, g))


@pytest.mark.parametrize("g", [0, 1])
def test_norms_of_a_batch(gctx, orc, g):
    """phi = 0: the residual is the right-hand side, so the ratio of the two norms is 1 exactly; in one
    problem the largest value is the last cell, in another the first, in a third it is the only one."""
    rhs, phi, per = [], [], []
    for k, (n, mb) in enumerate(SOLVES):
        ba, boxes = _boxes(gctx, n, mb)
        r = inputs.rng(11 + k)
        f = [r.standard_normal(v.shape) for v in orc.new_field(boxes, g)]
        if k % 3 == 0:
            gu.valid(f[-1], g)[0, -1, -1, -1] = -9.0 - k
        elif k % 3 == 1:
            gu.valid(f[0], g)[0, 0, 0, 0] = 1e3 * (k + 1)
        else:
            for a in f:
                a[...] = 0.0
            gu.valid(f[0], g)[0, 1, 1, 1] = 1e-300
        rhs.append(gu.to_fab(gctx, ba, f, g))
        phi.append(mg.mg_fab_alloc(gctx, ba, 1, 1))
        mg.mg_fab_set_val(gctx, phi[-1], 0.0)
    opt = mg.make_options(fixed_vcycles=0)
    bc = mg.make_bc((0, 0, 0))
    for a, b in zip(rhs, phi):
        assert mg.mg_solve(gctx, a, b, bc, 1e-10, opt).rel_resid == 1.0
    for res in mg.mg_solve_batch(gctx, rhs, phi, [bc] * len(rhs), 1e-10, opt):
        assert res.rel_resid == 1.0
