"""FP64 residual + restriction (csrc/mg_march.cu and the row kernel for small boxes and wide ones) against
the CPU oracle, bit for bit, with the values that the integer sums take, refuse and round at ties; the half-sweep
and the residual over boxes on both sides of the rule that chooses between the kernels; and the form that reads
stored residuals through solves.  Widths from one pair of cells to the widest taken and beyond, rows that end
inside warps and blocks, partial last blocks, boxes of 2^3 cells."""
import numpy as np
import pytest
import torch

from paper_2403_12179_gb300 import inputs, mg
from tests import gpu_util as gu
from tests.test_gpu_march import KINDS, _same, _values

pytestmark = pytest.mark.gpu
Z3 = (0, 0, 0)


@pytest.fixture(scope="module")
def gctx():
    ctx = mg.mg_init(0)
    yield ctx
    mg.mg_finalize(ctx)


WIDE = [((256, 16, 10), (256, 16, 10)), ((66, 30, 18), (66, 30, 18)), ((34, 34, 32), (34, 34, 32)),
        ((258, 16, 10), (258, 16, 10)), ((2, 128, 66), (2, 64, 66)), ((96, 24, 16), (32, 8, 4)),
        ((62, 6, 4), (62, 6, 4)), ((130, 22, 6), (130, 22, 6))]
SMALL = [((16, 16, 16), (2, 2, 2)), ((16, 16, 16), (4, 4, 4)), ((32, 16, 16), (8, 4, 4)), ((32, 32, 32), (8, 8, 8)),
         ((64, 8, 32), (32, 2, 32)), ((32, 32, 16), (8, 16, 8)), ((48, 40, 16), (16, 8, 4)), ((20, 24, 28), (12, 4, 16))]


def _case(gctx, orc, n, mb, kind, seed):
    dom = tuple(v - 1 for v in n)
    ba = mg.mg_box_array_create(gctx, Z3, dom, mb)
    boxes = mg.mg_box_array_info(gctx, ba)[1]
    g = inputs.rng(seed)
    phi = [_values(kind, f.shape, g) for f in orc.new_field(boxes, 1)]
    rhs = [_values("random" if kind == "inf" else kind, f.shape, g) for f in orc.new_field(boxes, 0)]
    return dom, ba, boxes, phi, rhs, 0.125 if kind == "ties" else 1.0 / 48


@pytest.mark.parametrize("n,mb", WIDE + SMALL)
@pytest.mark.parametrize("kind", KINDS)
def test_residual_restrict_bitwise(gctx, orc, n, mb, kind):
    dom, ba, boxes, phi, rhs, h = _case(gctx, orc, n, mb, kind, 53)
    cdom = tuple(v // 2 - 1 for v in n)
    cba = mg.mg_box_array_create(gctx, Z3, cdom, tuple(v // 2 for v in mb))
    cboxes = mg.mg_box_array_info(gctx, cba)[1]
    r, _ = orc.residual(Z3, dom, boxes, h, phi, 1, rhs, 0)
    ref = orc.restrict((Z3, dom, boxes), r, 0, (Z3, cdom, cboxes), 0)
    fp, fr = gu.to_fab(gctx, ba, phi, 1), gu.to_fab(gctx, ba, rhs, 0)
    crhs, cphi = mg.mg_fab_alloc(gctx, cba, 1, 0), mg.mg_fab_alloc(gctx, cba, 1, 1)
    for zero in (cphi, 0):
        mg.mg_fab_set_val(gctx, cphi, 7.0)
        mg.mg_residual_restrict(gctx, fp, fr, crhs, zero, h)
        for a, c in zip(gu.from_fab(gctx, crhs, len(cboxes)), ref):
            assert _same(a, c)
        for a in gu.from_fab(gctx, cphi, len(cboxes)):
            assert (gu.valid(a, 1) == (0.0 if zero else 7.0)).all()
    for f in (fp, fr, crhs, cphi):
        mg.mg_fab_free(gctx, f)


@pytest.mark.parametrize("n,mb", SMALL)
@pytest.mark.parametrize("kind", ["random", "ties", "inf"])
def test_small_boxes_bitwise(gctx, orc, n, mb, kind):
    dom, ba, boxes, phi, rhs, h = _case(gctx, orc, n, mb, kind, 54)
    fr = gu.to_fab(gctx, ba, rhs, 0)
    for color in (0, 1):
        ref = orc.rbgs(Z3, dom, boxes, h, phi, 1, rhs, 0, color)
        fp = gu.to_fab(gctx, ba, phi, 1)
        mg.mg_smooth(gctx, fp, fr, mg.make_bc((0, 0, 0)), h, color)
        for a, r in zip(gu.from_fab(gctx, fp, len(boxes)), ref):
            assert _same(gu.valid(a, 1), gu.valid(r, 1))
        mg.mg_fab_free(gctx, fp)
    fp, fo = gu.to_fab(gctx, ba, phi, 1), mg.mg_fab_alloc(gctx, ba, 1, 0)
    r_ref, n_ref = orc.residual(Z3, dom, boxes, h, phi, 1, rhs, 0)
    nrm = mg.mg_residual(gctx, fp, fr, fo, h)
    for a, r in zip(gu.from_fab(gctx, fo, len(boxes)), r_ref):
        assert _same(a, r)
    assert nrm == n_ref or not np.isfinite(n_ref) and not np.isfinite(nrm)
    for f in (fp, fr, fo):
        mg.mg_fab_free(gctx, f)


@pytest.mark.parametrize("n,mb", [((256, 16, 16), (256, 16, 16)), ((136, 24, 32), (136, 24, 32)),
                                  ((128, 32, 32), (32, 16, 32)), ((288, 16, 16), (288, 16, 16)),
                                  ((32, 32, 32), (4, 4, 4)), ((64, 32, 32), (8, 8, 8)), ((64, 64, 64), (16, 16, 16))])
@pytest.mark.parametrize("per", [(0, 0, 0), (1, 0, 1)])
def test_stored_residuals_equal_computed_ones(gctx, n, mb, per):
    """With direct reads the black residuals come from the last half-sweep before the restriction; without,
    all of them are computed from filled ghosts."""
    g = torch.Generator(device="cuda")
    g.manual_seed(6)
    f = torch.randn(n[2], n[1], n[0], generator=g, device="cuda", dtype=torch.float64)
    ba = mg.mg_box_array_create(gctx, Z3, tuple(v - 1 for v in n), mb)
    out = []
    for direct in (1, 0):
        r, u = gu.dense_fab(gctx, ba, f.cpu().numpy(), 0), mg.mg_fab_alloc(gctx, ba, 1, 1)
        res = mg.mg_solve(gctx, r, u, mg.make_bc(per), 1e-10, mg.make_options(fixed_vcycles=2, direct_reads=direct))
        out.append((gu.fab_dense(gctx, u, n[::-1]).tobytes(), res.rel_resid))
        mg.mg_fab_free(gctx, r)
        mg.mg_fab_free(gctx, u)
    assert out[0] == out[1]
