"""The marching FP64 half-sweep and residual (csrc/mg_march.cu) against the CPU oracle, bit for bit:
box widths from one pair of cells to the widest the kernels take and one beyond it, odd rows and
planes, odd widths (residual), row ends inside warps; values that the integer sums take, refuse
and round at ties: smooth, random, exponents far apart, exact zeros, short mantissas, tiny and
huge, infinite."""
import numpy as np
import pytest

from paper_2403_12179_gb300 import inputs, mg
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu
Z3 = (0, 0, 0)


@pytest.fixture(scope="module")
def gctx():
    ctx = mg.mg_init(0)
    yield ctx
    mg.mg_finalize(ctx)


@pytest.fixture(scope="module")
def orc():
    import oracle
    oracle.build()
    return oracle


def _values(kind, shape, g):
    a = g.standard_normal(shape)
    if kind == "smooth":
        x = np.arange(a.size, dtype=np.float64).reshape(shape)
        return 3.0 + np.sin(x * 1e-3) + 1e-9 * a
    if kind == "spread":
        return a * 2.0 ** g.integers(-45, 45, shape)
    if kind == "zeros":
        return np.where(g.random(shape) < 0.3, np.copysign(0.0, a), a)
    if kind == "ties":
        return g.integers(-64, 65, shape) * 2.0 ** g.integers(-30, 30, shape) + g.integers(-4, 5, shape)
    if kind == "tiny":
        return a * 1e-306
    if kind == "huge":
        return a * 1e306
    if kind == "inf":
        return np.where(g.random(shape) < 0.001, np.inf, a)
    return a


def _same(a, b):
    # (the sign of a NaN is not defined)
    n = np.isnan(a) & np.isnan(b)
    return np.array_equal(np.where(n, 0, np.ascontiguousarray(a).view(np.int64)),
                          np.where(n, 0, np.ascontiguousarray(b).view(np.int64)))


SHAPES = [((256, 16, 9), (256, 16, 9)), ((2, 130, 130), (2, 65, 130)), ((66, 30, 17), (66, 30, 17)),
          ((34, 33, 31), (34, 11, 31)), ((96, 24, 16), (32, 7, 5)), ((62, 3, 5), (62, 3, 5)),
          ((258, 16, 9), (258, 16, 9))]
KINDS = ["smooth", "random", "spread", "zeros", "ties", "tiny", "huge", "inf"]


def _case(gctx, orc, n, mb, kind, seed):
    dom = tuple(v - 1 for v in n)
    ba = mg.mg_box_array_create(gctx, Z3, dom, mb)
    boxes = mg.mg_box_array_info(gctx, ba)[1]
    g = inputs.rng(seed)
    phi = [_values(kind, f.shape, g) for f in orc.new_field(boxes, 1)]
    rhs = [_values("random" if kind == "inf" else kind, f.shape, g) for f in orc.new_field(boxes, 0)]
    return dom, ba, boxes, phi, rhs


@pytest.mark.parametrize("n,mb", SHAPES)
@pytest.mark.parametrize("kind", KINDS)
def test_half_sweep_bitwise(gctx, orc, n, mb, kind):
    h = 0.125 if kind == "ties" else 1.0 / 48
    dom, ba, boxes, phi, rhs = _case(gctx, orc, n, mb, kind, 51)
    for color in (0, 1):
        ref = orc.rbgs(Z3, dom, boxes, h, phi, 1, rhs, 0, color)
        fp, fr = gu.to_fab(gctx, ba, phi, 1), gu.to_fab(gctx, ba, rhs, 0)
        mg.mg_smooth(gctx, fp, fr, mg.make_bc((0, 0, 0)), h, color)
        for a, r in zip(gu.from_fab(gctx, fp, len(boxes)), ref):
            assert _same(gu.valid(a, 1), gu.valid(r, 1))
        mg.mg_fab_free(gctx, fp)
        mg.mg_fab_free(gctx, fr)


ODD = [((255, 16, 9), (255, 16, 9)), ((63, 33, 17), (63, 33, 17)), ((1, 180, 190), (1, 95, 190)),
       ((3, 110, 101), (3, 110, 101)), ((97, 31, 13), (33, 31, 6)), ((257, 16, 9), (257, 16, 9))]


@pytest.mark.parametrize("n,mb", SHAPES + ODD)
@pytest.mark.parametrize("kind", KINDS)
def test_residual_bitwise(gctx, orc, n, mb, kind):
    h = 0.125 if kind == "ties" else 1.0 / 48
    dom, ba, boxes, phi, rhs = _case(gctx, orc, n, mb, kind, 52)
    r_ref, n_ref = orc.residual(Z3, dom, boxes, h, phi, 1, rhs, 0)
    fp, fr = gu.to_fab(gctx, ba, phi, 1), gu.to_fab(gctx, ba, rhs, 0)
    fo = mg.mg_fab_alloc(gctx, ba, 1, 0)
    nrm = mg.mg_residual(gctx, fp, fr, fo, h)
    for a, r in zip(gu.from_fab(gctx, fo, len(boxes)), r_ref):
        assert _same(a, r)
    assert nrm == n_ref or not np.isfinite(n_ref) and not np.isfinite(nrm)
    for f in (fp, fr, fo):
        mg.mg_fab_free(gctx, f)
