"""FP64 solves over boxes that are not on a lattice: the same bits as over one box, for a solve on its
own and in a batch, from a guess, and again after the fabs have changed; phi's first ghost layer is
that of its own boxes."""
import numpy as np
import pytest
import torch

from paper_2403_12179_gb300 import mg
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu
CASES = [((24, 20, 28), (12, 12, 12)), ((96, 40, 24), (48, 24, 16)), ((256, 12, 8), (96, 8, 8)), ((288, 16, 24), (96, 16, 16))]


@pytest.mark.parametrize("n,mb", CASES)
@pytest.mark.parametrize("per", [(1, 1, 1), (0, 0, 0), (1, 0, 0)])
@pytest.mark.parametrize("kw", [{}, {"smoother": mg.MG_SMOOTH_HALF, "use_graph": 0}, {"prolong": mg.MG_PROLONG_TRILINEAR},
                                {"direct_reads": 0}])
def test_ragged_boxes_equal_one_box(n, mb, per, kw):
    ctx = mg.mg_init(0)
    try:
        g = np.random.default_rng(4)
        bc, opt = mg.make_bc(per), mg.make_options(fixed_vcycles=3, **kw)
        fabs = []
        for box in (mb, n):
            ba = mg.mg_box_array_create(ctx, (0, 0, 0), tuple(v - 1 for v in n), box)
            z = np.zeros(n[::-1])
            fabs.append((ba, gu.dense_fab(ctx, ba, z, 0), gu.dense_fab(ctx, ba, z, 2), gu.dense_fab(ctx, ba, z, 2)))
        for _ in range(2):
            f, p = g.standard_normal(n[::-1]), g.standard_normal(n[::-1])
            if all(per):
                f -= f.mean()
            out = []
            for ba, r, u, v in fabs:
                for a, b in ((r, f), (u, p), (v, p)):
                    t = torch.from_numpy(b).cuda()
                    mg.mg_fab_copy_from_dense(ctx, a, t.data_ptr(), False)
                    torch.cuda.synchronize()
                ru = mg.mg_solve(ctx, r, u, bc, 1e-10, opt)
                rv = mg.mg_solve_batch(ctx, [r], [v], [bc], 1e-10, opt)[0]
                out += [(gu.fab_dense(ctx, u, n[::-1]).tobytes(), ru.rel_resid), (gu.fab_dense(ctx, v, n[::-1]).tobytes(), rv.rel_resid)]
            assert all(o == out[0] for o in out)
        ba, _, u, _ = fabs[0]
        got = [torch.as_tensor(mg.BoxView(ctx, u, i), device="cuda").cpu().numpy()[0]
               for i in range(len(mg.mg_box_array_info(ctx, ba)[1]))]
        mg.mg_fill_boundary(ctx, u, bc)
        torch.cuda.synchronize()
        for i, a in enumerate(got):
            b = torch.as_tensor(mg.BoxView(ctx, u, i), device="cuda").cpu().numpy()[0]
            for s in ((slice(2, -2), slice(2, -2), slice(1, -1)), (slice(2, -2), slice(1, -1), slice(2, -2)),
                      (slice(1, -1), slice(2, -2), slice(2, -2))):
                assert np.array_equal(a[s], b[s])
    finally:
        mg.mg_finalize(ctx)
