"""The exact bottom solve with phi in rhs's own memory (one fab for both, or two fabs over the same
memory): the same bits as into another fab.  Several hundred rows, whose blocks would otherwise read
rhs while others write phi; one box and several, ghosts, both types."""
import numpy as np
import pytest
import torch

from paper_2403_12179_gb300 import mg
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,mb", [((3, 11, 1), (3, 11, 1)), ((7, 6, 5), (4, 6, 5)), ((10, 10, 10), (4, 4, 4)),
                                  ((16, 8, 8), (16, 8, 8))])
@pytest.mark.parametrize("dt", [mg.MG_F64, mg.MG_F32])
@pytest.mark.parametrize("wrapped", [False, True])
def test_in_place_equals_out_of_place(n, mb, dt, wrapped):
    ctx = mg.mg_init(0)
    try:
        ba = mg.mg_box_array_create(ctx, (0, 0, 0), tuple(v - 1 for v in n), mb)
        nb = len(mg.mg_box_array_info(ctx, ba)[1])
        g, tdt = np.random.default_rng(9), np.float64 if dt == mg.MG_F64 else np.float32
        mem = torch.zeros(mg.mg_fab_layout(ctx, ba, 1, 1, dt) + 256, dtype=torch.uint8, device="cuda")
        at = (mem.data_ptr() + 255) // 256 * 256
        size = mg.mg_fab_layout(ctx, ba, 1, 1, dt)
        rhs = mg.mg_fab_wrap(ctx, ba, 1, 1, dt, at, size)
        phi = mg.mg_fab_wrap(ctx, ba, 1, 1, dt, at, size) if wrapped else rhs
        other = mg.mg_fab_alloc(ctx, ba, 1, 1, dt)
        bc = mg.make_bc((0, 1, 0))
        for _ in range(10):
            for b in range(nb):
                v = torch.as_tensor(mg.BoxView(ctx, rhs, b), device="cuda")
                v.copy_(torch.from_numpy(g.standard_normal(tuple(v.shape)).astype(tdt)))
            torch.cuda.synchronize()
            mg.mg_bottom_solve(ctx, rhs, other, bc, 0.25)
            torch.cuda.synchronize()
            mg.mg_bottom_solve(ctx, rhs, phi, bc, 0.25)
            for a, r in zip(gu.from_fab(ctx, phi, nb), gu.from_fab(ctx, other, nb)):
                assert np.ascontiguousarray(gu.valid(a, 1)).tobytes() == np.ascontiguousarray(gu.valid(r, 1)).tobytes()
    finally:
        mg.mg_finalize(ctx)
