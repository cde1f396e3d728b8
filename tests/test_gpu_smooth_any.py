"""mg_smooth's whole sweep (color 2) on every layout it takes, against fill, red, fill, black on fabs
without the ghost layers of the fused route: valid cells bit for bit, and the ghost cells of rhs
(filled where the fused route's layout is met).  Boxes on a lattice and not, widths of whole strips
and not, both types, even and odd ghost widths."""
import numpy as np
import pytest
import torch

from paper_2403_12179_gb300 import mg

pytestmark = pytest.mark.gpu

SHAPES = [((32, 32, 32), (16, 16, 16)), ((40, 30, 22), (16, 30, 8)), ((64, 24, 20), (64, 24, 20)),
          ((48, 40, 32), (32, 16, 32)), ((22, 12, 14), (11, 12, 7)), ((144, 18, 10), (48, 6, 5))]


def _sweeps(ctx, n, box, per, dt, gp, gr, halves):
    tdt = torch.float64 if dt == mg.MG_F64 else torch.float32
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    a, b = (torch.randn(n[2], n[1], n[0], generator=g, device="cuda", dtype=torch.float64).to(tdt) for _ in range(2))
    ba = mg.mg_box_array_create(ctx, (0, 0, 0), tuple(v - 1 for v in n), box)
    fp, fr = mg.mg_fab_alloc(ctx, ba, 1, gp, dt), mg.mg_fab_alloc(ctx, ba, 1, gr, dt)
    bc, h = mg.make_bc(per), 1.0 / n[0]
    torch.cuda.synchronize()
    mg.mg_fab_copy_from_dense(ctx, fp, a.data_ptr(), False)
    mg.mg_fab_copy_from_dense(ctx, fr, b.data_ptr(), False)
    for _ in range(2):
        if halves:
            for color in (0, 1):
                mg.mg_fill_boundary(ctx, fp, bc)
                mg.mg_smooth(ctx, fp, fr, bc, h, color)
        else:
            mg.mg_smooth(ctx, fp, fr, bc, h, 2)
    if halves:
        mg.mg_fill_boundary(ctx, fr, bc)
    out = torch.empty_like(a)
    mg.mg_fab_copy_to_dense(ctx, fp, out.data_ptr(), False)
    torch.cuda.synchronize()
    boxes = range(len(mg.mg_box_array_info(ctx, ba)[1]))
    rhs = [torch.as_tensor(mg.BoxView(ctx, fr, i), device="cuda").cpu().numpy() for i in boxes]
    return out.cpu().numpy(), rhs


@pytest.mark.parametrize("n,box", SHAPES)
@pytest.mark.parametrize("per", [(0, 0, 0), (1, 1, 1), (0, 1, 0)])
@pytest.mark.parametrize("dt", [mg.MG_F64, mg.MG_F32])
@pytest.mark.parametrize("gp,gr", [(1, 0), (2, 1), (3, 2), (4, 4)])
def test_whole_sweep_equals_half_sweeps(n, box, per, dt, gp, gr):
    ctx = mg.mg_init(0)
    try:
        got, rhs = _sweeps(ctx, n, box, per, dt, gp, gr, False)
        ref, rref = _sweeps(ctx, n, box, per, dt, gp, gr, True)
        assert np.isfinite(got).all()
        assert got.tobytes() == ref.tobytes()
        if gp >= 2 and gr >= 1:
            for a, b in zip(rhs, rref):
                assert a.tobytes() == b.tobytes()
    finally:
        mg.mg_finalize(ctx)
