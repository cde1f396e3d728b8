"""A whole sweep (color 2) whose ghost fill cannot be built -- phi has more ghost layers than a Dirichlet
dimension has cells -- is refused with MG_EINVAL and changes neither fab, whatever route the layout
takes; the same fabs with that dimension periodic are taken."""
import numpy as np
import pytest
import torch

from paper_2403_12179_gb300 import mg
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("box", [(8, 8, 2), (4, 8, 2), (8, 5, 2)])
@pytest.mark.parametrize("dt", [mg.MG_F64, mg.MG_F32])
@pytest.mark.parametrize("gr", [0, 1, 2])
def test_refused_sweep_changes_nothing(box, dt, gr):
    ctx = mg.mg_init(0)
    try:
        ba = mg.mg_box_array_create(ctx, (0, 0, 0), (7, 7, 1), box)
        nb = len(mg.mg_box_array_info(ctx, ba)[1])
        g = np.random.default_rng(2)
        fp, fr = mg.mg_fab_alloc(ctx, ba, 1, 3, dt), mg.mg_fab_alloc(ctx, ba, 1, gr, dt)
        for f in (fp, fr):
            for b in range(nb):
                v = torch.as_tensor(mg.BoxView(ctx, f, b), device="cuda")
                v.copy_(torch.from_numpy(g.standard_normal(tuple(v.shape))).to(v.dtype))
        before = [a.tobytes() for f in (fp, fr) for a in gu.from_fab(ctx, f, nb)]
        with pytest.raises(mg.MgError) as e:
            mg.mg_smooth(ctx, fp, fr, mg.make_bc((1, 1, 0)), 0.125, 2)
        assert e.value.code == mg.MG_EINVAL
        assert before == [a.tobytes() for f in (fp, fr) for a in gu.from_fab(ctx, f, nb)]
        mg.mg_smooth(ctx, fp, fr, mg.make_bc((1, 1, 1)), 0.125, 2)
        torch.cuda.synchronize()
    finally:
        mg.mg_finalize(ctx)
