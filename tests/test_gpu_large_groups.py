"""Time groups of five to eight views: their kernels (three or five snapshots per cell, both
stores, every depth) against the oracle, with sample counts.  Their members lie within one
snapshot of each other, or within three, so that no rule cuts them smaller; where the
rule cuts is held elsewhere (test_time_group_rule.py, on the CPU)."""
import numpy as np
import pytest

import gen
import oracle
from tests._parity import assert_parity, beta_from_u, bf16_round, four_velocity_f16
from tests.test_gpu_schedule import even_grid

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2609_09322_gb300 as g
    c = g.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("views,span", [(5, 0.9), (8, 0.9), (8, 1.0), (6, 1.1), (7, 2.9), (8, 3.0)])
@pytest.mark.parametrize("store,paired", [("f32", False), ("f32", True), ("bf16", False), ("bf16", True)])
def test_groups_of_five_to_eight(ctx, views, span, store, paired):
    grid, j, beta = even_grid(views, (11, 9, 13), 6)
    vol = ctx.load_snapshots(grid, j, beta, store=store, paired=paired)
    jr, br, rel = j, beta, 1e-5
    if store == "bf16":
        jr, br, rel = bf16_round(j).astype(np.float64), beta_from_u(four_velocity_f16(beta)), 1e-4
    base = gen.view_from_angles(grid, 37.0, 205.0, size=19, fov=1.8 * float(np.max(grid.extent)), c=1.3)
    # times in snapshots from the later of the members' first ones; out of order
    offs = np.linspace(0.0, span, views)
    offs = np.concatenate([offs[1::2], offs[::2]])
    for first in (-0.6, 2.25):
        series = [base.with_(t_obs=grid.dt * (0.5 + first + float(o))) for o in offs]
        refs = [oracle.render(grid, jr, br, v, counts=True) for v in series]
        for depth in (1, 2, 4):
            img, cnt = ctx.render_batch(vol, series, samples=True, launch={"group": 8, "depth": depth})
            torch.cuda.synchronize()
            for k, (ref, rcnt) in enumerate(refs):
                assert_parity(img[k].cpu().numpy(), ref, rel=rel, what=f"{views} views over {span} depth {depth} view {k}")
                if store == "f32":
                    assert np.abs(cnt[k].cpu().numpy().astype(np.int64) - rcnt).max() <= 1
    ctx.unload(vol)
