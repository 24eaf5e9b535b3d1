"""Which kernel a launch gets decides nothing about its images: every stage depth
and register cap gives the same pixels bit for bit, and they match the oracle."""
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


def stored(j, beta, store):
    if store == "f32":
        return j, beta, 1e-5
    return bf16_round(j).astype(np.float64), beta_from_u(four_velocity_f16(beta)), 1e-4


# regions of 32 cells (one short of two, one more) and of 64 (the same)
@pytest.mark.parametrize("n,region", [((63, 17, 33), 32), ((65, 20, 18), 64), ((127, 9, 14), 64)])
@pytest.mark.parametrize("store,paired", [("f32", False), ("f32", True), ("bf16", False), ("bf16", True)])
def test_region_kernels_agree(ctx, n, region, store, paired):
    grid, j, beta = even_grid(sum(n), n, 3)
    vol = ctx.load_snapshots(grid, j, beta, store=store, paired=paired)
    # off the box centre: no ray lies in a face plane, where its cell would be a matter of rounding
    views = [gen.view_from_direction(grid, -d, size=21, c=20.0, t_obs=3.0) for d in gen.fibonacci_directions(9)]
    views = [v.with_(center=tuple(np.array(v.center) + (0.13, 0.07, 0.29))) for v in views]
    jr, br, rel = stored(j, beta, store)
    want = None
    for depth in (1, 2):
        for regcap in (0, 1):
            for warps in (1, 4, 8):
                img = ctx.render_batch(vol, views, launch={"packet": (4, 8), "cta_warps": warps, "depth": depth,
                                                           "persistent": 0, "regcap": regcap, "region": region})
                torch.cuda.synchronize()
                if want is None:
                    want = img.clone()
                    for k in (0, 4, 8):
                        assert_parity(want[k].cpu().numpy(), oracle.render(grid, jr, br, views[k]), rel=rel,
                                      what=f"{n} region {region} view {k}")
                assert torch.equal(img, want), (depth, regcap, warps)
    ctx.unload(vol)
