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
# and images of one ray through 50 cells to ten through one
@pytest.mark.parametrize("size", [9, 40, 360])
@pytest.mark.parametrize("store,paired", [("f32", False), ("f32", True), ("bf16", False), ("bf16", True)])
def test_region_kernels_agree(ctx, n, region, store, paired, size):
    grid, j, beta = even_grid(sum(n), n, 3)
    vol = ctx.load_snapshots(grid, j, beta, store=store, paired=paired)
    # off the box centre: no ray lies in a face plane, where its cell would be a matter of rounding
    views = [gen.view_from_direction(grid, -d, size=size, c=20.0, t_obs=3.0) for d in gen.fibonacci_directions(9)]
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
                    px = np.random.default_rng(size).integers(0, size, size=(60, 2))
                    for k in (0, 4, 8):
                        ref = oracle.render_pixels(grid, jr, br, views[k], px)
                        assert_parity(want[k].cpu().numpy()[px[:, 1], px[:, 0]], ref, rel=rel,
                                      what=f"{n} region {region} view {k}")
                assert torch.equal(img, want), (depth, regcap, warps)
    ctx.unload(vol)


@pytest.mark.parametrize("store", ["f32", "bf16"])
@pytest.mark.parametrize("size", [(64, 64), (23, 41), (700, 400)])
def test_views_side_by_side_equal_single_renders(ctx, store, size):
    """Views along different rays and along the same ones, in runs of every kind: a batch's
    images and a vector render's are the single renders' bit for bit."""
    w, h = size
    grid, j, beta = even_grid(9, (21, 15, 18), 4)
    vol = ctx.load_snapshots(grid, j, beta, store=store)
    ctx.load_channels(vol, np.stack([2.0 * j, j, -j]))
    fov = 1.8 * float(np.max(grid.extent))
    views = [gen.view_from_direction(grid, -d, size=w, fov=fov, height=h, c=1.3).with_(fov_v=fov, t_obs=3.0)
             for d in gen.fibonacci_directions(9)]
    series = [views[2].with_(t_obs=3.0 + 1.1 * k) for k in range(3)]
    batch = views[:5] + series + views[5:] + [series[0], views[0].with_(t_obs=9.5), views[0]]
    singles = [ctx.render(vol, v) for v in batch]
    got = ctx.render_batch(vol, batch, launch={"group": 1})
    vec = ctx.render_vector(vol, batch)
    one = torch.stack([ctx.render_vector(vol, [v])[0] for v in batch])
    torch.cuda.synchronize()
    assert torch.equal(got, torch.stack(singles)) and torch.equal(vec, one)
    assert float(got.max()) > 0
    ctx.unload(vol)


# 8000 warps of 8x4 pixels, one snapshot or three, dense rays or not, lone series
@pytest.mark.parametrize("w,h,views", [(512, 499, 1), (512, 500, 1), (512, 516, 1), (300, 290, 3)])
@pytest.mark.parametrize("m,paired", [(1, False), (3, False), (3, True)])
def test_stage_depths_agree(ctx, w, h, views, m, paired):
    grid, j, beta = even_grid(10 + m, (26, 33, 19), m)
    vol = ctx.load_snapshots(grid, j, beta, paired=paired)
    fov = 1.8 * float(np.max(grid.extent))
    base = gen.view_from_angles(grid, 37.0, 205.0, size=w, fov=fov, c=20.0).with_(height=h, fov_v=fov, t_obs=2.0)
    series = [base.with_(t_obs=2.0 + 0.3 * k) for k in range(views)]
    want = ctx.render_batch(vol, series, launch={"depth": 1, "group": 1})
    want = want.clone()
    assert float(want.max()) > 0
    for depth in (2, 4):
        for regcap in (0, 1):
            got = ctx.render_batch(vol, series, launch={"depth": depth, "group": 1, "regcap": regcap})
            assert torch.equal(got, want), (depth, regcap)
    px = np.random.default_rng(1).integers(0, (w, h), size=(40, 2))
    assert_parity(want[0].cpu().numpy()[px[:, 1], px[:, 0]], oracle.render_pixels(grid, j, beta, series[0], px),
                  what=f"{w}x{h} M {m}")
    ctx.unload(vol)
