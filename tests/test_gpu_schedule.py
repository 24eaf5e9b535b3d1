"""Where launches split their work: time groups at the spans that decide how
many snapshots they share and where a run is cut, and images at the edges of the
blocks of packets that CTAs take."""
import numpy as np
import pytest

import gen
import oracle
from tests._parity import assert_parity, beta_from_u, bf16_round, four_velocity_f16

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2609_09322_gb300 as g
    c = g.Context(0)
    yield c
    c.close()


def even_grid(seed, n, m):
    """Emissivities within a factor of 3 and |beta| <= 0.5, so within a factor
    of 9 in the squared boost: neighbouring snapshots differ by less than a factor of
    27, and an epoch coordinate that is off by 2 float ulps at 16 snapshots (2e-6)
    moves no sample by 1e-4 of its value."""
    rng = np.random.default_rng(seed)
    grid = gen.Grid(n=n, n_epochs=m, t0=0.0, dt=2.0)
    shape = (m, n[2], n[1], n[0])
    j = (0.5 + rng.random(shape)).astype(np.float32)
    d = rng.normal(size=(*shape, 3))
    d /= np.linalg.norm(d, axis=-1, keepdims=True)
    return grid, j, (d * rng.uniform(0.0, 0.5, size=(*shape, 1))).astype(np.float32)


# Observer times of a run in snapshots, from the later of its members' first
# ones.  A group spans at most `lim` = min(3, (M + 1) / 2) snapshots, and reads
# three per cell up to a span of 1, five beyond it.
EPS = 2.0 ** -20


def runs(lim):
    yield [0.0, 0.5, 1.0]                       # exactly 1
    yield [0.0, 1.0 + EPS]                      # just over it
    yield [lim, 0.0, 0.5 * lim, 0.5 * lim]      # the limit, out of order, a repeated time
    yield [0.0, lim + EPS]                      # just over it: two lone marches
    yield [lim + EPS, 0.25, 0.0, lim, 0.5]      # cut into a group and the rest
    yield list(np.linspace(-1.5, 6.5, 9))       # more than one group takes


@pytest.mark.parametrize("m", [1, 2, 6])
@pytest.mark.parametrize("store", ["f32", "bf16"])
@pytest.mark.parametrize("group,paired", [(4, True), (8, False)])
def test_time_groups_at_their_spans(ctx, m, store, group, paired):
    grid, j, beta = even_grid(100 * m + group, (11, 9, 13), m)
    vol = ctx.load_snapshots(grid, j, beta, store=store, paired=paired)
    j_r, b_r, rel = j, beta, 1e-5
    if store == "bf16":
        j_r, b_r, rel = bf16_round(j).astype(np.float64), beta_from_u(four_velocity_f16(beta)), 1e-4
    base = gen.view_from_angles(grid, 37.0, 205.0, size=19, fov=1.8 * float(np.max(grid.extent)), c=1.3)
    for offs in runs(min(3.0, 0.5 * (m + 1))):
        views = [base.with_(t_obs=grid.dt * (0.5 + o)) for o in offs]
        img, cnt = ctx.render_batch(vol, views, samples=True, launch={"group": group})
        torch.cuda.synchronize()
        for k, v in enumerate(views):
            ref, rcnt = oracle.render(grid, j_r, b_r, v, counts=True)
            assert_parity(img[k].cpu().numpy(), ref, rel=rel, what=f"M {m} times {offs} view {k}")
            if store == "f32":
                assert np.abs(cnt[k].cpu().numpy().astype(np.int64) - rcnt).max() <= 1
    ctx.unload(vol)


# one pixel, one row, one column, one more and one less than whole blocks
@pytest.mark.parametrize("size", [(1, 1), (129, 1), (1, 65), (31, 33), (64, 32), (65, 63)])
@pytest.mark.parametrize("store", ["f32", "bf16"])
def test_blocks_cover_images_once(ctx, size, store):
    """Whatever block a ray falls into, its pixel is the same bit for bit, in a
    single render and in a batch, and nothing outside the images is written."""
    w, h = size
    grid, j, beta = even_grid(7, (11, 9, 13), 3)
    vol = ctx.load_snapshots(grid, j, beta, store=store)
    fov = 1.8 * float(np.max(grid.extent))
    views = [gen.view_from_angles(grid, th, ph, size=w, fov=fov, c=1.3).with_(height=h, fov_v=fov, t_obs=3.0)
             for th, ph in ((37.0, 205.0), (90.0, 0.0), (121.0, 40.0))]
    want = torch.stack([ctx.render(vol, v) for v in views])
    assert float(want.max()) > 0
    guard = 4096
    for packet in ((8, 4), (4, 8), (32, 1), (1, 32)):
        for warps in (1, 2, 4, 8):
            buf = torch.full((3 * w * h + guard,), -1.0, device="cuda")
            out = buf[:3 * w * h].view(3, h, w)
            ctx.render_batch(vol, views, out=out, launch={"packet": packet, "cta_warps": warps, "regcap": 1})
            assert torch.equal(out, want), (packet, warps)
            assert bool((buf[3 * w * h:] == -1.0).all()), (packet, warps)
            assert torch.equal(ctx.render(vol, views[1], launch={"packet": packet, "cta_warps": warps, "regcap": 1}), want[1])
    ctx.unload(vol)
