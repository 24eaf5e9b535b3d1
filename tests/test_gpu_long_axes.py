"""Volumes with one long axis, whose march tables a CTA copies only where its rays can
read them: every way to render, from the sizes at which tables are still copied whole (32
loads of every thread) to the longest axis."""
import numpy as np
import pytest

import gen
from tests._parity import assert_parity
from tests.test_gpu_schedule import even_grid

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2609_09322_gb300 as g
    c = g.Context(0)
    yield c
    c.close()


def views_of(grid, axis):
    """Across the long axis, along it, and slowly along it; wide (nearly all rays miss) and
    close; far image planes."""
    long = float(grid.extent[axis])
    e = np.eye(3)
    dirs = [e[(axis + 1) % 3], -e[axis], e[axis] + 0.002 * e[(axis + 1) % 3], e[(axis + 2) % 3] - 0.01 * e[axis],
            np.array([0.5, -0.6, 0.4])]
    for k, d in enumerate(dirs):
        v = gen.view_from_direction(grid, d, size=23, height=18, fov=(6.0, 14.0, 3.0, 1.2 * long, 4.0)[k], c=40.0)
        off = 1.0e4 if k % 2 else 0.0
        yield v.with_(center=tuple(np.array(v.center) - off * np.array(v.dir)), t_obs=2.5 + off / 40.0)


def launch_of(warps, **kw):
    return dict({"packet": (8, 4), "cta_warps": warps, "depth": 2, "regcap": 1, "group": 1}, **kw)


# eight warps copy these whole (up to 8192 entries); one, two and four warps up to 1024, 2048 and 4096
@pytest.mark.parametrize("n", [(500, 5, 4), (5, 501, 4), (3, 7, 2035), (2038, 7, 3), (4, 4080, 3), (9, 3, 1020)])
@pytest.mark.parametrize("store,paired", [("f32", False), ("f32", True), ("bf16", False), ("bf16", True)])
def test_spans_give_what_whole_tables_give(ctx, n, store, paired):
    grid, j, beta = even_grid(sum(n), n, 3)
    vol = ctx.load_snapshots(grid, j, beta, store=store, paired=paired)
    for k, v in enumerate(views_of(grid, int(np.argmax(n)))):
        series = [v.with_(t_obs=v.t_obs + t) for t in (0.0, 0.3, 0.9, 1.6)]
        want = ctx.render_batch(vol, series, launch=launch_of(8))
        grouped = ctx.render_batch(vol, series, launch=launch_of(8, group=4))
        assert k == 3 or float(want.max()) > 0
        for warps in (1, 2, 4):
            assert torch.equal(ctx.render_batch(vol, series, launch=launch_of(warps)), want), (n, k, warps)
            got = ctx.render_batch(vol, series, launch=launch_of(warps, group=4))
            # one ray's sum whatever its kernel's member limit, to float32 rounding
            assert_parity(got.cpu().numpy(), grouped.cpu().numpy(), rel=1e-5, what=f"{n} view {k} groups {warps}")
    ctx.unload(vol)


@pytest.mark.parametrize("n", [(3, 4, 4096), (4096, 3, 4), (2, 4096, 2)])
@pytest.mark.parametrize("store", ["f32", "bf16"])
def test_longest_axes_against_the_region_schedule(ctx, n, store):
    """The region schedule stages each region's tables whole.  A crossing up to 4096 cells
    from its anchor is known to 4096 2^-23 cells (5e-4), a cell's boosted emissivity is
    at most 1.5 (sqrt(0.75) / 0.5)^2.6 = 6.3: the first and last chord of a ray differ by 6e-3 at
    most, and each inner crossing moves 5e-4 of a cell to its neighbour, which holds
    up to 27 times as much: 1.4e-2 of the sum."""
    grid, j, beta = even_grid(sum(n), n, 3)
    vol = ctx.load_snapshots(grid, j, beta, store=store)
    for k, v in enumerate(views_of(grid, int(np.argmax(n)))):
        want = ctx.render_batch(vol, [v] * 8, launch=launch_of(4, region=64))[0]
        for warps in (1, 4, 8):
            img = ctx.render(vol, v, launch=launch_of(warps))
            torch.cuda.synchronize()
            assert k == 3 or float(img.max()) > 0
            assert bool(((img - want).abs() <= 1.4e-2 * want.abs() + 6e-3).all()), (n, k, warps)
    ctx.unload(vol)


@pytest.mark.parametrize("n", [(4096, 3, 5), (6, 3000, 4)])
def test_served_and_vector_renders_of_long_volumes(ctx, n):
    grid, j, beta = even_grid(3, n, 2)
    vol = ctx.load_snapshots(grid, j, beta)
    short_grid, js, bs = even_grid(4, (9, 8, 7), 2)
    short = ctx.load_snapshots(short_grid, js, bs)
    ctx.load_channels(vol, torch.from_numpy(np.stack([j, -0.5 * j, 2.0 * j])).cuda())
    views = list(views_of(grid, int(np.argmax(n))))
    near = [gen.view_from_angles(short_grid, 40.0, 10.0, size=21, t_obs=t) for t in (3.0, 5.0)]
    ctx.serve_start()
    jobs = [(vol, v) for v in views] + [(short, v) for v in near]
    outs = [torch.full((v.height, v.width), -1.0, device="cuda") for _, v in jobs]
    torch.cuda.synchronize()
    tickets = [ctx.submit(w, v, o) for (w, v), o in zip(jobs, outs)]
    for t in tickets:
        ctx.wait(t)
    ctx.serve_stop()
    vec = [ctx.render_vector(vol, [v]) for v in views]
    for k, (w, v) in enumerate(jobs):
        want = ctx.render(w, v)
        torch.cuda.synchronize()
        assert torch.equal(outs[k], want)
        if w == vol:
            assert torch.equal(vec[k][0, 0], want)
            # -0.5 and 2 are exact factors of every term
            assert torch.equal(vec[k][0, 2], -0.5 * vec[k][0, 1]) and torch.equal(vec[k][0, 3], 2.0 * vec[k][0, 1])
    ctx.unload(vol)
    ctx.unload(short)
