"""Single-view renders inside a caller's stream capture, on the first use of an image
geometry: nothing is allocated or waited for, and a replay gives the direct render's image."""
import pytest

import gen
from tests.test_gpu_schedule import even_grid

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2609_09322_gb300 as g
    c = g.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("form", ["render", "render_persistent_0", "vector"])
def test_first_render_of_a_geometry_in_a_capture(ctx, form):
    grid, j, beta = even_grid(5, (12, 10, 9), 2)
    vol = ctx.load_snapshots(grid, j, beta)
    ctx.load_channels(vol, j[None].copy())
    size = {"render": 61, "render_persistent_0": 62, "vector": 63}[form]
    view = gen.view_from_angles(grid, 37.0, 205.0, size=size, c=1.3, t_obs=2.0)
    shape = (1, 2, size, size) if form == "vector" else (size, size)
    out = torch.full(shape, -1.0, device="cuda")

    def run():
        if form == "vector":
            ctx.render_vector(vol, [view], out=out)
        else:
            ctx.render(vol, view, out=out,
                       launch={"packet": (8, 4), "persistent": 0} if form.endswith("0") else None)

    warm = gen.view_from_angles(grid, 37.0, 205.0, size=17, c=1.3, t_obs=2.0)  # kernels loaded, another geometry
    ctx.render(vol, warm)
    ctx.render_vector(vol, [warm])
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        run()
    assert float(out.max()) == -1.0
    graph.replay()
    torch.cuda.synchronize()
    replayed = out.clone()
    run()
    torch.cuda.synchronize()
    assert float(replayed.max()) > 0 and torch.equal(replayed, out)
    ctx.unload(vol)
