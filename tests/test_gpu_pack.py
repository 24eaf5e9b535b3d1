"""Packing of float32 fields decides the limit of |beta| and rounds the float16
four-velocity without float64 where float32 can tell; the same values given as
float64 take the float64 path.  Both have to store the same records, so their
images are equal bit for bit, and to accept and refuse the same fields."""
import numpy as np
import pytest

import gen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2609_09322_gb300 as g
    c = g.Context(0)
    yield c
    c.close()


def hard_velocities(rng, shape, top):
    """|beta| from 0 up to ``top``, dense towards it, with zeros of both signs,
    tiny components and velocities along an axis."""
    d = rng.normal(size=(*shape, 3))
    d[rng.random(shape) < 0.1, 0] = 0.0
    d[rng.random(shape) < 0.1, 1:] *= 1e-6
    d /= np.maximum(np.linalg.norm(d, axis=-1, keepdims=True), 1e-30)
    mag = np.minimum(1.0 - 10.0 ** rng.uniform(-6.5, 0.0, size=(*shape, 1)), top)
    mag[rng.random((*shape, 1)) < 0.05] = 0.0
    return (d * mag * rng.choice([-1.0, 1.0], size=(*shape, 1))).astype(np.float32)


# no padding (whole super-bricks, nothing cleared beforehand), padding, one cell; unpaired and paired
@pytest.mark.parametrize("n", [(64, 32, 32), (33, 17, 9), (1, 1, 1)])
@pytest.mark.parametrize("store,top", [("f32", 1.0 - 1e-6), ("bf16", 1.0 - 1e-7), ("bf16", 0.99)])
@pytest.mark.parametrize("paired", [False, True])
def test_float32_and_float64_input_store_the_same(ctx, n, store, top, paired):
    rng = np.random.default_rng([*n, int(paired)])
    m = 3
    grid = gen.Grid(n=n, n_epochs=m, t0=0.0, dt=4.0)
    shape = (m, n[2], n[1], n[0])
    j = (rng.random(shape) * 10.0 ** rng.uniform(-6, 3, size=shape)).astype(np.float32)
    beta = hard_velocities(rng, shape, top)
    views = [gen.view_from_direction(grid, d, size=40, c=1.0, t_obs=4.0) for d in ((1, 0.2, 0.3), (-0.3, 1, 0.1), (0.2, -0.1, -1))]
    # memory that a load without clearing would otherwise find clean
    torch.full((4 << 20,), float("nan"), device="cuda")
    torch.cuda.empty_cache()
    imgs = []
    for dtype in (np.float32, np.float64):
        vol = ctx.load_snapshots(grid, j.astype(dtype), beta.astype(dtype), store=store, paired=paired)
        imgs.append(ctx.render_batch(vol, views).cpu().numpy())
        ctx.unload(vol)
    assert np.isfinite(imgs[0]).all() and imgs[0].max() > 0
    assert np.array_equal(imgs[0], imgs[1])


@pytest.mark.parametrize("store", ["f32", "bf16"])
def test_limit_of_beta_is_the_same_for_both_inputs(ctx, store):
    from paper_2609_09322_gb300 import GbdError
    grid = gen.Grid(n=(4, 4, 4), n_epochs=1, t0=0.0, dt=1.0)
    j = np.ones((1, 4, 4, 4), np.float32)
    took = []
    for b in np.float32([1.0 - 2.0 ** -k for k in range(14, 25)] + [1.0, 1.5, np.nan, np.inf]):
        beta = np.zeros((1, 4, 4, 4, 3), np.float32)
        beta[0, 1, 2, 3, 2] = b
        got = []
        for dtype in (np.float32, np.float64):
            try:
                ctx.unload(ctx.load_snapshots(grid, j.astype(dtype), beta.astype(dtype), store=store))
                got.append(True)
            except GbdError:
                got.append(False)
        assert got[0] == got[1], b
        took.append(got[0])
    # float32 storage: |beta|^2 <= 1 - 2^-20, so 1 - 2^-20 (|beta|^2 = 1 - 2^-19) is the largest of these; otherwise
    # the float16 four-velocity has to be finite, which it is up to 1 - 2^-24
    assert took == [True] * (7 if store == "f32" else 11) + [False] * (8 if store == "f32" else 4)
