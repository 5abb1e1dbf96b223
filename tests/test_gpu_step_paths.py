"""The paths of the time step: every launch form gives the bits of the general one."""
import numpy as np
import pytest

from paper_0707_1581_gb300 import flb

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_0707_1581_gb300 import build as B
    B.build()


def raw(ctx, box=0):
    out = np.empty(ctx.flb_state_bytes(box), dtype=np.uint8)
    ctx.flb_state_download(out, box)
    return out


def box(nx, ny, nz, store, pattern, **kw):
    kw = dict(dict(kT=1e-4, gamma_shear=0.3, gamma_bulk=0.2, seed=5), **kw)
    return flb.config(nx, ny, nz, store=store, pattern=pattern, **kw)


# boxes of a few blocks (a step is far shorter than a launch) and of several waves; every number of
# sites per thread; both lattices
CHAINED = [(16, 16, 16, "f64", {}), (48, 40, 44, "f64", {}), (16, 16, 16, "f32", {}), (33, 7, 5, "f32", {}),
           (64, 64, 64, "f32", {}), (64, 64, 64, "f16dev", {}), (128, 96, 60, "f32", {}), (96, 50, 70, "bf16sr", {}),
           (64, 48, 1, "f32", dict(lattice="d2q9")), (33, 48, 1, "bf16dev", dict(lattice="d2q9"))]


@pytest.mark.parametrize("pattern", ["ab", "aa"])
@pytest.mark.parametrize("nx,ny,nz,store,kw", CHAINED)
def test_chained_steps_equal_steps_waited_for_one_by_one(nx, ny, nz, store, kw, pattern):
    with flb.flb_create_ex(box(nx, ny, nz, store, pattern, **kw)) as ctx:
        for _ in range(48):
            ctx.flb_step(1)
            ctx.flb_sync()
        want = raw(ctx)
    for graph in (0, 6):
        with flb.flb_create_ex(box(nx, ny, nz, store, pattern, graph_steps=graph, **kw)) as ctx:
            ctx.flb_step(48)
            assert np.array_equal(raw(ctx), want)


def test_chained_steps_of_a_batch_of_several_launches_per_step():
    """More boxes than one launch's table holds: a step is two launches."""
    cfgs = [box(16 + 8 * (b % 3), 12, 10, "f32", "ab", replica=b) for b in range(70)]
    with flb.flb_create_batch(cfgs) as ctx:
        for _ in range(20):
            ctx.flb_step(1)
            ctx.flb_sync()
        want = [raw(ctx, b) for b in range(70)]
    with flb.flb_create_batch(cfgs) as ctx:
        ctx.flb_step(20)
        assert all(np.array_equal(raw(ctx, b), want[b]) for b in range(70))
