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


# (nx, sites per thread, block): the exchanges of the single-box kernel, with row counts that are and are not
# multiples of the rows of a block, rows shorter than a warp, longer, and of whole warps
SHAPES = [(12, 4, (128, 1)), (20, 4, (96, 1)), (40, 4, (128, 1)), (96, 4, (96, 1)), (100, 4, (256, 1)),
          (132, 4, (64, 1)), (500, 4, (128, 1)), (256, 4, (64, 1)), (1024, 4, (256, 1)), (128, 4, (128, 1)),
          (6, 2, (128, 1)), (50, 2, (32, 1)), (126, 2, (64, 1)), (250, 2, (128, 1)), (128, 2, (64, 1)),
          (300, 4, (64, 1)), (500, 4, (64, 1)), (1000, 4, (128, 1)), (250, 2, (64, 1)), (1, 1, (7, 3)),
          (37, 1, (128, 1)), (64, 2, (32, 4)), (16, 4, (4, 32))]
# steps of FP32 arithmetic on deviations of order 0.1: 5 x 16 roundings of 2^-24; one unit of binary16 or
# bfloat16 at 0.1 where a rounding falls the other way, carried through 5 steps
TOLERANCE = {"f64": 1e-13, "f32": 5 * 16 * 2.0 ** -24 * 0.1, "f16dev": 4 * 2.0 ** -14, "bf16dev": 4 * 2.0 ** -11}


@pytest.mark.parametrize("pattern", ["ab", "aa"])
@pytest.mark.parametrize("store", ["f64", "f32", "f16dev"])
@pytest.mark.parametrize("nx,V,block", SHAPES)
def test_every_exchange_gives_the_state_of_the_scalar_path(nx, V, block, store, pattern):
    if store == "f64" and V == 4:
        pytest.skip("FP64 takes at most two sites per thread")
    for ny, nz in ((1, 1), (5, 7), (3, 32)):
        cfg = box(nx, ny, nz, store, pattern, kT=1e-3, gamma_ghost=0.2, force_amp=1e-3)
        got = []
        for launch in ((1, 64, 1), (V,) + block):
            with flb.flb_create_ex(cfg) as ctx:
                ctx.flb_set_launch(*launch)
                ctx.flb_step(5)
                got.append(ctx.flb_get_populations())
        assert np.abs(got[0] - got[1]).max() <= TOLERANCE[store], (ny, nz)


@pytest.mark.parametrize("pattern", ["ab", "aa"])
@pytest.mark.parametrize("store", ["f64", "f32", "f16dev"])
def test_batch_of_every_row_length_equals_the_boxes_alone(store, pattern):
    edges = [(e, 3 + e % 5, 4) for e in (1, 2, 6, 12, 20, 28, 36, 40, 64, 100, 128, 132, 260, 516)]
    for V in (1, 2, 4):
        cfgs = [box(*(e if V == 1 else ((e[0] + V - 1) // V * V,) + e[1:]), store, pattern, kT=1e-3, replica=r)
                for r, e in enumerate(edges)]
        with flb.flb_create_batch(cfgs) as ctx:
            ctx.flb_set_launch(2 if store == "f64" and V == 4 else V, 32, 4)
            ctx.flb_step(5)
            got = [ctx.flb_get_populations(b) for b in range(len(cfgs))]
        for b, cfg in enumerate(cfgs):
            with flb.flb_create_ex(cfg) as ctx:
                ctx.flb_set_launch(1, 64, 1)
                ctx.flb_step(5)
                assert np.abs(ctx.flb_get_populations() - got[b]).max() <= TOLERANCE[store], (V, b)


@pytest.mark.parametrize("nx", [8, 12, 13, 16, 24, 36, 48, 64, 72, 100, 125, 128, 160, 250, 256, 300, 400, 512, 1000])
@pytest.mark.parametrize("store", ["f64", "f32", "f16dev"])
def test_automatic_launch_fits_its_box_and_is_accepted_back(nx, store):
    with flb.flb_create_ex(box(nx, 6, 4, store, "ab")) as ctx:
        V, bx, by = ctx.flb_get_launch()
        assert nx % V == 0 and 1 <= bx * by <= 256 and (V == 1 or bx * by % 32 == 0)
        ctx.flb_step(2)
        want = raw(ctx)
    with flb.flb_create_ex(box(nx, 6, 4, store, "ab")) as ctx:
        ctx.flb_set_launch(V, bx, by)
        ctx.flb_step(2)
        assert np.array_equal(raw(ctx), want)


@pytest.mark.parametrize("nx,ny,nz,nsteps", [(256, 130, 8, 2), (256, 117, 9, 2), (256, 100, 31, 4), (256, 129, 32, 5),
                                             (256, 104, 40, 5)] +
                         [(24, 6, nz, n) for nz, n in [(8, 2), (9, 2), (31, 4), (32, 5), (40, 5), (40, 6), (7, 3)]])
@pytest.mark.parametrize("pattern,start", [("ab", 0), ("ab", 1), ("aa", 0), ("aa", 1)])
def test_host_resident_steps_in_a_wave_equal_device_steps(pattern, start, nx, ny, nz, nsteps):
    """Several steps per call, each a few chunks behind the one before (20 MB of state for each; less: whole boxes)."""
    cfg = box(nx, ny, nz, "f32", pattern, kT=1e-3, force_amp=1e-4)
    with flb.flb_create_ex(cfg) as ref:
        ref.flb_step(6 + start)
        host = raw(ref)
        ref.flb_step(nsteps)
        want = raw(ref)
        ref.flb_step(3)
        later = raw(ref)
    with flb.flb_create_ex(cfg) as ctx:
        ctx.flb_step(6 + start)
        ctx.flb_init_velocity(None)
        ctx.flb_step_host(host, nsteps)
        assert np.array_equal(host, want) and ctx.flb_get_step() == 6 + start + nsteps
        assert np.array_equal(raw(ctx), want)
        ctx.flb_step(3)
        assert np.array_equal(raw(ctx), later)


@pytest.mark.parametrize("nx,store,kw", [(16, "f32", {}), (64, "f16dev", {}), (128, "f32", {}), (16, "f64", {}),
                                         (64, "f32", dict(lattice="d2q9"))])
def test_chained_launches_in_a_callers_graph(nx, store, kw):
    """Steps and a statistics sample captured from the caller's stream do what they do outside a capture."""
    import torch

    stream = torch.cuda.Stream()
    ny, nz = (nx, 1) if kw else (nx, nx // 2)
    with flb.flb_create_ex(box(nx, ny, nz, store, "ab", **kw)) as ctx:
        ctx.flb_step(4)
        ctx.flb_stats_sample()
        want, stats = raw(ctx), ctx.flb_mode_stats()
    with flb.flb_create_ex(box(nx, ny, nz, store, "ab", stream=stream, **kw)) as ctx:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            ctx.flb_step(4)
            ctx.flb_stats_sample()
        with torch.cuda.stream(stream):
            graph.replay()
        assert np.array_equal(raw(ctx), want)
        got = ctx.flb_mode_stats()
        assert got["nsamples"] == 1 and np.array_equal(got["mode_m2"], stats["mode_m2"])
        del graph


@pytest.mark.parametrize("nx,ny", [(236, 551), (512, 512), (752, 437), (1024, 1024), (2048, 2100)])
@pytest.mark.parametrize("store", ["f64", "f32", "f16dev", "bf16sr"])
@pytest.mark.parametrize("pattern,graph_steps", [("ab", 0), ("aa", 0), ("ab", 10), ("aa", 10)])
def test_chained_d2q9_steps_equal_steps_one_at_a_time(pattern, graph_steps, store, nx, ny):
    """Boxes of one block per SM, two, more, and beyond L2: each start point of the next step."""
    cfg = dict(lattice="d2q9", kT=1e-4, force_amp=1e-5)
    with flb.flb_create_ex(box(nx, ny, 1, store, pattern, **cfg)) as ctx:
        for _ in range(21):
            ctx.flb_step(1)
            ctx.flb_sync()
        want = raw(ctx)
    with flb.flb_create_ex(box(nx, ny, 1, store, pattern, graph_steps=graph_steps, **cfg)) as ctx:
        ctx.flb_step(21)
        assert np.array_equal(raw(ctx), want)


@pytest.mark.parametrize("nx,ny", [(7, 9), (51, 301), (117, 300), (301, 301), (501, 601), (1001, 601)])
@pytest.mark.parametrize("store", ["f64", "f32", "bf16dev", "bf16sr"])
@pytest.mark.parametrize("pattern,graph_steps", [("ab", 0), ("aa", 0), ("ab", 10), ("aa", 10)])
def test_chained_one_site_d2q9_steps_equal_steps_one_at_a_time(pattern, graph_steps, store, nx, ny):
    """Odd rows: every start point of the one-site kernel (half a block per SM, one, several, many)."""
    cfg = dict(lattice="d2q9", kT=1e-4, force_amp=1e-5)
    with flb.flb_create_ex(box(nx, ny, 1, store, pattern, **cfg)) as ctx:
        for _ in range(21):
            ctx.flb_step(1)
            ctx.flb_sync()
        want = raw(ctx)
    with flb.flb_create_ex(box(nx, ny, 1, store, pattern, graph_steps=graph_steps, **cfg)) as ctx:
        ctx.flb_step(21)
        assert np.array_equal(raw(ctx), want)


@pytest.mark.parametrize("nx,ny,force", [(256, 456, 0.0), (256, 458, 0.0), (256, 608, 0.0), (256, 610, 0.0),
                                         (256, 480, 1e-5)])
@pytest.mark.parametrize("pattern,graph_steps", [("ab", 0), ("aa", 0), ("ab", 10)])
def test_chained_fp64_d2q9_steps_of_two_blocks_per_sm(pattern, graph_steps, nx, ny, force):
    """On either side of the range of unchained FP64 steps; a statistics sample after them."""
    cfg = dict(lattice="d2q9", kT=1e-4, force_amp=force)
    with flb.flb_create_ex(box(nx, ny, 1, "f64", pattern, **cfg)) as ctx:
        for _ in range(21):
            ctx.flb_step(1)
            ctx.flb_sync()
        ctx.flb_stats_sample()
        want, stats = raw(ctx), ctx.flb_mode_stats()
    with flb.flb_create_ex(box(nx, ny, 1, "f64", pattern, graph_steps=graph_steps, **cfg)) as ctx:
        ctx.flb_step(21)
        ctx.flb_stats_sample()
        assert np.array_equal(raw(ctx), want)
        assert np.array_equal(ctx.flb_mode_stats()["mode_m2"], stats["mode_m2"])


@pytest.mark.parametrize("nx,ny,nz,store", [(16, 1, 70000, "f32"), (16, 2097153, 1, "f32"), (256, 1, 66000, "f32"),
                                            (250, 1, 66000, "f32"), (250, 66000, 1, "f32"), (1000, 1, 66000, "f16dev"),
                                            (1000, 66000, 1, "f16dev"), (32, 1, 70000, "f64")])
def test_boxes_of_more_planes_or_rows_than_a_grid_dimension(nx, ny, nz, store):
    """Rows that tile the warps, whole rows, blocks inside a row: against the scalar path, at sampled sites."""
    cfg = box(nx, ny, nz, store, "aa", kT=1e-3, force_amp=1e-3)
    N = nx * ny * nz
    sites = np.unique(np.concatenate([[0, N - 1, N - nx, 65535 * nx, min(N - 1, 65536 * nx + nx - 1)],
                                      np.random.default_rng(1).integers(0, N, 2000)]))
    got = []
    for launch in (None, (1, 128, 1)):
        with flb.flb_create_ex(cfg) as ctx:
            if launch:
                ctx.flb_set_launch(*launch)
            else:
                assert ctx.flb_get_launch()[0] > 1
            ctx.flb_step(3)
            got.append(ctx.flb_get_sites(sites))
    assert np.abs(got[0] - got[1]).max() <= TOLERANCE[store]


@pytest.mark.parametrize("nx,ny", [(256, 608), (256, 610), (1000, 601)])
@pytest.mark.parametrize("force,kT", [(0.0, 1e-4), (1e-5, 1e-4), (1e-5, 0.0)])
def test_fp64_d2q9_steps_in_place_equal_the_one_site_kernel(nx, ny, force, kT):
    """AA steps on either side of two blocks per SM against the one-site kernel: the same arithmetic, so FP64 bounds."""
    cfg = box(nx, ny, 1, "f64", "aa", lattice="d2q9", kT=kT, force_amp=force)
    got = []
    for launch in ((2, 128, 2), (1, 128, 2)):
        with flb.flb_create_ex(cfg) as ctx:
            ctx.flb_set_launch(*launch)
            ctx.flb_step(6)
            got.append(ctx.flb_get_populations())
    assert np.abs(got[0] - got[1]).max() <= TOLERANCE["f64"]
