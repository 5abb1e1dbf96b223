"""Plane and row averages (flb_box_z_profile) against sums of the canonical populations."""
import math

import numpy as np
import pytest

from paper_0707_1581_gb300 import flb
from paper_0707_1581_gb300.inputs import relative_perturbation

pytestmark = pytest.mark.gpu

WX = {19: [0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 0, 0, 0, 0, 1, -1, -1, 1], 9: [0, 1, -1, 0, 0, 1, -1, 1, -1]}
WY = {19: [0, 0, 0, 1, -1, 0, 0, 1, -1, -1, 1, 1, -1, 1, -1, 0, 0, 0, 0], 9: [0, 0, 0, 1, -1, 1, -1, -1, 1]}
WZ = {19: [0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, -1, -1, 1, 1, -1, 1, -1], 9: [0] * 9}


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_0707_1581_gb300 import build as B
    B.build()


def reference(n, two):
    """rho[units], j[3][units] of populations n[q, ..., x], summed over all but the unit axis in FP64."""
    q = n.shape[0]
    m = n.sum(2) / n.shape[2] if two else n.sum((2, 3)) / (n.shape[2] * n.shape[3])
    with np.errstate(invalid="ignore"):
        return m.sum(0), np.stack([(np.array(w[q])[:, None] * m).sum(0) for w in (WX, WY, WZ)])


# units of odd length (misaligned for vector loads), of fewer elements than a warp and than a block's
# threshold, and few large ones (several blocks per unit)
BOXES = [(1, 1, 1), (3, 5, 7), (17, 3, 6), (45, 46, 9), (64, 64, 8), (61, 67, 5), (301, 211, 2), (256, 256, 1)]


@pytest.mark.parametrize("steps", [0, 1, 2])
@pytest.mark.parametrize("pattern", ["ab", "aa"])
@pytest.mark.parametrize("store", ["f64", "f32", "f16dev", "bf16dev", "bf16sr"])
def test_profile_is_the_mean_of_the_populations(store, pattern, steps):
    for two in (False, True):
        for nx, ny, nz in BOXES:
            cfg = flb.config(nx, ny * nz if two else ny, 1 if two else nz, kT=1e-3, gamma_shear=0.3, seed=2, store=store,
                             pattern=pattern, lattice="d2q9" if two else "d3q19")
            with flb.flb_create_ex(cfg) as ctx:
                ctx.flb_step(steps)
                rho, j = ctx.flb_z_profile()
                want_rho, want_j = reference(ctx.flb_get_populations(), two)
            # both sides round in FP64 (or 48 bits, of the small deviations): 1e-15 per unit of rho
            assert np.abs(rho - want_rho).max() <= 2e-14 and np.abs(j - want_j).max() <= 2e-14, (two, nx, ny, nz)


@pytest.mark.parametrize("store", ["f64", "f32", "f16dev"])
def test_profile_of_values_beyond_the_ordinary(store):
    """Sums beyond FP32's range stay finite; an infinity or NaN shows in its plane and nowhere else."""
    shape = (19, 4, 40, 64)
    big = {"f64": 1e300, "f32": 2e38, "f16dev": 6e4}[store]
    with flb.flb_create_ex(flb.config(64, 40, 4, store=store, pattern="aa")) as ctx:
        n = relative_perturbation(shape[1:], seed=3, amp=0.02) / 19
        n[3, 1] = big
        ctx.flb_set_populations(n)
        n = ctx.flb_get_populations()
        rho, j = ctx.flb_z_profile()
        want_rho, want_j = reference(n, False)
        assert np.isfinite(rho).all() and np.allclose(rho, want_rho, rtol=1e-12) and np.allclose(j, want_j, rtol=1e-12, atol=1e-13)
        for bad in (np.inf, -np.inf, np.nan):
            m = relative_perturbation(shape[1:], seed=3, amp=0.02) / 19
            m[5, 2, 7, 9] = bad
            ctx.flb_set_populations(m)
            rho, j = ctx.flb_z_profile()
            with np.errstate(invalid="ignore"):
                want_rho, want_j = reference(ctx.flb_get_populations(), False)
            assert np.array_equal(np.isnan(rho), np.isnan(want_rho)) and np.array_equal(np.isinf(rho), np.isinf(want_rho))
            assert np.array_equal(np.isnan(j), np.isnan(want_j)) and np.array_equal(np.isinf(j), np.isinf(want_j))


def test_profile_of_more_than_2_to_27_rows():
    """D2Q9 rows of four sites; one thermal step, rows around 2^27 and the ends against their populations."""
    torch = pytest.importorskip("torch")
    ny = 2 ** 27 + 100                      # 2^29 sites, 9.7 GB of bfloat16 state
    if torch.cuda.mem_get_info()[0] < 24e9:
        pytest.skip("needs 24 GB of free device memory")
    rows = np.array([0, 1, 99, 100, 2 ** 26, 2 ** 27 - 1, 2 ** 27, 2 ** 27 + 1, ny - 2, ny - 1])
    cfg = flb.config(4, ny, 1, kT=1e-3, gamma_shear=0.3, seed=2, store="bf16dev", pattern="aa", lattice="d2q9")
    with flb.flb_create_ex(cfg) as ctx:
        ctx.flb_step(1)
        n = ctx.flb_get_sites((4 * rows[:, None] + np.arange(4)).ravel()).reshape(len(rows), 4, 9)
        rho, j = ctx.flb_z_profile()
    want_rho, want_j = reference(n.transpose(2, 0, 1), True)
    # as in the test above
    assert np.abs(rho[rows] - want_rho).max() <= 2e-14 and np.abs(j[:, rows] - want_j).max() <= 2e-14


@pytest.mark.parametrize("units", [65536, 65537, 131072 + 5])
@pytest.mark.parametrize("pattern,steps", [("ab", 2), ("aa", 2), ("aa", 3)])
@pytest.mark.parametrize("two", [False, True])
def test_profile_of_several_passes(two, pattern, steps, units):
    """Boxes of more units than one pass takes: the ends of the passes and of the box."""
    cfg = flb.config(3, units if two else 1, 1 if two else units, kT=1e-3, gamma_shear=0.3, seed=2, pattern=pattern,
                     lattice="d2q9" if two else "d3q19")
    with flb.flb_create_ex(cfg) as ctx:
        ctx.flb_step(steps)
        rho, j = ctx.flb_z_profile()
        want_rho, want_j = reference(ctx.flb_get_populations(), two)
    # as in the first test
    assert np.abs(rho - want_rho).max() <= 2e-14 and np.abs(j - want_j).max() <= 2e-14


@pytest.mark.parametrize("store,w", [("f32", 2.0 ** -26 * (1 + 2.0 ** -22 + 2.0 ** -23)), ("f32", 2.0 ** -27 * 1.7320508),
                                     ("bf16dev", 2.0 ** -27 * 1.75)])
def test_profile_keeps_the_bits_of_an_fp64_sum(store, w):
    """A few ones before many values below their 24 bits: the partial sums have to hold more than 48 bits."""
    nx = ny = 1024
    with flb.flb_create_ex(flb.config(nx, ny, 1, store=store, pattern="ab")) as ctx:
        x = np.full(nx * ny, w, np.float32)
        if store == "bf16dev":                       # the stored values: bfloat16 bits, of several sizes
            x[::3] *= 2.0 ** -9
            x[1::7] *= 2.0 ** -17
        x[np.arange(nx * ny) % 16384 < 1024] = 1.0
        raw = np.zeros(ctx.flb_state_bytes(), np.uint8)
        planes = raw.view(np.float32 if store == "f32" else np.uint16).reshape(19, -1)
        planes[5, :nx * ny] = x if store == "f32" else x.view(np.uint32) >> 16
        ctx.flb_state_upload(raw)
        j = ctx.flb_z_profile()[1]
    stored = x if store == "f32" else ((x.view(np.uint32) >> 16) << 16).view(np.float32)
    want = math.fsum(stored.astype(np.float64)) / (nx * ny)
    # slot 5 moves along z.  At most two roundings per thread, 8 warps, 64 pieces of the plane and the division, each
    # of 2^-53 of a sum no larger than the total
    assert abs(j[2, 0] - want) <= 75 * 2.0 ** -53 * want


@pytest.mark.parametrize("nx,ny", [(64, 40), (16, 16)])
def test_profile_of_values_beyond_fp32_only_together(nx, ny):
    """Four of 3e38 a row apart: no thread's own sum leaves FP32's range, that of the warp or block does."""
    with flb.flb_create_ex(flb.config(nx, ny, 4, store="f32", pattern="aa")) as ctx:
        n = relative_perturbation((4, ny, nx), seed=3, amp=0.02) / 19
        n[3, 1, :8:2, 5] = 3e38
        ctx.flb_set_populations(n)
        n = ctx.flb_get_populations()
        rho, j = ctx.flb_z_profile()
    want_rho, want_j = reference(n, False)
    assert np.isfinite(rho).all() and np.allclose(rho, want_rho, rtol=1e-12) and np.allclose(j, want_j, rtol=1e-12, atol=1e-13)


@pytest.mark.parametrize("store", ["f64", "f32", "bf16sr"])
def test_profile_on_either_side_of_warps_and_blocks(store):
    """Planes of 1023, 1024, 2025 and 2048 elements; 64 and 65 planes (1216 and 1235 sums)."""
    for nx, ny, nz in ((33, 31, 20), (32, 32, 64), (32, 32, 65), (45, 45, 8), (64, 32, 3)):
        with flb.flb_create_ex(flb.config(nx, ny, nz, kT=1e-3, gamma_shear=0.3, seed=2, store=store)) as ctx:
            ctx.flb_step(2)
            rho, j = ctx.flb_z_profile()
            want_rho, want_j = reference(ctx.flb_get_populations(), False)
        # as in the first test
        assert np.abs(rho - want_rho).max() <= 2e-14 and np.abs(j - want_j).max() <= 2e-14, (nx, ny, nz)
