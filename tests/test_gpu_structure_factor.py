"""S(q) where the transform's general stages can go wrong: prime edges (direct sums), small and large, and
edges so short that several threads share a column of the shell sums."""
import numpy as np
import pytest

from paper_0707_1581_gb300 import flb

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_0707_1581_gb300 import build as B
    B.build()


def shell_means(rho, nshells):
    """Mean of |FFT(rho)|^2 / N over the wave vectors of every shell, and their number (numpy, FP64)."""
    # k / n by one division, as the library's shell decision takes it (fftfreq multiplies by 1 / n)
    f = [np.where(np.arange(n) <= n // 2, np.arange(n), np.arange(n) - n) / n for n in rho.shape]
    nmax = max(rho.shape)
    shell = np.floor(nmax * np.sqrt((f[2][None, None, :] ** 2 + f[1][None, :, None] ** 2) + f[0][:, None, None] ** 2))
    shell = shell.astype(int).ravel()
    shell[0] = nshells
    power = (np.abs(np.fft.fftn(rho)) ** 2 / rho.size).ravel()
    keep = shell < nshells
    count = np.bincount(shell[keep], minlength=nshells)
    total = np.bincount(shell[keep], power[keep], minlength=nshells)
    return total / np.maximum(count, 1), count


VELOCITIES = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
              (1, -1, 0), (-1, 1, 0), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1), (1, 0, 1), (-1, 0, -1), (-1, 0, 1),
              (1, 0, -1)]


def density_deviation(ctx, nx, ny, nz, dtype):
    """rho - rho0 from the stored deviations of a two-buffer box (slot i at r - c_i), without the rounding of
    rho - 1 from whole populations."""
    raw = np.empty(ctx.flb_state_bytes() // np.dtype(dtype).itemsize, dtype=dtype)
    ctx.flb_state_download(raw)
    planes = raw.reshape(19, -1)[:, :nx * ny * nz].reshape(19, nz, ny, nx).astype(np.float64)
    return sum(np.roll(p, (c[2], c[1], c[0]), (0, 1, 2)) for p, c in zip(planes, VELOCITIES))


# (nx, ny, nz): primes alone, with factors of the other radices before them, along each direction; z edges of
# one to eight threads per kz
BOXES = [(11, 13, 17), (101, 6, 16), (8, 97, 5), (6, 4, 211), (88, 26, 34), (491, 3, 2), (3, 491, 4), (2, 3, 509),
         (253, 2, 3), (12, 7, 1), (16, 8, 2), (9, 5, 8), (10, 10, 32), (12, 20, 64), (6, 6, 100), (5, 8, 128),
         (4, 4, 144), (4, 3, 300)]


@pytest.mark.parametrize("store", ["f32", "f64"])
@pytest.mark.parametrize("nx,ny,nz", BOXES)
def test_structure_factor_of_prime_and_short_edges(nx, ny, nz, store):
    nsh = int(np.ceil(np.sqrt(3.0) * max(nx, ny, nz) / 2)) + 2
    with flb.flb_create_ex(flb.config(nx, ny, nz, kT=1e-3, gamma_shear=0.2, seed=4, store=store)) as ctx:
        ctx.flb_enable_structure_factor()
        ctx.flb_step(6)
        ctx.flb_stats_sample()
        S, count = ctx.flb_structure_factor(nsh)
        rho = density_deviation(ctx, nx, ny, nz, np.float32 if store == "f32" else np.float64)
    want, n = shell_means(rho, nsh)
    assert np.array_equal(count, n)
    # a line of L elements summed directly rounds to about eps sqrt(L) of the field's power per wave vector, the
    # radix stages to less; a shell averages its wave vectors' errors
    eps = (2.0 ** -24 if store == "f32" else 2.0 ** -53) * np.sqrt(max(nx, ny, nz))
    sel = n > 0
    bound = 4 * eps * (want[sel] + np.sqrt(want[sel] * want[sel].mean()) * 2)
    assert np.all(np.abs(S[sel] - want[sel]) <= bound), np.max(np.abs(S[sel] - want[sel]) / bound)
