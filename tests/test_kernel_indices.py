"""Index arithmetic that kernels share with the host, over its whole range, compiled for the host (no GPU)."""
import subprocess

import pytest

from paper_0707_1581_gb300 import build as B


def run_host(tmp_path, body: str, include: str) -> str:
    """Compiles a program of the library's own functions and returns what it prints."""
    src, exe = tmp_path / "t.cu", tmp_path / "t"
    src.write_text(f'#include "{include}"\n#include <cstdio>\n#include <cstdlib>\nusing namespace flb;\n'
                   f"int main() {{\n{body}\n    return 0;\n}}\n")
    cmd = [B.nvcc(), *B.ARCH, "-std=c++17", "-O1", f"-I{B.INCLUDE}", f"-I{B.CSRC}", str(src), "-o", str(exe)]
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    res = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert res.returncode == 0, res.stdout + res.stderr
    return res.stdout


@pytest.mark.parametrize("units", [1, 5, 2 ** 27 - 1, 2 ** 27, 2 ** 27 + 100, 2 ** 31 - 1])
def test_every_unit_has_its_own_warp_of_the_plane_means(tmp_path, units):
    """Block b of 128 threads holds the units 4 b .. 4 b + 3, to the largest number of units a box can have."""
    run_host(tmp_path, f"""
    const long long units = {units}, blocks = (units + 3) / 4;
    for (long long b : {{0ll, 1ll, blocks / 2, blocks - 1}})
        for (unsigned t = 0; t < 128; ++t) {{
            const long long u = 4 * b + t / 32;
            if (b < blocks && u < units && profile::unit_of((unsigned)b, 128, t) != u) {{
                printf("block %lld thread %u: unit %d\\n", b, t, profile::unit_of((unsigned)b, 128, t));
                return 1;
            }}
        }}""", "profile.cuh")


@pytest.mark.parametrize("xch", ["kRows", "kRagRow", "kOneRow"])
def test_row_exchange_slots_lie_in_the_arrays_and_pair_up(tmp_path, xch):
    """Every thread of every block shape that the exchange can have, the idle ones among them: slots inside the
    arrays; a thread with a site group reads what its neighbour in the (periodic) row wrote."""
    run_host(tmp_path, f"""
    constexpr int X = {xch}, slots = RowExchange<float, X>::kSlots;
    int bad = 0;
    for (int g = 1; g <= 256; ++g)
        for (int rows = 1; rows <= kXchRows && rows * g <= 256; ++rows)
            for (int T = (rows * g + 31) / 32 * 32; T <= 256; T += 32) {{
                if (X != kRows && rows > 1) continue;
                if (X == kOneRow && T != g) continue;
                auto place = [&](int t) {{
                    const int tr = t / g, tx = X == kRows ? t - tr * g : (t < g ? t : g - 1);
                    return row_place<X>(t & 31, t >> 5, T / 32, tx, g, X == kRows ? (tr < kXchRows ? tr : kXchRows - 1) : 0);
                }};
                int last[slots], first[slots];
                for (int k = 0; k < slots; ++k) last[k] = first[k] = -1;
                for (int t = 0; t < T; ++t) {{
                    const RowPlace p = place(t);
                    for (int k : {{p.mine_last, p.mine_first, p.from_left, p.from_right}})
                        if (k < 0 || k >= slots) {{
                            if (!bad++) printf("g %d rows %d T %d thread %d: slot %d of %d\\n", g, rows, T, t, k, slots);
                        }}
                    if (t >= rows * g) continue;
                    if (p.give_last) last[p.mine_last] = last[p.mine_last] < 0 ? t : -2;      // -2: two writers
                    if (p.give_first) first[p.mine_first] = first[p.mine_first] < 0 ? t : -2;
                }}
                for (int t = 0; t < rows * g; ++t) {{
                    const RowPlace p = place(t);
                    const int r = t / g, x = t - r * g, left = r * g + (x + g - 1) % g, right = r * g + (x + 1) % g;
                    if (p.take_left ? last[p.from_left] != left : left != t - 1) ++bad;
                    if (p.take_right ? first[p.from_right] != right : right != t + 1) ++bad;
                }}
            }}
    if (bad) printf("%d\\n", bad);
    return bad != 0;""", "kernels.cuh")


@pytest.mark.parametrize("units", [1, 2, 3, 65535, 65536, 65537, 65538, 131073, 2 ** 29 + 1, 2 ** 31 - 1])
def test_passes_of_the_plane_averages_cover_every_unit(tmp_path, units):
    """Each unit is a mean of one pass; slot i's sum that goes into unit u is that of unit u - c_i (periodic)."""
    run_host(tmp_path, f"""
    const long long units = {units};
    long long done = 0;
    for (long long u0 = 0, k = 0; u0 < units; ++k) {{
        const profile::Pass p = profile::pass_from((int)u0, (int)units);
        if (p.n < 1 || p.nsum > profile::kPassUnits + 2) return 1;
        const bool look = k < 3 || u0 + 3ll * profile::kPassUnits > units;      // the first and last passes, whole
        for (int m = 0; m < p.n; m += look ? 1 : 32767)
            for (int shift = -1; shift <= 1; ++shift) {{
                const int s = profile::sum_of_mean(p, m, shift);
                const long long want = (u0 + m - shift + units) % units;
                if (s < 0 || s >= p.nsum || profile::unit_of_sum(p, s, (int)units) != want) {{
                    printf("unit %lld shift %d: sum %d\\n", u0 + m, shift, s);
                    return 1;
                }}
            }}
        done += p.n;
        u0 += p.n;
    }}
    return done != units;""", "profile.cuh")
