"""The launch shape rules (host code, no GPU): the autotuner's candidates."""
import pytest

from test_kernel_indices import run_host

STORES = {"f64": 0, "f32": 1, "f16dev": 2, "bf16dev": 3, "bf16sr": 4}


@pytest.mark.parametrize("store", list(STORES))
def test_candidates_hold_the_shape_in_use_and_the_automatic_ones(tmp_path, store):
    """The shape in use first, the automatic shape for every number of sites per thread, the fixed blocks; every
    candidate fits the boxes, none twice."""
    run_host(tmp_path, f"""
    const int store = {STORES[store]};
    const std::vector<std::vector<int>> boxes = {{{{1}}, {{16}}, {{24}}, {{32}}, {{45}}, {{64}}, {{90}}, {{96}}, {{250}}, {{300}},
                                                 {{512}}, {{640}}, {{1000}}, {{4096}}, {{32, 64, 96}}, {{264, 508}}, {{33, 64}}}};
    auto same = [](const Launch &a, const Launch &b) {{
        return a.V == b.V && a.bx == b.bx && a.by == b.by && a.warprow == b.warprow && a.rows == b.rows &&
               a.edgerow == b.edgerow;
    }};
    for (const auto &nx : boxes)
        for (int d2 = 0; d2 < 2; ++d2)
            for (long long sites : {{1000ll, 90000ll, 3000000ll}}) {{
                if (d2 && nx.size() > 1) continue;
                const LaunchBoxes B{{store, d2 != 0, nx, sites}};
                for (Launch now : {{automatic_launch(B, 0, 0, 0), automatic_launch(B, 1, 7, 3)}}) {{
                    const std::vector<Launch> c = launch_candidates(B, now);
                    if (!same(c[0], now)) return 1;
                    for (int V : {{0, 1, 2, 4}}) {{
                        const Launch a = automatic_launch(B, V, 0, 0);
                        int n = 0;
                        for (const Launch &L : c) n += same(L, a);
                        if (n != 1) return printf("%d %d: %d x (%d, %d, %d)\\n", nx[0], d2, n, a.V, a.bx, a.by), 2;
                    }}
                    for (const Launch &L : c) {{
                        if (L.bx < 1 || L.by < 1 || L.bx * L.by > 256 || usable_V(B, L.V, L.bx, L.by) != L.V) return 3;
                        if (d2 && L.V != 1 && L.V != (store == 0 ? 2 : 4)) return 4;
                        int n = 0;
                        for (const Launch &o : c) n += o.V == L.V && o.bx == L.bx && o.by == L.by;
                        if (n != 1) return 5;
                    }}
                    const int fixed[3][2] = {{{{128, 1}}, {{32, 4}}, {{256, 1}}}};
                    for (const auto &s : fixed) {{
                        int n = 0;
                        for (const Launch &L : c) n += L.V == 1 && L.bx == s[0] && L.by == s[1];
                        if (n != 1 && nx[0] >= 128) return 6;
                    }}
                }}
            }}
    return 0;""", "launch_shape.h")


def test_automatic_shapes_outside_the_fixed_blocks_are_candidates(tmp_path):
    """Boxes whose automatic block is none of the fixed ones: 16^3 FP64 (32 threads), 96 and 640 wide FP32."""
    assert run_host(tmp_path, """
    const LaunchBoxes boxes[3] = {{FLB_STORE_F64, false, {16}, 4096}, {FLB_STORE_F32, false, {96}, 96 * 96 * 96},
                                  {FLB_STORE_F32, false, {640}, 640 * 64 * 64}};
    for (const LaunchBoxes &B : boxes) {
        Launch now;                       // something else in use
        now.V = 1, now.bx = 64, now.by = 4;
        const Launch a = automatic_launch(B, 0, 0, 0);
        int n = 0;
        for (const Launch &L : launch_candidates(B, now)) n += L.V == a.V && L.bx == a.bx && L.by == a.by;
        printf("%d %d %d %d\\n", a.V, a.bx, a.by, n);
    }""", "launch_shape.h").split() == "1 32 1 1 4 96 1 1 4 160 1 1".split()


def test_whole_rows_of_a_batch_leave_few_threads_idle(tmp_path):
    """Boxes of a batch take whole rows only where they fill the blocks: rows of 66, 80 and 96 threads in blocks of
    128, or of 3 in blocks of 256 (at most 32 rows), are packed densely; 24, 32 - 1 and 127 keep whole rows."""
    run_host(tmp_path, """
    for (int aa = 0; aa < 2; ++aa)
        for (int V : {2, 4})
            for (int T = 32; T <= 256; T += 32)
                for (int g = 1; g <= 1024; ++g) {
                    const int r = batch_rows(g, T, V, aa != 0);
                    if (r < 0 || r > kXchRows || r * g > T) return 1;
                    if (r && r * g < 0.7 * T) return 2;              // idle threads
                    if (T >= 64 && g <= T && r == 0 && std::min(T / g, kXchRows) * g >= 0.96 * T) return 3;
                }
    for (int g : {66, 80}) if (batch_rows(g, 128, 4, false) || batch_rows(g, 128, 4, true)) return 4;
    if (batch_rows(96, 128, 4, false) || batch_rows(3, 256, 4, false) || batch_rows(3, 256, 4, true)) return 5;
    if (batch_rows(24, 128, 4, false) != 5 || batch_rows(31, 128, 4, false) != 4 || batch_rows(127, 128, 4, true) != 1)
        return 6;
    return 0;""", "launch_shape.h")
