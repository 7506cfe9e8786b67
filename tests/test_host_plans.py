"""Sizes and splits the host decides (csrc/host_plans.h), walked over every size the entry points accept: no GPU.

The header is compiled with g++ into a small program per property; a line of its output is a violation."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def violations(tmp_path, body: str) -> str:
    src, exe = tmp_path / "walk.cpp", tmp_path / "walk"
    src.write_text('#include "host_plans.h"\n#include <cstdio>\nusing namespace bwla;\nint main() {\n' + body + "\n}\n")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2605_00422_b200", "csrc"), "-o", str(exe), str(src)], check=True)
    return subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout[:2000]


def test_partial_sums_of_the_low_rank_term_fit_their_section(tmp_path):
    """What the blocks that split K write ([tile][part][16][columns], whole tiles) against what the workspace holds for it; ranks
    above 64 whose padded columns do not fill the last tile are the narrow case."""
    assert violations(tmp_path, """
    for (int r = 1; r <= 256; ++r)
        for (int M = 1; M <= 80; ++M)
            for (int K = 32; K <= 25600; K += 32)
                for (int warps = 1; warps <= 16; ++warps) {
                    const int cols = lowrank_cols(r), ks = lowrank_ksplit(M, K, cols, warps);
                    const size_t wrote = ks > 1 ? (size_t)lowrank_tiles(M, cols) * ks * 16 * lowrank_tile_cols(M) * 4 : 0;
                    if (wrote > lowrank_split_bytes(M, cols)) { std::printf("r %d M %d K %d warps %d\\n", r, M, K, warps); return 0; }
                }""") == ""


def test_the_workspace_has_that_room(tmp_path):
    from paper_2605_00422_b200 import bwla
    rows = violations(tmp_path, """
    for (int r : {64, 65, 72, 88, 104, 120, 128, 136, 256})
        for (int M : {1, 8, 16, 17, 32, 33, 64}) std::printf("%d %d %zu\\n", r, M, lowrank_split_bytes(M, lowrank_cols(r)));""")
    for line in rows.splitlines():
        r, M, need = map(int, line.split())
        off_T, n_T = bwla.bwla_workspace_section(M, 4096, 64, r, 6, bwla.BWLA_WS_T)
        off_codes, _ = bwla.bwla_workspace_section(M, 4096, 64, r, 6, bwla.BWLA_WS_CODES)
        assert off_codes - (off_T + n_T) >= need, f"r {r}, {M} tokens"


SIZES = (32, 128, 512, 1152, 4096, 5120, 8192, 11008, 13824, 16384, 16416, 20480, 25600)
RANKS = (0, 1, 32, 64, 65, 72, 128, 256)


def test_a_workspace_for_many_tokens_serves_fewer():
    """A program that allocates for its largest batch calls with every smaller one."""
    from paper_2605_00422_b200 import bwla
    for K in SIZES:
        for r in RANKS:
            sizes = [bwla.bwla_workspace_bytes(M, K, 4096, r, 6) for M in range(1, 700)]
            drops = [M for M, (a, b) in enumerate(zip(sizes, sizes[1:]), 2) if b < a]
            assert not drops, f"K {K}, rank {r}: {drops[:5]} tokens need less than one token fewer"


def test_a_weight_only_workspace_for_many_tokens_serves_fewer(tmp_path):
    assert violations(tmp_path, """
    for (long K = 64; K <= 25600; K += 64)
        for (long M = 1; M <= 200; ++M)
            if (a16_value_bytes(M + 1, K) < a16_value_bytes(M, K) || a16_sum_bytes(M + 1) < a16_sum_bytes(M) || a16_value_bytes(M, K) < (size_t)(2 * M * K) ||
                (M <= kDigitTokens && (a16_value_bytes(M, K) < (size_t)(3 * M * K) || a16_sum_bytes(M) < (size_t)(96 * M)))) { std::printf("%ld tokens, K %ld\\n", M, K); return 0; }""") == ""


def test_problems_of_the_built_in_scratch():
    """bwla_w1ax_linear_static: 4 MiB hold the codes and at most 688 KiB of everything that does not grow with the tokens."""
    from paper_2605_00422_b200 import bwla
    for M, K in ((64, 25600), (134, 25600), (167, 20480), (246, 13824), (512, 5120)):
        for r in (0, 16, 64):
            assert bwla.bwla_workspace_bytes(M, K, 4096, r, 6) <= bwla.BWLA_STATIC_SCRATCH_BYTES, (M, K, r)
    for K in SIZES:
        for r in RANKS:
            for M in range(1, 256):
                per_token = K + 40 + 6 * max(64, r + r % 2)
                assert bwla.bwla_workspace_bytes(M, K, 4096, r, 6) <= M * per_token + 688 * 1024 + 256 * 6, (M, K, r)


def test_partial_sums_of_many_tokens_fit_where_the_codes_go(tmp_path):
    assert violations(tmp_path, """
    for (long M = 1; M <= 5000; ++M)
        for (long K = 64; K <= 25600; K += 64)
            if (lowrank_umma_part_bytes(M, K) > (size_t)(M * K) || lowrank_umma_parts(M, K) > K / 64) { std::printf("%ld tokens, K %ld\\n", M, K); return 0; }""") == ""


def test_operands_of_the_rotations_lie_inside_the_block(tmp_path):
    """Every pair of factor sizes, every number of tokens the few-token plan distinguishes: what ldmatrix reads of x and of P1's terms
    (whole column tiles of every warp, also beyond n1), what an MMA reads of P2's (128 rows), and the chains of sums (none empty)."""
    assert violations(tmp_path, """
    long seen = 0;
    auto check = [&](const RotGeom& g) {
        const int total = g.group_off + g.group_bytes, rows = g.cw * g.ntw * 8;
        const bool ok = total <= kRotMaxSmem && g.group_off + rows * g.s2 <= total && g.p1_off + (g.na * 8 + rows) * g.s1 <= total &&
                        (g.alias_z ? 0 : rows * (g.pad ? g.s2 : 0)) <= g.red_rel && g.red_rel + kRotRedBytes <= g.group_bytes &&
                        g.group_off + g.max_groups * g.group_bytes <= kRotMaxSmem &&
                        (g.group_off | g.group_bytes | g.p1_off | g.z_rel | g.red_rel | g.s1 | g.s2) % 16 == 0 && g.dc * g.dtc * 16 >= g.n2;
        if (!ok) std::printf("%d x %d: cluster %d, %d warps of %d tiles\\n", g.n1, g.n2, g.dc, g.cw, g.ntw);
        return ok;
    };
    for (int n1 = 1; n1 <= 192; ++n1)
        for (int n2 = 8; n2 <= 256; n2 += 8) {
            RotGeom g{};
            if (n1 * n2 % 32 || n1 * n2 > 25600 || !rot_geometry(n1, n2, &g)) continue;
            ++seen;
            if (!check(g)) return 0;
            for (int clusters = 1; clusters <= 148; ++clusters) {
                RotGeom few = g;
                if (few_tokens_geometry(g, clusters % 2 == 0, &few, [&](const RotGeom& t) { return clusters * t.dc <= 148; }) && (clusters * few.dc > 148 || !check(few))) return 0;
            }
            if (rot_okt_factors(g) && (n1 > 128 || n2 > 128 || rot_mma_always(g))) { std::printf("%d x %d: okt_umma.cu does not take them\\n", n1, n2); return 0; }
            for (int size = 1; size <= 2; ++size) {
                RotUmmaGeom u{};
                if (!rot_umma_geometry(g, size, &u)) continue;
                const int ks2 = n2 / 16, ks1 = u.nc / 16;
                if (u.total > kRotMaxSmem || u.p1_off - u.dt * 64 + 128 * 64 > u.total || 3 * u.ntot > 512 || u.dc * u.dt < n2 ||
                    (ks2 + 1) / 2 >= ks2 || (ks1 + 1) / 2 >= ks1) { std::printf("%d x %d on tcgen05\\n", n1, n2); return 0; }
            }
        }
    if (seen < 2000) std::printf("only %ld pairs\\n", seen);""") == ""


def test_operands_of_the_rotation_with_rows_on_the_lanes_lie_inside_the_block(tmp_path):
    """What its MMAs read of P1's terms (128 rows from any atom, and from 64 rows before them for a step's second token), its tensor memory and
    shared memory, every column with a warp, no empty chain of sums; one x, and fp32 rows."""
    assert violations(tmp_path, """
    long seen = 0;
    for (int n1 = 1; n1 <= 192; ++n1)
        for (int n2 = 8; n2 <= 256; n2 += 8)
            for (int size = 0; size <= 2; ++size)
                for (int terms = 1; terms <= 3; terms += 2) {
                    RotRowsGeom g{};
                    if (!rot_rows_geometry(n1, n2, size, &g, terms)) continue;
                    ++seen;
                    for (int xb = g.xb; xb >= 1; --xb) {
                        RotRowsGeom one = g;
                        const bool ok = rot_rows_places(one, xb, terms) && one.total <= kRotMaxSmem && one.x_off - one.lanes * 64 + 128 * 64 <= one.total &&
                                        one.p1_off >= (one.tps - 1) * 64 * 64 && (one.p1_off | one.x_off) % 1024 == 0 && (2 * one.nv + 2) * n2 <= 512 &&
                                        one.groups * one.chunks * 16 >= n2 && (one.groups - 1) * one.chunks * 16 < n2 && one.groups <= 5 && one.tps * one.lanes == 128 &&
                                        one.lanes >= n1 && one.ks1 >= 3 && one.ks1 <= 8 && one.ks2 >= 2 && one.ks2 <= 8 && one.ks2 * 16 == n2 &&
                                        one.st_off + (one.staged ? 2 * one.out_bytes : 0) <= one.sh_off && (n1 * n2 % 32 != 0 || one.out_bytes % 16 == 0);
                        if (!ok) { std::printf("%d x %d, %d bytes, %d terms\\n", n1, n2, size, terms); return 0; }
                    }
                }
    if (seen < 1000) std::printf("only %ld\\n", seen);""") == ""


def test_a_rotation_that_takes_all_tensor_memory_has_one_block_an_sm(tmp_path):
    """Whatever registers and shared memory would let stay: the problems' blocks together are no more than the SMs, every problem has one
    and none more than it has steps."""
    assert violations(tmp_path, """
    for (int sms : {1, 4, 132, 148})
        for (int per_sm = 1; per_sm <= 4; ++per_sm)
            for (int n = 1; n <= 4; ++n)
                for (long steps : {1L, 2L, 36L, 37L, 49L, 74L, 148L, 149L, 1000L}) {
                    const int ctas = rot_rows_ctas(per_sm * sms, sms, n, steps);
                    if (ctas * n > sms || ctas > steps || (n <= sms && ctas < 1)) { std::printf("%d SMs, %d an SM, %d problems, %ld steps: %d\\n", sms, per_sm, n, steps, ctas); return 0; }
                }""") == ""


def test_the_launch_asks_that_plan():
    """The rows kernel's grid comes from rot_rows_ctas and from nowhere else."""
    text = open(os.path.join(ROOT, "paper_2605_00422_b200", "csrc", "rot_rows.cu")).read()
    assert text.count("p.ctas_per_problem = ") == 1 and "p.ctas_per_problem = rot_rows_ctas(" in text


def test_the_rotation_with_rows_on_the_lanes_takes_no_factors_that_are_more_exact_elsewhere(tmp_path):
    """T = V x in the same launch kept factors of up to 80 rows on the warp-level kernel unless it had more exact ones to offer: 64 x 128 1.44e-7 of a
    row's 2-norm against 1.55e-7.  Up to 80 rows, and for bf16 values, the other kernel is rot_umma.cu: the second contraction has three chains of sums."""
    assert violations(tmp_path, """
    long window = 0;
    for (int n1 = 33; n1 <= 128; ++n1)
        for (int n2 = 32; n2 <= 128; n2 += 16) {
            RotGeom g{};
            RotRowsGeom rows{};
            if (n1 * n2 % 32 || !rot_geometry(n1, n2, &g) || !rot_rows_geometry(n1, n2, 1, &rows)) continue;
            const bool larger = n1 <= 80 && (n1 > 64 || n2 > 80);
            window += larger;
            RotRowsGeom values{};
            if (rot_rows_exact(g, true) == larger || !rot_rows_exact(g, false) || (n1 <= 80 && n2 > 32 && rows.y_chains != 3) ||
                (rot_rows_geometry(n1, n2, 2, &values) && n2 > 32 && values.y_chains != 3)) { std::printf("%d x %d\\n", n1, n2); return 0; }
        }
    if (window < 100) std::printf("only %ld\\n", window);""") == ""


def test_which_kernel_rotates(tmp_path):
    """The rule's two sides at its lines, on 148 SMs: r(factors, values, raw, T beside, T first, tokens x linears) and c(factors, T first, tokens,
    SMs of either kernel)."""
    got = violations(tmp_path, """
    auto geom = [](int n1, int n2) { RotGeom g{}; if (!rot_geometry(n1, n2, &g)) std::printf("no geometry "); return g; };
    auto r = [&](int n1, int n2, bool values, bool raw, bool beside, bool first, long t) {
        std::printf("%d", (int)rot_rows_faster(geom(n1, n2), values, raw, beside, first, t, 148));
    };
    auto c = [&](int n1, int n2, bool first, long t, int few, int behind) { std::printf("%d", (int)rot_rows_crowded(geom(n1, n2), first, t, few, behind, 148)); };
    for (long t : {149, 259, 260, 296, 297, 370, 371}) { r(64, 64, 0, 0, 0, 0, t); r(64, 64, 0, 1, 0, 0, t); r(64, 80, 0, 0, 0, 1, t); }
    std::printf(" ");
    for (long t : {150, 185, 186, 256}) { r(64, 64, 0, 0, 1, 0, t); r(64, 80, 0, 0, 1, 0, t); }
    std::printf(" ");
    for (long t : {444, 445, 592, 593}) { r(48, 64, 0, 0, 0, 0, t); r(48, 64, 1, 0, 0, 0, t); r(48, 80, 0, 0, 0, 0, t); r(64, 80, 1, 0, 0, 0, t); }
    std::printf(" ");
    for (long t : {149, 4096}) { r(47, 80, 0, 0, 0, 0, t); r(64, 48, 0, 0, 0, 0, t); r(48, 80, 1, 0, 0, 0, t); r(64, 64, 1, 0, 0, 0, t); r(64, 128, 0, 1, 0, 0, t); r(128, 64, 0, 0, 0, 0, t); }
    std::printf(" ");
    for (long t : {149, 222, 223}) { r(80, 64, 0, 0, 0, 0, t); r(72, 96, 0, 0, 0, 0, t); r(72, 96, 1, 0, 0, 0, t); }
    std::printf(" ");
    c(64, 80, 0, 20, 20, 128); c(64, 80, 0, 25, 25, 128); c(64, 80, 0, 64, 64, 140); c(64, 80, 0, 64, 64, 141); c(64, 80, 0, 17, 17, 146); c(64, 80, 0, 4, 4, 144); c(64, 80, 0, 5, 5, 144);
    std::printf(" ");
    c(64, 64, 0, 2, 2, 148); c(64, 64, 0, 3, 3, 148); c(64, 64, 0, 50, 25, 0); c(64, 80, 1, 128, 128, 40); c(64, 80, 1, 129, 129, 40); c(64, 64, 1, 140, 70, 148);
    c(64, 128, 0, 50, 50, 128); c(64, 48, 0, 50, 50, 128);""")
    assert got.split() == ["111111101101001001111", "11110101", "0000001100111111", "000111000111", "000000101", "0110001", "01001000"], got


def test_which_kernel_binarises(tmp_path):
    got = violations(tmp_path, """
    auto b = [](int n1, int n2, bool f32, long rows) { RotGeom g{}; rot_geometry(n1, n2, &g); std::printf("%d", (int)rot_rows_binarizes(g, f32, rows, 148)); };
    for (int f32 = 0; f32 < 2; ++f32) { b(64, 64, f32, 74); b(64, 64, f32, 75); b(48, 64, f32, 4000); b(48, 80, f32, 4000); b(56, 48, f32, 4000); b(48, 48, f32, 4000); b(64, 32, f32, 4000); b(64, 128, f32, 4000); std::printf(" "); }""")
    assert got.split() == ["01111000", "01011000"], got
