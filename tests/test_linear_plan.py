"""The few-token layer forward's launch plan, walked on the host: no plan may ask for more shared memory than its kernel's limit,
more slabs than the scratch is sized for, or slices that leave out a row of the codebook; the padded codebook starts where its widest
load may, whatever the workspace starts at.  Numbers of centroids are taken
densely around the ends of every slice, where rounding to whole groups of 16 rows decides."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2503_13089_b200", "csrc")

WALK = r"""
#include <cstdio>
#include "cc_linear_plan.h"

static long plans = 0, bad = 0;

static void check(int64_t d_out, int64_t d_in, int g, int M, int K, bool quant, bool words) {
    if (!gemv_applies(M, K, g, quant)) return;
    const int mt = gemv_pad(M);
    const GemvPlan p = gemv_plan(d_in, (int)((d_out + g - 1) / g), 148, K, g, mt, quant, words);
    const size_t row = gemv_row_bytes(g, quant);
    const int step = gemv_batch(g, mt) * LG_SUB;
    const size_t x = (size_t)((p.rows_per_split + step - 1) / step * step) * mt * 4;
    const size_t table = (size_t)p.slice_rows * row + gemv_tail_bytes(g, quant);
    const bool ok = p.fits && p.smem <= (size_t)LG_SMEM && LG_HEAD + x + table <= p.smem &&
                    (p.slice_rows * row) % 16 == 0 && p.slices >= 1 && p.slices <= LG_SLICES_MAX && (!quant || p.slices == 1) &&
                    (int64_t)p.slices * p.slice_rows >= K && (int64_t)(p.slices - 1) * p.slice_rows < K &&
                    (int64_t)p.splits * p.rows_per_split >= d_in && (int64_t)(p.splits - 1) * p.rows_per_split < d_in &&
                    (int64_t)p.splits * p.slices <= gemv_slabs_most(d_out, d_in, 148);
    ++plans;
    if (!ok && bad++ < 10)
        printf("M=%d %ldx%ld g=%d K=%d quant=%d: %d x %d rows, %d splits of %d, %zu bytes\n", M, (long)d_out, (long)d_in, g, K, quant,
               p.slices, p.slice_rows, p.splits, p.rows_per_split, p.smem);
}

int main() {
    const int64_t layers[][2] = {{28672, 4096}, {28672, 8192}, {11008, 2048}, {8192, 2048}, {14336, 2048}, {128256, 4096}, {11008, 4096},
                                 {32000, 4096}, {4096, 4096}, {1024, 4096}, {700, 900}, {1, 1}, {65, 100003}};
    for (const auto& l : layers)
        for (int g = 1; g <= 16; ++g)
            for (int quant = 0; quant <= (g % 2 ? 0 : 1); ++quant) {
                const int most = gemv_slice_most(g, quant), k_max = quant && 131072 / (g / 2) < 65536 ? 131072 / (g / 2) : 65536;
                for (int K = 1; K <= k_max; ++K) {
                    bool edge = K <= 17 || K > k_max - 17 || K % 997 == g;
                    for (int n = 1; n <= 5; ++n) edge |= K > n * most - 40 && K < n * most + 40;
                    if (!edge) continue;
                    for (int M = 1; M <= 4; ++M) check(l[0], l[1], g, M, K, quant, (K + M) % 2);
                }
            }
    // more in_features than a grid has rows of blocks for: the plan says so
    const GemvPlan far = gemv_plan((int64_t)1 << 30, 1, 148, 100, 1, 1, false, false);
    if (far.fits) { printf("a plan of %d splits fits\n", far.splits); ++bad; }
    // the padded codebook: rows of 16 values are loads of 32 bytes, a workspace starts on any 16-byte boundary
    const size_t from = 4096, to = from + 65536 * 32;
    for (uintptr_t ws = 1 << 20; ws < (1 << 20) + 256; ws += 16)
        for (int K = 1; K <= 65536; K += K < 65000 ? 97 : 1)
            for (int pad = 4; pad <= 16; pad *= 2) {
                const size_t at = padded_table_at(ws, from, to, K, pad);
                const bool must = from + 16 + (size_t)K * pad * 2 <= to;
                if (at ? (ws + at) % 32 || at < from || at + (size_t)K * pad * 2 > to : must) { printf("table at %zu, K=%d pad=%d\n", at, K, pad); ++bad; }
            }
    printf("%ld plans, %ld bad\n", plans, bad);
    return bad || plans < 100000;
}
"""


def test_no_plan_of_the_few_token_forward_exceeds_its_limits(tmp_path):
    src, exe = tmp_path / "walk.cpp", tmp_path / "walk"
    src.write_text(WALK)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], stdout=subprocess.PIPE, text=True)
    assert out.returncode == 0, out.stdout
