"""The planes' layer forward (cc_linear_planes.cu): its launch plans, walked on the host.  No plan may ask for more shared memory or
tensor memory than there is, longer chains than allowed, or blocks without work; the layers that the GPU tests give it are layers it takes."""
import os
import subprocess

# M, d_out, d_in, g, K, 4-bit codebook: layers for the planes; coordinates a look-up and stages that their plans have on 148 SMs.
LAYERS = [
    ((65, 3134, 640, 1, 65536, False), (1, 2)), ((200, 3000, 2760, 4, 65536, False), (1, 2)), ((256, 2050, 4160, 4, 65536, False), (1, 2)),
    ((33, 10000, 1300, 6, 65500, False), (1, 4)), ((48, 14000, 1100, 7, 65536, False), (1, 4)),
    ((91, 244, 453, 9, 30917, False), (2, 2)), ((129, 793, 523, 2, 25467, False), (2, 2)), ((256, 1030, 2800, 8, 32768, False), (2, 2)),
    ((70, 1030, 1200, 8, 32768, True), (2, 2)), ((192, 1030, 1200, 4, 16384, True), (2, 4)), ((12, 903, 1300, 9, 3000, False), (2, 4)),
    ((129, 453, 895, 2, 968, False), (2, 4)), ((60, 1030, 1025, 2, 20000, False), (2, 4)),
    # the last whole stage is the first of a block of the grid, in_features end behind it
    ((26, 1085, 4491, 16, 19780, False), (4, 2)), ((91, 260, 2380, 16, 17185, False), (4, 2)),
    ((192, 202, 3008, 3, 8722, False), (4, 2)), ((255, 212, 2827, 3, 7899, False), (4, 2)), ((192, 568, 1920, 4, 8753, True), (4, 2)),
    ((16, 514, 1000, 4, 300, False), (4, 4)), ((128, 777, 900, 4, 3000, False), (4, 4)), ((129, 737, 1088, 4, 858, True), (4, 4)),
    ((6, 207, 64, 16, 22, False), (4, 4)),
]

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2503_13089_b200", "csrc")

WALK = r"""
#include <cstdio>
#include <initializer_list>
#include "cc_linear_plan.h"

int main() {
    long plans = 0, bad = 0;
    const int64_t layers[][2] = {{28672, 8192}, {11008, 4096}, {128256, 4096}, {4096, 4096}, {1024, 11008}, {700, 900}, {1, 1}, {65, 30000}, {512, 513}};
    const int tokens[] = {1, 5, 16, 17, 33, 48, 64, 65, 100, 128, 192, 255, 256};
    const int books[] = {1, 2, 300, 4096, 12287, 12288, 16384, 24575, 32768, 32769, 50000, 65535, 65536};
    for (const auto& l : layers)
        for (int g = 1; g <= 16; ++g)
            for (int M : tokens)
                for (int K : books)
                    for (int chain : {1, 3, 16}) {
                        const PlanesPlan p = planes_plan(M, l[0], l[1], 148, K, g, chain);
                        const int chunks = (int)((l[1] + 63) / 64);
                        const size_t table = ((size_t)K * p.PP * 2 + 15) / 16 * 16;
                        bool ok = p.fits && p.PP * p.groups >= g && p.PP * (p.groups - 1) < g && p.NT >= M && p.NT % 16 == 0 && p.nt_cols >= p.NT &&
                                  p.nt_cols % 32 == 0 && 2 * p.nt_cols <= p.tmem_cols && p.tmem_cols <= 512 && (p.stages == 2 || p.stages == 4);
                        ok = ok && p.smem <= PL_SMEM && p.smem >= table + p.stages * (size_t)(128 * 64 * 2 + p.NT * 128) + PL_HEAD;
                        const int64_t out_groups = (l[0] + g - 1) / g, items = (int64_t)p.tiles * p.splits;
                        ok = ok && (int64_t)p.tiles * (128 / p.PP) >= out_groups && p.ctas >= 1 && p.ctas <= items && p.ctas * p.groups <= 148;
                        ok = ok && p.splits >= 1 && p.splits <= chunks && (chunks + p.splits - 1) / p.splits <= chain;
                        ok = ok && p.bytes == p.x_bytes + (size_t)p.groups * items * p.NT * 512 && p.x_bytes == (size_t)p.NT * chunks * 128;
                        ++plans;
                        if (!ok && bad++ < 10)
                            printf("M=%d %ldx%ld g=%d K=%d chain=%d: PP %d groups %d ctas %d tiles %d splits %d NT %d stages %d smem %zu\n", M, (long)l[0],
                                   (long)l[1], g, K, chain, p.PP, p.groups, p.ctas, p.tiles, p.splits, p.NT, p.stages, p.smem);
                    }
    printf("%ld plans, %ld bad\n", plans, bad);
    return bad != 0;
}
"""


def test_no_plan_of_the_planes_exceeds_its_limits(tmp_path):
    src, exe = tmp_path / "walk.cpp", tmp_path / "walk"
    src.write_text(WALK)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], stdout=subprocess.PIPE, text=True)
    assert out.returncode == 0, out.stdout


def test_the_layers_of_the_gpu_tests_take_the_planes(tmp_path):
    rows = "\n".join("    {%s}," % ", ".join(str(int(v)) for v in layer + plan) for layer, plan in LAYERS)
    src, exe = tmp_path / "layers.cpp", tmp_path / "layers"
    src.write_text("#include <cstdio>\n#include \"cc_linear_plan.h\"\nstatic const int L[][8] = {\n%s\n};\n" % rows + r"""
int main() {
    int bad = 0;
    for (const auto& l : L)
        for (int words = 0; words < 2; ++words) {
            const PlanesPlan p = planes_for(l[0], l[1], l[2], 148, l[4], l[3], l[5]);
            if (!p.fits || p.PP != l[6] || p.stages != l[7] || gemv_for(l[0], l[1], l[2], 148, l[4], l[3], l[5], words).fits) {
                printf("M=%d %dx%d g=%d K=%d q4=%d: fits %d, PP %d, stages %d\n", l[0], l[1], l[2], l[3], l[4], l[5], p.fits, p.PP, p.stages);
                ++bad;
            }
        }
    return bad != 0;
}
""")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], stdout=subprocess.PIPE, text=True)
    assert out.returncode == 0, out.stdout


REQUESTS = r"""
#include <cstdio>
#include <vector>
#include "cc_linear_plan.h"

// The look-up threads' requests in the order of linear_planes_kernel: the first block of a thread's first stage before the loop, in the loop
// always the next one; `item` starts at any stage.  No request may lie past the layer, and every in_feature has to have been asked for.
int main() {
    long asked = 0, bad = 0;
    for (int PP = 1; PP <= 4; PP *= 2)
        for (int stages = 2; stages <= 4; stages += 2)
            for (int d_in : {1, 7, 8, 63, 64, 65, 72, 127, 128, 130, 191, 192, 200, 256, 515, 4491, 2380})
                for (int from = 0; from < (d_in + 63) / 64; ++from) {
                    const int chunks = (d_in + 63) / 64, pairs = 64 / PP, threads = PL_LOOK_WARPS / stages * 32;
                    std::vector<int> seen((size_t)pairs * d_in, 0);
                    auto request = [&](int stage, const PlaneShare& t, int block) {
                        if (!plane_has_block(t.step, block)) return;
                        for (int r = 0; r < 8; ++r) {
                            const int i = stage * 64 + block * 8 + r;
                            if ((stage + 1) * 64 > d_in && i >= d_in) break;       // a stage that is not whole is looked at row by row
                            ++asked;
                            if (i < 0 || i >= d_in || i >= (stage + 1) * 64) { if (bad++ < 10) printf("PP=%d stages=%d d_in=%d: row %d\n", PP, stages, d_in, i); }
                            else ++seen[(size_t)t.pair * d_in + i];
                        }
                    };
                    for (int sg = 0; sg < stages; ++sg)
                        for (int thread = 0; thread < threads; ++thread) {
                            const PlaneShare t = plane_share(PP, stages, thread);
                            int c = from + sg;
                            if (t.pair < 0 || t.pair >= pairs || t.step < 1) { ++bad; continue; }
                            if (c < chunks) request(c, t, t.first);
                            for (; c < chunks; c += stages)
                                for (int b = t.first; b < 8; b += t.step) {
                                    if (b + t.step < 8) request(c, t, b + t.step);
                                    else if (c + stages < chunks) request(c + stages, t, t.first);
                                }
                        }
                    for (size_t e = 0; e < seen.size(); ++e)
                        if (seen[e] != ((int)(e % d_in) >= from * 64 ? 1 : 0) && bad++ < 10) printf("PP=%d stages=%d d_in=%d: %d times\n", PP, stages, d_in, seen[e]);
                }
    printf("%ld requests, %ld bad\n", asked, bad);
    return bad != 0;
}
"""


def test_no_look_up_thread_asks_for_codes_past_the_layer(tmp_path):
    src, exe = tmp_path / "requests.cpp", tmp_path / "requests"
    src.write_text(REQUESTS)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], stdout=subprocess.PIPE, text=True)
    assert out.returncode == 0, out.stdout
