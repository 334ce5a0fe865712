// Host-side plans of the layer forward: the few-token kernel's launch, the tensor kernel's (both cc_linear.cu), the one by planes
// (cc_linear_planes.cu), the place of the padded codebook.  No CUDA in here: what a plan asks for can be checked against the kernels'
// limits without a device.
#pragma once

#include <stddef.h>
#include <stdint.h>

#ifdef __CUDACC__
#define CC_PLAN_FN __host__ __device__
#else
#define CC_PLAN_FN
#endif

// ---- Layer forward plane by plane (cc_linear_planes.cu).
// PP: coordinates side by side in a table row; groups: plane groups (a table each); ctas: per plane group; an item is a tile of
// 128 / PP code groups and one of `splits` parts of the in_features.
struct PlanesPlan { int PP, groups, ctas, tiles, splits, NT, nt_cols, stages, tmem_cols; size_t smem, x_bytes, bytes; bool fits; double clocks; };

namespace {

constexpr int LG_THREADS = 1024, LG_GRPS = 64, LG_SUB = 16, LG_M_MAX = 4;
constexpr int LG_SMEM = 226 * 1024;                    // bytes of shared memory the kernel may have
constexpr int LG_HEAD = 128;                           // barrier, flag, 4-bit levels
constexpr int LG_X_MAX = 16 * 1024;                    // bytes of x (FP32) beside the table
constexpr int LG_SLICES_MAX = 4;
constexpr int LG_SPLITS_MAX = 65535;                   // gridDim.y

// Rows of codes a thread requests together; the next ones are under way while these are used.
CC_PLAN_FN constexpr int gemv_batch(int g, int mt) { return g * mt <= 8 ? 8 : 4; }
// Neighbouring code groups per thread: two codes come in one word and share the loads of x.  For short rows of the FP16
// codebook and layers of many codes (calls back to back, codes in L2): one token, g = 4, K = 65536, 11008 x 4096 39.8 -> 33.7 us, 4096 x
// 4096 18.7 -> 17.2;
// with few codes the wider exchange at the end costs more (g = 3, 700 x 900 7.7 -> 9.3; g = 8, 4096 x 4096 16.2 -> 17.1).
constexpr bool gemv_pair(int g, bool quant) { return g <= 4 && !quant; }
constexpr int64_t LG_PAIR_FROM = 1 << 21;              // codes

// Bytes of a codebook row, and of what lies behind the rows of a slice: a row of zeros and a word that the loads of odd rows
// may touch.
constexpr size_t gemv_row_bytes(int g, bool quant) { return quant ? (size_t)(g / 2) : (size_t)(2 * g); }
constexpr size_t gemv_tail_bytes(int g, bool quant) { return quant ? 0 : gemv_row_bytes(g, quant) + 4; }

// Rows of a slice: whole groups of 16 (so that a slice starts on a 16-byte boundary), as many as leave room for a full x.
constexpr int gemv_slice_most(int g, bool quant) {
    return (int)((LG_SMEM - LG_HEAD - LG_X_MAX - 15 - gemv_tail_bytes(g, quant)) / gemv_row_bytes(g, quant) / 16 * 16);
}

// Where the look-up kernel is the faster one.  M x g accumulators must fit the registers of 1024 threads per SM; the
// FP16 codebook is read once per slice, which costs the less the fewer gathers it saves (4096 x 4096: g = 4, K = 65536
// 26.9 -> 18.4 us at one token, 26.7 -> 25.7 at four; g = 6, K = 65500, four slices 30.8 -> 22.2 at one, on 11008 x 4096
// 98 -> 94 at four, where the tensor kernel with padded rows takes 70; g = 16, K = 20000, three slices, two tokens 20.2
// -> 24.4, not used).
constexpr int gemv_tokens(int g) { return g <= 8 ? 4 : 2; }                  // 4-bit codebook
inline bool gemv_applies(int64_t M, int K, int g, bool quant) {
    if (quant) return M <= gemv_tokens(g);
    return M <= (g <= 4 ? 4 : 2) && K <= (g <= 8 ? LG_SLICES_MAX : 2) * gemv_slice_most(g, false);
}
constexpr int gemv_pad(int64_t M) { return M <= 2 ? (int)M : 4; }

// fits: within what a launch may ask for; pays: not slower than the tensor kernel.  Where not both, that kernel takes the call.
struct GemvPlan { int pw, o_blocks, slices, slice_rows, splits, rows_per_split; size_t smem; bool fits, pays; };

// Whether a plan for the FP16 codebook beats the tensor kernel.  What costs is its end, where one CTA adds up the slabs of a
// block of code groups, eight loads a thread at a time: `tail` counts those rounds.  A layer with few code groups has few
// blocks and many slabs, and the tensor kernel is quick on it where a row of the codebook is one load.  One and two tokens, look-up / tensor
// kernel in us (tail): 1024 x 4096, g = 16, K = 4096 13.7 / 9.5 (19) and 21.1 / 9.5 (38), g = 9, K = 20000 12.0 / 12.2 (10) and 15.9 /
// 12.3 (20); 128 x 4096, K = 256 (19) g = 8 9.7 / 8.8 and 11.1 / 8.8, g = 4 9.1 / 8.8 and 10.9 / 8.8, g = 2 8.5 / 9.4 and 10.0 / 9.4;
// 512 x 512, g = 16, K = 4096 8.7 / 8.3 (2) and 11.2 / 8.5 (4); one token, g = 16: 2048 x 2048, K = 5000 12.0 / 9.6, 700 x 900 9.3 /
// 10.5; four, 1536 x 6144, g = 4, K = 300 14.7 / 12.3 (14).  Slices read every code once more each, which a layer of about a
// million codes does not make up for: 1024 x 4096, g = 4, K = 65536 10.4 / 12.0 and, at four tokens, 13.9 / 12.0, g = 8, K = 20000 10.7 /
// 10.0 and 12.1 / 10.1; but 700 x 900, g = 4, K = 65536, four tokens 10.3 / 14.0.
inline bool gemv_pays(const GemvPlan& p, int64_t d_in, int out_groups, int g, int mt) {
    const int slabs = p.splits * p.slices, groups = out_groups < LG_GRPS * p.pw ? out_groups : LG_GRPS * p.pw;
    const int tail = (slabs + 7) / 8 * ((mt * g * groups + LG_THREADS - 1) / LG_THREADS);
    if (tail >= 20) return false;
    if (g != 4 && g != 8 && g != 16) return true;                           // several loads a row, or two values
    if (mt * g >= 8 && tail >= 14) return false;
    if (g == 16 && p.o_blocks <= 2 && (mt > 1 || d_in % 8 == 0)) return false;   // x in 16-byte pieces there
    const int64_t codes = out_groups * d_in;
    return !(p.slices > 1 && mt * g * p.slices >= 32 && codes >= 500000 && codes <= 1100000);
}

// Slices of the codebook as its bytes ask for, splits of the in_features by a count of clocks: a CTA pays for its
// table (about 40 bytes a clock), some 4000 for its beginning and end, and 8 a row of codes (16 where a thread has two
// groups); CTAs come in waves of one per SM.  mt: tokens rounded up to 1, 2 or 4; words: the codes start on a word boundary.
inline GemvPlan gemv_plan(int64_t d_in, int out_groups, int sm_count, int K, int g, int mt, bool quant, bool words) {
    GemvPlan p;
    p.pw = (words && out_groups % 2 == 0 && gemv_pair(g, quant) && out_groups * d_in >= LG_PAIR_FROM) ? 2 : 1;
    p.o_blocks = (out_groups / p.pw + LG_GRPS - 1) / LG_GRPS;
    const size_t row = gemv_row_bytes(g, quant);
    const int slice_most = gemv_slice_most(g, quant);
    p.slices = (K + slice_most - 1) / slice_most;
    p.slice_rows = ((K + p.slices - 1) / p.slices + 15) / 16 * 16;          // at most slice_most
    p.slices = (K + p.slice_rows - 1) / p.slice_rows;
    const int step = gemv_batch(g, mt) * LG_SUB, rows_max = LG_X_MAX / (4 * mt) / step * step;
    const int ctas = p.o_blocks * p.slices;
    int most = 3 * sm_count / ctas, least = (int)((d_in + rows_max - 1) / rows_max);
    if ((int64_t)most * LG_SUB > d_in) most = (int)((d_in + LG_SUB - 1) / LG_SUB);   // at least 16 in_features per CTA
    if (most < least) most = least;
    double best = 0.0;
    p.splits = 0;
    for (int s = least; s <= most; ++s) {
        const int64_t rows = (d_in + s - 1) / s;
        const double t = (double)(((int64_t)ctas * s + sm_count - 1) / sm_count) * ((double)(p.slice_rows * row) / 40.0 + 4000.0 + 8.0 * p.pw * (double)rows);
        if (p.splits == 0 || t < best) { best = t; p.splits = s; }
    }
    p.rows_per_split = (int)((d_in + p.splits - 1) / p.splits);
    p.splits = (int)((d_in + p.rows_per_split - 1) / p.rows_per_split);
    size_t table = (size_t)p.slice_rows * row + gemv_tail_bytes(g, quant);
    const size_t red = (size_t)(LG_SUB - 1) * g * p.pw * LG_GRPS * 4;       // the exchange takes the table's place
    if (table < red) table = red;
    p.smem = LG_HEAD + (size_t)((p.rows_per_split + step - 1) / step * step) * mt * 4 + (table + 15) / 16 * 16;
    p.fits = p.smem <= (size_t)LG_SMEM && p.splits <= LG_SPLITS_MAX;
    p.pays = quant || gemv_pays(p, d_in, out_groups, g, mt);
    return p;
}

// The plan with which the look-up kernel takes a call; .fits is false where it does not.
inline GemvPlan gemv_for(int64_t M, int64_t d_out, int64_t d_in, int sm_count, int K, int g, bool quant, bool words) {
    GemvPlan p = {};
    if (!gemv_applies(M, K, g, quant)) return p;
    p = gemv_plan(d_in, (int)((d_out + g - 1) / g), sm_count, K, g, gemv_pad(M), quant, words);
    p.fits = p.fits && p.pays;
    return p;
}

// Slabs of partial sums that any plan of such a layer may write: three CTAs per SM at the most, or as many splits as x asks
// for.  The most come with the fewest blocks of code groups, i.e. at g = 16.
inline int64_t gemv_slabs_most(int64_t d_out, int64_t d_in, int sm_count) {
    const int o_blocks = (int)((d_out / 32 + LG_GRPS - 1) / LG_GRPS);
    const int64_t least = LG_SLICES_MAX * ((d_in + 511) / 512);
    const int64_t most = 3 * sm_count / (o_blocks < 1 ? 1 : o_blocks) + LG_SLICES_MAX;
    return most > least ? most : least;
}

// Where a copy of the codebook with rows of `pad` values goes between byte `from` and byte `to` of a workspace at address `ws`,
// which need only be on a 16-byte boundary while a row of 16 values is one load of 32 bytes: its offset, or 0 if it does not fit.
inline size_t padded_table_at(uintptr_t ws, size_t from, size_t to, int K, int pad) {
    const size_t at = ((ws + from + 31) & ~(uintptr_t)31) - ws;
    return at + (size_t)K * pad * 2 <= to ? at : 0;
}

// ---- The tensor kernel.
constexpr int LM = 128;                 // out_features per CTA = MMA M = TMEM lanes
constexpr int LKB = 64;                 // in_features per pipeline stage
constexpr int LSTAGES = 4;              // at most; two where the 4-bit table leaves room for no more wide tiles
constexpr int LPROD = 512;              // producer threads (16 warps); warps 0..3 also run the epilogue
constexpr int LTHREADS = LPROD + 32;    // + the MMA warp
constexpr int LNT_MAX = 256;            // tokens per CTA = MMA N
// Operand tiles in shared memory: the K-major no-swizzle layout of 8 x 16-byte core matrices, with the two
// strides of the descriptor chosen against bank conflicts of the producers' 16-byte stores.  Neighbouring
// lanes of an A-tile store hold neighbouring code groups, i.e. rows g apart in one column of core matrices:
// 144 instead of 128 bytes between 8-row groups puts row r at 16-byte slot 9 (r / 8) + r % 8, and the eight
// lanes of a store phase then fall into eight different slots mod 8 for g = 2, 4, 8 (two by two for g = 16;
// at 128 bytes they all shared one or two).  Neighbouring lanes of a B-tile store hold neighbouring
// 8-column pieces of one token's row: 16 bytes more between the columns of core matrices does the same.
// Measured (4096 x 4096, g 4, K 65536): the B stride alone 0.772 -> 0.585 ms at 4096 tokens, 64 -> 50 us at
// 256; the A stride on top 35.7 -> 33.6 us at 64 tokens (87 -> 64 us at g = 8 on 8192 x 8192, 16 tokens) but
// 0.585 -> 0.807 ms at 4096 tokens, where the MMA's own reads of the wider-spaced A tile come to matter:
// the A tile is widened for token blocks of at most 64 only, and never beside the 4-bit table (no room).
CC_PLAN_FN constexpr int a_sbo(bool pad) { return pad ? 144 : 128; }
CC_PLAN_FN constexpr int a_lbo(bool pad) { return (LM / 8) * a_sbo(pad); }
CC_PLAN_FN constexpr int a_stage(bool pad) { return (LKB / 8) * a_lbo(pad); }   // bytes
CC_PLAN_FN constexpr int b_lbo(int nt) { return nt * 16 + 16; }
CC_PLAN_FN constexpr int b_stage_bytes(int nt) { return (LKB / 8) * b_lbo(nt); }
// Quantised codebook (4 bits per value, two values per byte, low nibble first; Section 5.3): the whole
// table sits in shared memory, and a 256-entry table turns a byte into its two dequantised FP16 values.
constexpr int LQ_TABLE_MAX = 128 * 1024;   // bytes of packed codebook that fit beside the stages
constexpr int LQ_BULK_PIECE = 32 * 1024;   // bytes per bulk copy of the table
constexpr int LQ_WIDE_FROM = 256;
constexpr int LQ_NT_MAX = 64;              // tokens per CTA when the table takes most of the shared memory

constexpr int LINEAR_SPLITS_MORE = 8;   // splits beyond those that fill the SMs once are tried up to this many

struct LinearPlan { int NT, a_pad, stages, tmem_cols, o_tiles, tok_blocks, splits, chunks_per_split, fill; size_t smem; };   // fill: splits that fill the SMs once

// nt_max: tokens per CTA (256, or 64 with a quantised codebook in shared memory); table_bytes: that codebook.
inline LinearPlan linear_plan(int64_t M, int64_t d_out, int64_t d_in, int sm_count, int nt_max = LNT_MAX, size_t table_bytes = 0,
                       int g = 4) {
    LinearPlan p;
    const int64_t mt = M < nt_max ? M : nt_max;
    p.NT = (int)((mt + 15) / 16 * 16);
    // FP16 codebook with rows of at most 8 bytes, many tokens (of a layer too narrow for cc_linear_wide.cu, which the figures here
    // were taken before): the gathers of the weight tile bound a stage, so
    // one tile serves 512 tokens (two MMAs of 256 columns, all 512 TMEM columns) and the pipeline has two stages
    // of that size: 4096 x 4096, g 4, 4096 tokens 0.571 -> 0.464 ms.  With 16-byte rows (g = 8) there are half as
    // many gathers per weight and the coarser grid costs more than the reuse saves (1.62 -> 1.70 ms on 8192 x 8192).
    const bool wide = table_bytes == 0 && nt_max == LNT_MAX && M >= 2 * LNT_MAX && g <= 4;
    if (wide) p.NT = 2 * LNT_MAX;
    p.tmem_cols = 32;
    while (p.tmem_cols < p.NT) p.tmem_cols *= 2;
    p.o_tiles = (int)((d_out + LM - 1) / LM);
    p.tok_blocks = (int)((M + p.NT - 1) / p.NT);
    const int chunks = (int)((d_in + LKB - 1) / LKB);
    int splits = sm_count / (p.o_tiles * p.tok_blocks);             // fill the SMs when there are few tiles
    if (splits > chunks / 4) splits = chunks / 4;                   // at least four stages of work per CTA
    if (splits < 1) splits = 1;
    p.fill = splits;
    // More splits where the last wave would leave most SMs idle (86 tiles on 148 SMs: five splits make 2.9 waves of a
    // fifth each; 33 tokens, 11008 x 4096, g = 6: 80 -> 62 us): clocks of a wave count as its stages, two stages' worth of
    // setting up, and the slabs' traffic.  A stage is 8192 / g gathers at 0.73 a clock.
    const double stage_clk = 8192.0 / g / 0.73 + 4.0 * p.NT, slab_clk = (double)M * (double)d_out * 8.0 / 2000.0;
    double least = 0.0;
    const int most = chunks / 4 < LINEAR_SPLITS_MORE ? chunks / 4 : LINEAR_SPLITS_MORE;
    for (int cand = splits; cand <= most || cand == splits; ++cand) {
        const int cps = (chunks + cand - 1) / cand, real = (chunks + cps - 1) / cps;
        const int64_t ctas = (int64_t)p.o_tiles * p.tok_blocks * real;
        const double t = (double)((ctas + sm_count - 1) / sm_count) * (cps + 2) * stage_clk + (real > 1 ? 4000.0 + real * slab_clk : 0.0);
        if (cand == splits || t < 0.95 * least) { least = t; p.splits = real; p.chunks_per_split = cps; }
    }
    p.a_pad = (table_bytes == 0 && p.NT <= 64) ? 1 : 0;
    p.stages = (wide || (table_bytes != 0 && p.NT > LQ_NT_MAX)) ? 2 : LSTAGES;
    p.smem = (size_t)p.stages * (a_stage(p.a_pad) + (size_t)b_stage_bytes(p.NT)) + 256;
    if (table_bytes) p.smem += 1024 + (table_bytes + 15) / 16 * 16;
    return p;
}

// Tokens from which decoding the weight once and multiplying it afterwards (cc_linear_wide.cu) is the faster way, gathering /
// decoding in us: 4096 x 4096, g = 4, K = 65536, 128 tokens 42 / 46, 192 tokens 52 / 46, 512 tokens 85 / 52.  Earlier where
// the tiles of this kernel fill the SMs by themselves, so that its waves are the coarser (11008 x 4096, g = 8, 128 tokens
// 95 / 67; g = 6, 33 tokens 83 / about 80).  Later where it splits the in_features and so keeps the SMs busier than the few whole
// tiles of the product do: from 224 tokens on for long in_features and short rows (4096 x 11008, g = 4: K = 256, 192 tokens 58 / 67,
// K = 8000 65 / 71, at 224 tokens 82 / 71; g = 8, K = 16000, 192 tokens 82 / 75), from 256 on for the 4-bit codebook in shared
// memory with four splits or more (1024 x 4096, g = 6, 192 tokens 19 / 26, 224 tokens 23 / 26; FP16, 2048 x 2048, eight splits, g = 8,
// 224 tokens 19 / 16).
constexpr int LINEAR_WIDE_FEWEST = 96, LINEAR_WIDE_FROM = 192, LINEAR_WIDE_LONG = 224, LINEAR_WIDE_Q4 = 256;
inline int linear_wide_from(int fill, int64_t d_in, int g, bool quant) {
    if (fill == 1) return LINEAR_WIDE_FEWEST;
    if (quant && fill >= 4) return LINEAR_WIDE_Q4;
    return !quant && fill > 2 && g <= 6 && d_in > 8192 ? LINEAR_WIDE_LONG : LINEAR_WIDE_FROM;
}

// ---- Layer forward plane by plane.
constexpr int PL_ROWS = 128, PL_KB = 64, PL_NT_MAX = 256, PL_SPLITS_MAX = 64;
constexpr size_t PL_SMEM = 226 * 1024, PL_HEAD = 256;
constexpr int PL_LOOK_WARPS = 16;

// How the look-up warps share out a stage.  The warps of a stage are PL_LOOK_WARPS / stages; a thread of them has one pair of
// neighbouring code groups and blocks of eight in_features first, first + step, ...  With four coordinates a look-up and two stages
// there are twice as many threads as blocks: half of them have none, their first is behind the last of the stage.
struct PlaneShare { int pair, first, step; };
CC_PLAN_FN constexpr PlaneShare plane_share(int PP, int stages, int thread) {
    const int pairs = PL_ROWS / PP / 2;
    return {thread % pairs, thread / pairs, PL_LOOK_WARPS / stages * 32 / pairs};
}

// Whether a stage has the block, i.e. whether its codes may be asked for (those of its in_features that exist).
CC_PLAN_FN constexpr bool plane_has_block(int step, int block) { return step <= PL_KB / 8 || block < PL_KB / 8; }

// Clocks of an SM for a stage of 64 in_features: its 2 CW look-ups by 32 lanes take 3.5 clocks each (rows of 2 or 4 bytes) or 6.2
// (8 bytes), half a clock goes to the codes and half to each 16-byte piece of the operand.
constexpr double planes_stage_clocks(int PP) { return 2.0 * (PL_ROWS / PP) * ((PP == 4 ? 6.2 : 3.5) + 0.5 + 0.5 * PP); }

constexpr size_t PL_SLABS_MOST = 48u << 20;           // bytes of partial sums, unless the shortest chains ask for more

// chain: stages of 64 in_features that may be added up in one accumulator.
inline PlanesPlan planes_plan(int64_t M, int64_t d_out, int64_t d_in, int sm_count, int K, int g, int chain) {
    PlanesPlan best = {};
    const int chunks = (int)((d_in + PL_KB - 1) / PL_KB);
    const int out_groups = (int)((d_out + g - 1) / g);
    if (M > PL_NT_MAX) return best;
    for (int PP = 1; PP <= 4; PP *= 2) {
        PlanesPlan p = {};
        p.PP = PP;
        p.groups = (g + PP - 1) / PP;
        if (PP > 1 && p.groups == (g + PP / 2 - 1) / (PP / 2)) continue;      // no fewer tables than with shorter rows
        p.NT = (int)((M + 15) / 16 * 16);
        p.nt_cols = (p.NT + 31) / 32 * 32;
        const size_t table = ((size_t)K * PP * 2 + 15) / 16 * 16, stage = PL_ROWS * PL_KB * 2 + (size_t)p.NT * PL_KB * 2;
        p.stages = 4 * stage + table + PL_HEAD <= PL_SMEM ? 4 : 2;
        p.smem = p.stages * stage + table + PL_HEAD;
        if (p.smem > PL_SMEM) continue;
        p.tmem_cols = 64;
        while (p.tmem_cols < 2 * p.nt_cols) p.tmem_cols *= 2;
        const int cw = PL_ROWS / PP, most_ctas = sm_count / p.groups;
        if (most_ctas < 1) continue;
        p.tiles = (out_groups + cw - 1) / cw;
        int least = (chunks + chain - 1) / chain, most = chunks < PL_SPLITS_MAX ? chunks : PL_SPLITS_MAX;
        if (least < 1) least = 1;
        if (most < least) most = least;
        p.x_bytes = (size_t)p.NT * chunks * (PL_KB * 2);
        p.fits = true;
        for (int s = least; s <= most; ++s) {
            const int64_t items = (int64_t)p.tiles * s;
            const size_t slabs = (size_t)p.groups * items * p.NT * PL_ROWS * 4;
            if (s > least && slabs > PL_SLABS_MOST) break;
            const int rounds = (int)((items + most_ctas - 1) / most_ctas);
            const double t = rounds * ((double)chunks / s * planes_stage_clocks(PP) + 400.0 + 4.0 * p.NT) +
                             (double)s * p.tiles * p.groups * p.NT * PL_ROWS * 8.0 / 4000.0 + (double)table / 50.0;
            if (best.fits && t >= best.clocks) continue;
            p.splits = s;
            p.clocks = t;
            p.ctas = items < most_ctas ? (int)items : most_ctas;
            p.bytes = p.x_bytes + slabs;
            best = p;
        }
    }
    return best;
}

// Whether the planes' three launches beat the kernels they stand in for.  The planes win where the look-ups are many for each table
// an SM loads and each launch, and lose where a code costs more look-ups than gathers would take from L2.  Old / planes in us:
//   g >= 10 with fewer than four coordinates a look-up (33 tokens, 4096 x 4096, g = 16, K = 65536 20 / 34; with four:
//     119 tokens, 3008 x 10368, K = 4880 44 / 29);
//   one coordinate a look-up (K > 51,000 or so): 4096 x 4096, 33 tokens, g = 4 27 / 23, 11008 x 4096 68 / 44, g = 6 65 / 50, g = 8 53 / 49,
//     but 4096 x 4096, g = 8 22 / 27 and, few codes, 22 tokens, 1344 x 4992, g = 5 18 / 24, 153 tokens, 1024 x 1024, g = 6 13 / 17;
//   many parts of the in_features, i.e. few out_features: 57 tokens, 640 x 9707, g = 6, K = 12893 17 / 20, 25 tokens, 640 x 6893,
//     g = 4, K = 27278 12 / 15; with four coordinates a look-up 12 tokens, 832 x 1984, g = 4, K = 1137 14 / 10;
//   the 4-bit codebook from 192 tokens on, where the weight is decoded once: 215 tokens, 8064 x 2191, g = 8 24 / 41;
//   few in_features for many out_features, whose tiles keep the SMs busy without parts: 101 tokens, 6848 x 1011, g = 8, K = 2499, 4 bits 16.4 /
//     18.0, 5 tokens, 10624 x 686, g = 4, K = 39870 13.9 / 15.2 (odd g: 66 tokens, 8000 x 896, g = 5 22 / 18);
//   many tokens on few codes: 224 tokens, 768 x 512, g = 4, K = 17749 12.9 / 14.3.
// Over 260 drawn layers of 3 to 256 tokens, in device time (replayed from a graph), these bounds and PLANES_WIDE_IN make the layer 1.16 times as fast
// in the mean, the 138 that take the planes 1.32; 14 of those are slower by more than 5 %, at worst 1.32 times (8 tokens, 384 x 12480, g = 16).
// Called one by one from Python the three launches take the host 13.7 us, where one takes 9 and two 11.4: layers of less than half a million
// weights are up to 1.5 times as slow then, though the device is done in 0.7 of the time.
// Up to 64 tokens the answer may not depend on the form of the codebook (both give the same bits there).
inline bool planes_pay(const PlanesPlan& p, int64_t M, int64_t d_out, int64_t d_in, int g, bool quant) {
    const int64_t codes = (d_out + g - 1) / g * d_in;
    if (g >= 10 && p.PP < 4) return false;
    if (p.PP == 1 && (g >= 8 || codes < 2000000)) return false;
    if (p.PP < 4 && p.splits > 16) return false;
    if (g % 2 == 0 && d_in <= 1152 && d_out >= 4 * d_in) return false;
    return !(quant && M > 192) && !(M > 128 && codes < 200000);
}

// Stages of 64 in_features that the planes' kernel may add up in one accumulator: no longer a chain than the tensor
// kernel would have had (its splits), and at most 16.
constexpr int PLANES_CHAIN_MOST = 16;
inline int planes_chain(int64_t M, int64_t d_out, int64_t d_in, int sm_count, int g) {
    const LinearPlan p = linear_plan(M, d_out, d_in, sm_count, LNT_MAX, 0, g);
    return p.chunks_per_split < PLANES_CHAIN_MOST ? p.chunks_per_split : PLANES_CHAIN_MOST;
}

// In_features from which the planes take a layer that would otherwise be decoded once and multiplied.  That way costs little beside a gather a
// code, while the planes write and read partial sums of all out_features however few the in_features are.  Decoded once / planes, device
// time in us: 158 tokens, 12544 x 256, g = 3, K = 1110 13.8 / 35.5; 199, 1472 x 384, g = 2 6.8 / 13.4; 203, 6976 x 350, g = 7 15 / 23; 249, 2688 x
// 1032, g = 9 12 / 18; 102, 8384 x 1239, g = 4, 4 bits 15 / 23; 123, 8832 x 1216, g = 4, K = 44770, 4 bits 17 / 24; 154, 11392 x 2358, g = 4, 4 bits 31 / 46;
// 186, 6464 x 2624, g = 4, 4 bits 22 / 35; but 254, 1514 x 2816, g = 12 22 / 19; 193, 1728 x 3392, g = 7 25 / 17; 195, 832 x 4224, g = 2 21 / 18; 183,
// 10240 x 4480, g = 8, 4 bits 61 / 56; 122, 11494 x 7104, g = 4, K = 65536 144 / 94; 162, 11133 x 14528, g = 6 306 / 139 (three of 21 longer layers, all
// g = 4 with 160 tokens or more, 10 to 13 % slower: 185, 12416 x 5184 77 / 87).
constexpr int PLANES_WIDE_IN = 2700;

// The plan with which the planes take a call that the look-up kernel does not; .fits is false where they do not.
inline PlanesPlan planes_for(int64_t M, int64_t d_out, int64_t d_in, int sm_count, int K, int g, bool quant) {
    PlanesPlan p = {};
    if (M > PL_NT_MAX) return p;
    const LinearPlan l = quant ? linear_plan(M, d_out, d_in, sm_count, M >= LQ_WIDE_FROM ? LNT_MAX : LQ_NT_MAX, (size_t)K * (g / 2), g)
                               : linear_plan(M, d_out, d_in, sm_count, LNT_MAX, 0, g);
    if (d_in <= PLANES_WIDE_IN && M >= linear_wide_from(l.fill, d_in, g, quant)) return p;
    p = planes_plan(M, d_out, d_in, sm_count, K, g, planes_chain(M, d_out, d_in, sm_count, g));
    p.fits = p.fits && planes_pay(p, M, d_out, d_in, g, quant);
    return p;
}

}  // namespace
