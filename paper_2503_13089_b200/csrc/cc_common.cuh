// Shared host-side declarations of the library's translation units.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "cluscomp.h"

// Bits of the device status word (workspace, word 0).
#define CC_DEV_NONFINITE 1u
#define CC_DEV_TIMEOUT 2u

// Kernel classes for the optional per-kernel event timing (cc_profile_*).
enum { CC_K_ASSIGN_MAIN = 0, CC_K_ASSIGN_PREP = 1, CC_K_RESOLVE = 2, CC_K_OBJECTIVE = 3, CC_K_UPDATE_ACCUM = 4,
       CC_K_UPDATE_FINISH = 5, CC_K_RESHAPE = 6, CC_K_DECODE = 7, CC_K_OTHER = 8, CC_K_ASSIGN_FINISH = 9, CC_K_UPDATE_DELTA = 10,
       CC_K_LINEAR = 11, CC_K_LINEAR_REDUCE = 12, CC_K_COUNT = 13 };
constexpr int CC_PROF_CAP = 8192;

struct cc_prof_slot { cudaEvent_t a, b; int kind; };

struct cc_ctx {
    int device;
    int sm_count;
    int path;             // CC_PATH_*
    void* ws;             // caller-owned workspace
    size_t ws_bytes;
    int64_t launches;     // kernels launched so far
    int64_t* pos_host;    // staging for cc_init_codebook (K positions)
    int pos_cap;
    int prof_on;          // record an event pair around every kernel launch
    int prof_used, prof_made;
    cc_prof_slot* prof;   // CC_PROF_CAP slots, events created on first use
    void* e2e_buf;        // device memory of cc_compress_host, grown on demand, freed by cc_destroy
    size_t e2e_bytes;
    size_t e2e_refused;   // smallest size that was refused for want of memory (0: none yet); not asked for again
    void* stage;          // CC_STAGE_BYTES of page-locked host memory for small results, made on first use, freed by cc_destroy
    int empty_rule;       // CC_EMPTY_*
};

constexpr size_t CC_STAGE_BYTES = 512 * 1024;

// Brackets one kernel launch with events on its stream when timing is enabled, and counts it.
struct ProfScope {
    cc_ctx* c; cudaStream_t st; cc_prof_slot* slot;
    ProfScope(cc_ctx* ctx, int kind, cudaStream_t s) : c(ctx), st(s), slot(nullptr) {
        c->launches++;
        if (!c->prof_on || !c->prof || c->prof_used >= CC_PROF_CAP) return;
        cc_prof_slot* sl = c->prof + c->prof_used;
        if (c->prof_used >= c->prof_made) {
            if (cudaEventCreate(&sl->a) != cudaSuccess || cudaEventCreate(&sl->b) != cudaSuccess) return;
            c->prof_made = c->prof_used + 1;
        }
        sl->kind = kind;
        cudaEventRecord(sl->a, st);
        slot = sl;
        c->prof_used++;
    }
    ~ProfScope() { if (slot) cudaEventRecord(slot->b, st); }
};

// In a kernel that launch_after starts: everything in front of it has ended and is visible from here on; and the next such kernel may
// start (its blocks take the places that become free, and wait here in turn).  Calls back to back save about a
// microsecond each.  Kernels that fill an SM's shared memory do not let the next one start before they end where that lives off
// L1: its blocks would keep the small L1 they found (35,000 points, g = 16, K = 6971, twelve iterations 1189 -> 1294 us).
#ifdef __CUDACC__
__device__ __forceinline__ void after_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
#endif

// Launch that may begin before the kernel in front of it has ended; what it needs of that one stands behind
// after_previous().
template <class... Args, class... Given>
cudaError_t launch_after(dim3 grid, dim3 block, size_t smem, cudaStream_t st, void (*kernel)(Args...), Given... args) {
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<Args>(args)...);
}

// Status block at the start of every workspace: cleared by cc_set_workspace.
constexpr size_t CC_STATUS_BYTES = 4096;
constexpr int CC_ARRIVAL_WORD = 64, CC_ARRIVAL_COUNTERS = 960, CC_GATE_WORD = 56;

// Carving of the workspace for a problem (N, g, K).  All offsets 256-byte aligned.
struct WsLayout {
    size_t status;     // CC_STATUS_BYTES: 1024 x u32: [0] status bits, [2..3] flagged counter (u64), [8] last-block counter of the objective
                       // sum, [32..35] tensor-path parameters, [36] codebook quantiser's maximum, [40] largest distance, [41] a counter,
                       // [48..53] exact objective sum, [56..57] the counters at which the blocks of a small
                       // fit meet (both zero between calls), [64..1023] arrival
                       // counters of the layer forward's split reduction (zero between calls)
    size_t cprep;      // staged codebook for the FFMA E-step
    size_t flagged;    // u32 list of points sent to the exact stage
    size_t partials;   // doubles: per-block objective partial sums
    size_t sum_lo;     // int64 R x K x g: sums of |x| < 8 in units of 2^-24 (R = cc_sum_copies)
    size_t sum_hi;     // int64 R x K x g: sums of |x| >= 8 in units of 2^-7
    size_t count_copies;  // int32 R x K: per-copy member counts of the M-step (R > 1)
    size_t tmp_c;      // float K x g: widened FP16 codebook (finalize)
    size_t positions;  // int64 K: initial positions
    size_t dist_tmp;   // float N: distances when the caller passes dist == NULL
    size_t tensor;     // staging of the tensor-core E-step (split codebook operand)
    size_t tstate;     // float2 N: (second-best chunk minimum, best chunk id) from the tensor-core scan
    size_t idx_prev;   // u16 N: codes of the previous M-step inside cc_fit
    size_t total;      // what every call needs
    // pruned E-step (nothing where it does not apply, see cc_prune_applies)
    size_t xs;         // u16 N x g: points in spatial order
    size_t pos;        // u32 N: point -> position
    size_t idx_s;      // u16 N: codes by position
    size_t ub;         // float N: upper bounds of the last E-step
    size_t rise;       // float per row block of 32 points
    size_t gap;        // float row blocks x chunks (only where it is used, see cc_prune_gap_words)
    size_t list;       // u16 tiles of 128 points x chunks
    size_t list_n;     // u32 tiles
    size_t order;      // u32 Kp: position -> centroid
    size_t tree;       // u32 Kp: nodes of the k-d tree
    size_t first;      // u32 Kp: leaf -> position of its first point; scratch of the tree
    size_t cs;         // float K x g: codebook by position
    size_t c_prev;     // float K x g: codebook of the last E-step
    size_t boxes;      // float chunks x (2 g + 2 g + 3)
    size_t moved;      // float chunks
    size_t total_preferred;
};

// Buffers of the pruned E-step (cc_assign_pruned.cu), carved from the workspace.
struct PruneBuffers {
    int64_t N;
    int K, ld;
    uint16_t* Xs; unsigned* pos; uint16_t* idx_s; float* dist_s;
    float* ub; float* rise; float* gap;
    uint16_t* list; unsigned* list_n; unsigned* order; unsigned* tree; unsigned* first;
    float* Cs; float* C_prev; float* box_t; float* box_c; float* moved;
    unsigned char* gB; float* rescan; float2* tstate; unsigned* status; unsigned* flagged; long long* acc;
};
enum { CC_PRUNE_COLD = 0,      // first E-step: bounds from the tree leaf each point falls into
       CC_PRUNE_RESTART = 1,   // bounds from the previous codes; the chunks may have been redrawn, kept gaps start anew
       CC_PRUNE_NEXT = 2 };    // same chunks as in the previous E-step

constexpr int CC_KPAD = 1024;          // staged codebook is padded to a multiple of this
constexpr int CC_OBJ_BLOCKS = 1024;    // partial sums of the objective reduction

WsLayout cc_ws_layout(int64_t N, int g, int K);

// Copies of the M-step's sums (at most CC_SUM_COPY_ELEMS words per array).
#ifndef CC_SUM_COPIES_MAX
#define CC_SUM_COPIES_MAX 16
#endif
constexpr int CC_SUM_COPY_ELEMS = 1048576;
static inline int cc_sum_copies(int K, int g) {
    const int r = CC_SUM_COPY_ELEMS / (K * g);
    return r < 1 ? 1 : (r > CC_SUM_COPIES_MAX ? CC_SUM_COPIES_MAX : r);
}

// Copies for N points: few points do not queue up, and every copy is cleared and added up (8192 points, g = 16, K = 4096 with
// four copies 9.1 us, with sixteen 12.2; 65,000 points, g = 12 12.9 and 15.5; but 524,000 points, g = 8, K = 20000 with one 33.5, with
// six 22.9; 4.2 M points, g = 4, K = 65536 with one 65, with four 47).
constexpr int CC_SUM_COPY_FEW = 262144;              // words an array up to CC_SUM_COPY_POINTS points
constexpr int64_t CC_SUM_COPY_POINTS = 131072;
static inline int cc_sum_copies_for(int64_t N, int K, int g) {
    const int most = cc_sum_copies(K, g), few = CC_SUM_COPY_FEW / (K * g) < 1 ? 1 : CC_SUM_COPY_FEW / (K * g);
    return N > CC_SUM_COPY_POINTS || few > most ? most : few;
}

static inline size_t cc_align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// Launchers (each returns cudaGetLastError() of its launches and bumps ctx->launches).
cudaError_t cc_launch_reshape(cc_ctx*, const uint16_t* W, int64_t d_out, int64_t d_in, int g, int layout,
                              uint16_t* X, cudaStream_t);
cudaError_t cc_launch_decode(cc_ctx*, const uint16_t* C16, int K, int g, const uint16_t* idx, int64_t d_out,
                             int64_t d_in, int layout, uint16_t* W_hat, cudaStream_t);
// The same by coordinates (cc_decode_planes.cu).
bool cc_decode_planes_applies(int K, int g, int64_t d_out, int64_t d_in, const void* W_hat);
cudaError_t cc_launch_decode_planes(cc_ctx*, const uint16_t* C16, int K, int g, const uint16_t* idx, int64_t d_out, int64_t d_in,
                                    uint16_t* W_hat, cudaStream_t);
cudaError_t cc_launch_gather_init(cc_ctx*, const uint16_t* X, int g, int K, const int64_t* pos_dev, float* C,
                                  cudaStream_t);
constexpr int CC_INIT_ARGS = 480;      // initial positions that travel as a kernel argument instead of a copy
cudaError_t cc_launch_gather_init_args(cc_ctx*, const uint16_t* X, int g, int K, const int64_t* pos_host, float* C, cudaStream_t);
cudaError_t cc_launch_to_half(cc_ctx*, const float* C, int64_t n, uint16_t* C16, float* C_widened, cudaStream_t);

cudaError_t cc_launch_assign_ffma(cc_ctx*, const WsLayout&, const uint16_t* X, int64_t N, int g, const float* C,
                                  int K, uint16_t* idx, float* dist, double* objective, int64_t* n_resolved,
                                  cudaStream_t);
cudaError_t cc_launch_prep_ffma(cc_ctx*, const WsLayout&, int g, const float* C, int K, cudaStream_t);
bool cc_tensor_path_supported(int g, int K);
cudaError_t cc_launch_assign_tensor(cc_ctx*, const WsLayout&, const uint16_t* X, int64_t N, int g, const float* C,
                                    int K, uint16_t* idx, float* dist, double* objective, int64_t* n_resolved,
                                    cudaStream_t);
// Verification aid: every comparison score of the tensor-core scan, N x cc_tensor_score_ld(K) floats.
int cc_tensor_score_ld(int K);
cudaError_t cc_launch_gate_selftest(unsigned* gates_dev, long long limit_cycles, int* out_dev, long long* cycles_dev, cudaStream_t);
cudaError_t cc_launch_wait_selftest(long long limit_cycles, int* out_dev, long long* cycles_dev, cudaStream_t);
cudaError_t cc_launch_tensor_scores(cc_ctx*, const WsLayout&, const uint16_t* X, int64_t N, int g, const float* C,
                                    int K, float* scores, cudaStream_t);
cudaError_t cc_launch_tensor_finish_only(cc_ctx*, const WsLayout&, const uint16_t* X, int64_t N, int g, const float* C,
                                         int K, const void* scan, uint16_t* idx, float* dist, cudaStream_t);
// Second stage shared by both E-step paths: exact FP64 decision for the flagged points, then
// the deterministic objective sum.
cudaError_t cc_launch_assign_tail(cc_ctx*, const WsLayout&, const uint16_t* X, int64_t N, int g, const float* C,
                                  int K, uint16_t* idx, float* dist, double* objective, int64_t* n_resolved,
                                  cudaStream_t);

// Spatial order and pruned E-step.
bool cc_prune_applies(int64_t N, int g, int K);
constexpr int CC_PRUNE_G = 8;          // longest sub-vectors for which it is ever the faster
size_t cc_prune_gap_words(int64_t N, int K);
int cc_tree_positions(int K);
cudaError_t cc_launch_tree(cc_ctx*, const float* C, int K, int g, unsigned* order, unsigned* scratch, unsigned* tree, cudaStream_t);
cudaError_t cc_launch_sort_points(cc_ctx*, const uint16_t* X, int64_t N, int g, const unsigned* tree, int levels, uint16_t* leaf,
                                  unsigned* pos, unsigned* first, uint16_t* Xs, cudaStream_t);
cudaError_t cc_launch_unsort(cc_ctx*, const unsigned* pos, int64_t N, const uint16_t* idx_s, const float* dist_s, uint16_t* idx,
                             float* dist, unsigned* marks, unsigned* status, unsigned* flagged, cudaStream_t);
cudaError_t cc_launch_assign_pruned(cc_ctx*, const PruneBuffers&, int g, const float* C, int mode, cudaStream_t);
cudaError_t cc_launch_sum_exact(cc_ctx*, const PruneBuffers&, bool have_max, double* objective, int64_t* n_resolved, cudaStream_t);

cudaError_t cc_launch_update_means(cc_ctx*, const WsLayout&, int g, int K, float* C, int32_t* counts, cudaStream_t);

// Small problems (cc_small.cu): the E-step by direct distances, with the M-step behind it in the same launch.
enum { SMALL_E = 0, SMALL_FIRST = 1, SMALL_NEXT = 2 };
constexpr int SMALL_SMEM = 96 * 1024;                // bytes of codebook
constexpr int64_t SMALL_WORK = 350000000;            // point-centroid pairs times instructions each
bool cc_small_applies(const cc_ctx*, int64_t N, int g, int K);
bool cc_small_fit_applies(const cc_ctx*, int64_t N, int g, int K);   // whole iterations
cudaError_t cc_launch_small(cc_ctx*, const WsLayout&, const uint16_t* X, int64_t N, int g, float* C, int K, int mode, uint16_t* idx,
                            float* dist, int32_t* counts, double* objective, int64_t* n_flagged, cudaStream_t);
bool cc_small_loop_applies(const cc_ctx*, int64_t N, int g, int K);                        // all iterations in one launch
cudaError_t cc_launch_small_loop(cc_ctx*, const WsLayout&, const uint16_t* X, int64_t N, int g, float* C, int K, int iters, uint16_t* idx,
                                 float* dist, int32_t* counts, double* objective_trace, cudaStream_t);

// Scratch of the layer forward in the workspace: the status block, a copy of the codebook with padded rows, the rest.
constexpr size_t CC_LINEAR_SCRATCH_FROM = CC_STATUS_BYTES + (size_t)65536 * 32;

// Compressed linear layer: y = x . decode(C16, idx)^T (+ bias).
size_t cc_linear_scratch_bytes(int64_t M, int64_t d_out, int64_t d_in, int sm_count);             // what every call needs
size_t cc_linear_scratch_bytes_preferred(int64_t M, int64_t d_out, int64_t d_in, int sm_count, int K, int g);   // what the fastest way needs
int cc_linear_q_table_max(void);
// The same for many tokens (cc_linear_wide.cu): the weight is decoded once into tiles in the workspace.
bool cc_linear_wide_applies(int64_t M, int64_t d_out, int64_t d_in, int splits, int sm_count);
size_t cc_linear_wide_bytes(int64_t M, int64_t d_out, int64_t d_in);
cudaError_t cc_launch_linear_wide(cc_ctx*, const uint16_t* x, int64_t M, const uint16_t* C16, bool padded, const unsigned char* qtab,
                                  const float* qscale, int K, int g, const uint16_t* idx, int64_t d_out, int64_t d_in,
                                  const float* bias, float* y, int splits, cudaStream_t);
cudaError_t cc_launch_linear_forward(cc_ctx*, const uint16_t* x, int64_t M, const uint16_t* C16, const unsigned char* qtab,
                                     const float* qscale, int K, int g, const uint16_t* idx, int64_t d_out, int64_t d_in,
                                     const float* bias, float* y, cudaStream_t);

cudaError_t cc_launch_quantize_codebook(cc_ctx*, const uint16_t* C16, int64_t n, int bits, uint8_t* q, float* scale,
                                        uint16_t* deq, cudaStream_t);
cudaError_t cc_launch_gather_rows(cc_ctx*, const uint16_t* X, int g, const unsigned* pos_dev, int64_t n, uint16_t* out,
                                  cudaStream_t);
cudaError_t cc_launch_split_empty(cc_ctx*, const WsLayout&, float* C, int K, int g, const int32_t* counts, cudaStream_t);

cudaError_t cc_launch_update(cc_ctx*, const WsLayout&, const uint16_t* X, int64_t N, int g, const uint16_t* idx,
                             int K, float* C, int32_t* counts, cudaStream_t);
cudaError_t cc_launch_codebook_grad(cc_ctx*, const WsLayout&, const uint16_t* dX, int64_t N, int g, const uint16_t* idx,
                                    int K, float* dC, cudaStream_t);
cudaError_t cc_launch_update_delta(cc_ctx*, const WsLayout&, const uint16_t* X, int64_t N, int g, const uint16_t* idx,
                                   uint16_t* idx_prev, int K, float* C, int32_t* counts, cudaStream_t);
