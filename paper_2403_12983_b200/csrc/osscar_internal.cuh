// Internal declarations shared by the translation units of libosscar.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include <stddef.h>
#include "osscar.h"

namespace osscar {

constexpr int kTracePartials = 1184;   // blocks of a trace reduction; the context owns that many doubles
constexpr int64_t kMaxPairs = 1 << 20;     // PAIR_EXACT scores at most this many (kept, pruned) pairs per step
constexpr int kLoopMaxBlocks = 2048;   // most blocks the persistent swap loop is launched with (size of its candidate lists)
constexpr double kTinyProduct = 16777216.0;   // multiply-adds (256^3) up to which a product is one launch on the fp64 pipe
constexpr size_t kFreeDynSmem = 40 * 1024;   // dynamic shared memory above which a kernel asks for more (48 KB less its static arrays)
// g x g doubles of the widest groups.  A kernel's limit of dynamic shared memory belongs to the process: it is set to the most any layer needs, never
// to what this one needs, which another thread may be about to exceed.
constexpr int kGroupBytes = OSSCAR_MAX_GROUP * OSSCAR_MAX_GROUP * (int)sizeof(double);
constexpr int kPadF = 32;   // leading dimensions of internal fp32 matrices are padded to this many floats

extern unsigned long long g_launches;      // kernels launched by the library (host-side count)
static inline void count_launches(unsigned long long n) { g_launches += n; }

static inline int64_t round_up(int64_t x, int64_t a) { return (x + a - 1) / a * a; }

// Device-side control block of the swap loop.  Lives in the context's small device allocation.
struct SearchCtl {
    int32_t done;            // set once the loop has stopped; later kernels return at once
    int32_t stop_reason;
    int32_t status;          // OSSCAR_OK or an error raised on the device
    int32_t n_swaps;
    int32_t n_refresh;
    int32_t sel_slot;        // kept slot leaving
    int32_t sel_t;           // pruned slot (0-based among pruned slots) entering
    int32_t pending;         // rank-two terms not yet written into the matrices (search_lazy_g1.cuh)
    double  obj;             // running objective
    double  sel_D;           // drop score of the chosen slot
    double  delta;           // exact change of obj of the chosen swap
    double  const_term;
    double  acc[4];          // scratch accumulators (traces, objective reductions)
    long long wait_limit;    // cycles a bounded device-side wait may spin before it raises OSSCAR_E_TIMEOUT
    unsigned long long bar_count;   // arrivals at the grid barrier of the persistent swap loop (monotone)
    int32_t abort;           // set by a wait that ran out: every block of the persistent loop returns
    int32_t y_due;           // the step in flight made a swap (search_lazy_g1.cuh)
    int32_t dl_terms;        // pivots whose terms the matrices do not have yet (search_delayed_g1.cuh)
    int32_t dl_stop;         // 1: the swaps of this part of the search are made, 2: the terms have filled their memory
    int32_t dl_batches;      // batches of candidate columns of this search
    int32_t settled;         // the search made no swap: V is as refined as it was
    int32_t gram_skip[2];    // Gram of fp32 activations: the panel in flight skips the digits / the bf16 terms (gemm_i8.cu)
};

// Geometry of one layer's search state inside the caller's workspace.
struct Layout {
    int64_t d1, m, ng;       // rows of W, columns of W, number of groups
    int32_t g, k;
    int64_t nI, nJ;          // kept rows, pruned rows
    int64_t ldp;             // leading dimension of Hp (slot-permuted H)
    int64_t ldh;             // leading dimension of Hinv, and padded length of the n_I-vectors
    int64_t ldm;             // leading dimension of V, R, K, Vq
    // offsets in bytes from the workspace base
    size_t off_Hp, off_Hinv, off_V, off_R, off_big;
    size_t off_Hd;                                                     // fp64 copy of the inverse (g = 1 only, else a stub)
    size_t off_y, off_b, off_u2, off_bC, off_u2c, off_u, off_d, off_K, off_Vq;
    size_t off_vec_begin, off_vec_end;   // the staged vectors (zeroed once when the state is built)
    size_t off_vnorm, off_rnorm, off_D, off_A, off_c, off_small, off_gramV, off_gramR;
    size_t off_perm, off_slotof, off_energy, off_panel;
    size_t off_shard;                                                  // column shards: partial sums handed to the reduce hook
    size_t off_loop;                                                   // persistent swap loop: per-block candidates, phase timers
    size_t off_pairCinv, off_pairKK, off_pairScratch, off_pairDelta;   // PAIR_EXACT scoring
    size_t off_greedy;                                                 // scratch of the nested (greedy) phase
    size_t off_tc, tc_bytes;                                           // bf16 operand terms of the tensor-core GEMMs
    size_t off_block, block_bytes;                                     // panels of the block exchange (search_block.cuh)
    int32_t block_rows_max;                                            // largest s*g the block region holds
    int64_t pair_capacity;                                             // pairs the workspace can score
    size_t bytes;
};
// bytes of the block-exchange panels for G rows on each side (layout in search_block.cuh)
static inline size_t block_region_bytes(int64_t ldh, int64_t ldm, int64_t nJ, int64_t G)
{
    auto al = [](size_t b) { return (b + 255) / 256 * 256; };
    size_t n = 2 * al(sizeof(int32_t) * (size_t)G);
    n += 3 * al(sizeof(float) * (size_t)G * ldh);            // hT, yT, HrT
    n += 4 * al(sizeof(float) * 2 * (size_t)G * ldh);        // PB, PA and their transposes
    n += al(sizeof(float) * 2 * (size_t)G * ldm);            // KV
    n += 2 * al(sizeof(float) * (size_t)G * ldm);            // Vr, Rq
    n += al(sizeof(float) * (size_t)(nJ + G) * 2 * G);       // UD
    n += al(sizeof(double) * 18 * (size_t)G * G);            // small matrices
    return n;
}
int make_layout(int64_t d1, int64_t m, int32_t g, int32_t k, Layout* L);

}  // namespace osscar

struct osscar_ctx {
    int device;
    cudaStream_t stream;
    osscar::SearchCtl* ctl;          // device
    osscar::SearchCtl* ctl_host;     // pinned mirror
    double* partials;                // device, kTracePartials doubles: stage 1 of deterministic reductions
    volatile int32_t* done_flag_host; // pinned, device-mapped: copy of ctl->done pushed by the device
    int32_t* done_flag_dev;          // device alias of done_flag_host
    void* ws;
    size_t ws_bytes;
    osscar::Layout L;
    bool have_state;
    const float* H;                  // caller's matrices bound by init_support
    const float* G;
    const float* W;
    cudaEvent_t ev0, ev1;
    double gram_rows;                // rows accumulated since GRAM_BEGIN (bookkeeping only)
    bool have_const;                 // const term supplied by the caller (cross-term problems) instead of Tr(W^T G)
    double user_const;
    long long wait_limit;            // context default of SearchCtl::wait_limit
    bool hd_valid;                   // the fp64 copy of the inverse matches the state
    osscar_reduce_fn reduce;         // column shards: in-place sum over shards, enqueued by the caller's hook (or null)
    void* reduce_user;
};

namespace osscar {

// ---- dependent launches.  The kernels of a chain (swap steps, iterations of the nested phase, steps of the inversion) are
// launched so that the next one may start while the current one is still running.  A kernel of single-row groups first
// requests the rows it streams (written by kernels that finished long ago), all others begin with the wait; a kernel waits here for
// the kernel before it to complete before it reads anything that kernel wrote (staged vectors, scalars, the control
// block), and only then lets its own successor start: a successor's early part can thus overlap only the late part of its
// immediate predecessor, and its blocks are already resident when the predecessor drains.  Without the launch attribute both
// instructions do nothing.  What the predecessor wrote is read with ordinary loads only: the read-only (non-coherent)
// path may still hold a line from the step before, since no kernel boundary separates the two any more.
static __device__ __forceinline__ void pdl_wait_then_release() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Launch, with `dependent` set, as a programmatic dependent of the kernel before it on the stream.  Only a launch that directly
// follows another kernel launch of the chain may be one: behind an event record, a copy or a reduction by the caller's
// hook the launch is an ordinary, fully ordered one.
template <typename... KArgs, typename... Args>
static cudaError_t launch_pdl_smem(bool dependent, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = dependent ? 1 : 0;
    cfg.attrs = at; cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}
template <typename... KArgs, typename... Args>
static cudaError_t launch_pdl(bool dependent, void (*kernel)(KArgs...), dim3 grid, dim3 block, cudaStream_t st, Args... args)
{
    return launch_pdl_smem(dependent, kernel, grid, block, 0, st, args...);
}

// ---- sgemm.cu: C = alpha * op(A) * B + beta * C on the fp32 pipes ----------------------------
// A is M x K (lda) or, with transA, stored K x M; B is K x N (ldb) or, with transB, stored N x K.
// `done` (may be null): device flag; when non-zero the kernel returns without touching C.
cudaError_t sgemm(cudaStream_t st, bool transA, bool transB, int64_t M, int64_t N, int64_t K,
                  float alpha, const float* A, int64_t lda, const float* B, int64_t ldb,
                  float beta, float* C, int64_t ldc, const int32_t* done = nullptr);

// ---- dgemm.cu: C = beta * C0 + alpha * A * B (or I + alpha * A * B) with fp32 operands, products and sums in fp64;
// A (M x K) and B (K x N) row-major, C0 may alias C.
cudaError_t gemm_f64acc(cudaStream_t st, int64_t M, int64_t N, int64_t K, double alpha, const float* A, int64_t lda,
                        const float* B, int64_t ldb, double beta, const float* C0, int64_t ldc0, float* C, int64_t ldc,
                        bool identity_plus, const int32_t* done = nullptr);
cudaError_t gemm_f64out(cudaStream_t st, int64_t M, int64_t N, int64_t K, const float* A, int64_t lda,
                        const float* B, int64_t ldb, double* C, int64_t ldc, bool tri = false);

// ---- gemm_i8.cu: the same products from 8-bit digits of the operands on the int8 tensor cores (exact integer sums)
struct I8Scratch {                 // device memory for the digits of A and of B (256-byte aligned), and what A's part holds
    void* a = nullptr; size_t a_bytes = 0;
    void* b = nullptr; size_t b_bytes = 0;
    const float* have_A = nullptr; int64_t have_rows = 0, have_K = 0, have_ldk = 0; int have_S = 0;
};
struct I8Gemm {                    // C = beta * C0 + alpha * A * B, A (M x K) and B (K x N) row-major
    int64_t M, N, K;
    double alpha, beta;
    const float* A; int64_t lda;
    const float *B, *Bsub; const double* Bd; int64_t ldb;     // fp32 B (minus Bsub), or fp64 Bd
    const float* BT;               // or B transposed, N rows of K (without a balance: diag null)
    const float *C0, *C0sub; int64_t ldc0;
    void* C; int64_t ldc;
    bool identity;                 // I + alpha A B instead of beta C0 + alpha A B
    int64_t identity_col0;         // column of I that column 0 of the product is
    bool out64;                    // C in fp64
    bool tri;                      // B symmetric, K = N: its block upper triangle with halved diagonal blocks (see dgemm.cu)
    bool dot;                      // C (doubles, gemm_i8_dot_cols(N) per row) = partial sums of rows of A B times rows of C0 (- C0sub)
    const float* diag; int64_t diag_stride;            // diagonal of H_II: balances the contraction index (null: none)
    bool inverse_scale;            // the columns of A scale like those of the inverse of H, not like those of H
    const double* pivots;          // or: K factors 1 / S_kk of pivots, columns of A scale with their square roots and rows of B with the inverses
};
bool gemm_i8_usable(int64_t M, int64_t N, int64_t K, int S, const I8Scratch& sc);
cudaError_t gemm_i8(cudaStream_t st, const I8Gemm& p, int S, I8Scratch& sc, SearchCtl* ctl_dev, const int32_t* done);
int64_t gemm_i8_dot_cols(int64_t N);
// H (+)= Xc^T Xc (upper-triangle tiles) for fp32 Xc; cudaErrorMemoryAllocation: too small a product or scratch, take another path
cudaError_t gram_i8(cudaStream_t st, const float* X, int64_t n_rows, int64_t d1, float* C, bool accumulate,
                    void* scratch, size_t scratch_bytes, SearchCtl* ctl_dev);
// G = H W (H d1 x d1, W and G d1 x m, dense) from four digits of each operand, or as gemm_tc where they do not pay or fit
cudaError_t cross_term_tc(cudaStream_t st, const float* H, int64_t d1, const float* W, int64_t m, float* G,
                          void* scratch, size_t scratch_bytes, SearchCtl* ctl_dev);
// *out = sum of (W - Wt) o H (W - Wt) (H d1 x d1, W and Wt d1 x m, dense); `partials`: the context's reduction scratch.
// cudaErrorMemoryAllocation when the product is too small for digits or the scratch too small for them.
cudaError_t objective_i8(cudaStream_t st, const float* H, const float* W, const float* Wt, int64_t d1, int64_t m,
                         void* scratch, size_t scratch_bytes, double* partials, double* out_dev, SearchCtl* ctl_dev);
size_t gemm_i8_operand_bytes(int64_t rows, int64_t K, int S);      // scratch that holds the digits of a whole operand
int64_t gemm_i8_row_bytes(int64_t K);                              // one row of one digit, where whole operands fit

// ---- panel_tc.cu: Y[i*so_row + e*so_col] = sum_k A[i][k] * P[e][k] on the tensor cores; A (M x K, streamed once) is split
// into bf16 terms on the way (fp32-accurate); P is an N x K panel
// A 16-byte aligned with lda % 4 == 0; scratch at least panel_dot_tc_scratch bytes.
size_t panel_dot_tc_scratch(int64_t M, int64_t N, int64_t K);
cudaError_t panel_dot_tc(cudaStream_t st, int64_t M, int64_t N, int64_t K, const float* A, int64_t lda,
                         const float* P, int64_t ldp, float* Y, int64_t so_row, int64_t so_col,
                         void* scratch, size_t scratch_bytes, SearchCtl* ctl_dev, const int32_t* done = nullptr);

// ---- gemm_tc.cu: the same product on the tensor cores (three-term bf16 split, fp32-accurate); A and B row-major.
// `scratch` (256-byte aligned device memory, at least gemm_tc_min_scratch bytes) holds the bf16 terms of one K panel.  `upper`: only the tiles
// that reach the diagonal or lie above it.
size_t gemm_tc_min_scratch(int64_t M, int64_t N);
cudaError_t gemm_tc(cudaStream_t st, int64_t M, int64_t N, int64_t K, float alpha, const float* A, int64_t lda,
                    const float* B, int64_t ldb, float beta, float* C, int64_t ldc,
                    void* scratch, size_t scratch_bytes, SearchCtl* ctl_dev, const int32_t* done = nullptr,
                    bool upper = false);

// C += alpha * A * B for a short inner dimension (K <= 128 keeps the terms of A's row band in shared memory across a run
// of column tiles; larger K goes through gemm_tc).  Same operands and scratch as gemm_tc.  With row_sq (M floats) and
// sq_scratch (M * 2 * ceil(N / 128) floats) the squared norms of the updated rows are produced in the same pass (K <= 128 only).
cudaError_t rank_update_tc(cudaStream_t st, int64_t M, int64_t N, int64_t K, float alpha, const float* A, int64_t lda,
                           const float* B, int64_t ldb, float* C, int64_t ldc,
                           void* scratch, size_t scratch_bytes, SearchCtl* ctl_dev, const int32_t* done = nullptr,
                           float* row_sq = nullptr, float* sq_scratch = nullptr);

// H (+)= Xc^T Xc (upper-triangle tiles; Y null) or G (+)= Xc^T Yc with the drained-accumulator pipeline of gemm_tc.cu.
cudaError_t gram_tc2(cudaStream_t st, const void* X, int64_t n_rows, int64_t d1, const void* Y, int y_fp32, int64_t m,
                     float* C, bool accumulate, void* scratch, size_t scratch_bytes, SearchCtl* ctl_dev);
// H (+)= Xc^T Xc for fp32 Xc on the tensor cores (three-term bf16 split staged in `scratch`, row panels sized to it);
// cudaErrorMemoryAllocation when the scratch is too small for one panel.
cudaError_t gram_tc3(cudaStream_t st, const float* X, int64_t n_rows, int64_t d1, float* C, bool accumulate,
                     void* scratch, size_t scratch_bytes, SearchCtl* ctl_dev, const int32_t* done = nullptr);

// ---- gram_tc.cu ---------------------------------------------------------------------------------------------
cudaError_t set_device_double(cudaStream_t st, double* dst, double v);          // *dst = v on the stream
cudaError_t gram_mirror(cudaStream_t st, float* H, int64_t d1);   // copy upper triangle to lower

// ---- state.cu: support selection and state construction --------------------------------------
int select_support(osscar_ctx* ctx, int mode, int32_t* support);
int build_state(osscar_ctx* ctx);
// C = A B + beta C0 for A = Hinv or E (nI x nI): digits on the int8 tensor cores, or split bf16 where they do not pay or fit
cudaError_t inverse_product(osscar_ctx* ctx, int64_t N, const float* A, const float* B, int64_t ldb, float beta, const float* C0, float* C,
                            int64_t ldc, int digits, void* other, size_t other_bytes, const int32_t* skip = nullptr);
// E = I - H_II Hinv summed beyond fp32; `v_free`: V and R hold nothing yet, so their memory may take operand digits
cudaError_t inverse_residual(osscar_ctx* ctx, float* E, bool v_free);
// V += Hinv (G_I - H_II V), the residual summed beyond fp32.  GI: G_I in slot order (ldm), rV: as large, `other`: room for digits;
// nothing happens where *skip (device, may be null) is set
cudaError_t refine_v(osscar_ctx* ctx, const float* GI, float* rV, void* other, size_t other_bytes, const int32_t* skip = nullptr);
// ---- invert.cu
// Rows from which invert_spd_inplace sweeps on the tensor cores.  Sweeps against the steps of 64, ms: 2.25 / 3.05 at 3072 rows, 2.67 / 4.63 at 3584,
// 3.17 / 6.14 at 4096, 10.1 / 49 at 8602; at 2304, with blocks of 256, they took the same time.  I - H Hinv has the same or a smaller norm, at condition 1e5 (scaled)
// 8.4e-3 / 8.8e-3, but the largest error of an entry is 2.6e-4 against 1e-4 sqrt(Hinv_ii Hinv_jj) there.
constexpr int64_t kSweptRows = 3072;
int invert_spd_inplace(osscar_ctx* ctx, float* A, int64_t lda, int64_t n, const float* ref, int64_t ldref,
                       bool tensor_updates);
// H^-1 of the whole layer in the place of Hp (nested phase): one Newton-Schulz step from digit products, in column panels, and
// C = A B (d1 x d1 times d1 x m).  `correctable`: the layer is large enough and the free regions take the panels.
bool dense_inverse_correctable(const osscar_ctx* ctx);
cudaError_t correct_dense_inverse(osscar_ctx* ctx, float* A, int64_t lda);
cudaError_t dense_inverse_times(osscar_ctx* ctx, const float* A, int64_t lda, const float* B, float* C, int64_t ldc);
cudaError_t gather_rows(cudaStream_t st, const float* src, int64_t m, int g, const int32_t* perm,
                        int64_t slot_row0, int64_t nrows, float* dst, int64_t ld);
cudaError_t sum_partials(cudaStream_t st, const double* partials, int n, double* out_dev);   // *out = sum, fixed order
cudaError_t trace_product(cudaStream_t st, const float* A, int64_t lda, const float* B, int64_t ldb,
                          int64_t rows, int64_t cols, double* partials, double* out_dev);   // *out = sum A.*B

// ---- greedy.cu: nested phase of Algorithm 1 down to L.k groups (leaves the slot permutation in the workspace) -----
size_t greedy_scratch_bytes(int64_t d1, int64_t m, int g);
int greedy_support(osscar_ctx* ctx, int t_hat, int32_t* support, int32_t* drop_trace, int32_t* n_iters_out);

// ---- search.cu -------------------------------------------------------------------------------
int run_search(osscar_ctx* ctx, const osscar_search_params* p, int32_t* support_out, float* W_out,
               double* obj_trace, int32_t* swap_trace, osscar_search_result* res);
cudaError_t score_pass(osscar_ctx* ctx);   // full scoring pass from the current state (fills D, A)
// fp64 copy of the inverse from the fp32 one by a Newton-Schulz step summed in fp64 (single-row groups; uses `big`)
int build_hinv64(osscar_ctx* ctx, bool v_free);
// column shards: sum `count` values of `buf` (inside the workspace) over all shards through the context's hook
int shard_reduce(osscar_ctx* ctx, void* buf, int64_t count, int dtype);

}  // namespace osscar
