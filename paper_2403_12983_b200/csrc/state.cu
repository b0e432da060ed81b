// Starting support and construction of the search state for a given support:
// slot-permuted copy of H, (H_II)^-1 (invert.cu) and its correction,
// V = (H_II)^-1 G_I (Eq. tmp5), residual R, Schur complements c (Case 2 of Proposition 1).
#include "osscar_internal.cuh"
#include <math.h>

namespace osscar {
namespace {

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
// Block-wide sum (blockDim.x multiple of 32, <= 1024); result valid in thread 0.
__device__ double block_sum(double v) {
    __shared__ double red[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    v = warp_sum(v);
    __syncthreads();
    if (lane == 0) red[w] = v;
    __syncthreads();
    if (w == 0) {
        v = (lane < (int)((blockDim.x + 31) >> 5)) ? red[lane] : 0.0;
        v = warp_sum(v);
    }
    return v;
}

// e_q = Tr(W_q^T H_qq W_q) (mode 0) or ||W_q||_F^2 (mode 1); one block per group.
__global__ void k_energy(const float* __restrict__ H, const float* __restrict__ W, int64_t d1, int64_t m,
                         int g, int mode, double* __restrict__ e)
{
    const int64_t q = blockIdx.x;
    const float* Wq = W + q * g * m;
    double acc = 0.0;
    for (int64_t c = threadIdx.x; c < m; c += blockDim.x) {
        if (mode == OSSCAR_INIT_MAGNITUDE) {
            for (int a = 0; a < g; ++a) { double w = Wq[a * m + c]; acc += w * w; }
        } else {
            for (int a = 0; a < g; ++a) {
                double t = 0.0;
                const float* Hrow = H + (q * g + a) * d1 + q * g;
                for (int b = 0; b < g; ++b) t += (double)Hrow[b] * (double)Wq[b * m + c];
                acc += (double)Wq[a * m + c] * t;
            }
        }
    }
    acc = block_sum(acc);
    if (threadIdx.x == 0) e[q] = acc;
}

__device__ __forceinline__ int warp_count(int v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// kept[q] = 1 iff fewer than k groups beat q (larger energy, or equal energy and smaller id); a warp per group.  NaN ranks
// below every number: exactly k groups are marked whatever the energies are, and the slot permutation is complete.
__global__ void k_rank_select(const double* __restrict__ e, int64_t ng, int k, int32_t* __restrict__ kept)
{
    const int64_t q = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (q >= ng) return;
    auto ordered = [](double x) { return x == x ? x : -INFINITY; };
    const double eq = ordered(e[q]);
    int rank = 0;
#pragma unroll 4
    for (int64_t p = threadIdx.x & 31; p < ng; p += 32) {
        const double ep = ordered(e[p]);
        rank += (ep > eq) || (ep == eq && p < q);
    }
    rank = warp_count(rank);
    if ((threadIdx.x & 31) == 0) kept[q] = rank < k;
}

__global__ void k_user_support(const int32_t* __restrict__ support, int k, int64_t ng,
                               int32_t* __restrict__ kept, SearchCtl* ctl)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= k) return;
    const int q = support[i];
    if (q < 0 || q >= ng) { ctl->status = OSSCAR_E_ARG; return; }
    if (atomicExch(&kept[q], 1) != 0) ctl->status = OSSCAR_E_ARG;   // duplicate id
}

// After k_user_support: a list that was rejected (id out of range, duplicate) marks fewer than k groups.  The kernels
// that follow index H and G through the slot permutation, so the marks are replaced by a valid set (the first k
// groups) and the error stays in ctl->status; nothing downstream can then leave its buffers.  One block.
__global__ void __launch_bounds__(1024) k_user_support_guard(int32_t* __restrict__ kept, int64_t ng, int k, SearchCtl* ctl)
{
    __shared__ int cnt;
    if (threadIdx.x == 0) cnt = 0;
    __syncthreads();
    int local = 0;
    for (int64_t q = threadIdx.x; q < ng; q += blockDim.x) local += kept[q] != 0;
    if (local) atomicAdd(&cnt, local);
    __syncthreads();
    if (ctl->status == OSSCAR_OK && cnt == k) return;
    for (int64_t q = threadIdx.x; q < ng; q += blockDim.x) kept[q] = q < k;
    if (threadIdx.x == 0 && ctl->status == OSSCAR_OK) ctl->status = OSSCAR_E_ARG;
}

// Slots: kept groups in ascending id order take slots 0..k-1, pruned groups k..ng-1; a warp per group.
__global__ void k_build_perm(const int32_t* __restrict__ kept, int64_t ng, int k,
                             int32_t* __restrict__ perm, int32_t* __restrict__ slotof,
                             int32_t* __restrict__ support)
{
    const int64_t q = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (q >= ng) return;
    int before_kept = 0;
#pragma unroll 4
    for (int64_t p = threadIdx.x & 31; p < q; p += 32) before_kept += kept[p];
    before_kept = warp_count(before_kept);
    if ((threadIdx.x & 31) != 0) return;
    const int slot = kept[q] ? before_kept : k + (int)(q - before_kept);
    if (slot < 0 || slot >= ng || (kept[q] && slot >= k)) return;       // cannot happen with exactly k marks
    perm[slot] = (int32_t)q;
    slotof[q] = slot;
    if (kept[q]) support[slot] = (int32_t)q;
}

// Hp[i][j] = H[row(i)][row(j)], row(i) = perm[i / g] * g + i % g.  A thread owns four columns, whose source columns it looks up
// once for GS_R rows: 32 independent loads in flight and 16-byte stores.  Bound: HBM, 8 d1^2 bytes.  With one element and
// one look-up (two 64-bit divisions) per thread and step this copy took 6.4 ms at d1 = 28672, now 1.3 ms.
constexpr int GS_R = 8;
__global__ void __launch_bounds__(256) k_gather_sym(const float* __restrict__ H, int64_t d1, int g, const int32_t* __restrict__ perm,
                             float* __restrict__ Hp, int64_t ldp)
{
    const int64_t j0 = ((int64_t)blockIdx.x * 256 + threadIdx.x) * 4, i0 = (int64_t)blockIdx.y * GS_R;
    if (j0 >= ldp) return;
    const uint32_t ug = (uint32_t)g;
    int64_t col[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const uint32_t j = (uint32_t)j0 + k;
        col[k] = j < d1 ? (int64_t)perm[j / ug] * g + j % ug : -1;
    }
    float v[GS_R][4];
#pragma unroll
    for (int r = 0; r < GS_R; ++r) {
        const uint32_t i = (uint32_t)i0 + r;
        const float* row = H + (i < d1 ? (int64_t)perm[i / ug] * g + i % ug : 0) * d1;
#pragma unroll
        for (int k = 0; k < 4; ++k) v[r][k] = i < d1 && col[k] >= 0 ? row[col[k]] : 0.f;
    }
#pragma unroll
    for (int r = 0; r < GS_R; ++r)
        if (i0 + r < d1) *reinterpret_cast<float4*>(Hp + (i0 + r) * ldp + j0) = make_float4(v[r][0], v[r][1], v[r][2], v[r][3]);
}

// dst[i][0..ld) = src[row(slot0*g + i)][0..m) zero-padded, for i in [0, nrows).
__global__ void k_gather_rows(const float* __restrict__ src, int64_t m, int g, const int32_t* __restrict__ perm,
                              int64_t slot_row0, float* __restrict__ dst, int64_t ld)
{
    const int64_t i = blockIdx.x;
    const int64_t s = slot_row0 + i;
    const float* row = src + ((int64_t)perm[s / g] * g + s % g) * m;
    for (int64_t c = threadIdx.x; c < ld; c += blockDim.x) dst[i * ld + c] = c < m ? row[c] : 0.f;
}

// dst (rows x ldd, zero padded) = src[0:rows, 0:cols] (lds)
__global__ void k_copy_pad(const float* __restrict__ src, int64_t lds, int64_t rows, int64_t cols,
                           float* __restrict__ dst, int64_t ldd)
{
    const int64_t i = blockIdx.x;
    for (int64_t c = threadIdx.x; c < ldd; c += blockDim.x) dst[i * ldd + c] = c < cols ? src[i * lds + c] : 0.f;
}

// c_t[a][b] = Hp[J_ta][J_tb] - twice * sum_s Pm[ta][s] * Hp[J_tb][s]  for pruned slot t; grid (slots, shares of the g * g
// entries): 16 slots of 80 rows on one block each kept 16 SMs busy for 3.26 ms.
// Pm holds the rows of the pruned slots [t0, t0 + gridDim.x) in fp64 (row stride ldpm): H_JI Hinv (twice = 1), or, for
// single-row groups, H_JI U with U the halved block upper triangle of Hinv (twice = 2: h^T Hinv h = 2 h^T U h).
__global__ void k_schur(const float* __restrict__ Hp, int64_t ldp, const double* __restrict__ Pm, int64_t ldpm,
                        int64_t nI, int g, double* __restrict__ c, int64_t t0, double twice)
{
    const int64_t t = t0 + blockIdx.x;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int pair = blockIdx.y * nw + w; pair < g * g; pair += nw * gridDim.y) {
        const int a = pair / g, b = pair % g;
        const double* pr = Pm + ((t - t0) * g + a) * ldpm;
        const float* hr = Hp + (nI + t * g + b) * ldp;
        double s = 0.0;
        for (int64_t x = lane; x < nI; x += 32) s = fma(pr[x], (double)hr[x], s);
        s = warp_sum(s);
        if (lane == 0) c[(t * g + a) * g + b] = (double)Hp[(nI + t * g + a) * ldp + nI + t * g + b] - twice * s;
    }
}

// c_t = Hp[J_t][J_t] - 2 * (partial sums of the quadratic form, in column order); one warp per pruned row.
__global__ void k_schur_sum(const float* __restrict__ Hp, int64_t ldp, const double* __restrict__ part, int64_t ldpart, int np,
                            int64_t nI, int64_t nJ, double* __restrict__ c)
{
    const int64_t t = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (t >= nJ) return;
    double s = 0.0;
    for (int i = lane; i < np; i += 32) s += part[t * ldpart + i];
    s = warp_sum(s);
    if (lane == 0) c[t] = (double)Hp[(nI + t) * ldp + nI + t] - 2.0 * s;
}

// Two deterministic stages: per-block partial sums, then one block adds them in a fixed order.
__global__ void k_trace_product(const float* __restrict__ A, int64_t lda, const float* __restrict__ B, int64_t ldb,
                                int64_t rows, int64_t cols, double* __restrict__ partial)
{
    double acc = 0.0;
    for (int64_t r = blockIdx.x; r < rows; r += gridDim.x)
        for (int64_t c = threadIdx.x; c < cols; c += blockDim.x)
            acc += (double)A[r * lda + c] * (double)B[r * ldb + c];
    acc = block_sum(acc);
    if (threadIdx.x == 0) partial[blockIdx.x] = acc;
}
__global__ void k_sum_partials(const double* __restrict__ partial, int n, double* __restrict__ out)
{
    double acc = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) acc += partial[i];
    acc = block_sum(acc);
    if (threadIdx.x == 0) *out = acc;
}

// A := sym(A + D) (D may be null) on the n x n leading block: the blocked inversion leaves its two triangles different in the last bits
// times cond, and the correction of that difference is the antisymmetric part of D, so both are symmetrised together.
// A thread owns the pair (r, c), (c, r) with c >= r; tiles below the diagonal have nothing to do.
__global__ void k_add_sym(float* __restrict__ A, int64_t lda, const float* __restrict__ D, int64_t ldd, int64_t n)
{
    if (blockIdx.x < blockIdx.y) return;
    const int64_t c = (int64_t)blockIdx.x * 32 + threadIdx.x;
    for (int64_t r = (int64_t)blockIdx.y * 32 + threadIdx.y; r < (int64_t)blockIdx.y * 32 + 32 && r < n; r += 8) {
        if (c >= n || c < r) continue;
        const float v = 0.5f * ((A[r * lda + c] + A[c * lda + r]) + (D ? D[r * ldd + c] + D[c * ldd + r] : 0.f));
        A[r * lda + c] = v;
        A[c * lda + r] = v;
    }
}

// acc[0], acc[1] -> sh[0], sh[1] (back = 0) or back again (back = 1)
__global__ void k_pack2(SearchCtl* ctl, double* sh, int back)
{
    if (back) { ctl->acc[0] = sh[0]; ctl->acc[1] = sh[1]; } else { sh[0] = ctl->acc[0]; sh[1] = ctl->acc[1]; }
}

__global__ void k_set_obj(SearchCtl* ctl)   // obj = const - Tr(G_I^T V), with acc[0] = const, acc[1] = trace
{
    ctl->const_term = ctl->acc[0];
    ctl->obj = ctl->acc[0] - ctl->acc[1];
}

#define CK(x) do { cudaError_t e_ = (x); if (e_ != cudaSuccess) return OSSCAR_E_CUDA; } while (0)

}  // namespace

__global__ void k_set_double(double* dst, double v) { *dst = v; }
cudaError_t set_device_double(cudaStream_t st, double* dst, double v)
{
    k_set_double<<<1, 1, 0, st>>>(dst, v);
    count_launches(1);
    return cudaGetLastError();
}
cudaError_t gather_rows(cudaStream_t st, const float* src, int64_t m, int g, const int32_t* perm,
                        int64_t slot_row0, int64_t nrows, float* dst, int64_t ld)
{
    if (nrows > 0) { k_gather_rows<<<(unsigned)nrows, 256, 0, st>>>(src, m, g, perm, slot_row0, dst, ld); count_launches(1); }
    return cudaGetLastError();
}

cudaError_t trace_product(cudaStream_t st, const float* A, int64_t lda, const float* B, int64_t ldb,
                          int64_t rows, int64_t cols, double* partials, double* out_dev)
{
    if (rows <= 0 || cols <= 0) return cudaMemsetAsync(out_dev, 0, sizeof(double), st);
    const int grid = (int)(rows < kTracePartials ? rows : kTracePartials);
    k_trace_product<<<grid, 256, 0, st>>>(A, lda, B, ldb, rows, cols, partials);
    k_sum_partials<<<1, 256, 0, st>>>(partials, grid, out_dev);
    count_launches(2);
    return cudaGetLastError();
}

cudaError_t sum_partials(cudaStream_t st, const double* partials, int n, double* out_dev)
{
    k_sum_partials<<<1, 256, 0, st>>>(partials, n, out_dev);
    count_launches(1);
    return cudaGetLastError();
}

int make_layout(int64_t d1, int64_t m, int32_t g, int32_t k, Layout* L)
{
    if (d1 <= 0 || m <= 0 || g <= 0 || g > OSSCAR_MAX_GROUP || d1 % g != 0) return OSSCAR_E_SHAPE;
    const int64_t ng = d1 / g;
    if (k < 1 || k > ng) return OSSCAR_E_SHAPE;
    L->d1 = d1; L->m = m; L->ng = ng; L->g = g; L->k = k;
    L->nI = (int64_t)k * g; L->nJ = d1 - L->nI;
    L->ldp = round_up(d1, kPadF); L->ldh = round_up(L->nI, kPadF); L->ldm = round_up(m, kPadF);
    size_t off = 0;
    auto take = [&](size_t bytes) { size_t o = off; off += (bytes + 255) / 256 * 256; return o; };
    const int64_t nI = L->nI, nJ = L->nJ, ldh = L->ldh, ldm = L->ldm;
    // `big` first: osscar_objective uses the start of the workspace as 2 * d1 * ldm floats
    int64_t big = nI * ldm;
    if (nJ * ldh > big) big = nJ * ldh;
    if (2 * d1 * ldm > big) big = 2 * d1 * ldm;
    if (2 * nI * ldh > big) big = 2 * nI * ldh;             // residual and correction of the refinement step on Hinv
    const int64_t npairs = (int64_t)k * (ng - k);
    L->pair_capacity = npairs <= kMaxPairs ? npairs : 0;
    if (L->pair_capacity > 0 && nJ * ldh + nI * round_up(nJ, kPadF) > big) big = nJ * ldh + nI * round_up(nJ, kPadF);
    {   // the nested phase keeps V of all rows plus up to 256 staged rows of Hinv (twice, and their transposes) and of V in `big`
        const int64_t gneed = d1 * ldm + 2 * 256 * L->ldp + 256 * ldm + 2 * 256 * d1;
        if (gneed > big) big = gneed;
    }
    L->off_big = take(sizeof(float) * big);
    L->off_Hp = take(sizeof(float) * d1 * L->ldp);
    L->off_Hinv = take(sizeof(float) * nI * ldh);
    L->off_Hd = take(g == 1 ? sizeof(double) * nI * ldh : 256);
    L->off_V = take(sizeof(float) * nI * ldm);
    L->off_R = take(sizeof(float) * (nJ > 0 ? nJ : 1) * ldm);
    L->off_y = take(sizeof(float) * ldh * g);
    L->off_vec_begin = L->off_y;
    L->off_b = take(sizeof(float) * ldh * g);
    L->off_u2 = take(sizeof(float) * ldh * g);
    L->off_bC = take(sizeof(float) * ldh * g);
    L->off_u2c = take(sizeof(float) * ldh * g);
    L->off_u = take(sizeof(float) * (nJ + g) * g);
    L->off_d = take(sizeof(float) * (nJ + g) * g);
    L->off_K = take(sizeof(float) * g * ldm);
    L->off_Vq = take(sizeof(float) * g * ldm);
    L->off_vec_end = off;
    L->off_vnorm = take(sizeof(float) * (nI + nJ + 1));      // row norms of V, then of R: one buffer of d1 floats (shards sum it)
    L->off_rnorm = L->off_vnorm + sizeof(float) * nI;
    L->off_shard = take(sizeof(double) * 8);
    L->off_D = take(sizeof(double) * k);
    L->off_A = take(sizeof(double) * (ng - k > 0 ? ng - k : 1));
    L->off_c = take(sizeof(double) * (ng - k > 0 ? ng - k : 1) * g * g);
    L->off_small = take(sizeof(double) * 16 * g * g + 256);
    L->off_gramV = take(sizeof(double) * k * g * g);
    L->off_gramR = take(sizeof(double) * (ng - k > 0 ? ng - k : 1) * g * g);
    L->off_perm = take(sizeof(int32_t) * ng);
    L->off_slotof = take(sizeof(int32_t) * ng);
    L->off_energy = take(sizeof(double) * ng + sizeof(int32_t) * ng);
    constexpr int64_t NB = 64;                              // pivot block of the inversion (invert.cu)
    L->off_panel = take(sizeof(float) * (d1 * NB + 2 * NB * L->ldp + NB * NB));
    L->off_loop = take(2 * (size_t)kLoopMaxBlocks * 16 + 64);
    const size_t gg8 = sizeof(double) * g * g;
    const bool pairs_ok = L->pair_capacity > 0;
    L->off_pairCinv = take(pairs_ok ? gg8 * k : 8);
    L->off_pairKK = take(pairs_ok ? gg8 * k : 8);
    L->off_pairScratch = take(pairs_ok ? gg8 * 8 * 296 : 8);
    L->off_pairDelta = take(pairs_ok ? sizeof(double) * L->pair_capacity : 8);
    L->off_greedy = take(greedy_scratch_bytes(d1, m, g));
    {   // K panels of up to 2048 for the widest products of the state build (M <= d1, N <= max(m, n_I))
        const int64_t nmax = ldm > ldh ? ldm : ldh;
        L->tc_bytes = 3 * ((size_t)d1 * 2048 * 2 + (size_t)2048 * nmax * 2) + 16 * 1024;
        if (L->tc_bytes < gemm_tc_min_scratch(d1, nmax)) L->tc_bytes = gemm_tc_min_scratch(d1, nmax);
        L->off_tc = take(L->tc_bytes);
    }
    {   // block exchange: panels for up to min(OSSCAR_MAX_GROUP, n_I, n_J) rows on each side (a multiple of g)
        int64_t G = OSSCAR_MAX_GROUP;
        if (nI < G) G = nI;
        if (nJ < G) G = nJ;
        G = G / g * g;
        L->block_rows_max = (int32_t)G;
        const size_t n = G > 0 ? block_region_bytes(ldh, ldm, nJ, G) : 256;
        L->block_bytes = n;
        L->off_block = take(n);
    }
    L->bytes = off;
    return OSSCAR_OK;
}

int select_support(osscar_ctx* ctx, int mode, int32_t* support)
{
    const Layout& L = ctx->L;
    cudaStream_t st = ctx->stream;
    char* ws = (char*)ctx->ws;
    double* e = (double*)(ws + L.off_energy);
    int32_t* kept = (int32_t*)(e + L.ng);
    int32_t* perm = (int32_t*)(ws + L.off_perm);
    int32_t* slotof = (int32_t*)(ws + L.off_slotof);
    const unsigned nb = (unsigned)((L.ng + 7) / 8);          // eight groups per block
    if (mode == OSSCAR_INIT_USER) {
        CK(cudaMemsetAsync(kept, 0, sizeof(int32_t) * L.ng, st));
        k_user_support<<<(L.k + 255) / 256, 256, 0, st>>>(support, L.k, L.ng, kept, ctx->ctl);
        k_user_support_guard<<<1, 1024, 0, st>>>(kept, L.ng, L.k, ctx->ctl);
        count_launches(1);
    } else {
        k_energy<<<(unsigned)L.ng, 128, 0, st>>>(ctx->H, ctx->W, L.d1, L.m, L.g, mode, e);
        if (ctx->reduce) { const int rr = shard_reduce(ctx, e, L.ng, OSSCAR_FP64); if (rr != OSSCAR_OK) return rr; }   // energies are sums over columns
        k_rank_select<<<nb, 256, 0, st>>>(e, L.ng, L.k, kept);
    }
    k_build_perm<<<nb, 256, 0, st>>>(kept, L.ng, L.k, perm, slotof, support);
    count_launches(mode == OSSCAR_INIT_USER ? 2 : 3);
    CK(cudaGetLastError());
    return OSSCAR_OK;
}

// Scratch for a product of `rows` x K digits against N columns: B's digits go to the front of the tensor-core region, A's
// into what is left of it or into [other, other + bytes), whichever is larger.
static I8Scratch i8_scratch(osscar_ctx* ctx, int64_t N, int64_t K, int S, void* other, size_t other_bytes)
{
    const Layout& L = ctx->L;
    I8Scratch sc;
    char* tc = (char*)ctx->ws + L.off_tc;
    const size_t need_b = (gemm_i8_operand_bytes(N, K, S) + 255) / 256 * 256;
    sc.b = tc; sc.b_bytes = L.tc_bytes;
    sc.a = (void*)(((uintptr_t)other + 255) & ~(uintptr_t)255);
    sc.a_bytes = other_bytes > 256 ? other_bytes - 256 : 0;
    if (need_b < L.tc_bytes && L.tc_bytes - need_b > sc.a_bytes) {
        sc.b_bytes = need_b;
        sc.a = tc + need_b; sc.a_bytes = L.tc_bytes - need_b;
    }
    return sc;
}

// blocks per pruned slot of k_schur: about eight blocks per SM in all, each warp with at least one entry
static unsigned schur_shares(int64_t slots, int g)
{
    const int64_t want = (148 * 8 + slots - 1) / slots, most = ((int64_t)g * g + 7) / 8;
    return (unsigned)(want < 1 ? 1 : (want < most ? want : most));
}

constexpr int kResidualDigits = 6, kDirectDigits = 5;      // see gemm_i8.cu

// The products that only have to be as good as fp32 ones: four digits of an operand (31 bits below the largest entry of a row or
// column, balanced), three where the result is itself a small correction.  (Three for V left its error at d1 = 8192 at 3.8e-8
// against the 2.5e-8 of its fp32 rounding.)
cudaError_t inverse_product(osscar_ctx* ctx, int64_t N, const float* A, const float* B, int64_t ldb, float beta, const float* C0, float* C,
                            int64_t ldc, int digits, void* other, size_t other_bytes, const int32_t* skip)
{
    const Layout& L = ctx->L;
    char* ws = (char*)ctx->ws;
    const float* Hp = (const float*)(ws + L.off_Hp);
    I8Scratch sc = i8_scratch(ctx, N, L.nI, digits, other, other_bytes);
    if (gemm_i8_usable(L.nI, N, L.nI, digits, sc)) {
        I8Gemm p = {};
        p.M = L.nI; p.N = N; p.K = L.nI; p.alpha = 1.0; p.beta = beta;
        p.A = A; p.lda = L.ldh; p.B = B; p.ldb = ldb; p.C0 = beta != 0.f ? C0 : nullptr; p.ldc0 = ldc; p.C = C; p.ldc = ldc;
        p.diag = Hp; p.diag_stride = L.ldp + 1; p.inverse_scale = true;
        return gemm_i8(ctx->stream, p, digits, sc, ctx->ctl, skip);
    }
    // the smallest layers: one launch on the fp64 pipe instead of three (two splits and a product with a handful of tiles)
    if ((double)L.nI * L.nI * (double)N <= kTinyProduct)
        return gemm_f64acc(ctx->stream, L.nI, N, L.nI, 1.0, A, L.ldh, B, ldb, (double)beta, C0, ldc, C, ldc, false, skip);
    if (beta != 0.f && C0 != C) {
        const cudaError_t e = cudaMemcpyAsync(C, C0, sizeof(float) * L.nI * ldc, cudaMemcpyDeviceToDevice, ctx->stream);
        if (e != cudaSuccess) return e;
    }
    return gemm_tc(ctx->stream, L.nI, N, L.nI, 1.f, A, L.ldh, B, ldb, beta, C, ldc, ws + L.off_tc, L.tc_bytes, ctx->ctl, skip);
}

cudaError_t inverse_residual(osscar_ctx* ctx, float* E, bool v_free)
{
    const Layout& L = ctx->L;
    char* ws = (char*)ctx->ws;
    const float* Hp = (const float*)(ws + L.off_Hp);
    const float* Hinv = (const float*)(ws + L.off_Hinv);
    // the fp64 inverse is made from this residual, so its place (and, before V exists, the ones behind it) is free
    const size_t free_end = v_free ? L.off_y : L.off_V;
    I8Scratch sc = i8_scratch(ctx, L.nI, L.nI, kResidualDigits, ws + L.off_Hd, free_end - L.off_Hd);
    if (gemm_i8_usable(L.nI, L.nI, L.nI, kResidualDigits, sc)) {
        I8Gemm p = {};
        p.M = p.N = p.K = L.nI; p.alpha = -1.0; p.identity = true;
        p.A = Hp; p.lda = L.ldp; p.B = Hinv; p.ldb = L.ldh; p.C = E; p.ldc = L.ldh;
        p.diag = Hp; p.diag_stride = L.ldp + 1;
        return gemm_i8(ctx->stream, p, kResidualDigits, sc, ctx->ctl, nullptr);
    }
    return gemm_f64acc(ctx->stream, L.nI, L.nI, L.nI, -1.0, Hp, L.ldp, Hinv, L.ldh, 0.0, nullptr, 0, E, L.ldh, true);
}

cudaError_t refine_v(osscar_ctx* ctx, const float* GI, float* rV, void* other, size_t other_bytes, const int32_t* skip)
{
    const Layout& L = ctx->L;
    char* ws = (char*)ctx->ws;
    const float* Hp = (const float*)(ws + L.off_Hp);
    float* V = (float*)(ws + L.off_V);
    const int64_t nI = L.nI;
    I8Scratch sc = i8_scratch(ctx, L.m, nI, kResidualDigits, other, other_bytes);
    cudaError_t e;
    if (gemm_i8_usable(nI, L.m, nI, kResidualDigits, sc)) {
        I8Gemm p = {};
        p.M = nI; p.N = L.m; p.K = nI; p.alpha = -1.0; p.beta = 1.0;
        p.A = Hp; p.lda = L.ldp; p.B = V; p.ldb = L.ldm; p.C0 = GI; p.ldc0 = L.ldm; p.C = rV; p.ldc = L.ldm;
        p.diag = Hp; p.diag_stride = L.ldp + 1;
        e = gemm_i8(ctx->stream, p, kResidualDigits, sc, ctx->ctl, skip);
    } else
        e = gemm_f64acc(ctx->stream, nI, L.m, nI, -1.0, Hp, L.ldp, V, L.ldm, 1.0, GI, L.ldm, rV, L.ldm, false, skip);
    if (e != cudaSuccess) return e;
    return inverse_product(ctx, L.m, (const float*)(ws + L.off_Hinv), rV, L.ldm, 1.f, V, V, L.ldm, 4, other, other_bytes, skip);
}

// Free while the nested phase prepares H^-1 in the place of Hp: the regions behind it, up to the staged vectors, and the
// tensor-core region.  A column panel of E and its digits go into the latter, the digits of H or of H^-1 into the former.
struct DensePanels { int64_t np; float* E; I8Scratch sc; int digits; };
static bool dense_panels(const osscar_ctx* ctx, DensePanels* d)
{
    const Layout& L = ctx->L;
    char* ws = (char*)ctx->ws;
    const int64_t n = L.d1;
    d->digits = n <= 131071 / 5 ? 5 : 4;                             // contraction lengths that five (four) digits allow, see gemm_i8.cu
    const size_t per_col = sizeof(float) * (size_t)n + (size_t)d->digits * gemm_i8_row_bytes(n) + 16, fixed = 4 * (size_t)n + 8192;
    int64_t np = L.tc_bytes > fixed ? (int64_t)((L.tc_bytes - fixed) / per_col) / 256 * 256 : 0;
    if (np > n) np = round_up(n, 4);
    if (n < 4096 || np < 256) return false;
    d->np = np;
    const size_t e_bytes = (sizeof(float) * (size_t)n * np + 255) / 256 * 256;
    if (e_bytes >= L.tc_bytes) return false;
    d->E = (float*)(ws + L.off_tc);
    d->sc.b = ws + L.off_tc + e_bytes; d->sc.b_bytes = L.tc_bytes - e_bytes;
    d->sc.a = ws + L.off_Hinv; d->sc.a_bytes = L.off_y - L.off_Hinv;
    return gemm_i8_usable(n, 256, n, d->digits, d->sc);
}
bool dense_inverse_correctable(const osscar_ctx* ctx) { DensePanels d; return dense_panels(ctx, &d); }

cudaError_t correct_dense_inverse(osscar_ctx* ctx, float* A, int64_t lda)
{
    const int64_t n = ctx->L.d1;
    DensePanels d;
    if (!dense_panels(ctx, &d)) return cudaErrorInvalidValue;
    cudaStream_t st = ctx->stream;
    for (int64_t j0 = 0; j0 < n; j0 += d.np) {
        const int64_t w = n - j0 < d.np ? n - j0 : d.np;
        I8Gemm p = {};                       // E[:, j0:] = (I - H A)[:, j0:]
        p.M = p.K = n; p.N = w; p.alpha = -1.0; p.identity = true; p.identity_col0 = j0;
        p.A = ctx->H; p.lda = n; p.B = A + j0; p.ldb = lda; p.C = d.E; p.ldc = d.np;
        p.diag = ctx->H; p.diag_stride = n + 1;
        I8Scratch sc = d.sc;
        cudaError_t e = gemm_i8(st, p, d.digits, sc, ctx->ctl, nullptr);
        if (e != cudaSuccess) return e;
        // A[:, j0:] += A E[:, j0:]: a row's digits are taken before the row changes, and the columns already corrected only help
        p = {};
        p.M = p.K = n; p.N = w; p.alpha = 1.0; p.beta = 1.0;
        p.A = A; p.lda = lda; p.B = d.E; p.ldb = d.np; p.C0 = A + j0; p.ldc0 = lda; p.C = A + j0; p.ldc = lda;
        p.diag = ctx->H; p.diag_stride = n + 1; p.inverse_scale = true;
        sc = d.sc;
        e = gemm_i8(st, p, 3, sc, ctx->ctl, nullptr);
        if (e != cudaSuccess) return e;
    }
    k_add_sym<<<dim3((unsigned)((n + 31) / 32), (unsigned)((n + 31) / 32)), dim3(32, 8), 0, st>>>(A, lda, nullptr, 0, n);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t dense_inverse_times(osscar_ctx* ctx, const float* A, int64_t lda, const float* B, float* C, int64_t ldc)
{
    const Layout& L = ctx->L;
    const int64_t n = L.d1;
    DensePanels d;
    if (!dense_panels(ctx, &d)) return cudaErrorInvalidValue;
    I8Scratch sc;
    sc.a = d.sc.a; sc.a_bytes = d.sc.a_bytes;
    sc.b = (char*)ctx->ws + L.off_tc; sc.b_bytes = L.tc_bytes;
    if (!gemm_i8_usable(n, L.m, n, 4, sc))
        return sgemm(ctx->stream, false, false, n, L.m, n, 1.f, A, lda, B, L.m, 0.f, C, ldc);
    I8Gemm p = {};
    p.M = p.K = n; p.N = L.m; p.alpha = 1.0;
    p.A = A; p.lda = lda; p.B = B; p.ldb = L.m; p.C = C; p.ldc = ldc;
    p.diag = ctx->H; p.diag_stride = n + 1; p.inverse_scale = true;
    return gemm_i8(ctx->stream, p, 4, sc, ctx->ctl, nullptr);
}

// Builds every piece of the search state from H, G and the current slot permutation.
int build_state(osscar_ctx* ctx)
{
    const Layout& L = ctx->L;
    cudaStream_t st = ctx->stream;
    char* ws = (char*)ctx->ws;
    float* Hp = (float*)(ws + L.off_Hp);
    float* Hinv = (float*)(ws + L.off_Hinv);
    float* V = (float*)(ws + L.off_V);
    float* R = (float*)(ws + L.off_R);
    float* big = (float*)(ws + L.off_big);
    double* c = (double*)(ws + L.off_c);
    const int32_t* perm = (const int32_t*)(ws + L.off_perm);
    void* tc = ws + L.off_tc;
    const int64_t nI = L.nI, nJ = L.nJ;

    {   // slot-permuted copy of H
        dim3 grid((unsigned)((L.ldp + 1023) / 1024), (unsigned)((L.d1 + GS_R - 1) / GS_R));
        k_gather_sym<<<grid, 256, 0, st>>>(ctx->H, L.d1, L.g, perm, Hp, L.ldp);
    }
    CK(cudaMemsetAsync(ws + L.off_vec_begin, 0, L.off_vec_end - L.off_vec_begin, st));
    k_copy_pad<<<(unsigned)nI, 256, 0, st>>>(Hp, L.ldp, nI, nI, Hinv, L.ldh);
    count_launches(2);
    CK(cudaGetLastError());
    { const int rc_inv = invert_spd_inplace(ctx, Hinv, L.ldh, nI, Hp, L.ldp, true); if (rc_inv != OSSCAR_OK) return rc_inv; }
    // Every product below that forms a small difference of large sums is summed far beyond fp32 (digit products on the
    // int8 tensor cores, gemm_i8; small ones on the fp64 pipe, gemm_f64acc): the scores of Eq. impact are compared at 1e-5
    // relative, and fp32 accumulation leaves cond(H_II) * 2^-24 in them.
    // (1) the inverse.  Single-row groups: fp64 copy by a third-order correction from one fp64 residual, and the fp32
    //     inverse rounded from it (build_hinv64).  Groups of several rows: one Newton-Schulz step, E = I - H_II Hinv in
    //     fp64, Hinv := sym(Hinv + Hinv E) (E is tiny: any product will do), from kSweptRows rows up with E^2 as well
    ctx->hd_valid = false;
    if (L.g == 1) {
        const int rc_d = build_hinv64(ctx, true);
        if (rc_d != OSSCAR_OK) return rc_d;
    } else {
        float* E = big;
        float* Dlt = big + nI * L.ldh;
        CK(inverse_residual(ctx, E, true));
        if (nI >= kSweptRows) {          // Hinv + Hinv (E + E^2): the sweeps leave more in single entries, see kSweptRows
            CK(inverse_product(ctx, nI, E, E, L.ldh, 1.f, E, Dlt, L.ldh, 3, ws + L.off_Hd, L.off_y - L.off_Hd));
            float* t = E; E = Dlt; Dlt = t;
        }
        CK(inverse_product(ctx, nI, Hinv, E, L.ldh, 0.f, nullptr, Dlt, L.ldh, 3, ws + L.off_Hd, L.off_y - L.off_Hd));
        k_add_sym<<<dim3((unsigned)((nI + 31) / 32), (unsigned)((nI + 31) / 32)), dim3(32, 8), 0, st>>>(Hinv, L.ldh, Dlt, L.ldh, nI);
        count_launches(1);
    }
    // (2) V = Hinv G_I, then one refinement step with the residual G_I - H_II V
    float* GI = big;
    float* rV = big + nI * L.ldm;
    k_gather_rows<<<(unsigned)nI, 256, 0, st>>>(ctx->G, L.m, L.g, perm, 0, GI, L.ldm);
    count_launches(1);
    if (L.ldm != L.m) CK(cudaMemsetAsync(V, 0, sizeof(float) * nI * L.ldm, st));     // padding columns stay zero
    const int64_t big_floats = (int64_t)((L.off_Hp - L.off_big) / sizeof(float));
    {   // digits beside GI and rV, or in the place of R
        const size_t used = sizeof(float) * 2 * (size_t)nI * L.ldm, tail = sizeof(float) * (size_t)big_floats - used;
        const size_t rbytes = L.off_y - L.off_R;
        void* other = tail > rbytes ? (void*)((char*)big + used) : (void*)R;
        const size_t other_bytes = tail > rbytes ? tail : rbytes;
        CK(inverse_product(ctx, L.m, Hinv, GI, L.ldm, 0.f, nullptr, V, L.ldm, 4, other, other_bytes));
        CK(refine_v(ctx, GI, rV, other, other_bytes));
    }
    // obj = Tr(W^T G) - Tr(G_I^T V)
    if (ctx->have_const) CK(set_device_double(st, &ctx->ctl->acc[0], ctx->user_const));
    else CK(trace_product(st, ctx->W, L.m, ctx->G, L.m, L.d1, L.m, ctx->partials, &ctx->ctl->acc[0]));
    CK(trace_product(st, GI, L.ldm, V, L.ldm, nI, L.m, ctx->partials, &ctx->ctl->acc[1]));
    if (ctx->reduce) {      // both traces are sums over this shard's columns (a constant given by the caller is the layer's)
        double* sh = (double*)(ws + L.off_shard);
        k_pack2<<<1, 1, 0, st>>>(ctx->ctl, sh, 0);
        const int rr = shard_reduce(ctx, sh, 2, OSSCAR_FP64);
        if (rr != OSSCAR_OK) return rr;
        k_pack2<<<1, 1, 0, st>>>(ctx->ctl, sh, 1);
        if (ctx->have_const) CK(set_device_double(st, &ctx->ctl->acc[0], ctx->user_const));
        count_launches(2);
    }
    k_set_obj<<<1, 1, 0, st>>>(ctx->ctl);
    count_launches(1);
    if (nJ > 0) {
        // (3) R_J = G_J - Hp[J, I] V
        k_gather_rows<<<(unsigned)nJ, 256, 0, st>>>(ctx->G, L.m, L.g, perm, nI, R, L.ldm);
        count_launches(1);
        const float* HJI = Hp + nI * L.ldp;
        // single-row groups: partial sums of the quadratic forms at the end of `big`, the digits of H_JI in front of them
        // (used by both products); wider groups: Pm in `big`
        const bool one = L.g == 1;
        const size_t part_bytes = one ? sizeof(double) * (size_t)nJ * gemm_i8_dot_cols(nI) : 0;
        const size_t big_bytes = (sizeof(float) * (size_t)big_floats) / 256 * 256;
        const size_t room = big_bytes > part_bytes + 512 ? (big_bytes - part_bytes) / 256 * 256 : 0;
        double* part = (double*)((char*)big + room);
        I8Scratch scR;
        scR.a = big; scR.a_bytes = room; scR.b = tc; scR.b_bytes = L.tc_bytes;
        if (gemm_i8_usable(nJ, L.m, nI, kDirectDigits, scR)) {
            I8Gemm p = {};
            p.M = nJ; p.N = L.m; p.K = nI; p.alpha = -1.0; p.beta = 1.0;
            p.A = HJI; p.lda = L.ldp; p.B = V; p.ldb = L.ldm; p.C0 = R; p.ldc0 = L.ldm; p.C = R; p.ldc = L.ldm;
            p.diag = Hp; p.diag_stride = L.ldp + 1;
            CK(gemm_i8(st, p, kDirectDigits, scR, ctx->ctl, nullptr));
        } else
            CK(gemm_f64acc(st, nJ, L.m, nI, -1.0, HJI, L.ldp, V, L.ldm, 1.0, R, L.ldm, R, L.ldm, false));
        // (4) Schur complements H_qq - H_qI Hinv H_Iq.  Single-row groups need one quadratic form per pruned row, for which
        // half of the symmetric inverse is enough: from the fp64 inverse, with the dot products in the product's epilogue.
        if (one && gemm_i8_usable(nJ, nI, nI, kDirectDigits, scR)) {
            I8Gemm p = {};
            p.M = nJ; p.N = nI; p.K = nI; p.alpha = 1.0; p.tri = true; p.dot = true;
            p.A = HJI; p.lda = L.ldp; p.Bd = (const double*)(ws + L.off_Hd); p.ldb = L.ldh; p.C0 = HJI; p.ldc0 = L.ldp;
            p.C = part; p.ldc = gemm_i8_dot_cols(nI);
            p.diag = Hp; p.diag_stride = L.ldp + 1;
            CK(cudaMemsetAsync(part, 0, part_bytes, st));        // 256-column tiles fill half of the columns
            CK(gemm_i8(st, p, kDirectDigits, scR, ctx->ctl, nullptr));
            k_schur_sum<<<(unsigned)((nJ + 7) / 8), 256, 0, st>>>(Hp, L.ldp, part, p.ldc, (int)p.ldc, nI, nJ, c);
            count_launches(1);
        } else {
            // Pm = Hp[J, I] Hinv kept in fp64, in panels of whole pruned groups that fit the scratch, then fp64 dot products
            double* Pm = (double*)big;
            int64_t gpp = (big_floats / 2) / (L.ldh * L.g);                 // pruned groups per panel
            if (gpp < 1) return OSSCAR_E_WORKSPACE;
            for (int64_t t0 = 0; t0 < L.ng - L.k; t0 += gpp) {
                const int64_t ngr = L.ng - L.k - t0 < gpp ? L.ng - L.k - t0 : gpp;
                const float* At = Hp + (nI + t0 * L.g) * L.ldp;
                I8Scratch sc = i8_scratch(ctx, nI, nI, kResidualDigits, nullptr, 0);
                if (!one && gemm_i8_usable(ngr * L.g, nI, nI, kResidualDigits, sc)) {
                    I8Gemm p = {};
                    p.M = ngr * L.g; p.N = nI; p.K = nI; p.alpha = 1.0; p.out64 = true;
                    p.A = At; p.lda = L.ldp; p.B = Hinv; p.ldb = L.ldh; p.C = Pm; p.ldc = L.ldh;
                    p.diag = Hp; p.diag_stride = L.ldp + 1;
                    CK(gemm_i8(st, p, kResidualDigits, sc, ctx->ctl, nullptr));
                } else
                    CK(gemm_f64out(st, ngr * L.g, nI, nI, At, L.ldp, Hinv, L.ldh, Pm, L.ldh, one));
                k_schur<<<dim3((unsigned)ngr, schur_shares(ngr, L.g)), 256, 0, st>>>(Hp, L.ldp, Pm, L.ldh, nI, L.g, c, t0, one ? 2.0 : 1.0);
                count_launches(1);
            }
        }
    }
    CK(cudaGetLastError());
    return OSSCAR_OK;
}

}  // namespace osscar
