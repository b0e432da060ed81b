// Swap loop of single-row groups on one device with delayed updates: between two batches of candidate columns a swap touches vectors
// of d1 entries only, and no matrix of the state is read or written.  Included by search.cu after search_loop_g1.cuh.
//
// The state is one symmetric matrix S (the sweep of H on the kept rows) and the Gram matrix Gam = M M^T of M = [V; R],
//     S_II = -Hinv,  S_IJ = Hinv H_IJ,  S_JJ = H_JJ - H_JI Hinv H_IJ (the Schur complements c on its diagonal),
// and a swap is two pivots, the leaving row i and then the entering row q.  A pivot on p with s = S[:, p], a = 1 / S_pp,
// b = a s, g = Gam[:, p], n = Gam_pp, w = g - b n / 2 changes, outside row and column p,
//     S -= a s s^T,   Gam -= b w^T + w b^T,   M_r -= b_r M_p,
// and row p becomes |a| s (S_pp: -a), M_p becomes |a| M_p.  The scores are Gam_rr / |S_rr|, the exact change of obj of a swap
// needs entries (i, q) besides: diagonals and two columns per swap are all that the search reads.  So the matrices of the
// state stay as they were (the base), every pivot leaves its vectors s and w, kept in fp64, and a column as it is now is its base
// column less the terms.  Base columns are formed in batches for the DL_B best candidates of each side, one pass over
// H_JI, Hinv, V and R for all of them; the swaps that follow mostly stay inside the batch (27 to 31 of 32, or 8 to 9 where every swap moves the scores of many
// groups, as from the energy start at d1 = 28672 and 1024), and the first one that does not ends it: every choice is made from all scores,
// so the swaps are those of any other driver.  V, R, Hinv and Hp are brought up to date once, at the end (or when the terms fill
// their memory).
//
// Bound: the panel products of a batch (fp64 tensor path) at large sizes, the latency of a swap at small ones: about 11000 cycles,
// a third of them the grid barrier, the rest a chain of reductions, loads from L2 and fp64 operations.  A swap, its share of the
// batches and of the rewrite included, took before (matrices streamed in every step, or kept in L2 with three barriers) and takes
// now: 490 -> 160 us at d1 = 28672, m = 7168, k = 8602, 97 -> 30 us at 8192, 2048, 4096, 43 -> 16 us at 5000, 1283, 1777, 20 -> 11 us at
// 1024, 1024, 512, 14 -> 8 us at 64, 64, 32.  Where a batch lasts 8.6 swaps (28672, energy start) it is 490 -> 390 us.
//   select     candidates of both sides          stage, panel     base columns: products with up to 64 columns on the fp64
//   terms      sums over earlier pivots            apply              tensor path (mma m8n8k4), operands streamed once
//   loop       the swaps                           history ... rank   the matrices after a search
#pragma once

constexpr int DL_B = 32, DL_N = 2 * DL_B;        // candidates per side, columns of a batch
constexpr int DL_KB = 2 * DL_B;                  // pivots (terms) of a batch
constexpr int DL_T = 512;                        // threads of the loop
constexpr int DL_MAX_BLOCKS = DL_T / 2;          // blocks of the loop: a thread for each of their candidates
constexpr int DL_MAX_TERMS = 1024;               // terms between two rewrites of the matrices
// Swaps asked for from which AUTO takes this loop.  Its fixed cost is the first batch and the rewrite, and AUTO cannot see how early a search stops.
// Search of 4, 8, 12 and 16 swaps in us, this loop / the one AUTO took before it: 130 / 96, 145 / 152, 164 / 207, 179 / 264 at d1 = 64;
// 187 / 117, 220 / 194, 246 / 268, 272 / 344 at 1024; 289 / 242, 317 / 411, 352 / 573, 378 / 744 at 5000, 1283; 557 / 444, 582 / 830, 640 / 1219,
// 670 / 1600 at 8192, 2048; 5350 / 2350, 5380 / 4470, 5390 / 6690, 5590 / 8670 at 28672, 7168; 427 / 146, 456 / 263, 492 / 381, 518 / 506 at 90, 20001.
// A search that may make hundreds and finds nothing to swap takes 105 / 41, 104 / 45, 182 / 72, 316 / 726, 3300 / 3100.
constexpr int DL_MIN_SWAPS = 10, DL_MIN_SWAPS_WIDE = 16;

// Best row of a block: score (smallest is best), diagonals, group, slot, last pivot on it, column in the batch.
struct __align__(16) DlCand { double val, S, G; int32_t id, idx, last, col; double pad; };
struct DlPtrs {
    double *s, *w;               // terms [k][ld]
    double *alpha, *nu;          // 1 / S_pp and Gam_pp of a pivot
    double *S0, *G0;             // columns of the batch [c][ld]
    double *cs, *cw;             // terms at the candidates [k][DL_N]
    double *Sd, *Gd, *hd, *val;  // diagonals by slot; diagonal of H; scores, the best one smallest (infinite: not a candidate)
    double *By, *Bh, *Bg;        // right-hand sides of the panel products: [k][DL_B], [k][DL_N], [k][DL_N]
    double *py, *ph, *pg;        // their partial sums [z][c][rows]
    double *ts, *tg;             // sums over the terms [z][c][d1]
    DlCand* cands;               // [2][2][DL_MAX_BLOCKS]
    int32_t *last, *kept, *cidx, *cand, *src;      // by slot: last pivot (-1: none), kept now, column in the batch (-1: none); slots of the columns; slot of the group that moves here
    float *coef, *mk;            // rewrite: coefficients [d1][kp], rows of the pivots [k][ldm]
    int64_t ld;
    int kcap, zy, zh, zg, zt;    // terms that fit; k-slices of the panel products and of the sums over terms
};

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Score of a slot: rise of obj if a kept one leaves, fall if a pruned one enters; false where it cannot be chosen.
__device__ __forceinline__ bool dl_score(bool kept, double S, double G, double hd, double* v) {
    if (kept) { *v = -S > 0.0 ? G / -S : INFINITY; }
    else *v = S > kAddPivotTol * hd ? G / S : -INFINITY;
    return isfinite(*v);
}

// Diagonals of S and Gam from the matrices of the state; a warp per row.
__global__ void __launch_bounds__(256) k_dl_init(Ptrs p, DlPtrs z)
{
    if (p.ctl->done) return;
    const int64_t r = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (blockIdx.x == 0 && threadIdx.x == 0) { p.ctl->dl_terms = 0; p.ctl->dl_stop = 0; }
    if (r >= p.nI + p.nJ) return;
    const int lane = threadIdx.x & 31;
    const bool kept = r < p.nI;
    const float4* row = reinterpret_cast<const float4*>(kept ? p.V + r * p.ldm : p.R + (r - p.nI) * p.ldm);
    double n = 0.0;
    for (int64_t c = lane; c < p.ldm / 4; c += 32) {
        const float4 v = row[c];
        n += ((double)v.x * v.x + (double)v.y * v.y) + ((double)v.z * v.z + (double)v.w * v.w);
    }
    n = warp_sum_d(n);
    if (lane == 0) {
        z.Gd[r] = n;
        z.Sd[r] = kept ? -p.Hd[r * p.ldh + r] : p.c[r - p.nI];
        z.hd[r] = (double)p.Hp[r * p.ldp + r];
        z.last[r] = -1; z.kept[r] = kept ? 1 : 0; z.cidx[r] = -1;
        double v;
        const bool ok = dl_score(kept, z.Sd[r], n, z.hd[r], &v);
        z.val[r] = ok ? (kept ? v : -v) : INFINITY;
    }
}

// Lane l has entry l of a list: score and group, ordered by score, then by group.
__device__ __forceinline__ void dl_exchange(double& v, int& id, int j, bool low) {
    const double ov = __shfl_xor_sync(0xffffffffu, v, j);
    const int oid = __shfl_xor_sync(0xffffffffu, id, j);
    const bool less = ov < v || (ov == v && oid < id), same = ov == v && oid == id;
    if (less == low && !same) { v = ov; id = oid; }
}
__device__ __forceinline__ void dl_sort32(double& v, int& id, int lane) {
#pragma unroll
    for (int k = 2; k <= 32; k <<= 1)
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) dl_exchange(v, id, j, ((lane & j) == 0) == ((lane & k) == 0));
}
// The 32 first of two sorted lists of 32, sorted.
__device__ __forceinline__ void dl_merge32(double& v, int& id, double ov, int oid, int lane) {
    ov = __shfl_sync(0xffffffffu, ov, 31 - lane);
    oid = __shfl_sync(0xffffffffu, oid, 31 - lane);
    if (ov < v || (ov == v && oid < id)) { v = ov; id = oid; }
#pragma unroll
    for (int j = 16; j > 0; j >>= 1) dl_exchange(v, id, j, (lane & j) == 0);
}
// Candidates: block 0 the kept slots with the smallest scores, block 1 the pruned ones with the largest: the first DL_B of the 2048 slots
// that are among the two best of a thread's share.  The best slot is always there (the swap that comes next); a third one of the first 32
// in one share is rare, and the set only decides how long a batch lasts.  (One per thread ended batches of 28 swaps after 24 at
// d1 = 28672.)  Lists of 32 are sorted and merged by warps, in registers: a sort of all 2048 entries in shared memory, with a barrier for each
// of its 66 steps, took 8 us longer, whatever the layer (51 swaps in 6 batches at d1 = 1024: 1.076 -> 1.034 ms).
__global__ void __launch_bounds__(1024) k_dl_select(Ptrs p, DlPtrs z)
{
    static_assert(DL_B == 32, "a candidate per lane");
    if (p.ctl->done || p.ctl->dl_stop) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) { p.ctl->bar_count = 0; p.ctl->abort = 0; }          // for the loop's grid barrier
    const int side = blockIdx.x, t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int64_t d1 = p.nI + p.nJ;
    __shared__ double sv[32][32];
    __shared__ int sx[32][32];
    double v0 = INFINITY, v1 = INFINITY; int i0 = INT_MAX, i1 = INT_MAX;
    for (int64_t r = t; r < d1; r += 1024) {
        if ((z.kept[r] != 0) != (side == 0)) continue;
        z.cidx[r] = -1;
        const double v = z.val[r];
        if (!(v < INFINITY) || v > v1) continue;
        const int id = p.perm[r];
        if (v < v0 || (v == v0 && id < i0)) { v1 = v0; i1 = i0; v0 = v; i0 = id; }
        else if (v < v1 || id < i1) { v1 = v; i1 = id; }
    }
    dl_sort32(v0, i0, lane);
    dl_sort32(v1, i1, lane);
    dl_merge32(v0, i0, v1, i1, lane);
    for (int n = 16; n > 0; n >>= 1) {               // the upper half of the lists into the lower one
        if (warp >= n && warp < 2 * n) { sv[warp][lane] = v0; sx[warp][lane] = i0; }
        __syncthreads();
        if (warp < n) dl_merge32(v0, i0, sv[warp + n][lane], sx[warp + n][lane], lane);
    }
    if (t < DL_B) {
        const int x = i0 != INT_MAX ? p.slotof[i0] : -1;
        z.cand[side * DL_B + t] = x;
        if (x >= 0) z.cidx[x] = side * DL_B + t;
    }
}

// Right-hand sides: columns of the inverse (kept candidates) and rows H_qI (pruned ones), rows of M.  A slot that was a pivot
// before has its column among the terms: zeros.  Blocks [0, nbI): 32 entries of the n_I-vectors, [nbI, nbI + nbM): of the rows of M,
// the rest: s and w of 32 earlier terms at the candidates, less those that a candidate's own pivot has replaced.
__global__ void __launch_bounds__(256) k_dl_stage(Ptrs p, DlPtrs z, unsigned nbI, unsigned nbM)
{
    pdl_wait_then_release();
    if (p.ctl->done || p.ctl->dl_stop) return;
    __shared__ double tile[DL_N][33];
    if (blockIdx.x >= nbI + nbM) {
        const int K0 = p.ctl->dl_terms, k0 = (int)(blockIdx.x - nbI - nbM) * 32;
        for (int i = threadIdx.x; i < 32 * DL_N; i += 256) {
            const int k = k0 + i / DL_N, c = i % DL_N;
            if (k >= K0) break;
            const int x = z.cand[c];
            const bool on = x >= 0 && k > z.last[x];
            const int64_t o = (int64_t)k * z.ld + (on ? x : 0);
            z.cs[(int64_t)k * DL_N + c] = on ? z.s[o] : 0.0;
            z.cw[(int64_t)k * DL_N + c] = on ? z.w[o] : 0.0;
        }
        return;
    }
    const bool rows = blockIdx.x >= nbI;
    const int64_t k0 = (int64_t)(rows ? blockIdx.x - nbI : blockIdx.x) * 32, K = rows ? p.ldm : p.nI;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t k = k0 + lane;
    for (int c = w; c < DL_N; c += 8) {
        const int x = z.cand[c];
        double v = 0.0;
        if (x >= 0 && z.last[x] < 0 && k < K) {
            if (rows) v = (double)(x < p.nI ? p.V[(int64_t)x * p.ldm + k] : p.R[(int64_t)(x - p.nI) * p.ldm + k]);
            else v = x < p.nI ? p.Hd[(int64_t)x * p.ldh + k] : (double)p.Hp[(int64_t)x * p.ldp + k];
        }
        tile[c][lane] = v;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 32 * DL_N; i += 256) {
        const int c = i % DL_N;
        const int64_t kk = k0 + i / DL_N;
        if (kk >= K) break;
        const double v = tile[c][i / DL_N];
        if (rows) z.Bg[kk * DL_N + c] = v;
        else if (c < DL_B) z.Bh[kk * DL_N + c] = v;
        else z.By[kk * DL_B + c - DL_B] = v;
    }
}
// Hinv h of the pruned candidates from the slices of the product: right-hand sides of the H pass, and the kept rows of their columns.
__global__ void __launch_bounds__(256) k_dl_stage_y(Ptrs p, DlPtrs z)
{
    pdl_wait_then_release();
    if (p.ctl->done || p.ctl->dl_stop) return;
    __shared__ double tile[DL_B][33];
    const int64_t k0 = (int64_t)blockIdx.x * 32;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t k = k0 + lane;
    for (int c = w; c < DL_B; c += 8) {
        double v = 0.0;
        if (k < p.nI) {
            for (int i = 0; i < z.zy; ++i) v += z.py[((int64_t)i * DL_B + c) * p.nI + k];
            z.S0[(int64_t)(DL_B + c) * z.ld + k] = v;
        }
        tile[c][lane] = v;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 32 * DL_B; i += 256) {
        const int c = i % DL_B;
        const int64_t kk = k0 + i / DL_B;
        if (kk >= p.nI) break;
        z.Bh[kk * DL_N + DL_B + c] = tile[c][i / DL_B];
    }
}

__device__ __forceinline__ void dl_dmma(double& d0, double& d1, double a, double b) {
    asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};" : "+d"(d0), "+d"(d1) : "d"(a), "d"(b));
}

__device__ __forceinline__ void dl_cp16(void* dst, const void* src, int bytes) {          // bytes of the 16 that exist; the rest is zero
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(bytes) : "memory");
}

// out[z][c][row] = sum over slice z of k of A[row][k] B[k][c], c < BN, sums in fp64.  Block: 128 rows, 16 k a step, 8 warps of
// 32 x 32 (BN = 64) or 16 x 32 (BN = 32); operands as they are through a ring of DL_PS steps of asynchronous copies, A converted when
// its fragments are read.  A: rows [0, split) of A0, the others of A1 (row starts 16-byte aligned, whole pieces inside the matrix).
// At d1 = 28672, m = 7168, k = 8602 the three products of a batch are 53 GFLOP; with one step of registers ahead and the operands
// converted on their way into shared memory they took 3.7 ms, and 512 swaps 13 ms more of a solve (376 -> 362 ms; 31.8 -> 30.1 ms at 8192, 2048,
// 7.20 -> 6.98 ms at 5000, 1283).
constexpr int DL_PS = 4;
template <typename TA, int BN> constexpr int dl_panel_smem() { return DL_PS * (128 * 20 * (int)sizeof(TA) + 16 * (BN + 4) * 8); }
template <typename TA, int BN>
__global__ void __launch_bounds__(256, 2)
k_dl_panel(int64_t M, int64_t K, const TA* A0, const TA* A1, int64_t split, int64_t lda, const double* B, double* out, int slices, const SearchCtl* ctl)
{
    pdl_wait_then_release();
    if (ctl->done || ctl->dl_stop) return;
    constexpr int BM = 128, BK = 16, AS = BK + 4, BS = BN + 4, WN = BN / 32, WM = 8 / WN, TI = BM / WM / 8;
    constexpr int PE = 16 / (int)sizeof(TA), PR = BK / PE, AV = BM * PR / 256, BV = BK * BN / 2 / 256;      // elements of a piece, pieces of a row, per thread
    extern __shared__ __align__(16) double dl_smem[];
    TA* const As = reinterpret_cast<TA*>(dl_smem);
    double* const Bs = reinterpret_cast<double*>(As + DL_PS * BM * AS);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, wm = warp / WN, wn = warp % WN;
    const int64_t m0 = (int64_t)blockIdx.x * BM;
    const int64_t steps = (K + BK - 1) / BK, kb = steps * blockIdx.y / slices, ke = steps * (blockIdx.y + 1) / slices;
    const TA* arow[AV];
#pragma unroll
    for (int q = 0; q < AV; ++q) {
        int64_t r = m0 + (tid + q * 256) / PR;
        if (r >= M) r = M - 1;
        arow[q] = r < split ? A0 + r * lda : A1 + (r - split) * lda;
    }
    double acc[TI][4][2];
#pragma unroll
    for (int i = 0; i < TI; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) { acc[i][j][0] = 0.0; acc[i][j][1] = 0.0; }
    auto load = [&](int64_t kt) {
        if (kt < ke) {
            const int64_t k0 = kt * BK;
            TA* a = As + (kt - kb) % DL_PS * (BM * AS);
            double* b = Bs + (kt - kb) % DL_PS * (BK * BS);
#pragma unroll
            for (int q = 0; q < AV; ++q) {
                const int i = tid + q * 256, c = (i % PR) * PE;
                const int64_t left = K - k0 - c;          // what lies behind the row's end is not part of the product, whatever it holds
                const int n = left >= PE ? 16 : (left > 0 ? (int)left * (int)sizeof(TA) : 0);
                dl_cp16(a + (i / PR) * AS + c, n > 0 ? arow[q] + k0 + c : arow[q], n);
            }
#pragma unroll
            for (int q = 0; q < BV; ++q) {
                const int i = tid + q * 256, kr = i / (BN / 2), c = (i % (BN / 2)) * 2;
                const bool in = k0 + kr < K;
                dl_cp16(b + kr * BS + c, in ? B + (k0 + kr) * BN + c : B, in ? 16 : 0);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    const int fr = lane >> 2, fk = lane & 3;
#pragma unroll
    for (int i = 0; i < DL_PS - 1; ++i) load(kb + i);
    for (int64_t kt = kb; kt < ke; ++kt) {
        asm volatile("cp.async.wait_group %0;" ::"n"(DL_PS - 2) : "memory");
        __syncthreads();
        load(kt + DL_PS - 1);                        // into the place that every warp has left behind
        const TA* a = As + (kt - kb) % DL_PS * (BM * AS) + (wm * TI * 8) * AS;
        const double* b = Bs + (kt - kb) % DL_PS * (BK * BS) + wn * 32;
#pragma unroll
        for (int ks = 0; ks < BK; ks += 4) {
            double af[TI], bf[4];
#pragma unroll
            for (int i = 0; i < TI; ++i) af[i] = (double)a[(i * 8 + fr) * AS + ks + fk];
#pragma unroll
            for (int j = 0; j < 4; ++j) bf[j] = b[(ks + fk) * BS + j * 8 + fr];
#pragma unroll
            for (int i = 0; i < TI; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) dl_dmma(acc[i][j][0], acc[i][j][1], af[i], bf[j]);
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
#pragma unroll
    for (int i = 0; i < TI; ++i) {
        const int64_t row = m0 + wm * TI * 8 + i * 8 + fr;
        if (row >= M) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int e = 0; e < 2; ++e) out[((int64_t)blockIdx.y * BN + wn * 32 + j * 8 + 2 * fk + e) * M + row] = acc[i][j][e];
    }
}

// Sums over the terms so far in the columns of the batch: ts[z][c][r] = sum_k alpha_k s_k[r] s_k[x_c] and
// tg = sum_k alpha_k (s_k[r] w_k[x_c] + w_k[r] s_k[x_c]), terms after the last pivot on r and on x_c only.  Tiles and layout as in k_dl_panel.
// (A thread per row with a loop over the terms took 55 us at d1 = 1024 and 650 us at d1 = 28672.)
__global__ void __launch_bounds__(256, 1) k_dl_terms(Ptrs p, DlPtrs z)
{
    pdl_wait_then_release();
    const int K = p.ctl->dl_terms;
    if (p.ctl->done || p.ctl->dl_stop || K == 0) return;
    constexpr int BM = 128, BK = 16, AS = BK + 4, BS = DL_N + 4, ABUF = BM * AS, BBUF = BK * BS;
    extern __shared__ double dl_smem[];
    double *As = dl_smem, *Bs = dl_smem + 4 * ABUF;               // [buffer][s, w]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, wm = warp >> 1, wn = warp & 1;
    const int64_t d1 = p.nI + p.nJ, m0 = (int64_t)blockIdx.x * BM;
    const int steps = (K + BK - 1) / BK, kb = steps * blockIdx.y / gridDim.y, ke = steps * (blockIdx.y + 1) / gridDim.y;
    const int64_t r = m0 + tid % BM;                              // this thread loads one row: terms tid / 128 + 2 q of a step
    const int lr = r < d1 ? z.last[r] : INT_MAX;
    double as[4][4][2], ag[4][4][2];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) as[i][j][0] = as[i][j][1] = ag[i][j][0] = ag[i][j][1] = 0.0;
    double rs[8], rw[8];
    double2 bs[2], bw[2];
    auto fetch = [&](int kt) {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int k = kt * BK + tid / BM + 2 * q;
            const bool on = k < K && k > lr;
            const double al = on ? z.alpha[k] : 0.0;
            rs[q] = on ? al * z.s[(int64_t)k * z.ld + r] : 0.0;
            rw[q] = on ? al * z.w[(int64_t)k * z.ld + r] : 0.0;
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int i = tid + q * 256, k = kt * BK + i / (DL_N / 2), c = (i % (DL_N / 2)) * 2;
            bs[q] = k < K ? *reinterpret_cast<const double2*>(z.cs + (int64_t)k * DL_N + c) : make_double2(0.0, 0.0);
            bw[q] = k < K ? *reinterpret_cast<const double2*>(z.cw + (int64_t)k * DL_N + c) : make_double2(0.0, 0.0);
        }
    };
    auto stash = [&](int buf) {
        double *a = As + buf * 2 * ABUF, *b = Bs + buf * 2 * BBUF;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int o = (tid % BM) * AS + tid / BM + 2 * q;
            a[o] = rs[q]; a[ABUF + o] = rw[q];
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int i = tid + q * 256, o = (i / (DL_N / 2)) * BS + (i % (DL_N / 2)) * 2;
            b[o] = bs[q].x; b[o + 1] = bs[q].y; b[BBUF + o] = bw[q].x; b[BBUF + o + 1] = bw[q].y;
        }
    };
    const int fr = lane >> 2, fk = lane & 3;
    if (kb < ke) { fetch(kb); stash(0); }
    __syncthreads();
    for (int kt = kb; kt < ke; ++kt) {
        const int buf = (kt - kb) & 1;
        if (kt + 1 < ke) fetch(kt + 1);
        const double *a = As + buf * 2 * ABUF + (wm * 32) * AS, *b = Bs + buf * 2 * BBUF + wn * 32;
#pragma unroll
        for (int ks = 0; ks < BK; ks += 4) {
            double fs[4], fw[4], gs[4], gw[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) { const int o = (i * 8 + fr) * AS + ks + fk; fs[i] = a[o]; fw[i] = a[ABUF + o]; }
#pragma unroll
            for (int j = 0; j < 4; ++j) { const int o = (ks + fk) * BS + j * 8 + fr; gs[j] = b[o]; gw[j] = b[BBUF + o]; }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    dl_dmma(as[i][j][0], as[i][j][1], fs[i], gs[j]);
                    dl_dmma(ag[i][j][0], ag[i][j][1], fs[i], gw[j]);
                    dl_dmma(ag[i][j][0], ag[i][j][1], fw[i], gs[j]);
                }
        }
        if (kt + 1 < ke) stash(buf ^ 1);
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int64_t row = m0 + wm * 32 + i * 8 + fr;
        if (row >= d1) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int64_t o = ((int64_t)blockIdx.y * DL_N + wn * 32 + j * 8 + 2 * fk + e) * d1 + row;
                z.ts[o] = as[i][j][e]; z.tg[o] = ag[i][j][e];
            }
    }
}

// The columns of the batch as they are now: the base, or what the last pivot on the row or on the column left, less the terms since.
constexpr int DL_AC = 2;                         // columns per block
__global__ void __launch_bounds__(128) k_dl_apply(Ptrs p, DlPtrs z)
{
    pdl_wait_then_release();
    if (p.ctl->done || p.ctl->dl_stop) return;
    const int K0 = p.ctl->dl_terms;
    const int64_t r = (int64_t)blockIdx.x * 128 + threadIdx.x, d1 = p.nI + p.nJ;
    if (r >= d1) return;
    const int lr = z.last[r];
#pragma unroll
    for (int i = 0; i < DL_AC; ++i) {
        const int c = blockIdx.y * DL_AC + i, x = z.cand[c];
        if (x < 0) continue;
        const int lx = z.last[x], m = lr > lx ? lr : lx;
        double v = 0.0, g = 0.0;
        if (m >= 0) {                        // entry (r, x) right after pivot m, which was on r or on x
            const int64_t o = (int64_t)m * z.ld + (lr > lx ? x : r);
            const double al = z.alpha[m], sv = z.s[o];
            v = fabs(al) * sv;
            g = fabs(al) * (z.w[o] - 0.5 * al * sv * z.nu[m]);
            if (r == x) { v = -al; g = al * al * z.nu[m]; }
        } else {
            const int64_t y = r - p.nI;
            for (int k = 0; k < z.zg; ++k) g += z.pg[((int64_t)k * DL_N + c) * d1 + r];
            if (r < p.nI) v = x < p.nI ? -p.Hd[(int64_t)x * p.ldh + r] : z.S0[(int64_t)c * z.ld + r];
            else {
                for (int k = 0; k < z.zh; ++k) v += z.ph[((int64_t)k * DL_N + c) * p.nJ + y];
                if (x >= p.nI) v = (double)p.Hp[(int64_t)x * p.ldp + r] - v;
            }
        }
        if (K0 > 0)
            for (int k = 0; k < z.zt; ++k) {
                const int64_t o = ((int64_t)k * DL_N + c) * d1 + r;
                v -= z.ts[o]; g -= z.tg[o];
            }
        z.S0[(int64_t)c * z.ld + r] = v;
        z.G0[(int64_t)c * z.ld + r] = g;
    }
}

struct DlArgs {
    Ptrs p; DlPtrs z;
    double* obj_trace; int32_t* swap_trace;
    double tol;
    int accept_mode, max_swaps;      // the loop ends when ctl->n_swaps reaches max_swaps
    int rows, kb;                    // rows per block, terms this launch may add
};
constexpr size_t DL_SMEM_MAX = 219 * 1024;       // beside 7.4 KB of static arrays
// dynamic shared memory of the loop: the batch's terms and the diagonals of the block's rows, partial sums of the k-slices
inline size_t dl_loop_smem(int rows, int kb) {
    const int nrp = (rows + 31) / 32 * 32;
    const int slices = nrp >= DL_T ? 1 : DL_T / nrp > 8 ? 8 : DL_T / nrp;
    return sizeof(double) * ((size_t)2 * kb * nrp + 3 * nrp + (size_t)(slices - 1) * 4 * nrp) + sizeof(int) * 4 * (size_t)nrp;
}

__device__ __forceinline__ uint64_t dl_ordered(double v) {              // whole numbers in the order of v; zeros of both signs alike, as in k_dl_select
    const uint64_t b = (uint64_t)__double_as_longlong(v + 0.0);
    return b ^ ((uint64_t)((int64_t)b >> 63) | 0x8000000000000000ull);
}
// Lane of the warp with the smallest (val, id); -1 where no lane has one.
__device__ __forceinline__ int dl_warp_best(const DlCand& c) {
    const uint64_t k = c.idx >= 0 ? dl_ordered(c.val) : ~0ull;
    const uint32_t hi = __reduce_min_sync(0xffffffffu, (uint32_t)(k >> 32));
    if (hi == 0xffffffffu) return -1;
    const uint32_t lo = __reduce_min_sync(0xffffffffu, (uint32_t)(k >> 32) == hi ? (uint32_t)k : 0xffffffffu);
    const bool mine = (uint32_t)(k >> 32) == hi && (uint32_t)k == lo;
    const uint32_t id = __reduce_min_sync(0xffffffffu, mine ? (uint32_t)c.id : 0xffffffffu);
    return __ffs(__ballot_sync(0xffffffffu, mine && (uint32_t)c.id == id)) - 1;
}
__device__ __forceinline__ void dl_keep(DlCand& b, double v, double S, double G, int id, int idx, int last, int col) {
    if (b.idx < 0 || cand_less(v, id, b.val, b.id)) { b.val = v; b.S = S; b.G = G; b.id = id; b.idx = idx; b.last = last; b.col = col; }
}
// The swaps of a batch: one cooperative kernel, a block owns `rows` slots, one grid barrier per swap.  Then every block
// takes the best leaving and entering slot of all blocks and decides the swap for itself, from the same numbers, moves the
// diagonals of its own slots and names its new candidates.  Ends when a choice has no column here,
// the terms are full, the loop stops or max_swaps is reached.
__global__ void __launch_bounds__(DL_T, 1) k_dl_loop(const DlArgs a)
{
    const Ptrs& p = a.p;
    const DlPtrs& z = a.z;
    SearchCtl* ctl = p.ctl;
    if (ctl->done || ctl->dl_stop) return;                     // set by an earlier kernel: the same in every block
    extern __shared__ double dl_smem[];
    __shared__ DlCand s_best[2][DL_T / 32], s_all[DL_T / 32], s_i, s_q;
    __shared__ double2 s_ci[DL_KB], s_cq[DL_KB];               // alpha_k (s_k, w_k) at the two slots
    __shared__ double s_co[4][DL_KB], s_al[DL_KB], s_nu[DL_KB], s_cross[2];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int nrp = (a.rows + 31) / 32 * 32;
    const int64_t d1 = p.nI + p.nJ, row0 = (int64_t)blockIdx.x * a.rows;
    const int nr = (int)(d1 - row0 < a.rows ? (d1 > row0 ? d1 - row0 : 0) : a.rows);
    const int slices = nrp >= DL_T ? 1 : DL_T / nrp > 8 ? 8 : DL_T / nrp;
    double* hs = dl_smem;                                      // [term][row]
    double* hw = hs + (size_t)a.kb * nrp;
    double *Sd = hw + (size_t)a.kb * nrp, *Gd = Sd + nrp, *hd = Gd + nrp, *red = hd + nrp;
    int* last = reinterpret_cast<int*>(red + (size_t)(slices - 1) * 4 * nrp);
    int *kept = last + nrp, *gid = kept + nrp, *col = gid + nrp;
    const int K0 = ctl->dl_terms;
    int n_swaps = ctl->n_swaps;
    double obj = ctl->obj;
    const long long limit = ctl->wait_limit;
    unsigned long long epoch = 0;
    __shared__ int s_flag;
    const int my0 = slices > 1 ? t % nrp : t, slice = slices > 1 ? t / nrp : 0, my_step = slices > 1 ? nrp : DL_T;
    const bool worker = slice < slices;

    DlCand bd, ba;
    bd.idx = -1; bd.val = 0.0; bd.S = bd.G = 0.0; bd.id = 0; bd.last = -1; bd.col = -1; bd.pad = 0.0; ba = bd;
    for (int lr = t; lr < nr; lr += DL_T) {
        const int64_t r = row0 + lr;
        Sd[lr] = z.Sd[r]; Gd[lr] = z.Gd[r]; hd[lr] = z.hd[r]; last[lr] = z.last[r]; kept[lr] = z.kept[r]; gid[lr] = p.perm[r]; col[lr] = z.cidx[r];
        double v;
        if (dl_score(kept[lr], Sd[lr], Gd[lr], hd[lr], &v)) dl_keep(kept[lr] ? bd : ba, kept[lr] ? v : -v, Sd[lr], Gd[lr], gid[lr], (int)r, last[lr], col[lr]);
    }
    int nb = 0, buf = 0, stop = 0;                             // terms of this launch; 1: search ends, 2: terms full, 3: batch ends
    for (;;) {
        // candidates of the block, then of all blocks
        {
            const int wd = dl_warp_best(bd), wa = dl_warp_best(ba);
            if (lane == (wd < 0 ? 0 : wd)) s_best[0][warp] = bd;
            if (lane == (wa < 0 ? 0 : wa)) s_best[1][warp] = ba;
        }
        __syncthreads();
        if (gridDim.x == 1) {
            if (warp < 2) {
                DlCand c = s_best[warp][lane < DL_T / 32 ? lane : 0];
                if (lane >= DL_T / 32) c.idx = -1;
                const int w = dl_warp_best(c);
                if (lane == (w < 0 ? 0 : w)) { if (warp == 0) s_i = c; else s_q = c; }
            }
        } else {
            DlCand* list = z.cands + (size_t)buf * 2 * DL_MAX_BLOCKS;
            if (warp < 2) {
                DlCand c = s_best[warp][lane < DL_T / 32 ? lane : 0];
                if (lane >= DL_T / 32) c.idx = -1;
                const int w = dl_warp_best(c);
                if (lane == (w < 0 ? 0 : w)) list[(size_t)warp * DL_MAX_BLOCKS + blockIdx.x] = c;
            }
            if (!grid_barrier(ctl, epoch, gridDim.x, limit, &s_flag)) return;
            DlCand c; c.idx = -1; c.val = c.S = c.G = c.pad = 0.0; c.id = 0; c.last = c.col = -1;
            const int from = t & (DL_MAX_BLOCKS - 1), side = t / DL_MAX_BLOCKS;
            if (from < (int)gridDim.x) c = list[(size_t)side * DL_MAX_BLOCKS + from];
            const int w = dl_warp_best(c);
            if (lane == (w < 0 ? 0 : w)) s_all[warp] = c;
            __syncthreads();
            if (warp < 2) {
                DlCand x = s_all[warp * (DL_MAX_BLOCKS / 32) + (lane & (DL_MAX_BLOCKS / 32 - 1))];
                const int b = dl_warp_best(x);
                if (lane == (b < 0 ? 0 : b)) { if (warp == 0) s_i = x; else s_q = x; }
            }
        }
        __syncthreads();
        const int i = s_i.idx, q = s_q.idx;
        if (i < 0 || q < 0) {
            if (blockIdx.x == 0 && t == 0) { ctl->done = 1; ctl->stop_reason = OSSCAR_STOP_GUARD; *p.done_host = 1; }
            stop = 1;
            break;
        }
        const int ci = s_i.col, cq = s_q.col, li = max(s_i.last - K0, -1), lq = max(s_q.last - K0, -1);      // -1: not a pivot of this batch
        if ((ci < 0 && li < 0) || (cq < 0 && lq < 0)) { stop = 3; break; }
        // terms at the two slots, and the entry (i, q)
        for (int x = t; x < 4 * nb; x += DL_T) {
            const int which = x / nb, k = x % nb;
            s_co[which][k] = ((which & 1) ? z.w : z.s)[(int64_t)(K0 + k) * z.ld + (which < 2 ? i : q)];
        }
        double bi0[2], bq0[2];                                 // base entries of this thread's row: requested early (first row only)
        {
            const int64_t r = row0 + my0;
            const bool on = worker && slice == 0 && my0 < nr;
            bi0[0] = on && ci >= 0 ? z.S0[(int64_t)ci * z.ld + r] : 0.0; bi0[1] = on && ci >= 0 ? z.G0[(int64_t)ci * z.ld + r] : 0.0;
            bq0[0] = on && cq >= 0 ? z.S0[(int64_t)cq * z.ld + r] : 0.0; bq0[1] = on && cq >= 0 ? z.G0[(int64_t)cq * z.ld + r] : 0.0;
        }
        double e0 = 0.0;
        const int m_iq = li > lq ? li : lq;
        if (warp < 2 && m_iq < 0) e0 = (warp == 0 ? z.S0 : z.G0)[(int64_t)ci * z.ld + q];
        __syncthreads();
        if (t < nb) { const double al = s_al[t]; s_ci[t] = make_double2(al * s_co[0][t], al * s_co[1][t]); s_cq[t] = make_double2(al * s_co[2][t], al * s_co[3][t]); }
        if (warp < 2) {
            double v = 0.0;
            for (int k = m_iq + 1 + lane; k < nb; k += 32) {
                const double al = s_al[k], si = s_co[0][k], sq = s_co[2][k];
                v -= warp == 0 ? al * si * sq : al * (sq * s_co[1][k] + si * s_co[3][k]);
            }
            v = warp_sum_d(v);
            if (m_iq >= 0) {                                   // right after pivot m_iq, which was on the one or the other
                const double al = s_al[m_iq], sv = lq > li ? s_co[0][m_iq] : s_co[2][m_iq], wv = lq > li ? s_co[1][m_iq] : s_co[3][m_iq];
                e0 = warp == 0 ? fabs(al) * sv : fabs(al) * (wv - 0.5 * al * sv * s_nu[m_iq]);
            }
            if (lane == 0) s_cross[warp] = e0 + v;
        }
        __syncthreads();
        const double Sii = s_i.S, nui = s_i.G, Sqi = s_cross[0], Gqi = s_cross[1];
        const double ali = 1.0 / Sii, aai = fabs(ali), beq = Sqi * ali, wiq = Gqi - 0.5 * beq * nui;
        const double Sq1 = s_q.S - Sqi * beq, nuq = s_q.G - 2.0 * beq * wiq, alq = 1.0 / Sq1, aaq = fabs(alq);
        const double delta = nui * -ali - nuq * alq;
        {
            int reason = -1;
            if (!(-Sii > 0.0) || !(Sq1 > 0.0) || !isfinite(delta)) reason = OSSCAR_STOP_GUARD;
            else if (a.accept_mode == OSSCAR_ACCEPT_IMPROVING && !(delta <= -a.tol * obj)) reason = OSSCAR_STOP_NO_IMPROVEMENT;
            if (reason >= 0) {
                if (blockIdx.x == 0 && t == 0) { ctl->done = 1; ctl->stop_reason = reason; ctl->delta = delta; *p.done_host = 1; }
                stop = 1;
                break;
            }
        }
        if (blockIdx.x == 0 && t == 0) {
            a.swap_trace[2 * n_swaps] = s_i.id; a.swap_trace[2 * n_swaps + 1] = s_q.id;
            a.obj_trace[n_swaps + 1] = obj + delta;
            z.alpha[K0 + nb] = ali; z.nu[K0 + nb] = nui; z.alpha[K0 + nb + 1] = alq; z.nu[K0 + nb + 1] = nuq;
        }
        obj += delta;
        ++n_swaps;
        // columns i and q of this block's rows
        bd.idx = ba.idx = -1;
        for (int lr = my0; lr < nrp && worker; lr += my_step) {
            double vi = 0.0, gi = 0.0, vq = 0.0, gq = 0.0;
            if (lr < nr) {
                const int64_t r = row0 + lr;
                const int lk = max(last[lr] - K0, -1), mi = lk > li ? lk : li, mq = lk > lq ? lk : lq;
                if (slice == 0) {
                    if (mi >= 0) {
                        const double al = s_al[mi], sv = lk > li ? s_co[0][mi] : hs[(size_t)mi * nrp + lr], wv = lk > li ? s_co[1][mi] : hw[(size_t)mi * nrp + lr];
                        vi = fabs(al) * sv; gi = fabs(al) * (wv - 0.5 * al * sv * s_nu[mi]);
                    } else if (lr == my0) { vi = bi0[0]; gi = bi0[1]; }
                    else { vi = z.S0[(int64_t)ci * z.ld + r]; gi = z.G0[(int64_t)ci * z.ld + r]; }
                    if (mq >= 0) {
                        const double al = s_al[mq], sv = lk > lq ? s_co[2][mq] : hs[(size_t)mq * nrp + lr], wv = lk > lq ? s_co[3][mq] : hw[(size_t)mq * nrp + lr];
                        vq = fabs(al) * sv; gq = fabs(al) * (wv - 0.5 * al * sv * s_nu[mq]);
                    } else if (lr == my0) { vq = bq0[0]; gq = bq0[1]; }
                    else { vq = z.S0[(int64_t)cq * z.ld + r]; gq = z.G0[(int64_t)cq * z.ld + r]; }
                }
                const int first = (mi < mq ? mi : mq) + 1, both = (mi < mq ? mq : mi) + 1;
                int k = slice;
                while (k < first) k += slices;
                for (; k < nb && k < both; k += slices) {          // rows and slots that were pivots of this batch
                    const double s = hs[(size_t)k * nrp + lr], w = hw[(size_t)k * nrp + lr];
                    if (k > mi) { vi = fma(-s, s_ci[k].x, vi); gi = fma(-w, s_ci[k].x, gi); gi = fma(-s, s_ci[k].y, gi); }
                    else { vq = fma(-s, s_cq[k].x, vq); gq = fma(-w, s_cq[k].x, gq); gq = fma(-s, s_cq[k].y, gq); }
                }
                double gi2 = 0.0, gq2 = 0.0;
#pragma unroll 4
                for (; k < nb; k += slices) {
                    const double s = hs[(size_t)k * nrp + lr], w = hw[(size_t)k * nrp + lr];
                    const double2 ci2 = s_ci[k], cq2 = s_cq[k];
                    vi = fma(-s, ci2.x, vi); gi = fma(-w, ci2.x, gi); gi2 = fma(-s, ci2.y, gi2);
                    vq = fma(-s, cq2.x, vq); gq = fma(-w, cq2.x, gq); gq2 = fma(-s, cq2.y, gq2);
                }
                gi += gi2; gq += gq2;
            }
            if (slices > 1) {
                if (slice > 0) { double* x = red + (size_t)(slice - 1) * 4 * nrp + lr; x[0] = vi; x[nrp] = gi; x[2 * nrp] = vq; x[3 * nrp] = gq; }
                else { bi0[0] = vi; bi0[1] = gi; bq0[0] = vq; bq0[1] = gq; }
                break;
            }
            bi0[0] = vi; bi0[1] = gi; bq0[0] = vq; bq0[1] = gq;
            if (lr >= nr) continue;
#define DL_FINISH() do { \
            const int64_t r = row0 + lr; \
            double sv = bi0[0], wv, s2, w2, Sn, Gn; \
            if (r == i) { sv = Sii; wv = 0.0; s2 = aai * Sqi; w2 = aai * (Gqi - beq * nui); Sn = -ali; Gn = ali * ali * nui; } \
            else { \
                const double be = sv * ali; \
                wv = bi0[1] - 0.5 * be * nui; \
                s2 = bq0[0] - be * Sqi; w2 = bq0[1] - be * wiq - wv * beq; \
                Sn = Sd[lr] - sv * be; Gn = Gd[lr] - 2.0 * be * wv; \
            } \
            if (r == q) { s2 = Sq1; w2 = 0.0; Sn = -alq; Gn = alq * alq * nuq; } \
            else { const double be = s2 * alq; w2 -= 0.5 * be * nuq; Sn -= s2 * be; Gn -= 2.0 * be * w2; } \
            hs[(size_t)nb * nrp + lr] = sv; hw[(size_t)nb * nrp + lr] = wv; \
            hs[(size_t)(nb + 1) * nrp + lr] = s2; hw[(size_t)(nb + 1) * nrp + lr] = w2; \
            const int64_t o = (int64_t)(K0 + nb) * z.ld + r; \
            z.s[o] = sv; z.w[o] = wv; z.s[o + z.ld] = s2; z.w[o + z.ld] = w2; \
            Sd[lr] = Sn; Gd[lr] = Gn; \
            if (r == i) { last[lr] = K0 + nb; kept[lr] = 0; } \
            if (r == q) { last[lr] = K0 + nb + 1; kept[lr] = 1; } \
            double v; \
            if (dl_score(kept[lr], Sn, Gn, hd[lr], &v)) dl_keep(kept[lr] ? bd : ba, kept[lr] ? v : -v, Sn, Gn, gid[lr], (int)r, last[lr], col[lr]); \
        } while (0)
            DL_FINISH();
        }
        if (slices > 1) {
            __syncthreads();
            const int lr = my0;
            if (slice == 0 && lr < nr) {
                for (int x = 0; x < slices - 1; ++x) {
                    const double* y = red + (size_t)x * 4 * nrp + lr;
                    bi0[0] += y[0]; bi0[1] += y[nrp]; bq0[0] += y[2 * nrp]; bq0[1] += y[3 * nrp];
                }
                DL_FINISH();
            }
        }
#undef DL_FINISH
        if (t == 0) { s_al[nb] = ali; s_nu[nb] = nui; s_al[nb + 1] = alq; s_nu[nb + 1] = nuq; }       // read again behind the barriers of the next step
        nb += 2;
        buf ^= 1;
        if (n_swaps >= a.max_swaps) { stop = 1; break; }
        if (K0 + nb + 2 > z.kcap) { stop = 2; break; }
        if (nb + 2 > a.kb) { stop = 3; break; }
    }
    __syncthreads();
    for (int lr = t; lr < nr; lr += DL_T) {
        const int64_t r = row0 + lr;
        z.Sd[r] = Sd[lr]; z.Gd[r] = Gd[lr]; z.last[r] = last[lr]; z.kept[r] = kept[lr];
        double v;
        const bool ok = dl_score(kept[lr], Sd[lr], Gd[lr], hd[lr], &v);
        z.val[r] = ok ? (kept[lr] ? v : -v) : INFINITY;
    }
    if (blockIdx.x == 0 && t == 0) {
        ctl->dl_terms = K0 + nb; ctl->n_swaps = n_swaps; ctl->obj = obj; ctl->dl_batches += 1;
        if (stop != 3) ctl->dl_stop = stop;
        // the best slots are among the candidates, so that a batch makes a swap at least: one that does not would be followed by the same for ever
        else if (nb == 0 && ctl->status == OSSCAR_OK) ctl->status = OSSCAR_E_TIMEOUT;
    }
}
// What the host looks at between batches: [0] stop (1: swaps of the segment made, search stopped or failed, 2: terms full), [1] terms,
// [2] swaps, [3] status.
__global__ void k_dl_report(const SearchCtl* ctl, int32_t* out) { out[0] = ctl->done || ctl->status != OSSCAR_OK ? 1 : ctl->dl_stop; out[1] = ctl->dl_terms; out[2] = ctl->n_swaps; out[3] = ctl->status; }

// ------------------------------------------------------------------ the matrices of the state after the terms
// What the K pivots of `swaps` (pairs of groups) were on: piv[k] the slot, prev[k] the pivot on the same slot before (-1: none); and where
// the groups are now: every swap exchanged the places of its two groups, so that src[x], the slot whose group sits at x now, is x but
// for the list[0 .. *count) of changed slots.  One block.
__global__ void __launch_bounds__(1024) k_dl_history(Ptrs p, DlPtrs z, int K, const int32_t* swaps, int32_t* piv, int32_t* prev, int32_t* list, int32_t* count)
{
    __shared__ int s_piv[DL_MAX_TERMS], s_prev[DL_MAX_TERMS], s_loc[DL_MAX_TERMS];
    __shared__ int s_n;
    const int t = threadIdx.x;
    const int64_t d1 = p.nI + p.nJ;
    for (int64_t x = t; x < d1; x += 1024) z.src[x] = (int)x;
    for (int k = t; k < K; k += 1024) s_piv[k] = p.slotof[swaps[k]];
    if (t == 0) s_n = 0;
    __syncthreads();
    for (int k = t; k < K; k += 1024) {
        const int x = s_piv[k];
        int pr = -1;
        for (int j = 0; j < k; ++j) if (s_piv[j] == x) pr = j;
        s_prev[k] = pr;
        s_loc[k] = pr < 0 ? x : -1;                  // where the group sits before its swap
        piv[k] = x; prev[k] = pr;
    }
    for (;;) {                                       // a group that was in a swap before sits where its partner of that swap did
        __syncthreads();
        int open = 0;
        for (int k = t; k < K; k += 1024)
            if (s_loc[k] < 0) {
                const int o = s_loc[s_prev[k] ^ 1];
                if (o >= 0) s_loc[k] = o; else open = 1;
            }
        if (!__syncthreads_or(open)) break;
    }
    for (int k = t; k < K; k += 1024)
        if (z.last[s_piv[k]] == k) {
            const int x = s_loc[k ^ 1];
            z.src[x] = s_piv[k];
            if (x != s_piv[k]) list[atomicAdd(&s_n, 1)] = x;
        }
    __syncthreads();
    if (t == 0) *count = s_n;
}

// Coefficients of the pivots' rows in the rows of the new V and R, [d1][kp] in the new order; rows that were pivots start from nothing.
__global__ void __launch_bounds__(256) k_dl_coef(Ptrs p, DlPtrs z, int K, int64_t kp)
{
    __shared__ float tile[32][33];
    const int64_t x0 = (int64_t)blockIdx.x * 32, d1 = p.nI + p.nJ;
    const int k0 = blockIdx.y * 32, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int64_t x = x0 + tx;
    const int64_t r = x < d1 ? z.src[x] : 0;
    const int lr = x < d1 ? z.last[r] : 0;
    for (int j = ty; j < 32; j += 8) {
        const int k = k0 + j;
        double c = 0.0;
        if (x < d1 && k < K && k >= lr) c = k == lr ? fabs(z.alpha[k]) : -z.alpha[k] * z.s[(int64_t)k * z.ld + r];
        tile[j][tx] = (float)c;
    }
    __syncthreads();
    for (int j = ty; j < 32; j += 8)
        if (x0 + j < d1 && k0 + tx < kp) z.coef[(x0 + j) * kp + k0 + tx] = tile[tx][j];
    if (blockIdx.y == 0) {
        for (int j = 0; j < 32 && x0 + j < d1; ++j) {
            const int64_t y = x0 + j;
            if (z.last[z.src[y]] < 0) continue;
            float* row = y < p.nI ? p.V + y * p.ldm : p.R + (y - p.nI) * p.ldm;
            for (int64_t c = threadIdx.x; c < p.ldm; c += 256) row[c] = 0.f;
        }
    }
}

// Rows M_p of the pivots at the time of their pivot: mk[k] = [p_k was no pivot before] M_p + sum over the terms between.  First the
// base rows and the coefficients f[k][j] of earlier pivots (fp32, row stride kp) for all k; then, DL_MT pivots at a time, a product with the
// rows before them and the triangle within.  (One thread per column over all terms took 0.48 ms for 256 terms of 1024 columns.)
constexpr int DL_MT = 64;
__device__ __forceinline__ double dl_pivot_coef(const DlPtrs& z, int k, int j, const int32_t* piv, const int32_t* prev) {      // of row j < k in row k
    const int pr = prev[k];
    if (j < pr) return 0.0;
    return j == pr ? fabs(z.alpha[j]) : -z.alpha[j] * z.s[(int64_t)j * z.ld + piv[k]];
}
__global__ void __launch_bounds__(256) k_dl_pivot_base(Ptrs p, DlPtrs z, const int32_t* piv, const int32_t* prev, float* f, int64_t kp)
{
    const int k = blockIdx.x;
    const int64_t x = piv[k];
    const bool fresh = prev[k] < 0;
    const float* row = x < p.nI ? p.V + x * p.ldm : p.R + (x - p.nI) * p.ldm;
    for (int64_t c = threadIdx.x; c < p.ldm; c += 256) z.mk[(int64_t)k * p.ldm + c] = fresh ? row[c] : 0.f;
    for (int64_t j = threadIdx.x; j < kp; j += 256) f[(int64_t)k * kp + j] = j < k ? (float)dl_pivot_coef(z, k, (int)j, piv, prev) : 0.f;
}
__global__ void __launch_bounds__(128) k_dl_pivot_rows(Ptrs p, DlPtrs z, int k0, int n, const int32_t* piv, const int32_t* prev)
{
    __shared__ double tri[DL_MT][DL_MT + 1];
    const int64_t c = (int64_t)blockIdx.x * 128 + threadIdx.x;
    for (int i = threadIdx.x; i < n * n; i += 128) {
        const int k = i / n, j = i % n;
        tri[k][j] = j < k ? dl_pivot_coef(z, k0 + k, k0 + j, piv, prev) : 0.0;
    }
    __syncthreads();
    if (c >= p.ldm) return;
    double m[DL_MT];
#pragma unroll
    for (int k = 0; k < DL_MT; ++k) m[k] = k < n ? (double)z.mk[(int64_t)(k0 + k) * p.ldm + c] : 0.0;
#pragma unroll
    for (int k = 1; k < DL_MT; ++k) {
        if (k >= n) break;
        double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
#pragma unroll
        for (int j = 0; j < k; ++j) {
            if ((j & 3) == 0) a0 = fma(tri[k][j], m[j], a0); else if ((j & 3) == 1) a1 = fma(tri[k][j], m[j], a1);
            else if ((j & 3) == 2) a2 = fma(tri[k][j], m[j], a2); else a3 = fma(tri[k][j], m[j], a3);
        }
        m[k] += (a0 + a1) + (a2 + a3);
        z.mk[(int64_t)(k0 + k) * p.ldm + c] = (float)m[k];
    }
}
// Hinv on the new kept slots: what the base or the last pivot on the row or the column left, plus alpha_k s_k s_k^T for the terms since
// (S_II = -Hinv), sums in fp64.  Tile 128 x 64, upper triangle and its mirror image.
__global__ void __launch_bounds__(256, 2) k_dl_rank(Ptrs p, DlPtrs z, int K)
{
    constexpr int BM = 128, BN = 64, BK = 16, AS = BK + 4, BS = BN + 4;
    extern __shared__ double dl_smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, wm = warp >> 1, wn = warp & 1;
    const int64_t m0 = (int64_t)blockIdx.y * BM, n0 = (int64_t)blockIdx.x * BN;
    if (n0 + BN <= m0) return;
    double* As[2] = { dl_smem, dl_smem + BM * AS };
    double* Bs[2] = { dl_smem + 2 * BM * AS, dl_smem + 2 * BM * AS + BK * BS };
    double acc[4][4][2];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) { acc[i][j][0] = 0.0; acc[i][j][1] = 0.0; }
    const int64_t ya = m0 + tid % BM, yb = n0 + tid % BN;          // this thread loads one row of each operand
    const int64_t xa = ya < p.nI ? z.src[ya] : 0, xb = yb < p.nI ? z.src[yb] : 0;
    const int la = ya < p.nI ? z.last[xa] : INT_MAX, lb = yb < p.nI ? z.last[xb] : INT_MAX;
    double ra[8], rb[4];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int q = 0; q < 8; ++q) { const int k = k0 + tid / BM + 2 * q; ra[q] = k < K && k > la ? z.alpha[k] * z.s[(int64_t)k * z.ld + xa] : 0.0; }
#pragma unroll
        for (int q = 0; q < 4; ++q) { const int k = k0 + tid / BN + 4 * q; rb[q] = k < K && k > lb ? z.s[(int64_t)k * z.ld + xb] : 0.0; }
    };
    auto stash = [&](int buf) {
#pragma unroll
        for (int q = 0; q < 8; ++q) As[buf][(tid % BM) * AS + tid / BM + 2 * q] = ra[q];
#pragma unroll
        for (int q = 0; q < 4; ++q) Bs[buf][(tid / BN + 4 * q) * BS + tid % BN] = rb[q];
    };
    const int fr = lane >> 2, fk = lane & 3, nk = (K + BK - 1) / BK;
    fetch(0);
    stash(0);
    __syncthreads();
    for (int kt = 0; kt < nk; ++kt) {
        const int buf = kt & 1;
        if (kt + 1 < nk) fetch((kt + 1) * BK);
        const double* a = As[buf] + (wm * 32) * AS;
        const double* b = Bs[buf] + wn * 32;
#pragma unroll
        for (int ks = 0; ks < BK; ks += 4) {
            double af[4], bf[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) af[i] = a[(i * 8 + fr) * AS + ks + fk];
#pragma unroll
            for (int j = 0; j < 4; ++j) bf[j] = b[(ks + fk) * BS + j * 8 + fr];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) dl_dmma(acc[i][j][0], acc[i][j][1], af[i], bf[j]);
        }
        if (kt + 1 < nk) stash(buf ^ 1);
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int64_t row = m0 + wm * 32 + i * 8 + fr;
        if (row >= p.nI) continue;
        const int64_t r = z.src[row];
        const int lr = z.last[r];
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int64_t col = n0 + wn * 32 + j * 8 + 2 * fk + e;
                if (col >= p.nI || col < row) continue;
                const int64_t x = z.src[col];
                const int lx = z.last[x], m = lr > lx ? lr : lx;
                double v;
                if (m < 0) v = p.Hd[row * p.ldh + col];
                else if (row == col) v = z.alpha[m];
                else v = -fabs(z.alpha[m]) * z.s[(int64_t)m * z.ld + (lr > lx ? x : r)];
                v += acc[i][j][e];
                p.Hd[row * p.ldh + col] = v;
                if (col != row) p.Hd[col * p.ldh + row] = v;
            }
    }
}
// Rows and columns of Hp of the changed slots, from H and the new permutation.
__global__ void __launch_bounds__(256) k_dl_hgather(Ptrs p, const float* __restrict__ H, const int32_t* list, const int32_t* count)
{
    const int64_t d1 = p.nI + p.nJ, y = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (y >= d1) return;
    const int64_t gy = p.perm[y];
    const int n = *count;
    for (int i = blockIdx.y; i < n; i += gridDim.y) {
        const int64_t x = list[i];
        const float v = H[(int64_t)p.perm[x] * d1 + gy];
        p.Hp[x * p.ldp + y] = v;
        p.Hp[y * p.ldp + x] = v;
    }
}
// Vectors by slot in the new order: diagonals, norms, scores; groups (old slots in, new slots out).
__global__ void __launch_bounds__(256) k_dl_vectors(Ptrs p, DlPtrs z, const int32_t* old_perm)
{
    const int64_t x = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (x >= p.nI + p.nJ) return;
    const int64_t r = z.src[x];
    const int id = old_perm[r];
    p.perm[x] = id; p.slotof[id] = (int)x;
    double v;
    const bool kept = x < p.nI;
    dl_score(kept, z.Sd[r], z.Gd[r], z.hd[r], &v);
    if (kept) { p.D[x] = v; p.vnorm[x] = (float)z.Gd[r]; }
    else { p.A[x - p.nI] = v; p.rnorm[x - p.nI] = (float)z.Gd[r]; p.c[x - p.nI] = z.Sd[r]; }
}

// ------------------------------------------------------------------ host side
struct DlPlan {
    DlPtrs z;
    int32_t *list, *piv, *prev, *count, *perm0;
    int grid, rows, kb;
    size_t smem;
    char* scratch; size_t scratch_bytes;          // what the rewrite may use for digits
    int64_t kp;
};

// Geometry and memory of the delayed loop: vectors and terms in `big`, partial sums (in the loop) or coefficients and the rows of the
// pivots (in the rewrite) in the tensor-core region; both are idle otherwise.  false where a layer does not fit.
inline bool dl_plan(osscar_ctx* ctx, DlPlan* d)
{
    const Layout& L = ctx->L;
    int dev = 0, coop = 0, sms = 0;
    if (L.nJ < 1 || cudaGetDevice(&dev) != cudaSuccess) return false;
    if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop) return false;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return false;
    // rows per block: a barrier costs more the more blocks meet at it
    int64_t grid = (L.d1 + 63) / 64;
    if (grid > sms) grid = sms;
    if (grid > DL_MAX_BLOCKS) grid = DL_MAX_BLOCKS;
    d->rows = (int)((L.d1 + grid - 1) / grid);
    d->grid = (int)((L.d1 + d->rows - 1) / d->rows);
    for (d->kb = DL_KB; d->kb >= 8 && dl_loop_smem(d->rows, d->kb) > DL_SMEM_MAX; d->kb -= 2) {}
    if (d->kb < 8) return false;
    d->smem = dl_loop_smem(d->rows, d->kb);
    DlPtrs& z = d->z;
    char* const ws = (char*)ctx->ws;
    size_t off = L.off_big;
    const size_t end = L.off_Hp;
    auto take = [&](size_t n) { char* q = ws + off; off += (n + 255) / 256 * 256; return q; };
    const size_t d1 = (size_t)L.d1, ld = (size_t)round_up(L.d1, 16);
    z.ld = (int64_t)ld;
    z.cands = (DlCand*)take(sizeof(DlCand) * 4 * DL_MAX_BLOCKS);
    z.alpha = (double*)take(8 * DL_MAX_TERMS); z.nu = (double*)take(8 * DL_MAX_TERMS);
    z.Sd = (double*)take(8 * d1); z.Gd = (double*)take(8 * d1); z.hd = (double*)take(8 * d1); z.val = (double*)take(8 * d1);
    z.last = (int32_t*)take(4 * d1); z.kept = (int32_t*)take(4 * d1); z.cidx = (int32_t*)take(4 * d1); z.src = (int32_t*)take(4 * d1);
    z.cand = (int32_t*)take(4 * DL_N);
    d->count = (int32_t*)take(16);
    d->list = (int32_t*)take(4 * DL_MAX_TERMS);
    d->perm0 = (int32_t*)take(4 * d1);
    d->piv = (int32_t*)take(4 * DL_MAX_TERMS); d->prev = (int32_t*)take(4 * DL_MAX_TERMS);
    z.S0 = (double*)take(8 * DL_N * ld); z.G0 = (double*)take(8 * DL_N * ld);
    z.By = (double*)take(8 * DL_B * (size_t)L.nI); z.Bh = (double*)take(8 * DL_N * (size_t)L.nI); z.Bg = (double*)take(8 * DL_N * (size_t)L.ldm);
    if (off >= end) return false;
    int64_t k = (int64_t)((end - off) / (16 * ld)) / 2 * 2 - 2;
    if (k > DL_MAX_TERMS) k = DL_MAX_TERMS;
    // the rewrite keeps coefficients and rows for all terms in the tensor-core region
    const int64_t kt = (int64_t)((L.tc_bytes - 4096) / (4 * (d1 + (size_t)L.ldm + DL_MAX_TERMS))) / 32 * 32;
    if (k > kt) k = kt;
    if (k < DL_KB) return false;
    z.kcap = (int)k;
    z.s = (double*)take(8 * ld * (size_t)k); z.w = (double*)take(8 * ld * (size_t)k);
    if (off > end) return false;
    // slices of the panel products: two blocks per SM, 64 k each at least, no more than eight (each is read again), sums that fit
    auto slices = [&](int64_t M, int64_t K) {
        int64_t n = 2 * sms / ((M + 127) / 128);
        if (n > K / 64) n = K / 64;
        if (n > 8) n = 8;
        return (int)(n < 1 ? 1 : n);
    };
    z.zy = slices(L.nI, L.nI); z.zh = slices(L.nJ, L.nI); z.zg = slices(L.d1, L.ldm); z.zt = slices(L.d1, 256);
    char* const tc = ws + L.off_tc + 2 * 8 * DL_N * (size_t)z.kcap;
    const size_t room = L.tc_bytes - 2 * 8 * DL_N * (size_t)z.kcap;
    if (L.tc_bytes < 2 * 8 * DL_N * (size_t)z.kcap) return false;
    z.cs = (double*)(ws + L.off_tc); z.cw = z.cs + DL_N * (size_t)z.kcap;
    for (;;) {
        const size_t ny = (8 * (size_t)z.zy * DL_B * (size_t)L.nI + 255) / 256 * 256, nh = (8 * (size_t)z.zh * DL_N * (size_t)L.nJ + 255) / 256 * 256;
        const size_t ng = 8 * (size_t)z.zg * DL_N * d1, nt = 8 * (size_t)z.zt * DL_N * d1;
        if (ny + nh + ng + 2 * nt <= room) {
            z.py = (double*)tc; z.ph = (double*)(tc + ny); z.pg = (double*)(tc + ny + nh);
            z.ts = (double*)(tc + ny + nh + ng); z.tg = (double*)(tc + ny + nh + ng + nt);
            break;
        }
        if (z.zy == 1 && z.zh == 1 && z.zg == 1 && z.zt == 1) return false;
        if (z.zt > 1) z.zt--;
        if (z.zy > 1) z.zy--;
        if (z.zh > 1) z.zh--;
        if (z.zg > 1) z.zg--;
    }
    return true;
}

constexpr int DL_TERMS_SMEM = 4 * (128 * 20 + 16 * 68) * (int)sizeof(double);
constexpr int DL_RANK_SMEM = (2 * 128 * 20 + 2 * 16 * 68) * (int)sizeof(double);

// Base columns of a batch and its swaps.  `marks` (or null): DL_MARKS events around its four parts.
constexpr int DL_MARKS = 5;
cudaError_t dl_batch(osscar_ctx* ctx, const Ptrs& p, const DlPlan& d, const DlArgs& args, cudaEvent_t* marks)
{
    const Layout& L = ctx->L;
    cudaStream_t st = ctx->stream;
    const DlPtrs& z = d.z;
    const unsigned nbI = (unsigned)((L.nI + 31) / 32), nbM = (unsigned)((L.ldm + 31) / 32);
    auto tiles = [](int64_t M, int n) { return dim3((unsigned)((M + 127) / 128), (unsigned)n); };
    auto mark = [&](int i) { if (marks) cudaEventRecord(marks[i], st); };
    mark(0);
    k_dl_select<<<2, 1024, 0, st>>>(p, z);
    // the kernels up to the columns are programmatic dependents, each of the one before it (ordinary launches between events): a batch is 15 to 20 us
    // shorter, 51 swaps in 6 batches at d1 = 1024 1.034 -> 0.924 ms
    const bool dep = !marks;
    const SearchCtl* ctl = ctx->ctl;
    const float *Vc = p.V, *Rc = p.R, *HJI = p.Hp + L.nI * L.ldp;
    const double* Hd = p.Hd;
    launch_pdl(dep, k_dl_stage, dim3(nbI + nbM + (unsigned)((z.kcap + 31) / 32)), dim3(256), st, p, z, nbI, nbM);
    launch_pdl_smem(dep, k_dl_terms, tiles(L.d1, z.zt), dim3(256), DL_TERMS_SMEM, st, p, z);
    mark(1);
    launch_pdl_smem(dep, k_dl_panel<double, DL_B>, tiles(L.nI, z.zy), dim3(256), dl_panel_smem<double, DL_B>(), st, L.nI, L.nI, Hd, Hd, L.nI, L.ldh, z.By, z.py, z.zy, ctl);
    launch_pdl_smem(dep, k_dl_panel<float, DL_N>, tiles(L.d1, z.zg), dim3(256), dl_panel_smem<float, DL_N>(), st, L.d1, L.ldm, Vc, Rc, L.nI, L.ldm, z.Bg, z.pg, z.zg, ctl);
    launch_pdl(dep, k_dl_stage_y, dim3(nbI), dim3(256), st, p, z);
    launch_pdl_smem(dep, k_dl_panel<float, DL_N>, tiles(L.nJ, z.zh), dim3(256), dl_panel_smem<float, DL_N>(), st, L.nJ, L.nI, HJI, HJI, L.nJ, L.ldp, z.Bh, z.ph, z.zh, ctl);
    mark(2);
    launch_pdl(dep, k_dl_apply, dim3((unsigned)((L.d1 + 127) / 128), DL_N / DL_AC), dim3(128), st, p, z);
    mark(3);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    void* kargs[] = { (void*)&args };
    e = cudaLaunchCooperativeKernel((const void*)k_dl_loop, dim3((unsigned)d.grid), dim3(DL_T), kargs, d.smem, st);
    if (e != cudaSuccess) return e;
    mark(4);
    count_launches(9);
    return cudaGetLastError();
}

cudaError_t dl_prepare(osscar_ctx* ctx, const Ptrs& p, const DlPlan& d)
{
    cudaError_t e = cudaFuncSetAttribute(k_dl_loop, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DL_SMEM_MAX);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_dl_panel<double, DL_B>, cudaFuncAttributeMaxDynamicSharedMemorySize, (dl_panel_smem<double, DL_B>()));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_dl_panel<float, DL_N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (dl_panel_smem<float, DL_N>()));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_dl_terms, cudaFuncAttributeMaxDynamicSharedMemorySize, DL_TERMS_SMEM);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_dl_rank, cudaFuncAttributeMaxDynamicSharedMemorySize, DL_RANK_SMEM);
    if (e != cudaSuccess) return e;
    k_dl_init<<<(unsigned)((ctx->L.d1 + 7) / 8), 256, 0, ctx->stream>>>(p, d.z);
    count_launches(1);
    return cudaGetLastError();
}

// V, R, the inverse, Hp and the vectors by slot after the K terms of `swaps` (pairs of groups); slot permutation included.
// `matrices` false: the permutation only (the state is about to be rebuilt).
cudaError_t dl_rewrite(osscar_ctx* ctx, const Ptrs& p, const DlPlan& d, int K, const int32_t* swaps, bool matrices)
{
    const Layout& L = ctx->L;
    cudaStream_t st = ctx->stream;
    DlPtrs z = d.z;
    const unsigned nbd = (unsigned)((L.d1 + 255) / 256);
    cudaError_t e = cudaMemcpyAsync(d.perm0, p.perm, sizeof(int32_t) * (size_t)L.d1, cudaMemcpyDeviceToDevice, st);
    if (e != cudaSuccess) return e;
    k_dl_history<<<1, 1024, 0, st>>>(p, z, K, swaps, d.piv, d.prev, d.list, d.count);
    count_launches(1);
    if (matrices && K > 0) {
        const int64_t kp = round_up(K, 32);
        char* tc = (char*)ctx->ws + L.off_tc;
        z.coef = (float*)tc;
        const size_t nc = (sizeof(float) * (size_t)L.d1 * kp + 255) / 256 * 256;
        z.mk = (float*)(tc + nc);
        const size_t nm = (sizeof(float) * (size_t)K * L.ldm + 255) / 256 * 256;          // behind the rows: coefficients, later digits
        float* f = (float*)(tc + nc + nm);
        k_dl_pivot_base<<<(unsigned)K, 256, 0, st>>>(p, z, d.piv, d.prev, f, kp);
        for (int k = 0; k < K; k += DL_MT) {
            const int n = K - k < DL_MT ? K - k : DL_MT;
            float* rows = z.mk + (int64_t)k * L.ldm;
            if (k > 0) {
                e = gemm_f64acc(st, n, L.ldm, k, 1.0, f + (int64_t)k * kp, kp, z.mk, L.ldm, 1.0, rows, L.ldm, rows, L.ldm, false);
                if (e != cudaSuccess) return e;
            }
            k_dl_pivot_rows<<<(unsigned)((L.ldm + 127) / 128), 128, 0, st>>>(p, z, k, n, d.piv, d.prev);
            count_launches(1);
        }
        k_dl_coef<<<dim3((unsigned)((L.d1 + 31) / 32), (unsigned)(kp / 32)), 256, 0, st>>>(p, z, K, kp);
        count_launches(2);
        // V and R: sums beyond fp32, as every other product that their values come from.  A leaving pivot has coefficients of the size of
        // sqrt(H_pp) and a row M_p of its inverse, an entering one the other way round: digits below one scale per row and column need
        // the index balanced, or the error grows with the units of H (1e-3 of V at 2600 rows whose activations have a size of 256).
        for (int side = 0; side < 2; ++side) {
            const int64_t M = side == 0 ? L.nI : L.nJ;
            float* C = side == 0 ? p.V : p.R;
            const float* A = z.coef + (side == 0 ? 0 : L.nI * kp);
            I8Scratch sc;
            const size_t used = (nc + nm + 255) / 256 * 256, room = used < L.tc_bytes ? (L.tc_bytes - used) / 256 * 256 : 0;
            size_t nb = (gemm_i8_operand_bytes(L.ldm, K, 5) + 255) / 256 * 256;
            if (nb > room / 2) nb = room / 2 / 256 * 256;
            sc.b = tc + used; sc.b_bytes = nb;
            sc.a = tc + used + nb; sc.a_bytes = room - nb;
            if (gemm_i8_usable(M, L.ldm, K, 5, sc)) {
                I8Gemm q = {};
                q.M = M; q.N = L.ldm; q.K = K; q.alpha = 1.0; q.beta = 1.0;
                q.A = A; q.lda = kp; q.B = z.mk; q.ldb = L.ldm; q.C0 = C; q.ldc0 = L.ldm; q.C = C; q.ldc = L.ldm;
                q.pivots = z.alpha;
                e = gemm_i8(st, q, 5, sc, ctx->ctl, nullptr);
            } else e = gemm_f64acc(st, M, L.ldm, K, 1.0, A, kp, z.mk, L.ldm, 1.0, C, L.ldm, C, L.ldm, false);
            if (e != cudaSuccess) return e;
        }
        k_dl_rank<<<dim3((unsigned)((L.nI + 63) / 64), (unsigned)((L.nI + 127) / 128)), 256, DL_RANK_SMEM, st>>>(p, z, K);
        count_launches(1);
    }
    k_dl_vectors<<<nbd, 256, 0, st>>>(p, z, d.perm0);
    count_launches(1);
    if (matrices && K > 0) {
        k_dl_hgather<<<dim3(nbd, (unsigned)(K < 64 ? K : 64)), 256, 0, st>>>(p, ctx->H, d.list, d.count);
        count_launches(1);
    }
    return cudaGetLastError();
}
