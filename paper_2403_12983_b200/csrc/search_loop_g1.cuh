// Persistent swap loop for single-row groups (g = 1, independent scores): ONE cooperative kernel runs every step of the
// search.  Included by search.cu after search_g1.cuh (same translation unit: uses its Ptrs, scalar slots and helpers).
//
// A step has three phases, separated by grid-wide barriers (all blocks are co-resident: cooperative launch):
//   A   every block, redundantly and identically: the leaving slot r (arg-min of the per-block candidates of D), the
//       cross term V_r . R_q, the exact change of obj, the accept test; block 0 records the swap.  The vectors of the
//       step, b = Hinv[r, :], u2 = y - b y_r / C, K = V_r / C, Vq = (R_q + (y_r / C) V_r) / c1, go to the block's own shared
//       memory.  Then V' = V - b K - u2 Vq with its row norms and drop scores D  ||  H pass (u_l, d_l of every pruned row and
//       of the leaving row).  Row r of V, which other blocks may still be reading, is replaced in B.
//   B   R' = R + u K - d Vq with row norms, Schur complements c' and add scores A  ||  exchange of the two slots in Hp.
//   C   every block: entering slot of the NEXT step (arg-max of the per-block candidates of A); then
//       Hinv' = Hinv - (b / C) b^T + (u2 / c1) u2^T fused with y_next = Hinv' Hp[q_next, 0:n_I]^T.
// Bound: latency.  The states that come here stay in L2, and a step is three barriers and a handful of dependent reads.
// One block of 24 warps per SM and a warp per row: a barrier collects at most 148 arrivals, no phase synchronises inside a
// block while it streams, rows of any length are handed out one by one (with four rows per 256-thread block, 445
// row groups on 444 blocks were two rounds), and fewer blocks take part where the layer has fewer than 8 rows per SM.
// Before (444 blocks of 256 threads, rows in groups of 1 / 2 / 4, vectors through global memory, four barriers) a swap took
// 20.9 / 25.0 / 61.7 us at d1 = 64 / 1024 / 5000 (m = 64 / 1024 / 1283), now 15.4 / 20.1 / 43.8 us.
// Every barrier wait is bounded by ctl->wait_limit cycles: the block that runs out sets ctl->abort and
// OSSCAR_E_TIMEOUT, every other block sees the flag in its own wait, and all return.
#pragma once

constexpr int PL_W = 24;                    // warps per block
constexpr int PL_T = PL_W * 32;
constexpr int PL_ROWS_PER_BLOCK = 8;        // rows a block should at least have before another block joins the barrier
constexpr int PL_CAND = kLoopMaxBlocks / 2; // entries of one of the two lists of drop candidates
constexpr int PL_SMEM_MAX = 200 * 1024;     // vectors of a step in shared memory, else in global memory behind one more barrier

struct LoopCand { double val; int32_t id; int32_t idx; };

struct LoopArgs {
    Ptrs p;
    LoopCand* candD;               // per block: cheapest drop among the rows it updated; entry gridDim.x: the entering row.  Two
                                   // lists: a block that is ahead fills the one while others still choose from the other
    LoopCand* candA;               // per block: most valuable add among the rows it updated
    unsigned long long* prof;      // [0..3] nanoseconds spent in the decision, the rest of A, B and C (block 0), [4] steps counted
    double* obj_trace;
    int32_t* swap_trace;
    double tol;
    int accept_mode;
    int max_steps;                 // steps this launch may run
    int max_swaps;                 // the loop ends when ctl->n_swaps reaches this
    int smem_vectors;              // the launch has shared memory for the vectors of a step
};

struct StepScal {                  // scalars of a step, identical in every block
    int64_t r0, t;                 // leaving kept slot, entering pruned slot
    float Cinv, c1inv, Q1, M2;     // 1/C, 1/c1, y_r / C, y_r / (C c1)
    double Cinv_d, c1inv_d, hdiag; // the same in double, H diagonal entry of the leaving row
    float dr;                      // d of the leaving row (valid after A)
};

__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long* ptr) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(ptr) : "memory");
    return v;
}
__device__ __forceinline__ int ld_volatile_s32(const int32_t* ptr) {
    int v;
    asm volatile("ld.volatile.global.s32 %0, [%1];" : "=r"(v) : "l"(ptr) : "memory");
    return v;
}
__device__ __forceinline__ unsigned long long global_timer_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// Grid-wide barrier over `nblocks` co-resident blocks on the monotone counter ctl->bar_count (zeroed by the host
// before the launch); `epoch` is the count this block expects after the barrier.  The block's barrier orders its writes
// before thread 0's release, and thread 0's acquire before what the block reads afterwards.  Returns false when the wait
// ran out or another block gave up.
__device__ __forceinline__ bool grid_barrier(SearchCtl* ctl, unsigned long long& epoch, unsigned nblocks, long long limit, int* s_flag)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        epoch += nblocks;
        asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(&ctl->bar_count), "l"(1ULL) : "memory");
        const long long t0 = clock64();
        int bad = 0;
        while (ld_acquire_u64(&ctl->bar_count) < epoch) {
            if (ld_volatile_s32(&ctl->abort)) { bad = 1; break; }
            if (clock64() - t0 > limit) {
                atomicExch(&ctl->abort, 1);
                ctl->status = OSSCAR_E_TIMEOUT;
                bad = 1;
                break;
            }
        }
        *s_flag = bad;
    }
    __syncthreads();
    return *s_flag == 0;
}

// lexicographic "better" for minimisation with ties to the smaller group id
__device__ __forceinline__ bool cand_less(double v, int id, double bv, int bid) { return v < bv || (v == bv && id < bid); }

// Arg-min over the per-block candidates (negate: arg-max); every thread of warp 0 takes part, result in lane 0.
__device__ __forceinline__ void reduce_cands(const LoopCand* cand, unsigned nblocks, bool negate, double* val, int* idx)
{
    const int lane = threadIdx.x & 31;
    double best = INFINITY; int bid = INT_MAX, bidx = -1;
    for (unsigned i = lane; i < nblocks; i += 32) {
        const LoopCand c = cand[i];
        const double v = negate ? -c.val : c.val;
        if (c.idx >= 0 && cand_less(v, c.id, best, bid)) { best = v; bid = c.id; bidx = c.idx; }
    }
    for (int o = 16; o > 0; o >>= 1) {
        const double ov = __shfl_xor_sync(0xffffffffu, best, o);
        const int oid = __shfl_xor_sync(0xffffffffu, bid, o), oidx = __shfl_xor_sync(0xffffffffu, bidx, o);
        if (cand_less(ov, oid, best, bid)) { best = ov; bid = oid; bidx = oidx; }
    }
    *val = negate ? -best : best;
    *idx = bidx;
}


__device__ __forceinline__ void keep_best(LoopCand& b, double v, int id, int64_t idx) {
    if (b.idx < 0 || cand_less(v, id, b.val, b.id)) { b.val = v; b.id = id; b.idx = (int)idx; }
}

struct LoopVecs { const float4 *K, *Q, *b, *u2; };       // vectors of the step: shared memory, or the staged global ones

// V'[s] = V[s] - b[s] K - u2[s] Vq and D'[s] (kind 0, all rows but r0), or R'[l] = R[l] + u[l] K - d[l] Vq, c'[l] and A'[l]
// (kind 1; row t := K - d_r Vq).  A warp per row, rows w0, w0 + W, ...; U 16-byte pieces of a row in flight per lane.
template <int U>
__device__ __noinline__ void pl_update_rows(const Ptrs& p, const int kind, const StepScal& sc, const LoopVecs& x, int64_t w0, int64_t W,
                                            LoopCand& best)
{
    float* M = kind == 0 ? p.V : p.R;
    const int64_t nrows = kind == 0 ? p.nI : p.nJ;
    const int n4 = (int)(p.ldm / 4);
    const int lane = threadIdx.x & 31;
    const float4 *K4 = x.K, *Q4 = x.Q;
    const float* bs = reinterpret_cast<const float*>(x.b);
    const float* us = reinterpret_cast<const float*>(x.u2);
    for (int64_t s = w0; s < nrows; s += W) {
        if (kind == 0 && s == sc.r0) continue;
        float4* row = reinterpret_cast<float4*>(M + s * p.ldm);
        const bool sp = kind == 1 && s == sc.t;
        float nrm[4] = {0.f, 0.f, 0.f, 0.f};
        float ck, cq;
        double e0, e1, cc = 0.0;
        int id;
        for (int base = lane; base < n4; base += 32 * U) {
            float4 v[U];
#pragma unroll
            for (int j = 0; j < U; ++j) v[j] = base + 32 * j < n4 ? row[base + 32 * j] : make_float4(0.f, 0.f, 0.f, 0.f);
            if (base == lane) {              // scalars of the row, requested behind the row itself
                id = p.perm[kind == 0 ? s : p.k + s];
                if (kind == 0) { ck = -bs[s]; cq = -us[s]; e0 = p.Hd[s * p.ldh + s]; e1 = 0.0; }
                else {
                    ck = p.u[s]; cq = -p.d[s]; e0 = p.c[s]; e1 = (double)p.Hp[(p.nI + s) * p.ldp + p.nI + s];
                    cc = e0 + (double)ck * (double)ck * sc.Cinv_d - (double)cq * (double)cq * sc.c1inv_d;
                }
                if (sp) { ck = 1.f; cq = -sc.dr; }
            }
#pragma unroll
            for (int j = 0; j < U; ++j) {
                const int c = base + 32 * j;
                if (c < n4) {
                    const float4 kk = K4[c], qq = Q4[c];
                    if (sp) v[j] = make_float4(0.f, 0.f, 0.f, 0.f);
                    fma4(v[j], ck, kk);
                    fma4(v[j], cq, qq);
                    row[c] = v[j];
                    nrm[j & 3] += dot4(v[j], v[j]);
                }
            }
        }
        const float nr = warp_sum((nrm[0] + nrm[1]) + (nrm[2] + nrm[3]));
        if (lane == 0) {
            if (kind == 0) {
                p.vnorm[s] = nr;
                const double bd = -(double)ck, ud = -(double)cq;
                const double hd = e0 - bd * bd * sc.Cinv_d + ud * ud * sc.c1inv_d;
                const double score = hd > 0.0 ? (double)nr / hd : INFINITY;
                p.D[s] = score;
                if (isfinite(score)) keep_best(best, score, id, s);
            } else {
                p.rnorm[s] = nr;
                double hd = e1;
                if (sp) { cc = sc.Cinv_d - (double)sc.dr * (double)sc.dr * sc.c1inv_d; hd = sc.hdiag; }
                p.c[s] = cc;
                const double score = cc > kAddPivotTol * hd ? (double)nr / cc : -INFINITY;
                p.A[s] = score;
                if (isfinite(score)) keep_best(best, -score, id, s);          // candidates are kept as minima
            }
        }
    }
}

// Row r0 of V' is Vq: one warp, in phase B (nobody reads the old row any more); its drop score joins the candidates.
__device__ void pl_entering_row(const Ptrs& p, const StepScal& sc, const LoopVecs& x, LoopCand* out)
{
    const int lane = threadIdx.x & 31;
    float4* row = reinterpret_cast<float4*>(p.V + sc.r0 * p.ldm);
    float nrm = 0.f;
    for (int c = lane; c < (int)(p.ldm / 4); c += 32) {
        const float4 q = x.Q[c];
        row[c] = q;
        nrm += dot4(q, q);
    }
    nrm = warp_sum(nrm);
    if (lane == 0) {
        p.vnorm[sc.r0] = nrm;
        const double score = sc.c1inv_d > 0.0 ? (double)nrm / sc.c1inv_d : INFINITY;
        p.D[sc.r0] = score;
        LoopCand b; b.idx = -1; b.val = 0.0; b.id = 0;
        if (isfinite(score)) keep_best(b, score, p.perm[sc.r0], sc.r0);
        *out = b;
    }
}

// H pass: u_l = Hp[l, 0:n_I] . b, d_l = Hp[l, q] - Hp[l, 0:n_I] . u2 for the pruned rows (items 0 .. n_J - 1) and the
// leaving row (item n_J); a warp per row.
template <int U>
__device__ __noinline__ void pl_hpass(const Ptrs& p, const StepScal& sc, const LoopVecs& x, int64_t w0, int64_t W)
{
    const int n4 = (int)(p.ldh / 4);
    const int lane = threadIdx.x & 31;
    const int64_t qcol = p.nI + sc.t;
    const float4 *bv = x.b, *uv = x.u2;
    for (int64_t l = w0; l < p.nJ + 1; l += W) {
        const float* rowf = p.Hp + (l < p.nJ ? p.nI + l : sc.r0) * p.ldp;
        const float4* row = reinterpret_cast<const float4*>(rowf);
        float au[4] = {0.f, 0.f, 0.f, 0.f}, ad[4] = {0.f, 0.f, 0.f, 0.f};
        float hq = 0.f;
        for (int base = lane; base < n4; base += 32 * U) {
            float4 v[U];
#pragma unroll
            for (int j = 0; j < U; ++j) v[j] = base + 32 * j < n4 ? row[base + 32 * j] : make_float4(0.f, 0.f, 0.f, 0.f);
            if (base == lane) hq = rowf[qcol];
#pragma unroll
            for (int j = 0; j < U; ++j) {
                const int c = base + 32 * j;
                if (c < n4) { au[j & 3] += dot4(v[j], bv[c]); ad[j & 3] += dot4(v[j], uv[c]); }
            }
        }
        const float su = warp_sum((au[0] + au[1]) + (au[2] + au[3])), sd = warp_sum((ad[0] + ad[1]) + (ad[2] + ad[3]));
        if (lane == 0) { p.u[l] = su; p.d[l] = hq - sd; }
    }
}

// C: rows of the inverse, kept in fp64 (row and column r0 replaced), and y_next = Hinv' h; a warp per row.
// The inverse is the one piece of the state that fp32 cannot carry: y = Hinv h cancels the common component of the
// rows of H to a few parts in 10^4, so an entry rounded to 2^-24 shows up in y, then in u2, and from there in every
// matrix (measured: the scores drift 3e-7 per swap with an fp32 inverse, 5e-9 with this one).  A piece is a double2.
template <int U>
__device__ __noinline__ void pl_update_hinv(const Ptrs& p, const StepScal& sc, const LoopVecs& x, int64_t t_next, int64_t w0, int64_t W)
{
    const float2* b2 = reinterpret_cast<const float2*>(x.b);
    const float2* u2v = reinterpret_cast<const float2*>(x.u2);
    const float* bs = reinterpret_cast<const float*>(x.b);
    const float* us2 = reinterpret_cast<const float*>(x.u2);
    const float2* h2 = reinterpret_cast<const float2*>(p.Hp + (p.nI + t_next) * p.ldp);
    const int n2 = (int)(p.ldh / 2);
    const int lane = threadIdx.x & 31;
    for (int64_t s = w0; s < p.nI; s += W) {
        double2* row = reinterpret_cast<double2*>(p.Hd + s * p.ldh);
        const bool srow = s == sc.r0;
        // row r0 becomes -u2 / c1: 0 * old - 0 * b + (-1 / c1) * u2
        const double nb = srow ? 0.0 : -(double)bs[s] * sc.Cinv_d;
        const double us = srow ? -sc.c1inv_d : (double)us2[s] * sc.c1inv_d;
        const double corner = srow ? sc.c1inv_d : -us;               // value of column r0 in this row
        double y0 = 0.0, y1 = 0.0;
        for (int base = lane; base < n2; base += 32 * U) {
            double2 h[U];
#pragma unroll
            for (int j = 0; j < U; ++j) h[j] = base + 32 * j < n2 ? row[base + 32 * j] : make_double2(0.0, 0.0);
#pragma unroll
            for (int j = 0; j < U; ++j) {
                const int c = base + 32 * j;
                if (c < n2) {
                    const float2 bb = b2[c], uu = u2v[c], hh = h2[c];
                    const int64_t rc = sc.r0 - (int64_t)c * 2;           // position of column r0 inside this piece, if any
                    double2 v = srow ? make_double2(0.0, 0.0) : h[j];
                    v.x = fma(us, (double)uu.x, fma(nb, (double)bb.x, v.x));
                    v.y = fma(us, (double)uu.y, fma(nb, (double)bb.y, v.y));
                    v.x = rc == 0 ? corner : v.x;
                    v.y = rc == 1 ? corner : v.y;
                    row[c] = v;
                    y0 = fma(v.x, (double)hh.x, y0);
                    y1 = fma(v.y, (double)hh.y, y1);
                }
            }
        }
        const double t = warp_sum(y0 + y1);
        if (lane == 0) p.y[s] = (float)t;
    }
}

// Best candidate of the block (one per warp in s_best) to *out; all threads call it.
__device__ __forceinline__ void merge_best(LoopCand* s_best, const LoopCand& mine, LoopCand* out)
{
    if ((threadIdx.x & 31) == 0) s_best[threadIdx.x >> 5] = mine;
    __syncthreads();
    if (threadIdx.x == 0) {
        LoopCand b = s_best[0];
        for (int r = 1; r < PL_W; ++r) {
            const LoopCand c = s_best[r];
            if (c.idx >= 0) keep_best(b, c.val, c.id, c.idx);
        }
        *out = b;
    }
}

// pieces in flight per lane by row length (16-byte pieces): short rows need fewer registers, long ones loop
#define PL_DISPATCH(fn, n, ...) do { if ((n) <= 128) fn<4>(__VA_ARGS__); else fn<8>(__VA_ARGS__); } while (0)

__global__ void __launch_bounds__(PL_T, 1) k_swap_loop_g1(LoopArgs a)
{
    // the phase routines are separate functions (their streaming loops get registers of their own); they read the
    // pointers, sizes and scalars from these shared copies
    extern __shared__ float4 pl_vectors[];
    __shared__ Ptrs s_p;
    __shared__ StepScal s_sc;
    __shared__ LoopVecs s_x;
    __shared__ LoopCand s_best[PL_W];
    __shared__ float red[PL_W];
    __shared__ int s_flag, s_stop, s_idx;
    __shared__ double s_val;
    const Ptrs& p = s_p;
    SearchCtl* ctl = a.p.ctl;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned nblocks = gridDim.x;
    const int nm4 = (int)(a.p.ldm / 4), nh4 = (int)(a.p.ldh / 4);
    if (tid == 0) {
        s_p = a.p;
        if (a.smem_vectors) { s_x.K = pl_vectors; s_x.Q = pl_vectors + nm4; s_x.b = pl_vectors + 2 * nm4; s_x.u2 = pl_vectors + 2 * nm4 + nh4; }
        else {
            s_x.K = reinterpret_cast<const float4*>(a.p.K); s_x.Q = reinterpret_cast<const float4*>(a.p.Vq);
            s_x.b = reinterpret_cast<const float4*>(a.p.b); s_x.u2 = reinterpret_cast<const float4*>(a.p.u2);
        }
    }
    if (ctl->done) return;                              // uniform: nothing writes `done` before every block has read it
    const long long limit = ctl->wait_limit;
    unsigned long long epoch = 0;
    double obj = ctl->obj;
    int n_swaps = ctl->n_swaps;
    const int64_t W = (int64_t)nblocks * PL_W;
    const int64_t w0 = (int64_t)warp * nblocks + blockIdx.x;          // neighbouring rows go to different SMs
    const int64_t w0h = ((w0 - a.p.nI) % W + W) % W;                  // H rows are dealt behind the rows of V

    // candidates from the score vectors that the host-side bootstrap left (D, A of the current state)
    if (tid == 0) {
        LoopCand bd; bd.idx = -1; bd.val = 0.0; bd.id = 0;
        for (int64_t s = blockIdx.x; s < a.p.nI; s += nblocks) {
            const double v = a.p.D[s];
            if (isfinite(v)) keep_best(bd, v, a.p.perm[s], s);
        }
        a.candD[blockIdx.x] = bd;
        if (blockIdx.x == 0) { LoopCand e; e.idx = -1; e.val = 0.0; e.id = 0; a.candD[nblocks] = e; }
        LoopCand ba; ba.idx = -1; ba.val = 0.0; ba.id = 0;
        for (int64_t s = blockIdx.x; s < a.p.nJ; s += nblocks) {
            const double v = -a.p.A[s];
            if (isfinite(v)) keep_best(ba, v, a.p.perm[a.p.k + s], s);
        }
        a.candA[blockIdx.x] = ba;
    }
    if (!grid_barrier(ctl, epoch, nblocks, limit, &s_flag)) return;
    int64_t t_cur;
    {
        if (tid < 32) {
            double v; int idx;
            reduce_cands(a.candA, nblocks, false, &v, &idx);
            if (tid == 0) s_idx = idx;
        }
        __syncthreads();
        t_cur = s_idx;
        __syncthreads();
    }
    if (t_cur < 0) {                                    // no eligible group to add
        if (blockIdx.x == 0 && tid == 0) { ctl->done = 1; ctl->stop_reason = OSSCAR_STOP_GUARD; *p.done_host = 1; }
        return;
    }
    unsigned long long tp = 0;
    const bool timer = blockIdx.x == 0 && tid == 0;
    if (timer) tp = global_timer_ns();
#define PL_LAP(phase) do { if (timer) { const unsigned long long now_ = global_timer_ns(); a.prof[phase] += now_ - tp; tp = now_; } } while (0)

    for (int step = 0; step < a.max_steps && n_swaps < a.max_swaps; ++step) {
        // ---------------------------------------------------------------- A: decision
        LoopCand* const cur = a.candD + (step & 1) * PL_CAND;
        LoopCand* const next = a.candD + ((step & 1) ^ 1) * PL_CAND;
        if (tid < 32) {
            double v; int idx;
            reduce_cands(cur, nblocks + 1, false, &v, &idx);
            if (tid == 0) s_idx = idx;
        }
        __syncthreads();
        const int slot = s_idx;
        if (slot < 0) {
            if (blockIdx.x == 0 && tid == 0) { ctl->done = 1; ctl->stop_reason = OSSCAR_STOP_GUARD; *p.done_host = 1; }
            return;
        }
        const int64_t r0 = slot, t = t_cur;
        const float4* v4 = reinterpret_cast<const float4*>(p.V + r0 * p.ldm);
        const float4* r4 = reinterpret_cast<const float4*>(p.R + t * p.ldm);
        const double2* h2 = reinterpret_cast<const double2*>(p.Hd + r0 * p.ldh);
        const float4* y4 = reinterpret_cast<const float4*>(p.y);
        float4 *sK = pl_vectors, *sQ = pl_vectors + nm4, *sB = pl_vectors + 2 * nm4, *sU = pl_vectors + 2 * nm4 + nh4;
        double C = 0.0, P = 0.0, cq = 0.0, GV = 0.0, GR = 0.0;
        float hdiag = 0.f;
        if (tid == 0) {
            C = p.Hd[r0 * p.ldh + r0]; P = p.y[r0]; cq = p.c[t]; GV = p.vnorm[r0]; GR = p.rnorm[t];
            hdiag = p.Hp[r0 * p.ldp + r0];
        }
        float gx = 0.f;
        for (int c = tid; c < nm4; c += PL_T) {
            const float4 v = v4[c], r = r4[c];
            if (a.smem_vectors) { sK[c] = v; sQ[c] = r; }
            gx += dot4(v, r);
        }
        if (a.smem_vectors)
            for (int c = tid; c < nh4; c += PL_T) {
                const double2 h0 = h2[2 * c], h1 = h2[2 * c + 1];
                sB[c] = make_float4((float)h0.x, (float)h0.y, (float)h1.x, (float)h1.y);
                sU[c] = y4[c];
            }
        gx = warp_sum(gx);
        if (lane == 0) red[warp] = gx;
        __syncthreads();
        if (tid == 0) {
            float g = 0.f;
            for (int i = 0; i < PL_W; ++i) g += red[i];
            const double GX = (double)g;
            const double Cinv = 1.0 / C;
            const double Ds = GV * Cinv;
            const double RR1 = GR + 2.0 * P * Cinv * GX + P * P * Cinv * Cinv * GV;
            const double c1 = cq + P * P * Cinv;
            const double c1inv = 1.0 / c1;
            const double delta = Ds - c1inv * RR1;
            int stop = 0, reason = 0;
            if (!(C > 0.0) || !(c1 > 0.0) || !isfinite(delta)) { stop = 1; reason = OSSCAR_STOP_GUARD; }
            else if (a.accept_mode == OSSCAR_ACCEPT_IMPROVING && !(delta <= -a.tol * obj)) { stop = 1; reason = OSSCAR_STOP_NO_IMPROVEMENT; }
            s_stop = stop;
            s_val = delta;
            s_sc.r0 = r0; s_sc.t = t;
            s_sc.Cinv_d = Cinv; s_sc.c1inv_d = c1inv;
            s_sc.Cinv = (float)Cinv; s_sc.c1inv = (float)c1inv;
            s_sc.Q1 = (float)(Cinv * P); s_sc.M2 = (float)(c1inv * P * Cinv);
            s_sc.hdiag = hdiag;
            s_sc.dr = 0.f;
            if (blockIdx.x == 0) {
                ctl->delta = delta; ctl->sel_D = Ds; ctl->sel_slot = slot; ctl->sel_t = (int)t;
                if (stop) { ctl->done = 1; ctl->stop_reason = reason; *p.done_host = 1; }
                else {
                    // the two groups trade slots now: the rows of A read the ids of kept slots other than r0, those of B all
                    // others
                    const int tt = p.k + (int)t;
                    const int gi = p.perm[slot], gj = p.perm[tt];
                    a.swap_trace[2 * n_swaps] = gi;
                    a.swap_trace[2 * n_swaps + 1] = gj;
                    a.obj_trace[n_swaps + 1] = obj + delta;
                    ctl->obj = obj + delta;
                    ctl->n_swaps = n_swaps + 1;
                    p.small[S_CINV] = Cinv; p.small[S_C1INV] = c1inv;
                    p.perm[slot] = gj; p.perm[tt] = gi;
                    p.slotof[gj] = slot; p.slotof[gi] = tt;
                }
            }
        }
        __syncthreads();
        if (s_stop) return;
        obj += s_val;
        ++n_swaps;
        const float Cinv = s_sc.Cinv, c1inv = s_sc.c1inv, Q1 = s_sc.Q1, M2 = s_sc.M2;
        auto stage_h = [&](int c, float4 bs, float4 yy, float4* ob, float4* ou) {
            float4 uu = make_float4(fmaf(-bs.x, Q1, yy.x), fmaf(-bs.y, Q1, yy.y), fmaf(-bs.z, Q1, yy.z), fmaf(-bs.w, Q1, yy.w));
            const int64_t rc = r0 - (int64_t)c * 4;
            uu.x = rc == 0 ? 0.f : uu.x; uu.y = rc == 1 ? 0.f : uu.y; uu.z = rc == 2 ? 0.f : uu.z; uu.w = rc == 3 ? 0.f : uu.w;
            ob[c] = bs;
            ou[c] = uu;
        };
        auto stage_m = [&](int c, float4 v, float4 r, float4* ok, float4* oq) {
            ok[c] = make_float4(Cinv * v.x, Cinv * v.y, Cinv * v.z, Cinv * v.w);
            oq[c] = make_float4(fmaf(c1inv, r.x, M2 * v.x), fmaf(c1inv, r.y, M2 * v.y), fmaf(c1inv, r.z, M2 * v.z), fmaf(c1inv, r.w, M2 * v.w));
        };
        if (a.smem_vectors) {                           // in place, by the threads that loaded the pieces
            for (int c = tid; c < nm4; c += PL_T) stage_m(c, sK[c], sQ[c], sK, sQ);
            for (int c = tid; c < nh4; c += PL_T) stage_h(c, sB[c], sU[c], sB, sU);
            __syncthreads();
        } else {                                        // a slice per block, through global memory
            for (int c = blockIdx.x * PL_T + tid; c < nh4; c += nblocks * PL_T) {
                const double2 h0 = h2[2 * c], h1 = h2[2 * c + 1];
                stage_h(c, make_float4((float)h0.x, (float)h0.y, (float)h1.x, (float)h1.y), y4[c], reinterpret_cast<float4*>(p.b), reinterpret_cast<float4*>(p.u2));
            }
            for (int c = blockIdx.x * PL_T + tid; c < nm4; c += nblocks * PL_T)
                stage_m(c, v4[c], r4[c], reinterpret_cast<float4*>(p.K), reinterpret_cast<float4*>(p.Vq));
            if (!grid_barrier(ctl, epoch, nblocks, limit, &s_flag)) return;
        }
        PL_LAP(0);

        // ---------------------------------------------------------------- A: V and the H pass
        LoopCand best; best.idx = -1; best.val = 0.0; best.id = 0;
        PL_DISPATCH(pl_update_rows, nm4, p, 0, s_sc, s_x, w0, W, best);
        PL_DISPATCH(pl_hpass, nh4, p, s_sc, s_x, w0h, W);
        merge_best(s_best, best, &next[blockIdx.x]);
        PL_LAP(1);
        if (!grid_barrier(ctl, epoch, nblocks, limit, &s_flag)) return;

        // ---------------------------------------------------------------- B
        if (tid == 0) s_sc.dr = p.d[p.nJ];
        __syncthreads();
        {   // exchange of the two slots in Hp: the strided column part first, its latency hides behind the row updates
            hswap_g1_at(p, r0, p.nI + t, (int64_t)blockIdx.x * PL_T + tid, (int64_t)nblocks * PL_T);
        }
        best.idx = -1;
        PL_DISPATCH(pl_update_rows, nm4, p, 1, s_sc, s_x, w0, W, best);
        if (w0 == W - 1) pl_entering_row(p, s_sc, s_x, &next[nblocks]);
        merge_best(s_best, best, &a.candA[blockIdx.x]);
        PL_LAP(2);
        if (!grid_barrier(ctl, epoch, nblocks, limit, &s_flag)) return;

        // ---------------------------------------------------------------- C
        if (tid < 32) {
            double v; int idx;
            reduce_cands(a.candA, nblocks, false, &v, &idx);
            if (tid == 0) s_idx = idx;
        }
        __syncthreads();
        const int64_t t_next = s_idx >= 0 ? s_idx : 0;
        const bool no_add = s_idx < 0;
        PL_DISPATCH(pl_update_hinv, 2 * nh4, p, s_sc, s_x, t_next, w0, W);
        t_cur = t_next;
        if (timer) a.prof[4] += 1;
        PL_LAP(3);
        if (no_add) {                                   // the state is complete; nothing can enter at the next step
            if (blockIdx.x == 0 && tid == 0) { ctl->sel_t = -1; ctl->done = 1; ctl->stop_reason = OSSCAR_STOP_GUARD; *p.done_host = 1; }
            return;
        }
        if (!grid_barrier(ctl, epoch, nblocks, limit, &s_flag)) return;
    }
    if (blockIdx.x == 0 && tid == 0) ctl->sel_t = (int)t_cur;
#undef PL_LAP
}
#undef PL_DISPATCH

inline size_t pl_smem_bytes(const Layout& L) { return sizeof(float) * 2 * (size_t)(L.ldm + L.ldh); }
