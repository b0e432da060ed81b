// Swap step for single-row groups streamed from HBM: a chain of six launches in which V, R and the inverse are READ once per
// step and written only every LZ_B-th one.  Included by search.cu after search_g1.cuh (same translation unit).
//
// Bound: HBM.  With every matrix updated in place a step moves 16 n_I^2 + 8 d1 m + 4 n_J n_I bytes, almost half of it writes
// of values that the next step reads back only to change them again.  Here the matrices are kept as a base plus the last
// few rank-two terms (at most LZ_B - 1 pending ones),
//     V = Vb + sum_e cv[s][e] KQ[e],   R = Rb + sum_e cr[l][e] KQ[e],   Hinv = Hb + sum_t (-b_t b_t^T / C_t + u_t u_t^T / c1_t),
// KQ[2t] = K_t, KQ[2t+1] = Vq_t, so that a step reads 8 n_I^2 + 4 d1 m + 4 n_J n_I bytes and every LZ_B-th one also writes:
// at d1 = 28672, m = 7168, k = 8602 2.46 GB a step against 3.52 GB.  The rows of V and R are formed in registers in every
// step, so norms and scores come from the same fp32 values as before (with fewer roundings on the way); y = Hinv h takes the
// pending terms as 2 LZ_B scalars.  The row and column of the leaving slot are replaced in the base at once, and the pending
// coefficients of that slot are cleared.  Per swap: 628 -> 490 us there, 107 -> 97 us at d1 = 8192, m = 2048, k = 4096.
//
//   decide   one cluster of blocks: i* from the candidates, exact change of obj, accept test, the new vectors and coefficients
//   hpass    u_l, d_l for every pruned row and the leaving row
//   rows     V' and R' with their row norms (partial sums per column tile)  ||  slot exchange in Hp
//   finish   D, A, c, the diagonal of the inverse; best candidate per block
//   select   q* for the NEXT step, and the scalars of the pending terms for its y
//   y        y = Hinv' h (and the update of the base in every LZ_B-th step)
#pragma once

constexpr int LZ_B = 4;              // steps between two writes of the matrices
constexpr int LZ_E = 2 * LZ_B;       // coefficient slots of a row
constexpr int LZ_T = 256;            // threads of the streaming kernels: eight warps, 128 columns each, per column tile
constexpr int LZ_R = 8;              // rows of a tile in flight per thread
constexpr int LZ_FB = 296;           // blocks of `finish` (candidates of a step)
constexpr int LZ_CL = 8, LZ_CT = 512;    // decide and select: one cluster of eight blocks

struct LazyPtrs {
    float *KQ;                       // LZ_E vectors of ldm floats
    float *cv, *cr;                  // coefficients [n_I][LZ_E], [n_J][LZ_E]
    double *bu;                      // LZ_E vectors of ldh entries: b_t (row r_t cleared), u_t: fp32 values kept as fp64, which
                                     // spares the passes over the inverse their conversions (16 per clock and SM)
    double *scal;                    // [2 t] = -1 / C_t, [2 t + 1] = 1 / c1_t; [LZ_E + e] = scal[e] * (bu[e] . h)
    double *xch;                     // exchange between the blocks of a cluster: LZ_CL x LZ_E
    double *dg;                      // diagonal of the inverse
    float *part;                     // row norms per column tile: [tile][n_I + n_J]
    LoopCand *candD, *candA;         // LZ_FB each
    double *ypart;                   // partial sums of y per column tile of k_lz_y_write
    int tiles;                       // column tiles
    int warps;                       // warps per column tile
};

// first piece of the area, LZ_FB candidates twice, then the arrays; all 256-byte aligned.  Returns the bytes used.
inline size_t lazy_layout(const Layout& L, char* base, LazyPtrs* z)
{
    size_t off = 0;
    auto take = [&](size_t bytes) { char* p = base + off; off += (bytes + 255) / 256 * 256; return p; };
    const int slabs = (int)((L.ldm + 127) / 128);
    z->tiles = (slabs + LZ_T / 32 - 1) / (LZ_T / 32);
    z->warps = (slabs + z->tiles - 1) / z->tiles;
    z->candD = (LoopCand*)take(sizeof(LoopCand) * LZ_FB);
    z->candA = (LoopCand*)take(sizeof(LoopCand) * LZ_FB);
    z->scal = (double*)take(sizeof(double) * 2 * LZ_E);
    z->xch = (double*)take(sizeof(double) * LZ_CL * LZ_E);
    z->KQ = (float*)take(sizeof(float) * LZ_E * (size_t)L.ldm);
    z->cv = (float*)take(sizeof(float) * LZ_E * (size_t)L.nI);
    z->cr = (float*)take(sizeof(float) * LZ_E * (size_t)L.nJ);
    z->bu = (double*)take(sizeof(double) * LZ_E * (size_t)L.ldh);
    z->dg = (double*)take(sizeof(double) * (size_t)L.nI);
    z->part = (float*)take(sizeof(float) * (size_t)z->tiles * (size_t)L.d1);
    z->ypart = (double*)take(sizeof(double) * (size_t)((L.ldh + 2 * LZ_T - 1) / (2 * LZ_T)) * (size_t)L.nI);
    return off;
}

// Pending terms after a state build: none.
__global__ void k_lz_reset(SearchCtl* ctl) { if (!ctl->done) { ctl->pending = 0; ctl->y_due = 0; } }

// Best of the LZ_FB candidates, by one warp with all its loads in flight at once; all threads of the block call it.
__device__ __forceinline__ void lz_argmin(const LoopCand* cand, double* val, int* idx)
{
    __shared__ double s_v; __shared__ int s_i;
    if (threadIdx.x < 32) {
        LoopCand c[LZ_FB / 32 + 1];
#pragma unroll
        for (int u = 0; u < LZ_FB / 32 + 1; ++u) {
            const int i = (int)threadIdx.x + 32 * u;
            c[u].idx = -1;
            if (i < LZ_FB) c[u] = cand[i];
        }
        double best = INFINITY; int bid = INT_MAX, bidx = -1;
#pragma unroll
        for (int u = 0; u < LZ_FB / 32 + 1; ++u)
            if (c[u].idx >= 0 && cand_less(c[u].val, c[u].id, best, bid)) { best = c[u].val; bid = c[u].id; bidx = c[u].idx; }
        for (int o = 16; o > 0; o >>= 1) {
            const double ov = __shfl_xor_sync(0xffffffffu, best, o);
            const int oid = __shfl_xor_sync(0xffffffffu, bid, o), oidx = __shfl_xor_sync(0xffffffffu, bidx, o);
            if (cand_less(ov, oid, best, bid)) { best = ov; bid = oid; bidx = oidx; }
        }
        if (threadIdx.x == 0) { s_v = best; s_i = bidx; }
    }
    __syncthreads();
    *val = s_v; *idx = s_i;
    __syncthreads();
}

// Barrier of the cluster; what a block wrote before it, in global memory too, is seen by the others after it.
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// P: pending terms before this step (the new one goes to slot P).  One cluster of blocks: every block chooses the leaving row
// and computes the scalars of the step for itself, the vectors are dealt by slices (one block alone took 22-32 us for them).
__global__ void __cluster_dims__(LZ_CL, 1, 1) __launch_bounds__(LZ_CT)
k_lz_decide(Ptrs p, LazyPtrs z, int P, int accept_mode, double accept_tol, double* __restrict__ obj_trace, int32_t* __restrict__ swap_trace)
{
    pdl_wait_then_release();
    SearchCtl* ctl = p.ctl;
    const bool first = blockIdx.x == 0;
    if (ctl->done) { if (first && threadIdx.x == 0) ctl->y_due = 0; return; }         // set by an earlier kernel: the same in every block
    __shared__ float redf[32];
    __shared__ int s_stop;
    __shared__ float s_q1, s_m2, s_cinv, s_c1inv;
    __shared__ float s_cv[LZ_E], s_cr[LZ_E];
    __shared__ double s_f[LZ_E];
    double Dbest; int slot;
    lz_argmin(z.candD, &Dbest, &slot);
    const int64_t t = ctl->sel_t, r0 = slot < 0 ? 0 : slot;
    const int ne = 2 * P;
    const int64_t me = (int64_t)blockIdx.x * LZ_CT + threadIdx.x, all = LZ_CL * LZ_CT;
    if (threadIdx.x < ne) {
        s_cv[threadIdx.x] = z.cv[r0 * LZ_E + threadIdx.x];
        s_cr[threadIdx.x] = z.cr[t * LZ_E + threadIdx.x];
        s_f[threadIdx.x] = z.scal[threadIdx.x] * z.bu[(int64_t)threadIdx.x * p.ldh + r0];
    }
    double C = 0.0, Pd = 0.0, cq = 0.0, GV = 0.0, GR = 0.0, obj = 0.0;
    float hdiag = 0.f;
    if (threadIdx.x == 0) {
        C = z.dg[r0]; Pd = p.y[r0]; cq = p.c[t]; GV = p.vnorm[r0]; GR = p.rnorm[t];
        hdiag = p.Hp[r0 * p.ldp + r0];
        obj = ctl->obj;
    }
    __syncthreads();
    // the two rows as they are now: parked in the new term's own places until the scalars are known
    const int64_t m4 = p.ldm / 4;
    const float4* vr = reinterpret_cast<const float4*>(p.V + r0 * p.ldm);
    const float4* rq = reinterpret_cast<const float4*>(p.R + t * p.ldm);
    float4* kn = reinterpret_cast<float4*>(z.KQ + (int64_t)(2 * P) * p.ldm);
    float4* qn = reinterpret_cast<float4*>(z.KQ + (int64_t)(2 * P + 1) * p.ldm);
    float acc = 0.f;
    for (int64_t c = me; c < m4; c += all) {
        float4 v = vr[c], r = rq[c];
#pragma unroll
        for (int e = 0; e < LZ_E - 2; ++e)
            if (e < ne) {
                const float4 x = reinterpret_cast<const float4*>(z.KQ + (int64_t)e * p.ldm)[c];
                fma4(v, s_cv[e], x);
                fma4(r, s_cr[e], x);
            }
        kn[c] = v; qn[c] = r;
        acc += dot4(v, r);
    }
    const float mine = block_sum_f(acc, redf);
    if (threadIdx.x == 0) z.xch[blockIdx.x] = (double)mine;
    cluster_barrier();
    if (threadIdx.x == 0) {
        double GX = 0.0;
#pragma unroll
        for (int i = 0; i < LZ_CL; ++i) GX += z.xch[i];
        const double Cinv = 1.0 / C;
        const double Ds = GV * Cinv;
        const double RR1 = GR + 2.0 * Pd * Cinv * GX + Pd * Pd * Cinv * Cinv * GV;
        const double c1 = cq + Pd * Pd * Cinv;
        const double c1inv = 1.0 / c1;
        const double delta = Ds - c1inv * RR1;
        bool stop = false; int reason = 0;
        if (slot < 0 || !(C > 0.0) || !(c1 > 0.0) || !isfinite(delta)) { stop = true; reason = OSSCAR_STOP_GUARD; }
        else if (accept_mode == OSSCAR_ACCEPT_IMPROVING && !(delta <= -accept_tol * obj)) { stop = true; reason = OSSCAR_STOP_NO_IMPROVEMENT; }
        if (first) {
            if (slot >= 0) { ctl->delta = delta; ctl->sel_D = Ds; ctl->sel_slot = slot; }
            if (stop) { ctl->done = 1; ctl->stop_reason = reason; ctl->y_due = 0; *p.done_host = 1; }
            else {
                const int n = ctl->n_swaps;
                swap_trace[2 * n] = p.perm[slot];
                swap_trace[2 * n + 1] = p.perm[p.k + t];
                obj_trace[n + 1] = obj + delta;
                ctl->obj = obj + delta;
                ctl->n_swaps = n + 1;
                ctl->pending = P + 1 == LZ_B ? 0 : P + 1;        // the last term of a round is written with the matrices
                ctl->y_due = 1;
                p.small[S_CINV] = Cinv; p.small[S_C1INV] = c1inv;
                p.small[G1_HDIAG] = hdiag;
                z.scal[2 * P] = -Cinv; z.scal[2 * P + 1] = c1inv;
            }
        }
        s_q1 = (float)(Cinv * Pd); s_m2 = (float)(c1inv * Pd * Cinv); s_cinv = (float)Cinv; s_c1inv = (float)c1inv;
        s_stop = stop;
    }
    __syncthreads();
    if (s_stop) return;
    const float Q1 = s_q1, fM2 = s_m2, fC = s_cinv, fc1 = s_c1inv;
    for (int64_t c = me; c < m4; c += all) {
        const float4 v = kn[c], r = qn[c];
        kn[c] = make_float4(fC * v.x, fC * v.y, fC * v.z, fC * v.w);
        qn[c] = make_float4(fmaf(fc1, r.x, fM2 * v.x), fmaf(fc1, r.y, fM2 * v.y), fmaf(fc1, r.z, fM2 * v.z), fmaf(fc1, r.w, fM2 * v.w));
    }
    // b = row r0 of the inverse as it is now, u2 = y - b Q1
    const double* hrow = p.Hd + r0 * p.ldh;
    double* bn = z.bu + (int64_t)(2 * P) * p.ldh;
    double* un = bn + p.ldh;
    for (int64_t j = me; j < p.ldh; j += all) {
        double h = hrow[j];
        const bool self = j == r0;
#pragma unroll
        for (int e = 0; e < LZ_E - 2; ++e)
            if (e < ne) h = fma(s_f[e], z.bu[(int64_t)e * p.ldh + j], h);
        const float bj = (float)h;
        const float uj = self ? 0.f : fmaf(-bj, Q1, p.y[j]);
        p.b[j] = bj; p.u2[j] = uj;
        bn[j] = self ? 0.0 : (double)bj; un[j] = (double)uj;
        if (j < p.nI) *reinterpret_cast<float2*>(z.cv + j * LZ_E + 2 * P) = make_float2(self ? 0.f : -bj, -uj);
        // the leaving slot has no part in the pending terms any more (the other blocks read its entries before the barrier)
        if (self) for (int e = 0; e < ne; ++e) z.bu[(int64_t)e * p.ldh + j] = 0.0;
    }
    if (first && threadIdx.x < ne) {
        z.cv[r0 * LZ_E + threadIdx.x] = 0.f;
        z.cr[t * LZ_E + threadIdx.x] = 0.f;
    }
}

// u_l = Hp[l, 0:n_I] . b and d_l = Hp[l, q] - Hp[l, 0:n_I] . u2 for the pruned rows (items 0 .. n_J - 1) and the leaving row
// (item n_J), RB rows per block with U pieces of each in flight per thread.
template <int RB, int U>
__global__ void __launch_bounds__(LZ_T) k_lz_hpass(Ptrs p, LazyPtrs z, int P)
{
    __shared__ float red[2 * RB][LZ_T / 32];
    const int64_t l0 = (int64_t)blockIdx.x * RB, items = p.nJ + 1;
    const int64_t n4 = p.ldh / 4;
    const bool early = l0 + RB <= p.nJ;          // the leaving row is named by the control block: its block waits first
    if (!early) pdl_wait_then_release();
    const float4* row[RB];
#pragma unroll
    for (int r = 0; r < RB; ++r) {
        const int64_t l = l0 + r < items ? l0 + r : items - 1;
        row[r] = reinterpret_cast<const float4*>(p.Hp + (l < p.nJ ? p.nI + l : (int64_t)p.ctl->sel_slot) * p.ldp);
    }
    const float4* bv = reinterpret_cast<const float4*>(p.b);
    const float4* uv = reinterpret_cast<const float4*>(p.u2);
    float au[RB], ad[RB];
#pragma unroll
    for (int r = 0; r < RB; ++r) { au[r] = 0.f; ad[r] = 0.f; }
    for (int64_t base = threadIdx.x; base < n4; base += (int64_t)LZ_T * U) {
        float4 x[RB][U];
#pragma unroll
        for (int r = 0; r < RB; ++r)
#pragma unroll
            for (int j = 0; j < U; ++j) {
                const int64_t c = base + LZ_T * j;
                x[r][j] = c < n4 ? row[r][c] : make_float4(0.f, 0.f, 0.f, 0.f);
            }
        if (early && base == threadIdx.x) pdl_wait_then_release();          // b and u2 come from the kernel before this one
#pragma unroll
        for (int j = 0; j < U; ++j) {
            const int64_t c = base + LZ_T * j;
            if (c < n4) {
                const float4 bb = bv[c], uu = uv[c];
#pragma unroll
                for (int r = 0; r < RB; ++r) { au[r] += dot4(x[r][j], bb); ad[r] += dot4(x[r][j], uu); }
            }
        }
    }
    if (early && threadIdx.x >= n4) pdl_wait_then_release();               // threads without a piece of the row
    if (p.ctl->done) return;
#pragma unroll
    for (int r = 0; r < RB; ++r) {
        const float a = warp_sum(au[r]), d = warp_sum(ad[r]);
        if ((threadIdx.x & 31) == 0) { red[2 * r][threadIdx.x >> 5] = a; red[2 * r + 1][threadIdx.x >> 5] = d; }
    }
    __syncthreads();
    if (threadIdx.x < RB && l0 + threadIdx.x < items) {
        const int64_t l = l0 + threadIdx.x, tq = p.ctl->sel_t;
        float su = 0.f, sd = 0.f;
#pragma unroll
        for (int i = 0; i < LZ_T / 32; ++i) { su += red[2 * threadIdx.x][i]; sd += red[2 * threadIdx.x + 1][i]; }
        const float d = p.Hp[(l < p.nJ ? p.nI + l : (int64_t)p.ctl->sel_slot) * p.ldp + p.nI + tq] - sd;
        p.u[l] = su;
        p.d[l] = d;
        // row t of R is replaced outright: the newest term has no part in it
        if (l < p.nJ) *reinterpret_cast<float2*>(z.cr + l * LZ_E + 2 * P) = l == tq ? make_float2(0.f, 0.f) : make_float2(su, -d);
    }
}

// Sums over the warp of eight values at once: after the call lane 4 i + (0..3) holds the sum of v[i'], i' = lz_row8(lane).
template <typename T> __device__ __forceinline__ T lz_sum8(const T (&v)[8])
{
    const int lane = threadIdx.x & 31;
    T a[4], b[2];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const T keep = lane & 16 ? v[i + 4] : v[i], give = lane & 16 ? v[i] : v[i + 4];
        a[i] = keep + __shfl_xor_sync(0xffffffffu, give, 16);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const T keep = lane & 8 ? a[i + 2] : a[i], give = lane & 8 ? a[i] : a[i + 2];
        b[i] = keep + __shfl_xor_sync(0xffffffffu, give, 8);
    }
    const T keep = lane & 4 ? b[1] : b[0], give = lane & 4 ? b[0] : b[1];
    T s = keep + __shfl_xor_sync(0xffffffffu, give, 4);
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    return s;
}
__device__ __forceinline__ int lz_row8(int lane) { return ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1); }

// Rows of V' (blocks [0, nbV)) and R' (the next nbR blocks), formed from the base and NT terms with the coefficient vectors held
// in registers: a warp owns 128 columns, a lane one 16-byte piece, rows pass by eight at a time.  A block takes one column
// tile of `rc` rows; the partial norms of its warps are added in order.  FLUSH also writes the rows back; the replaced rows
// (slot r0 of V: Vq, slot t of R: K - d_r Vq) are always written.  The remaining blocks exchange the two slots in Hp.
template <int NT, bool FLUSH>
__global__ void __launch_bounds__(LZ_T, 2) k_lz_rows(Ptrs p, LazyPtrs z, unsigned nbV, unsigned nbR, int rc)
{
    constexpr int NE = 2 * NT;
    if (blockIdx.x >= nbV + nbR) {
        pdl_wait_then_release();
        if (p.ctl->done) return;
        const unsigned b = blockIdx.x - nbV - nbR;
        hswap_g1(p, (int64_t)b * LZ_T + threadIdx.x, (int64_t)(gridDim.x - nbV - nbR) * LZ_T);
        if (b == 0 && threadIdx.x == 0) {
            const int s = p.ctl->sel_slot, t = p.k + p.ctl->sel_t;
            const int gi = p.perm[s], gj = p.perm[t];
            p.perm[s] = gj; p.perm[t] = gi;
            p.slotof[gj] = s; p.slotof[gi] = t;
        }
        return;
    }
    __shared__ float s_coef[128 * NE];
    __shared__ float s_nrm[LZ_T / 32][128];
    const bool isV = blockIdx.x < nbV;
    const unsigned blk = isV ? blockIdx.x : blockIdx.x - nbV;
    float* M = isV ? p.V : p.R;
    const int64_t nrows = isV ? p.nI : p.nJ;
    const int tile = (int)(blk % (unsigned)z.tiles);
    const int64_t row0 = (int64_t)(blk / (unsigned)z.tiles) * rc;
    const int nr = (int)(nrows - row0 < rc ? nrows - row0 : rc);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t c4 = ((int64_t)tile * z.warps + warp) * 32 + lane;
    const bool on = warp < z.warps && c4 < p.ldm / 4;
    float4* base = reinterpret_cast<float4*>(M + row0 * p.ldm) + c4;
    const int64_t ld4 = p.ldm / 4;
    float4 v[LZ_R];
#pragma unroll
    for (int i = 0; i < LZ_R; ++i) v[i] = on && i < nr ? base[i * ld4] : make_float4(0.f, 0.f, 0.f, 0.f);     // requested before the step's scalars arrive
    pdl_wait_then_release();
    if (p.ctl->done) return;
    const int64_t special = isV ? (int64_t)p.ctl->sel_slot : (int64_t)p.ctl->sel_t;
    const int sp = special >= row0 && special < row0 + nr ? (int)(special - row0) : -1;
    const float* coef = (isV ? z.cv : z.cr) + row0 * LZ_E;
    for (int i = threadIdx.x; i < nr * NE; i += LZ_T) s_coef[i] = coef[(i / NE) * LZ_E + i % NE];
    float4 x[NE];
#pragma unroll
    for (int e = 0; e < NE; ++e) x[e] = on ? reinterpret_cast<const float4*>(z.KQ + (int64_t)e * p.ldm)[c4] : make_float4(0.f, 0.f, 0.f, 0.f);
    __syncthreads();
    for (int i0 = 0; i0 < nr; i0 += LZ_R) {
        float nrm[LZ_R];
#pragma unroll
        for (int i = 0; i < LZ_R; ++i) {
            const int r = i0 + i;
            if (r < nr) {
                const float* cf = s_coef + r * NE;
#pragma unroll
                for (int e = 0; e < NE; ++e) fma4(v[i], cf[e], x[e]);
                if (FLUSH && on && r != sp) base[(int64_t)r * ld4] = v[i];
            }
            nrm[i] = dot4(v[i], v[i]);
        }
        const float s = lz_sum8(nrm);
        if ((lane & 3) == 0) s_nrm[warp][i0 + lz_row8(lane)] = s;
#pragma unroll
        for (int i = 0; i < LZ_R; ++i) v[i] = on && i0 + LZ_R + i < nr ? base[(int64_t)(i0 + LZ_R + i) * ld4] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    if (sp >= 0) {           // the replaced row: the newest term alone, and its pending coefficients are clear
        const float dr = isV ? 0.f : p.d[p.nJ];
        const float4 k = x[NE - 2], q = x[NE - 1];
        const float4 w = isV ? q : make_float4(fmaf(-dr, q.x, k.x), fmaf(-dr, q.y, k.y), fmaf(-dr, q.z, k.z), fmaf(-dr, q.w, k.w));
        if (on) base[(int64_t)sp * ld4] = w;
        const float s = warp_sum(dot4(w, w));
        __syncwarp();
        if (lane == 0) s_nrm[warp][sp] = s;
    }
    __syncthreads();
    if (threadIdx.x < nr) {
        float s = 0.f;
        for (int w = 0; w < z.warps; ++w) s += s_nrm[w][threadIdx.x];
        z.part[(int64_t)tile * (p.nI + p.nJ) + (isV ? 0 : p.nI) + row0 + threadIdx.x] = s;
    }
}

// Scores of the new state and the best candidates per block.  INIT: from the row norms and the matrices as they stand.
template <bool INIT>
__global__ void __launch_bounds__(256) k_lz_finish(Ptrs p, LazyPtrs z)
{
    pdl_wait_then_release();
    if (p.ctl->done) return;
    __shared__ LoopCand s_d[8], s_a[8];
    LoopCand bd, ba;
    bd.idx = -1; bd.val = 0.0; bd.id = 0; ba = bd;
    const int64_t d1 = p.nI + p.nJ;
    const double Cinv = INIT ? 0.0 : p.small[S_CINV], c1inv = INIT ? 0.0 : p.small[S_C1INV];
    const int64_t r0 = INIT ? -1 : (int64_t)p.ctl->sel_slot, tq = INIT ? -1 : (int64_t)p.ctl->sel_t;
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < d1; i += (int64_t)gridDim.x * 256) {
        float nr = 0.f;
        if (!INIT) for (int k = 0; k < z.tiles; ++k) nr += z.part[(int64_t)k * d1 + i];
        if (i < p.nI) {
            double hd;
            if (INIT) { hd = p.Hd[i * p.ldh + i]; nr = p.vnorm[i]; }
            else {
                p.vnorm[i] = nr;
                const double bs = p.b[i], us = p.u2[i];
                hd = i == r0 ? c1inv : z.dg[i] - bs * bs * Cinv + us * us * c1inv;
            }
            z.dg[i] = hd;
            const double score = hd > 0.0 ? (double)nr / hd : INFINITY;
            p.D[i] = score;
            if (isfinite(score)) keep_best(bd, score, p.perm[i], i);
        } else {
            const int64_t t = i - p.nI;
            double cc, hd;
            if (INIT) { cc = p.c[t]; hd = p.Hp[i * p.ldp + i]; nr = p.rnorm[t]; }
            else {
                p.rnorm[t] = nr;
                if (t == tq) { const double dr = p.d[p.nJ]; cc = Cinv - dr * dr * c1inv; hd = p.small[G1_HDIAG]; }
                else { const double uu = p.u[t], dd = p.d[t]; cc = p.c[t] + uu * uu * Cinv - dd * dd * c1inv; hd = p.Hp[i * p.ldp + i]; }
                p.c[t] = cc;
            }
            const double score = cc > kAddPivotTol * hd ? (double)nr / cc : -INFINITY;
            p.A[t] = score;
            if (isfinite(score)) keep_best(ba, -score, p.perm[i], t);          // candidates are kept as minima
        }
    }
    auto merge = [&](LoopCand& b) {
        for (int o = 16; o > 0; o >>= 1) {
            LoopCand c;
            c.val = __shfl_xor_sync(0xffffffffu, b.val, o);
            c.id = __shfl_xor_sync(0xffffffffu, b.id, o);
            c.idx = __shfl_xor_sync(0xffffffffu, b.idx, o);
            if (c.idx >= 0) keep_best(b, c.val, c.id, c.idx);
        }
    };
    merge(bd); merge(ba);
    if ((threadIdx.x & 31) == 0) { s_d[threadIdx.x >> 5] = bd; s_a[threadIdx.x >> 5] = ba; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) {
            if (s_d[w].idx >= 0) keep_best(bd, s_d[w].val, s_d[w].id, s_d[w].idx);
            if (s_a[w].idx >= 0) keep_best(ba, s_a[w].val, s_a[w].id, s_a[w].idx);
        }
        z.candD[blockIdx.x] = bd;
        z.candA[blockIdx.x] = ba;
    }
}

// q* for the next step, and for its y the products of h = Hp[q*, 0:n_I] with the NT pending terms; one cluster of blocks.
__global__ void __cluster_dims__(LZ_CL, 1, 1) __launch_bounds__(LZ_CT) k_lz_select(Ptrs p, LazyPtrs z, int NT)
{
    pdl_wait_then_release();
    SearchCtl* ctl = p.ctl;
    if (ctl->done) return;                       // set by an earlier kernel: the same in every block
    __shared__ double s_red[LZ_CT / 32][LZ_E];
    const bool first = blockIdx.x == 0;
    double best; int idx;
    lz_argmin(z.candA, &best, &idx);
    double s[LZ_E];
#pragma unroll
    for (int e = 0; e < LZ_E; ++e) s[e] = 0.0;
    const float* h = p.Hp + (p.nI + (int64_t)(idx < 0 ? 0 : idx)) * p.ldp;
    for (int64_t j = (int64_t)blockIdx.x * LZ_CT + threadIdx.x; j < p.nI && NT > 0; j += LZ_CL * LZ_CT) {
        const double hj = (double)h[j];
#pragma unroll
        for (int e = 0; e < LZ_E; ++e)
            if (e < 2 * NT) s[e] = fma(hj, z.bu[(int64_t)e * p.ldh + j], s[e]);
    }
#pragma unroll
    for (int e = 0; e < LZ_E; ++e)
        if (e < 2 * NT) {
            const double v = warp_sum(s[e]);
            if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5][e] = v;
        }
    __syncthreads();
    if (threadIdx.x < 2 * NT) {
        double v = 0.0;
#pragma unroll
        for (int w = 0; w < LZ_CT / 32; ++w) v += s_red[w][threadIdx.x];
        z.xch[blockIdx.x * LZ_E + threadIdx.x] = v;
    }
    cluster_barrier();
    if (!first) return;
    if (threadIdx.x < 2 * NT) {
        double v = 0.0;
#pragma unroll
        for (int i = 0; i < LZ_CL; ++i) v += z.xch[i * LZ_E + threadIdx.x];
        z.scal[LZ_E + threadIdx.x] = v * z.scal[threadIdx.x];
    }
    if (threadIdx.x == 0) {
        ctl->sel_t = idx;
        // the state moves on with this step's swap; only the next one has nothing to add
        if (idx < 0) { ctl->done = 1; ctl->stop_reason = OSSCAR_STOP_GUARD; *p.done_host = 1; }
    }
}

// y = Hinv' h, one row of the inverse per block; NT pending terms (the newest included) enter as scalars.  The row and column
// of slot r0 are replaced in the base: -u2 / c1, corner 1 / c1.  NT = 0: y of the plain base (start of a chain).
template <int NT, int TB>
__global__ void __launch_bounds__(TB) k_lz_y(Ptrs p, LazyPtrs z)
{
    constexpr int NE = 2 * NT;
    __shared__ double red[8];
    const int64_t s = blockIdx.x;
    const int64_t n2 = p.ldh / 2;
    double2* row = reinterpret_cast<double2*>(p.Hd + s * p.ldh);
    const float2* h2 = nullptr;
    const float2* un = nullptr;
    int64_t r0 = -1;
    bool srow = false;
    double c1inv = 0.0, corner = 0.0, yacc0 = 0.0, yacc1 = 0.0;
    for (int64_t base = threadIdx.x; base < n2; base += (int64_t)TB * G1_UH) {
        double2 v[G1_UH];
#pragma unroll
        for (int j = 0; j < G1_UH; ++j) {
            const int64_t c = base + TB * j;
            v[j] = c < n2 ? row[c] : make_double2(0.0, 0.0);          // requested before the step's scalars arrive
        }
        if (base == threadIdx.x) {
            pdl_wait_then_release();
            // a stop that this step's own selection found (nothing can enter next) leaves a swap whose base must follow; a step
            // that did not swap changes nothing
            if (p.ctl->done && (NT == 0 || !p.ctl->y_due)) return;
            h2 = reinterpret_cast<const float2*>(p.Hp + (p.nI + (int64_t)(p.ctl->sel_t < 0 ? 0 : p.ctl->sel_t)) * p.ldp);
            if (NT > 0) {
                r0 = p.ctl->sel_slot;
                c1inv = p.small[S_C1INV];
                un = reinterpret_cast<const float2*>(p.u2);
                srow = s == r0;
                corner = srow ? c1inv : -(double)p.u2[s] * c1inv;            // value of column r0 in this row
            }
        }
#pragma unroll
        for (int j = 0; j < G1_UH; ++j) {
            const int64_t c = base + TB * j;
            if (c < n2) {
                const float2 hh = h2[c];
                double2 w = v[j];
                if (NT > 0) {
                    const int64_t rc = r0 - c * 2;           // position of column r0 inside this piece, if any
                    if (srow) { const float2 uu = un[c]; w = make_double2(-(double)uu.x * c1inv, -(double)uu.y * c1inv); }
                    w.x = rc == 0 ? corner : w.x;
                    w.y = rc == 1 ? corner : w.y;
                    if (srow || rc == 0 || rc == 1) row[c] = w;
                }
                yacc0 = fma(w.x, (double)hh.x, yacc0);
                yacc1 = fma(w.y, (double)hh.y, yacc1);
            }
        }
    }
    if (threadIdx.x >= n2) {           // threads without a piece of the row
        pdl_wait_then_release();
        if (p.ctl->done && (NT == 0 || !p.ctl->y_due)) return;
    }
    const double t = warp_sum(yacc0 + yacc1);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        double sum = 0.0;
#pragma unroll
        for (int i = 0; i < TB / 32; ++i) sum += red[i];
#pragma unroll
        for (int e = 0; e < NE; ++e) sum = fma(z.scal[LZ_E + e], z.bu[(int64_t)e * p.ldh + s], sum);
        p.y[s] = (float)sum;
    }
}

// The last step of a round: the NT terms are added to the rows of the inverse, which are written, and y = Hinv' h in the same
// pass.  The layout of k_lz_rows: a lane owns one double2 of the columns and keeps the 2 NT pieces of the vectors in
// registers while eight rows at a time pass by (a row per block re-read 550 KB of vectors from L2 for every row: 0.36 ms
// at n_I = 8602, two rows per block 0.30 ms, now 0.22 ms).  Blocks of rc <= 64 rows x LZ_YC columns; the partial sums of y per
// column tile are added by k_lz_y_sum.
constexpr int LZ_YC = 2 * LZ_T;
template <int NT>
__global__ void __launch_bounds__(LZ_T, 2) k_lz_y_write(Ptrs p, LazyPtrs z, int tiles, int rc)
{
    constexpr int NE = 2 * NT;
    __shared__ double s_f[64][NE];
    __shared__ double s_y[LZ_T / 32][64];
    const int tile = (int)(blockIdx.x % (unsigned)tiles);
    const int64_t row0 = (int64_t)(blockIdx.x / (unsigned)tiles) * rc;
    const int nr = (int)(p.nI - row0 < rc ? p.nI - row0 : rc);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t c = (int64_t)tile * LZ_T + threadIdx.x, n2 = p.ldh / 2;
    const bool on = c < n2;
    double2* base = reinterpret_cast<double2*>(p.Hd + row0 * p.ldh) + c;
    double2 v[LZ_R];
#pragma unroll
    for (int i = 0; i < LZ_R; ++i) v[i] = on && i < nr ? base[i * n2] : make_double2(0.0, 0.0);
    pdl_wait_then_release();
    if (p.ctl->done && !p.ctl->y_due) return;           // see k_lz_y
    const int64_t r0 = p.ctl->sel_slot;
    const double c1inv = p.small[S_C1INV];
    const float2 hh = on ? reinterpret_cast<const float2*>(p.Hp + (p.nI + (int64_t)(p.ctl->sel_t < 0 ? 0 : p.ctl->sel_t)) * p.ldp)[c] : make_float2(0.f, 0.f);
    const double hx = (double)hh.x, hy = (double)hh.y;
    for (int i = threadIdx.x; i < nr * NE; i += LZ_T) s_f[i / NE][i % NE] = z.scal[i % NE] * z.bu[(int64_t)(i % NE) * p.ldh + row0 + i / NE];
    double2 x[NE];
#pragma unroll
    for (int e = 0; e < NE; ++e) x[e] = on ? reinterpret_cast<const double2*>(z.bu + (int64_t)e * p.ldh)[c] : make_double2(0.0, 0.0);
    const float2 uu = on ? reinterpret_cast<const float2*>(p.u2)[c] : make_float2(0.f, 0.f);
    const int64_t rcol = r0 - c * 2;                     // position of column r0 inside this piece, if any
    __syncthreads();
    for (int i0 = 0; i0 < nr; i0 += LZ_R) {
        double ys[LZ_R];
#pragma unroll
        for (int i = 0; i < LZ_R; ++i) {
            const int r = i0 + i;
            ys[i] = 0.0;
            if (r < nr) {
                double2 w = v[i];
#pragma unroll
                for (int e = 0; e < NE; ++e) { w.x = fma(s_f[r][e], x[e].x, w.x); w.y = fma(s_f[r][e], x[e].y, w.y); }
                const bool srow = row0 + r == r0;
                if (srow) w = make_double2(-(double)uu.x * c1inv, -(double)uu.y * c1inv);
                if (rcol == 0 || rcol == 1) {
                    const double corner = srow ? c1inv : -(double)p.u2[row0 + r] * c1inv;
                    if (rcol == 0) w.x = corner; else w.y = corner;
                }
                if (on) base[(int64_t)r * n2] = w;
                ys[i] = fma(w.x, hx, w.y * hy);
            }
        }
        const double s = lz_sum8(ys);
        if ((lane & 3) == 0) s_y[warp][i0 + lz_row8(lane)] = s;
#pragma unroll
        for (int i = 0; i < LZ_R; ++i) v[i] = on && i0 + LZ_R + i < nr ? base[(int64_t)(i0 + LZ_R + i) * n2] : make_double2(0.0, 0.0);
    }
    __syncthreads();
    if (threadIdx.x < nr) {
        double s = 0.0;
#pragma unroll
        for (int w = 0; w < LZ_T / 32; ++w) s += s_y[w][threadIdx.x];
        z.ypart[(int64_t)tile * p.nI + row0 + threadIdx.x] = s;
    }
}
__global__ void __launch_bounds__(256) k_lz_y_sum(Ptrs p, LazyPtrs z, int tiles)
{
    pdl_wait_then_release();
    if (p.ctl->done && !p.ctl->y_due) return;
    const int64_t s = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (s >= p.nI) return;
    double t = 0.0;
    for (int k = 0; k < tiles; ++k) t += z.ypart[(int64_t)k * p.nI + s];
    p.y[s] = (float)t;
}

// End of a search: the terms still pending (their number is on the device: a loop may stop anywhere) go into the matrices.
// blockIdx.y: 0 V, 1 R, 2 the inverse; one row per block.
__global__ void __launch_bounds__(256) k_lz_flush(Ptrs p, LazyPtrs z)
{
    const int ne = 2 * p.ctl->pending;
    const int64_t s = blockIdx.x;
    if (ne == 0) return;
    if (blockIdx.y == 2) {
        if (s >= p.nI) return;
        double* row = p.Hd + s * p.ldh;
        double f[LZ_E];
#pragma unroll
        for (int e = 0; e < LZ_E; ++e) f[e] = e < ne ? z.scal[e] * z.bu[(int64_t)e * p.ldh + s] : 0.0;
        for (int64_t c = threadIdx.x; c < p.ldh; c += 256) {
            double v = row[c];
#pragma unroll
            for (int e = 0; e < LZ_E; ++e) if (e < ne) v = fma(f[e], z.bu[(int64_t)e * p.ldh + c], v);
            row[c] = v;
        }
        return;
    }
    const bool isV = blockIdx.y == 0;
    if (s >= (isV ? p.nI : p.nJ)) return;
    float4* row = reinterpret_cast<float4*>((isV ? p.V : p.R) + s * p.ldm);
    float f[LZ_E];
#pragma unroll
    for (int e = 0; e < LZ_E; ++e) f[e] = e < ne ? (isV ? z.cv : z.cr)[s * LZ_E + e] : 0.f;
    for (int64_t c = threadIdx.x; c < p.ldm / 4; c += 256) {
        float4 v = row[c];
#pragma unroll
        for (int e = 0; e < LZ_E; ++e) if (e < ne) fma4(v, f[e], reinterpret_cast<const float4*>(z.KQ + (int64_t)e * p.ldm)[c]);
        row[c] = v;
    }
}
