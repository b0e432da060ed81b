// In-place inverse of an SPD matrix by the blocked exchange (Gauss-Jordan) scheme: per 64-wide pivot block P
//   Dinv = A[P,P]^-1 (fp64),  T = A[:,P] Dinv,  Un = -Dinv A[P,:],  A -= T A[P,:],  A[:,P] = T, A[P,:] = Un, A[P,P] = Dinv.
//
// Bound: the chain of n / 64 steps, about 26 us each.  A step is two launches, chained as programmatic dependents: the
// panels, and the update of the whole matrix with the write-back in its epilogue, in which block 0 meanwhile inverts the
// NEXT pivot block (from a copy that the panel kernel made, brought up to date by itself), so that the serial inverse
// hides behind the update.  Before (pivot inverse, two panel products, two copies, update, write-back: seven launches a
// step) the build of a state of 2304 rows took 4.0 ms with its correction, then 3.6 ms; 1777 rows 5.9 -> 3.1 ms with the digit
// products of the correction.
// From kSweptRows rows up the matrix is swept in blocks of 512 pivots on the tensor cores, and the scheme above inverts the 512 x 512
// pivot blocks: the matrix is read and written n / 512 times instead of n / 64 times.  4096 rows 4.8 -> 3.1 ms, 8602 rows 42 -> 8.5 ms;
// blocks of 256 at 2304 rows took as long as the steps of 64 (1.8 ms), which keep everything below.
#include "osscar_internal.cuh"
#include <math.h>

namespace osscar {
namespace {

constexpr int NB = 64;
constexpr double kPivotRelTol = 1e-7;
constexpr int GJ_T = 256;
constexpr int UP_M = 64, UP_N = 128;                     // tile of the update

struct PivotSmem {
    double rowj[2][NB];
    double hdiag[NB];
    float out[NB][NB + 1];
    int bad;
};

constexpr int PV_FLOATS = 5120;                          // shared memory of block 0: PivotSmem, then two 64 x 65 panels
constexpr int UP_SMEM = (PV_FLOATS + 2 * NB * (NB + 1)) * (int)sizeof(float);
static_assert(sizeof(PivotSmem) <= PV_FLOATS * sizeof(float) && UP_SMEM >= (UP_M * NB + NB * UP_N) * (int)sizeof(float), "shared memory of the update");

// Inverse of the nb x nb block whose entry (i, c) is x[i % 4][c % 4] of thread (i / 4) * 16 + c / 4 (zeros beyond nb), by
// Gauss-Jordan elimination without pivoting: 256 threads, 16 entries each in registers.  In step j the half-warp that owns
// row j publishes it scaled by the inverse pivot, with the inverse pivot itself in column j (double-buffered shared memory,
// one barrier per step); all others drop their entry of column j, whose old value they need as the factor of the rank-1
// update, and every entry is one multiply-add.  The pivots are the diagonal of the successive Schur complements (the
// squared diagonal of the Cholesky factor).  Dinv (row stride NB) receives the symmetrised inverse; OSSCAR_E_NOTPD is
// raised in ctl->status when a pivot is not positive.
__device__ void pivot_inverse(double (&x)[4][4], int nb, PivotSmem& sm, float* Dinv, SearchCtl* ctl)
{
    const int t = threadIdx.x, lane = t & 31, rg = t >> 4, cg = t & 15;
    for (int j4 = 0; j4 < NB / 4; ++j4) {
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) {
            const int j = j4 * 4 + jj;
            if (j < nb) {
                double* row = sm.rowj[j & 1];
                double f[4];
#pragma unroll
                for (int a = 0; a < 4; ++a) f[a] = __shfl_sync(0xffffffffu, x[a][jj], (lane & 16) | j4);      // entries (row, j)
                if (rg == j4) {
                    double d = f[jj];
                    // a pivot that fp32 data cannot tell from zero counts as not positive
                    if (!(d > kPivotRelTol * sm.hdiag[j])) { if (cg == 0) sm.bad = 1; d = 1.0; }
                    const double pinv = 1.0 / d;
#pragma unroll
                    for (int b = 0; b < 4; ++b) row[cg * 4 + b] = cg == j4 && b == jj ? pinv : x[jj][b] * pinv;
                }
                __syncthreads();
                double r[4];
#pragma unroll
                for (int b = 0; b < 4; ++b) r[b] = row[cg * 4 + b];
#pragma unroll
                for (int a = 0; a < 4; ++a) {
                    if (cg == j4) x[a][jj] = 0.0;
                    const bool own = a == jj && rg == j4;
#pragma unroll
                    for (int b = 0; b < 4; ++b) x[a][b] = own ? r[b] : x[a][b] - f[a] * r[b];
                }
            }
        }
    }
    // the two triangles differ by rounding only
    __syncthreads();
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) sm.out[rg * 4 + a][cg * 4 + b] = (float)x[a][b];
    __syncthreads();
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int i = rg * 4 + a, c = cg * 4 + b;
            if (i < nb && c < nb) Dinv[i * NB + c] = 0.5f * (sm.out[i][c] + sm.out[c][i]);
        }
    if (t == 0 && sm.bad && ctl->status == OSSCAR_OK) ctl->status = OSSCAR_E_NOTPD;       // the first error is the one reported
}

// The pivot block A[p0:, p0:] (nb x nb), by one block of GJ_T threads.
__device__ void pivot_block(const float* A, int64_t lda, int64_t p0, int nb, float* Dinv, const float* ref, int64_t ldref, SearchCtl* ctl)
{
    __shared__ PivotSmem sm;
    const int t = threadIdx.x, rg = t >> 4, cg = t & 15;
    double x[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int i = rg * 4 + a, c = cg * 4 + b;
            // symmetrise: the two triangles can differ in the last bits
            x[a][b] = i < nb && c < nb ? 0.5 * ((double)A[(p0 + i) * lda + p0 + c] + (double)A[(p0 + c) * lda + p0 + i]) : 0.0;
        }
    if (t == 0) sm.bad = 0;
    if (t < nb) sm.hdiag[t] = (double)ref[(p0 + t) * ldref + p0 + t];
    __syncthreads();
    pivot_inverse(x, nb, sm, Dinv, ctl);
}
__global__ void __launch_bounds__(GJ_T)
k_gj_pivot(const float* A, int64_t lda, int64_t p0, int nb, float* Dinv, const float* ref, int64_t ldref, SearchCtl* ctl)
{
    pivot_block(A, lda, p0, nb, Dinv, ref, ldref, ctl);
}

// Rows [32 b, 32 b + 32) of T = A[:,P] Dinv (zero in the pivot rows) and columns [32 b, 32 b + 32) of U = A[P,:] and
// Un = -Dinv U; block 0 also copies the next pivot block, before the update changes it.
__global__ void __launch_bounds__(GJ_T)
k_gj_panels(const float* A, int64_t lda, int64_t n, int64_t p0, int nb, const float* Dinv, float* T, float* U, float* Un, int64_t ldu,
            float* next)
{
    pdl_wait_then_release();
    __shared__ float sD[NB][NB];
    __shared__ float sA[NB][33];          // A[row, P] transposed: [k][row]
    __shared__ float sU[NB][33];          // A[P, col]: [k][col]
    const int t = threadIdx.x;
    const int64_t i0 = (int64_t)blockIdx.x * 32;
    {   // everything a thread needs is requested at once: Dinv four, A and U two 16-byte pieces each (A is padded to whole pieces)
        float4 d[4], av[2], uv[2];
#pragma unroll
        for (int q = 0; q < 4; ++q) d[q] = reinterpret_cast<const float4*>(Dinv)[t + q * GJ_T];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int ra = (t + q * GJ_T) >> 4, ka = ((t + q * GJ_T) & 15) * 4;          // row of the panel, first k
            const int ku = (t + q * GJ_T) >> 3, cu = ((t + q * GJ_T) & 7) * 4;           // k, first column
            av[q] = i0 + ra < n && p0 + ka < lda ? *reinterpret_cast<const float4*>(A + (i0 + ra) * lda + p0 + ka) : make_float4(0.f, 0.f, 0.f, 0.f);
            uv[q] = ku < nb && i0 + cu < lda ? *reinterpret_cast<const float4*>(A + (p0 + ku) * lda + i0 + cu) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int i = (t + q * GJ_T) >> 4, c = ((t + q * GJ_T) & 15) * 4;
            const float e[4] = {d[q].x, d[q].y, d[q].z, d[q].w};
#pragma unroll
            for (int k = 0; k < 4; ++k) sD[i][c + k] = i < nb && c + k < nb ? e[k] : 0.f;
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int ra = (t + q * GJ_T) >> 4, ka = ((t + q * GJ_T) & 15) * 4;
            const int ku = (t + q * GJ_T) >> 3, cu = ((t + q * GJ_T) & 7) * 4;
            const float ea[4] = {av[q].x, av[q].y, av[q].z, av[q].w}, eu[4] = {uv[q].x, uv[q].y, uv[q].z, uv[q].w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                sA[ka + k][ra] = ka + k < nb ? ea[k] : 0.f;
                sU[ku][cu + k] = i0 + cu + k < n ? eu[k] : 0.f;
            }
        }
    }
    if (blockIdx.x == 0 && next)
#pragma unroll
        for (int q = 0; q < 4; ++q) {               // pieces past the matrix are padding, of no use to the pivot block
            const int64_t i = p0 + NB + ((t + q * GJ_T) >> 4), c = p0 + NB + ((t + q * GJ_T) & 15) * 4;
            reinterpret_cast<float4*>(next)[t + q * GJ_T] = i < n && c < lda ? *reinterpret_cast<const float4*>(A + i * lda + c) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    __syncthreads();
    {   // T: a thread takes one row and 8 columns
        const int r = t & 31, c0 = (t >> 5) * 8;
        float acc[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[c] = 0.f;
#pragma unroll 8
        for (int k = 0; k < NB; ++k) {
            const float a = sA[k][r];
#pragma unroll
            for (int c = 0; c < 8; ++c) acc[c] = fmaf(a, sD[k][c0 + c], acc[c]);
        }
        const int64_t row = i0 + r;
        const bool pivot = row >= p0 && row < p0 + nb;
        if (row < n) {
            float4* dst = reinterpret_cast<float4*>(T + row * NB + c0);
            dst[0] = pivot ? make_float4(0.f, 0.f, 0.f, 0.f) : make_float4(acc[0], acc[1], acc[2], acc[3]);
            dst[1] = pivot ? make_float4(0.f, 0.f, 0.f, 0.f) : make_float4(acc[4], acc[5], acc[6], acc[7]);
        }
    }
    {   // U and Un: a thread takes one column and 8 rows
        const int c = t & 31, r0 = (t >> 5) * 8;
        float acc[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) acc[r] = 0.f;
#pragma unroll 8
        for (int k = 0; k < NB; ++k) {
            const float u = sU[k][c];
#pragma unroll
            for (int r = 0; r < 8; ++r) acc[r] = fmaf(sD[r0 + r][k], u, acc[r]);
        }
        if (i0 + c < n) {
#pragma unroll
            for (int r = 0; r < 8; ++r)
                if (r0 + r < nb) {
                    U[(r0 + r) * ldu + i0 + c] = sU[r0 + r][c];
                    Un[(r0 + r) * ldu + i0 + c] = -acc[r];
                }
        }
    }
}

// New value of entry (row, col) outside the plain update: the pivot block's row and column panels.
__device__ __forceinline__ float gj_entry(int64_t row, int64_t col, int64_t p0, int nb, float v, const float* T, const float* Un, int64_t ldu, const float* Dinv)
{
    const bool pr = row >= p0 && row < p0 + nb, pc = col >= p0 && col < p0 + nb;
    if (pr && pc) return Dinv[(row - p0) * NB + (col - p0)];
    if (pr) return Un[(row - p0) * ldu + col];
    if (pc) return T[row * NB + (col - p0)];
    return v;
}

// A -= T U with the write-back of the panels; tile UP_M x UP_N per block, 4 x 8 entries per thread.  Block 0 inverts the next
// pivot block instead (its tile-mates are the blocks 1, 2, ...).
__global__ void __launch_bounds__(GJ_T)
k_gj_update(float* A, int64_t lda, int64_t n, int64_t p0, int nb, const float* T, const float* U, const float* Un, int64_t ldu,
            const float* Dinv, const float* next, float* Dnext, const float* ref, int64_t ldref, int tiles_n, SearchCtl* ctl)
{
    pdl_wait_then_release();
    extern __shared__ __align__(16) float up_smem[];
    const int t = threadIdx.x;
    if (blockIdx.x == 0) {
        const int64_t q0 = p0 + NB;
        if (q0 >= n) return;
        const int nbq = (int)(n - q0 < NB ? n - q0 : NB);
        PivotSmem& sm = *reinterpret_cast<PivotSmem*>(up_smem);
        const int rg = t >> 4, cg = t & 15;
        float* sT = up_smem + PV_FLOATS;              // [row][k], [k][col]
        float* sU = sT + NB * (NB + 1);
        float4 tv[4], uv[4], nv[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int i = (t + q * GJ_T) >> 4, c = ((t + q * GJ_T) & 15) * 4;
            tv[q] = i < nbq ? *reinterpret_cast<const float4*>(T + (q0 + i) * NB + c) : make_float4(0.f, 0.f, 0.f, 0.f);
            uv[q] = i < nb && q0 + c < ldu ? *reinterpret_cast<const float4*>(U + i * ldu + q0 + c) : make_float4(0.f, 0.f, 0.f, 0.f);
            nv[q] = *reinterpret_cast<const float4*>(next + (rg * 4 + q) * NB + cg * 4);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int i = (t + q * GJ_T) >> 4, c = ((t + q * GJ_T) & 15) * 4;
            const float et[4] = {tv[q].x, tv[q].y, tv[q].z, tv[q].w}, eu[4] = {uv[q].x, uv[q].y, uv[q].z, uv[q].w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                sT[i * (NB + 1) + c + k] = c + k < nb ? et[k] : 0.f;
                sU[i * (NB + 1) + c + k] = c + k < nbq ? eu[k] : 0.f;
            }
        }
        __syncthreads();
        float v[4][4];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) v[a][b] = 0.f;
#pragma unroll 4
        for (int k = 0; k < NB; ++k) {
            float ta[4], ub[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) ta[a] = sT[(rg * 4 + a) * (NB + 1) + k];
#pragma unroll
            for (int b = 0; b < 4; ++b) ub[b] = sU[k * (NB + 1) + cg * 4 + b];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) v[a][b] = fmaf(ta[a], ub[b], v[a][b]);
        }
        if (t == 0) sm.bad = 0;
        if (t < nbq) sm.hdiag[t] = (double)ref[(q0 + t) * ldref + q0 + t];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const int i = rg * 4 + a, c = cg * 4 + b;
                v[a][b] = (b == 0 ? nv[a].x : b == 1 ? nv[a].y : b == 2 ? nv[a].z : nv[a].w) - v[a][b];
                sm.out[i][c] = v[a][b];
            }
        __syncthreads();
        double x[4][4];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const int i = rg * 4 + a, c = cg * 4 + b;
                x[a][b] = i < nbq && c < nbq ? 0.5 * ((double)v[a][b] + (double)sm.out[c][i]) : 0.0;
            }
        __syncthreads();
        pivot_inverse(x, nbq, sm, Dnext, ctl);
        return;
    }
    float* sT = up_smem;                              // [k][row]
    float* sU = up_smem + NB * UP_M;                  // [k][col]
    const int tile = blockIdx.x - 1;
    const int64_t m0 = (int64_t)(tile / tiles_n) * UP_M, n0 = (int64_t)(tile % tiles_n) * UP_N;
    {   // T: lanes along rows, four k per thread and round
        const int r = t & 63;
        for (int k4 = (t >> 6) * 4; k4 < NB; k4 += 16) {
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (m0 + r < n) v = *reinterpret_cast<const float4*>(T + (m0 + r) * NB + k4);
            sT[(k4 + 0) * UP_M + r] = k4 + 0 < nb ? v.x : 0.f; sT[(k4 + 1) * UP_M + r] = k4 + 1 < nb ? v.y : 0.f;
            sT[(k4 + 2) * UP_M + r] = k4 + 2 < nb ? v.z : 0.f; sT[(k4 + 3) * UP_M + r] = k4 + 3 < nb ? v.w : 0.f;
        }
        for (int idx = t; idx < NB * (UP_N / 4); idx += GJ_T) {
            const int k = idx / (UP_N / 4), c = (idx % (UP_N / 4)) * 4;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (k < nb) {
                const float* src = U + k * ldu + n0 + c;
                if (n0 + c + 3 < n) v = *reinterpret_cast<const float4*>(src);
                else {
                    if (n0 + c < n) v.x = src[0];
                    if (n0 + c + 1 < n) v.y = src[1];
                    if (n0 + c + 2 < n) v.z = src[2];
                }
            }
            *reinterpret_cast<float4*>(sU + k * UP_N + c) = v;
        }
    }
    const int tr = (t >> 4) * 4, tc = (t & 15) * 4;   // rows tr .. tr + 3, columns tc .. tc + 3 and tc + 64 .. tc + 67
    float4 old[4][2];
    const int64_t col0 = n0 + tc, col1 = n0 + 64 + tc;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        const int64_t row = m0 + tr + a;
        old[a][0] = row < n && col0 + 3 < n ? *reinterpret_cast<const float4*>(A + row * lda + col0) : make_float4(0.f, 0.f, 0.f, 0.f);
        old[a][1] = row < n && col1 + 3 < n ? *reinterpret_cast<const float4*>(A + row * lda + col1) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();
    float acc[4][8];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 8; ++b) acc[a][b] = 0.f;
#pragma unroll 4
    for (int k = 0; k < NB; ++k) {
        const float4 ta = *reinterpret_cast<const float4*>(sT + k * UP_M + tr);
        const float4 u0 = *reinterpret_cast<const float4*>(sU + k * UP_N + tc), u1 = *reinterpret_cast<const float4*>(sU + k * UP_N + 64 + tc);
        const float av[4] = {ta.x, ta.y, ta.z, ta.w}, uv[8] = {u0.x, u0.y, u0.z, u0.w, u1.x, u1.y, u1.z, u1.w};
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 8; ++b) acc[a][b] = fmaf(av[a], uv[b], acc[a][b]);
    }
    const bool panel = (m0 < p0 + nb && m0 + UP_M > p0) || (n0 < p0 + nb && n0 + UP_N > p0);      // the tile meets a pivot panel
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        const int64_t row = m0 + tr + a;
        if (row >= n) continue;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int64_t col = h ? col1 : col0;
            float* dst = A + row * lda + col;
            float4 o = old[a][h];
            float v[4] = {o.x - acc[a][4 * h], o.y - acc[a][4 * h + 1], o.z - acc[a][4 * h + 2], o.w - acc[a][4 * h + 3]};
            if (col + 3 < n) {
                if (panel) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) v[i] = gj_entry(row, col + i, p0, nb, v[i], T, Un, ldu, Dinv);
                }
                *reinterpret_cast<float4*>(dst) = make_float4(v[0], v[1], v[2], v[3]);
            } else {
                for (int i = 0; i < 4; ++i)
                    if (col + i < n) dst[i] = gj_entry(row, col + i, p0, nb, dst[i] - acc[a][4 * h + i], T, Un, ldu, Dinv);
            }
        }
    }
}

// Panel of a wide pivot block [p0, p0 + nb) of the upper triangle A: U (bw x n, rows of ldu) and Ut (n x bw), zero in the pivot rows and
// beyond nb, and the pivot block itself in D (bw x bw, identity beyond nb).  Tiles of 32 x 32.
__global__ void __launch_bounds__(256) k_sw_gather(const float* __restrict__ A, int64_t lda, int64_t n, int64_t p0, int nb, int bw, float* __restrict__ U, int64_t ldu,
                                                   float* __restrict__ Ut, float* __restrict__ D)
{
    __shared__ float tile[32][33];                   // [column of the panel][k] or the other way round
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int64_t j0 = (int64_t)blockIdx.x * 32;
    const int k0 = blockIdx.y * 32;
    for (int i = ty; i < 32; i += 8) {
        {   // columns left of the block lie transposed above it: read along k
            const int64_t j = j0 + i;
            const int k = k0 + tx;
            if (j < n && j < p0) tile[i][tx] = k < nb ? A[j * lda + p0 + k] : 0.f;
        }
    }
    __syncthreads();
    for (int i = ty; i < 32; i += 8) {               // the others: read along the columns; a thread writes what it alone reads
        const int64_t j = j0 + tx;
        const int k = k0 + i;
        if (j >= p0) tile[tx][i] = j >= p0 + nb && j < n && k < nb ? A[(p0 + k) * lda + j] : 0.f;
        if (j >= p0 && j < p0 + bw && k < bw) {
            const int a = k, b = (int)(j - p0);
            float v = a == b ? 1.f : 0.f;
            if (a < nb && b < nb) v = a <= b ? A[(p0 + a) * lda + p0 + b] : A[(p0 + b) * lda + p0 + a];
            D[(int64_t)a * bw + b] = v;
        }
    }
    __syncthreads();
    for (int i = ty; i < 32; i += 8) {
        if (j0 + i < n) Ut[(j0 + i) * bw + k0 + tx] = tile[i][tx];
        if (j0 + tx < ldu) U[(int64_t)(k0 + i) * ldu + j0 + tx] = j0 + tx < n ? tile[tx][i] : 0.f;
    }
}
// D = (D + D^T) / 2 where the two triangles differ by rounding (nb x nb, rows of bw).
__global__ void __launch_bounds__(256) k_sw_sym(float* D, int nb, int bw)
{
    const int i = blockIdx.x;
    for (int j = i + 1 + threadIdx.x; j < nb; j += 256) {
        const float v = 0.5f * (D[(int64_t)i * bw + j] + D[(int64_t)j * bw + i]);
        D[(int64_t)i * bw + j] = v; D[(int64_t)j * bw + i] = v;
    }
}
// The swept panel: A[i, P] = T[i] above the block, A[P, j] = T[j]^T right of it, A[P, P] = -Dinv (upper triangle).
__global__ void __launch_bounds__(256) k_sw_put(float* __restrict__ A, int64_t lda, int64_t n, int64_t p0, int nb, int bw, const float* __restrict__ T, const float* __restrict__ Dinv)
{
    __shared__ float tile[32][33];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int64_t j0 = (int64_t)blockIdx.x * 32;
    const int k0 = blockIdx.y * 32;
    for (int i = ty; i < 32; i += 8) {
        const int64_t j = j0 + i;
        const int k = k0 + tx;
        if (j >= n) continue;
        tile[i][tx] = T[j * bw + k];
        if (j < p0 && k < nb) A[j * lda + p0 + k] = tile[i][tx];
    }
    __syncthreads();
    for (int i = ty; i < 32; i += 8) {
        const int64_t j = j0 + tx;
        const int k = k0 + i;
        if (j >= n || k >= nb || j < p0) continue;
        if (j >= p0 + nb) A[(p0 + k) * lda + j] = tile[tx][i];
        else if (j - p0 >= k) A[(p0 + k) * lda + j] = -Dinv[(int64_t)k * bw + (j - p0)];
    }
}
// A = -A, the lower triangle as the mirror image of the upper one.
__global__ void __launch_bounds__(256) k_sw_finish(float* A, int64_t lda, int64_t n)
{
    if (blockIdx.x < blockIdx.y) return;
    __shared__ float tile[32][33];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int64_t c = (int64_t)blockIdx.x * 32 + tx, r0 = (int64_t)blockIdx.y * 32;
    for (int i = ty; i < 32; i += 8) {
        const int64_t r = r0 + i;
        if (r < n && c < n && c >= r) { const float v = -A[r * lda + c]; tile[i][tx] = v; A[r * lda + c] = v; }
    }
    __syncthreads();
    for (int i = ty; i < 32; i += 8) {               // row c' = block column + i, column r0 + tx
        const int64_t r = (int64_t)blockIdx.x * 32 + i, cc = r0 + tx;
        if (r < n && cc < r) A[r * lda + cc] = tile[tx][i];
    }
}

#define CK(x) do { cudaError_t e_ = (x); if (e_ != cudaSuccess) return OSSCAR_E_CUDA; } while (0)

constexpr int kWide = 512;

// Blocks of 512 pivots as symmetric sweeps of the upper triangle, A_ij -= A_iP A_PP^-1 A_Pj, A_iP := A_iP A_PP^-1, A_PP := -A_PP^-1:
// the matrix is read and written once per block, on the tensor cores (three bf16 terms, half of the tiles), and the chain of
// 64-wide pivot blocks runs inside the small A_PP.  The result is -A^-1.  0: not enough memory, 1: done.
int invert_wide(osscar_ctx* ctx, float* A, int64_t lda, int64_t n, const float* ref, int64_t ldref, int* done)
{
    const Layout& L = ctx->L;
    cudaStream_t st = ctx->stream;
    *done = 0;
    constexpr int bw = kWide;
    char* base = (char*)ctx->ws + L.off_tc;
    size_t off = 65536;                              // in front: what the inversion of the pivot block keeps here
    auto take = [&](size_t floats) { float* q = (float*)(base + off); off += (floats * sizeof(float) + 1023) / 1024 * 1024; return q; };
    float* D = take((size_t)bw * bw);
    float* U = take((size_t)bw * lda);
    float* Ut = take((size_t)bw * n);
    float* T = take((size_t)bw * n);
    if (off + gemm_tc_min_scratch(n, lda) * 4 > L.tc_bytes) return OSSCAR_OK;
    void* scratch = base + off;
    const size_t scratch_bytes = L.tc_bytes - off;
    for (int64_t p0 = 0; p0 < n; p0 += bw) {
        const int nb = (int)(n - p0 < bw ? n - p0 : bw);
        const int64_t cols = lda > p0 + bw ? lda : p0 + bw;          // all of D, also where the last block reaches past the matrix
        const dim3 grid((unsigned)((cols + 31) / 32), (unsigned)(bw / 32));
        k_sw_gather<<<grid, 256, 0, st>>>(A, lda, n, p0, nb, bw, U, lda, Ut, D);
        const int rc = invert_spd_inplace(ctx, D, bw, nb, ref + p0 * (ldref + 1), ldref, false);
        if (rc != OSSCAR_OK) return rc;
        k_sw_sym<<<(unsigned)nb, 256, 0, st>>>(D, nb, bw);
        CK(gemm_tc(st, n, bw, bw, 1.f, Ut, bw, D, bw, 0.f, T, bw, scratch, scratch_bytes, ctx->ctl));
        CK(gemm_tc(st, n, lda, bw, -1.f, T, bw, U, lda, 1.f, A, lda, scratch, scratch_bytes, ctx->ctl, nullptr, true));
        k_sw_put<<<dim3((unsigned)((n + 31) / 32), (unsigned)(bw / 32)), 256, 0, st>>>(A, lda, n, p0, nb, bw, T, D);
        count_launches(3);
        CK(cudaGetLastError());
    }
    const unsigned nt = (unsigned)((n + 31) / 32);
    k_sw_finish<<<dim3(nt, nt), 256, 0, st>>>(A, lda, n);
    count_launches(1);
    CK(cudaGetLastError());
    *done = 1;
    return OSSCAR_OK;
}

}  // namespace

// In-place inverse of the n x n SPD matrix A (row stride lda, a multiple of 4; A 16-byte aligned).
// `ref` (row stride ldref) supplies the original diagonal, the scale of the positive-definiteness test.
// With `tensor_updates` large matrices are swept on the tensor cores (three bf16 terms per operand): what their truncating accumulator
// loses, the correction of the inverse from a residual summed beyond fp32, which the caller then applies, removes.
int invert_spd_inplace(osscar_ctx* ctx, float* A, int64_t lda, int64_t n, const float* ref, int64_t ldref,
                       bool tensor_updates)
{
    const Layout& L = ctx->L;
    cudaStream_t st = ctx->stream;
    if (tensor_updates && n >= kSweptRows) {
        int done = 0;
        const int rc = invert_wide(ctx, A, lda, n, ref, ldref, &done);
        if (rc != OSSCAR_OK || done) return rc;
    }
    float* T = (float*)((char*)ctx->ws + L.off_panel);
    float* U = T + L.d1 * NB;
    float* Un = U + NB * L.ldp;
    float* Dinv = Un + NB * L.ldp;
    const int nb0 = (int)(n < NB ? n : NB);
    const unsigned pgrid = (unsigned)((n + 31) / 32);
    k_gj_pivot<<<1, GJ_T, 0, st>>>(A, lda, 0, nb0, Dinv, ref, ldref, ctx->ctl);
    count_launches(1);
    // the tensor-core region is idle here: the copy of the next pivot block and the second inverse live in it
    float* next = (float*)((char*)ctx->ws + L.off_tc);
    float* Dbuf[2] = { Dinv, next + NB * NB };
    CK(cudaFuncSetAttribute(k_gj_update, cudaFuncAttributeMaxDynamicSharedMemorySize, UP_SMEM));
    const int tiles_n = (int)((n + UP_N - 1) / UP_N);
    const unsigned ugrid = (unsigned)(1 + (int64_t)tiles_n * ((n + UP_M - 1) / UP_M));
    for (int64_t p0 = 0, s = 0; p0 < n; p0 += NB, ++s) {
        const int nb = (int)(n - p0 < NB ? n - p0 : NB);
        const float* D = Dbuf[s & 1];
        CK(launch_pdl(true, k_gj_panels, dim3(pgrid), dim3(GJ_T), st, (const float*)A, lda, n, p0, nb, D, T, U, Un, lda, next));
        CK(launch_pdl_smem(true, k_gj_update, dim3(ugrid), dim3(GJ_T), UP_SMEM, st, A, lda, n, p0, nb, (const float*)T, (const float*)U, (const float*)Un, lda,
                            D, (const float*)next, Dbuf[(s & 1) ^ 1], ref, ldref, tiles_n, ctx->ctl));
        count_launches(2);
    }
    CK(cudaGetLastError());
    return OSSCAR_OK;
}

}  // namespace osscar
