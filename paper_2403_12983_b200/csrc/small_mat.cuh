// Block-cooperative small dense algebra in fp64 (g x g matrices in shared or global memory) and warp sums,
// shared by the search and the greedy phase.
#pragma once
#include <float.h>

namespace osscar {
namespace smallmat {

static __device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
static __device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
// Inverse of the g x g SPD matrix M (ld g, shared memory where possible) by Gauss-Jordan elimination without pivoting, the
// matrix in registers: of NW warps, warp w owns the rows w, w + NW, ... (A of them), a lane the columns lane, lane + 32, ...
// (B of them; B = 1 or NW = 32).  A step is one shuffle per owned row (its entry of the pivot column), the scaled pivot row
// through double-buffered shared memory and ONE barrier.  Out receives the symmetrised inverse, M is overwritten.  Returns
// the smallest pivot, i.e. the smallest diagonal entry of the successive Schur complements = the squared diagonal of the
// Cholesky factor (<= 0 when M is not positive definite).
template <int NW, int A, int B>
static __device__ double spd_inverse_reg(double* M, double* Out, int g)
{
    static_assert(B == 1 || (NW == 32 && A == B), "row and column of the pivot in the same register");
    __shared__ double rows[2][32 * B];
    __shared__ double s_pinv[2], s_piv[NW], s_min;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    double x[A][B];
    __syncthreads();
#pragma unroll
    for (int a = 0; a < A; ++a)
#pragma unroll
        for (int b = 0; b < B; ++b) {
            const int i = w + NW * a, c = lane + 32 * b;
            x[a][b] = i < g && c < g ? M[i * g + c] : 0.0;
        }
    double minpiv = DBL_MAX;                       // kept by the owner of each pivot row
#pragma unroll
    for (int kk = 0; kk < A; ++kk) {
        constexpr int kB = B;
        const int bk = kB == 1 ? 0 : kk;
        for (int jj = 0; jj < NW; ++jj) {
            const int j = kk * NW + jj;
            if (j >= g) break;
            double* rowj = rows[j & 1];
            double col[A];
#pragma unroll
            for (int a = 0; a < A; ++a) col[a] = __shfl_sync(0xffffffffu, x[a][bk], j & 31);      // entry (row, j)
            if (w == jj) {                         // row j is this warp's row kk
                double d = col[kk];
                const bool bad = !(d > 0.0);
                if (bad) { minpiv = -1.0; d = 1.0; }
                else if (d < minpiv) minpiv = d;
                const double pinv = 1.0 / d;
#pragma unroll
                for (int b = 0; b < B; ++b) rowj[lane + 32 * b] = x[kk][b] * pinv;
                if (lane == 0) s_pinv[j & 1] = pinv;
            }
            __syncthreads();
            const double pinv = s_pinv[j & 1];
#pragma unroll
            for (int b = 0; b < B; ++b) {
                const int c = lane + 32 * b;
                const double r = rowj[c];
#pragma unroll
                for (int a = 0; a < A; ++a) {
                    double v;
                    if (a == kk && w == jj) v = c == j ? pinv : r;
                    else if (c == j) v = -col[a] * pinv;
                    else v = x[a][b] - col[a] * r;
                    x[a][b] = v;
                }
            }
        }
    }
#pragma unroll
    for (int a = 0; a < A; ++a)
#pragma unroll
        for (int b = 0; b < B; ++b) {
            const int i = w + NW * a, c = lane + 32 * b;
            if (i < g && c < g) M[i * g + c] = x[a][b];
        }
    if (lane == 0) s_piv[w] = minpiv;
    __syncthreads();
#pragma unroll
    for (int a = 0; a < A; ++a)                    // the two triangles differ by rounding only
#pragma unroll
        for (int b = 0; b < B; ++b) {
            const int i = w + NW * a, c = lane + 32 * b;
            if (i < g && c < g) Out[i * g + c] = 0.5 * (x[a][b] + M[c * g + i]);
        }
    if (threadIdx.x == 0) {
        double mp = s_piv[0];
        for (int i = 1; i < NW; ++i) mp = s_piv[i] < mp ? s_piv[i] : mp;
        s_min = mp;
    }
    __syncthreads();
    return s_min;
}

// Block-cooperative inverse of the g x g SPD matrix M (ld g) by in-place Gauss-Jordan elimination without pivoting:
// g steps of one rank-1 update over all g^2 entries, so every thread of the block works in every step.
// M is overwritten (keep it in shared memory where possible); Out receives the symmetrised inverse; Lw: scratch of
// at least 2 g doubles.  Returns the smallest pivot, i.e. the smallest diagonal entry of the successive Schur
// complements = the squared diagonal of the Cholesky factor (<= 0 when M is not positive definite).
// The register form takes over where its thread layouts fit (blocks of 32 warps up to g = 96, of 8 warps up to g = 32):
// with the two-barrier form below the scores of 32 groups of 80 rows took 0.21 ms, now 0.094 ms; larger matrices (the nested phase's joint downdates) stay here.
static __device__ double spd_inverse(double* M, double* Lw, double* Out, int g)
{
    if (blockDim.x == 1024 && g > 32 && g <= 64) return spd_inverse_reg<32, 2, 2>(M, Out, g);
    if (blockDim.x == 1024 && g > 64 && g <= 96) return spd_inverse_reg<32, 3, 3>(M, Out, g);
    if (blockDim.x == 1024 && g <= 32) return spd_inverse_reg<32, 1, 1>(M, Out, g);
    if (blockDim.x == 256 && g <= 32) return spd_inverse_reg<8, 4, 1>(M, Out, g);
    __shared__ double minpiv;
    const int t = threadIdx.x, nt = blockDim.x;
    double* colj = Lw; double* rowj = Lw + g;
    __syncthreads();
    if (t == 0) minpiv = DBL_MAX;
    __syncthreads();
    for (int j = 0; j < g; ++j) {
        double d = M[j * g + j];
        const bool bad = !(d > 0.0);
        if (t == 0) { if (bad) minpiv = -1.0; else if (d < minpiv) minpiv = d; }
        if (bad) d = 1.0;
        const double pinv = 1.0 / d;
        for (int i = t; i < g; i += nt) { colj[i] = M[i * g + j]; rowj[i] = M[j * g + i] * pinv; }
        __syncthreads();
        for (int idx = t; idx < g * g; idx += nt) {
            const int i = idx / g, c = idx % g;
            double v;
            if (i == j) v = (c == j) ? pinv : rowj[c];
            else if (c == j) v = -colj[i] * pinv;
            else v = M[idx] - colj[i] * rowj[c];
            M[idx] = v;
        }
        __syncthreads();
    }
    for (int idx = t; idx < g * g; idx += nt) {          // the two triangles differ by rounding only
        const int i = idx / g, c = idx % g;
        Out[idx] = 0.5 * (M[idx] + M[c * g + i]);
    }
    __syncthreads();
    return minpiv;
}
// C = op(A) * op(B), all g x g (ld g), block-cooperative, on the fp64 tensor-core path: every warp of the block takes
// 8 x 8 tiles of C in turn and runs g / 4 steps of mma.m8n8k4 (A fragment: row lane / 4, column lane % 4; B fragment:
// row lane % 4, column lane / 4; C fragment: row lane / 4, columns 2 (lane % 4) and + 1).  Entries beyond g read as 0.
// C must not overlap A or B.  blockDim.x must be a multiple of 32.
static __device__ __forceinline__ void mat_tile(const double* A, bool tA, const double* B, bool tB, double* C, int g, int tile)
{
    const int lane = threadIdx.x & 31, nt = (g + 7) >> 3;
    const int r4 = lane >> 2, c4 = lane & 3;
    const int i0 = (tile / nt) * 8, j0 = (tile % nt) * 8;
    const int ai = i0 + r4, bj = j0 + r4;
    double d0 = 0.0, d1 = 0.0;
#pragma unroll 4
    for (int k0 = 0; k0 < g; k0 += 4) {
        const int kk = k0 + c4;
        const bool ka = kk < g;
        const double a = (ka && ai < g) ? (tA ? A[kk * g + ai] : A[ai * g + kk]) : 0.0;
        const double b = (ka && bj < g) ? (tB ? B[bj * g + kk] : B[kk * g + bj]) : 0.0;
        asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};"
                     : "+d"(d0), "+d"(d1) : "d"(a), "d"(b));
    }
    const int ci = i0 + r4, cj = j0 + 2 * c4;
    if (ci < g) {
        if (cj < g) C[ci * g + cj] = d0;
        if (cj + 1 < g) C[ci * g + cj + 1] = d1;
    }
}
static __device__ void mat_mul(const double* A, bool tA, const double* B, bool tB, double* C, int g)
{
    const int warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5, nt = (g + 7) >> 3;
    for (int tile = warp; tile < nt * nt; tile += nwarps) mat_tile(A, tA, B, tB, C, g, tile);
    __syncthreads();
}
// Several products at once, their tiles dealt to the warps together (a product of 80 x 80 has 100 tiles for 32 warps).
struct MatJob { const double *A, *B; bool tB; double* C; };
template <int N> static __device__ void mat_mul_jobs(const MatJob (&jobs)[N], int g)
{
    const int warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5, nt = (g + 7) >> 3, n = nt * nt;
    for (int tile = warp; tile < N * n; tile += nwarps) {
        MatJob j = jobs[0];
#pragma unroll
        for (int i = 1; i < N; ++i) if (tile >= i * n) j = jobs[i];
        mat_tile(j.A, false, j.B, j.tB, j.C, g, tile % n);
    }
    __syncthreads();
}
static __device__ double mat_trace_prod(const double* A, const double* B, int g, double* red)   // sum A .* B^T = Tr(A B)
{
    double s = 0.0;
    for (int idx = threadIdx.x; idx < g * g; idx += blockDim.x) s += A[idx] * B[(idx % g) * g + idx / g];
    s = warp_sum(s);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    double tot = 0.0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) tot += red[i];
    __syncthreads();
    return tot;
}


}  // namespace smallmat
}  // namespace osscar
