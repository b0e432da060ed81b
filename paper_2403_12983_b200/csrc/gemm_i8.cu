// C = beta * C0 + alpha * A * B to (nearly) fp64 accuracy on the int8 tensor cores: error-free splitting of the operands
// into 8-bit digits, exact integer products and sums (the scheme of Ootomo, Ozaki and Yokota, "DGEMM on integer matrix
// multiplication unit", 2024, with balanced radix-256 digits).
//
// What it replaces and why.  The residuals of the refinement steps, R = G_J - H_JI V and the Schur products have to be
// summed far beyond fp32 (see dgemm.cu).  On the fp64 pipe they run at 29-30 TFLOP/s, which was 218 of the 306 ms of the
// state build of a d1 = 28672 layer.  kind::i8 multiplies at twice the bf16 rate and adds without any rounding: 2.6 POPS here,
// so 21 or 15 digit products replace an fp64 product 6 to 9 times faster.  At d1 = 28672, m = 7168, k = 8602 the two residuals
// take 18.4 ms, R 14.3 ms and the Schur products with their dot products 10.7 ms (230 ms for all on the fp64 pipe, and
// 1.4 GB of fp64 panels written and read again); at d1 = 8192, m = 2048, k = 4096 2.9 ms against 12.7 ms.
//
// Splitting.  Row i of A and column j of B are scaled by powers of two so that their largest entry is below one; the
// contraction index k is first balanced by 2^(-+ck), ck = half the exponent of H_kk, so that channels of very different
// scale do not cost digits.  An entry becomes a fixed-point number of 8 S - 1 bits, cut into S signed digits
// d_1 .. d_S (weight 2^(1 - 8 i)).  Digit products of order o = i + j <= S + 1 are kept, S (S + 1) / 2 of them; all
// products of one order have one weight and accumulate in ONE int32 TMEM chain over the whole of K, exactly:
// S * K * 2^14 < 2^31 (max_k).  What is dropped is below 2^(-8 S + 5) sqrt(K) of (row maximum x column maximum):
// S = 6 for the residuals of the inverse and of V and for the Schur panels of wide groups, 5 for R and the Schur products of single
// rows, 4 for products that have to be as good as fp32 ones (V, G = H W, X0 T, pair scores, the objective), 3 for corrections
// and, with the products of order 5 as well, for the Gram of fp32 activations.
//
// Per output tile (128 x 256) the orders run from the smallest products to the largest; orders above 3 are added up in
// fp32 registers as they finish (their weight is 2^-16 of the leading one and less), the last two stay in the two TMEM
// buffers until the epilogue forms the sum in fp64.  Tiles of 128 columns where those of 256 leave SMs idle.
//
// Two orders o and o - 1 share one pass over the operands, one TMEM buffer each: in step i of a k-block, A_i B_(o-i) of the one order
// is followed by A_i B_(o-1-i) of the other, whose digit of B is the one the next step has loaded.  A step moves 48 KB from
// L2 for 1024 cycles of MMA; a pass per order moved them for 512.  MMAs issued back to back reach 4.3 Pop/s here; what the kernel
// lost against that were the L2 requests of its loads and an epilogue that held both TMEM buffers for 50000 to 75000 cycles per tile,
// spent on instruction fetches (it was unrolled over the chunks of a row), on conversions to 64 bits, on C0 and on spills.  Now
// 28000 to 40000.  The objective at d1 = 8192, m = 2048: 1.69 -> 1.53 ms; a layer of d1 = 28672, m = 7168, k = 8602 with its products
// 197 -> 164 ms under the power cap; G = H W at 5000 x 1283 (240 tiles) 0.30 -> 0.25 ms.
//   warp 0: TMA producer     warp 1: MMA issuer     warps 4-11: TMEM -> registers -> C
#include "osscar_internal.cuh"
#include "tc_common.cuh"
#include <math.h>

namespace osscar {
namespace {

using namespace tc;

constexpr int I8_TM = 128, I8_BK = 128, I8_UK = 32;           // rows per tile; bytes (= digits) per k-block and per MMA
constexpr int I8_A_BYTES = I8_TM * I8_BK;
constexpr int I8_RING = 196608;                               // bytes of the operand ring
constexpr int I8_STG = 32 * 16 * 8;                           // staging block of one accumulate warp: 32 rows x 16 doubles
constexpr int I8_SMEM = I8_RING + 1024 + 256 + 8 * I8_STG;
constexpr int I8_THREADS = 384;                               // warps 2 and 3 idle: registers are dealt by groups of four warps
constexpr int64_t max_k(int S) { return 131071 / S; }         // S products of 2^14 per k in one int32 sum
constexpr int I8_BAND = 8;
constexpr int64_t digit_stride(int64_t K) { return K >= 1024 ? (K + 127) / 128 * 128 : (K + 15) / 16 * 16; }      // bytes from row to row of a digit plane

enum { EPI_F32 = 0, EPI_F64 = 1, EPI_DOT = 2 };

__device__ __forceinline__ double pow2d(int e) {              // 2^e, |e| <= 1000
    e = e < -1000 ? -1000 : (e > 1000 ? 1000 : e);
    return __hiloint2double((e + 1023) << 20, 0);
}
// Exponent e with m < 0.99 * 2^e (0 for m = 0): the top digit of a value scaled by it, carry included, stays below 128.
__device__ __forceinline__ int scale_exponent(double m) {
    if (m == 0.0) return 0;
    int e;
    const double f = frexp(m, &e);
    return f > 0.99 ? e + 1 : e;
}
// (double)t of a whole number below 2^51 by one addition: conversions to 64 bits run at a quarter of the rate of fp64 additions.
__device__ __forceinline__ double whole_double(long long t) { return __longlong_as_double(t + 0x4338000000000000ll) - 6755399441055744.0; }
__device__ __forceinline__ void sts64(uint32_t a, double v) { asm volatile("st.shared.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory"); }
__device__ __forceinline__ double lds64(uint32_t a) { double v; asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory"); return v; }
__device__ __forceinline__ unsigned long long abs_bits(double x) {      // orders like |x|; NaN above everything
    return (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
}
__device__ __forceinline__ bool finite_bits(unsigned long long b) { return b < 0x7ff0000000000000ull; }

// Balanced radix-256 digits of q: byte i of q + 0x80..80, with its top bit flipped, is the digit of weight 256^i.
template <int S> __device__ __forceinline__ uint64_t digit_bytes(long long q) {
    constexpr uint64_t kBias = 0x8080808080808080ull >> (64 - 8 * S);
    return ((uint64_t)q + kBias) ^ kBias;
}

// ck[k] = half the binary exponent of the k-th diagonal entry of H_II; negated where A scales with the inverse of H.
__global__ void k_i8_balance(const float* __restrict__ diag, int64_t stride, int64_t K, int flip, int32_t* __restrict__ ck)
{
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= K) return;
    const float d = diag[k * stride];
    int e = 0;
    if (d > 0.f && isfinite(d)) frexpf(d, &e);
    ck[k] = flip ? -(e >> 1) : e >> 1;
}
// The same for an index that runs over pivots: half the binary exponent of |1 / S_kk|.
__global__ void k_i8_balance_pivots(const double* __restrict__ alpha, int64_t K, int32_t* __restrict__ ck)
{
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= K) return;
    const double a = alpha[k];
    int e = 0;
    if (a != 0.0 && isfinite(a)) frexp(a, &e);
    ck[k] = e >> 1;
}

// Digits of the rows of A (rows x K, row stride lda): plane s holds digit s + 1, rows ldk bytes apart.  One block per
// row: a pass for the largest entry, a second one (from L1 / L2) for the digits, 16 per thread and plane store.
template <int S>
__global__ void __launch_bounds__(256) k_i8_slice_rows(const float* __restrict__ A, int64_t lda, int64_t K, const int32_t* __restrict__ ck,
                                int8_t* __restrict__ planes, int64_t plane, int64_t ldk, double* __restrict__ scale,
                                int vec, const int32_t* __restrict__ done)
{
    if (done && *done) return;
    __shared__ unsigned long long red[8];
    const int64_t row = blockIdx.x;
    const float* a = A + row * lda;
    unsigned long long mx = 0;
    for (int64_t k = threadIdx.x; k < K; k += 256) {
        const unsigned long long b = abs_bits((double)a[k] * pow2d(-ck[k]));
        mx = b > mx ? b : mx;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) { const unsigned long long b = __shfl_xor_sync(0xffffffffu, mx, o); mx = b > mx ? b : mx; }
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < 8; ++w) mx = red[w] > mx ? red[w] : mx;
    const bool fin = finite_bits(mx);
    const int e = fin ? scale_exponent(__longlong_as_double((long long)mx)) : 0;
    if (threadIdx.x == 0) scale[row] = fin ? pow2d(e) : __longlong_as_double(0x7ff8000000000000ll);
    for (int64_t k0 = (int64_t)threadIdx.x * 16; k0 < ldk; k0 += 256 * 16) {
        uint32_t w[S][4];
#pragma unroll
        for (int q4 = 0; q4 < 4; ++q4) {
            float x[4];
            int c[4];
            if (vec && k0 + q4 * 4 + 4 <= K) {
                const float4 v = *reinterpret_cast<const float4*>(a + k0 + q4 * 4);
                const int4 cv = *reinterpret_cast<const int4*>(ck + k0 + q4 * 4);
                x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
                c[0] = cv.x; c[1] = cv.y; c[2] = cv.z; c[3] = cv.w;
            } else {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int64_t k = k0 + q4 * 4 + i;
                    x[i] = k < K ? a[k] : 0.f;
                    c[i] = k < K ? ck[k] : 0;
                }
            }
            uint64_t d[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) d[i] = fin ? digit_bytes<S>(__double2ll_rn((double)x[i] * pow2d(8 * S - 1 - e - c[i]))) : 0ull;
#pragma unroll
            for (int s = 0; s < S; ++s) {
                uint32_t p = 0;
#pragma unroll
                for (int i = 0; i < 4; ++i) p |= (uint32_t)((d[i] >> (8 * (S - 1 - s))) & 0xff) << (8 * i);
                w[s][q4] = p;
            }
        }
#pragma unroll
        for (int s = 0; s < S; ++s)
            *reinterpret_cast<uint4*>(planes + s * plane + row * ldk + k0) = make_uint4(w[s][0], w[s][1], w[s][2], w[s][3]);
    }
}

// Largest entry of every column of B (K x N) after balancing, as ordered bits; grid (column tiles of 64, chunks of 256 rows).
// `sub` (same layout, fp32 only): the matrix is B - sub.
template <typename T>
__global__ void __launch_bounds__(256) k_i8_colmax(const T* __restrict__ B, const T* __restrict__ sub, int64_t ldb, int64_t K, int64_t N, const int32_t* __restrict__ ck,
                            unsigned long long* __restrict__ cmax, const int32_t* __restrict__ done)
{
    if (done && *done) return;
    __shared__ unsigned long long red[4][64];
    const int64_t n = (int64_t)blockIdx.x * 64 + (threadIdx.x & 63);
    const int64_t k1 = min(K, ((int64_t)blockIdx.y + 1) * 256);
    unsigned long long mx = 0;
    if (n < N)
        for (int64_t k = (int64_t)blockIdx.y * 256 + (threadIdx.x >> 6); k < k1; k += 4) {
            const T x = sub ? B[k * ldb + n] - sub[k * ldb + n] : B[k * ldb + n];
            const unsigned long long b = abs_bits((double)x * pow2d(ck[k]));
            mx = b > mx ? b : mx;
        }
    red[threadIdx.x >> 6][threadIdx.x & 63] = mx;
    __syncthreads();
    if (threadIdx.x < 64 && n < N) {
#pragma unroll
        for (int i = 1; i < 4; ++i) mx = red[i][threadIdx.x] > mx ? red[i][threadIdx.x] : mx;
        atomicMax(&cmax[n], mx);
    }
}

// Digits of the columns of B, stored transposed (column n of B = row n of the planes): tiles of 128 k x 32 columns turned
// in shared memory.  tri_block > 0: entries of the diagonal blocks of that width are halved (column n is column col0 + n
// of the whole matrix).  spread (or null): sums over a column of the squares of its entries, each rounded to 15 bits below the
// column's scale; as whole numbers they do not depend on the order of the additions.
template <int S, typename T, bool SPREAD = false>
__global__ void __launch_bounds__(256) k_i8_slice_cols(const T* __restrict__ B, const T* __restrict__ sub, int64_t ldb, int64_t K, int64_t N, const int32_t* __restrict__ ck,
                                const unsigned long long* __restrict__ cmax, int8_t* __restrict__ planes, int64_t plane, int64_t ldk,
                                double* __restrict__ scale, int tri_block, int64_t col0, const int32_t* __restrict__ done,
                                unsigned long long* __restrict__ spread = nullptr)
{
    if (done && *done) return;
    __shared__ T tile[128][33];
    const int64_t n0 = (int64_t)blockIdx.x * 32, k0 = (int64_t)blockIdx.y * 128;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const int64_t k = k0 + ty + 8 * i, n = n0 + tx;
        tile[ty + 8 * i][tx] = (k < K && n < N) ? (sub ? B[k * ldb + n] - sub[k * ldb + n] : B[k * ldb + n]) : (T)0;
    }
    __syncthreads();
    const int nl = threadIdx.x >> 3, kg = (threadIdx.x & 7) * 16;
    const int64_t n = n0 + nl;
    if (!SPREAD && n >= N) return;
    const unsigned long long mb = n < N ? cmax[n] : 0ull;
    const bool fin = finite_bits(mb);
    const int e = fin ? scale_exponent(__longlong_as_double((long long)mb)) : 0;
    if (blockIdx.y == 0 && kg == 0 && n < N) scale[n] = fin ? pow2d(e) : __longlong_as_double(0x7ff8000000000000ll);
    if (!SPREAD && k0 + kg >= ldk) return;
    uint32_t w[S][4];
    unsigned long long sq = 0;                     // entries beyond the matrix are zero in the tile
#pragma unroll
    for (int q4 = 0; q4 < 4; ++q4) {
        uint64_t d[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int64_t k = k0 + kg + q4 * 4 + i;
            const int half = tri_block > 0 && k / tri_block == (col0 + n) / tri_block ? 1 : 0;
            const int c = k < K ? ck[k] : 0;
            const long long q = fin ? __double2ll_rn((double)tile[kg + q4 * 4 + i][nl] * pow2d(8 * S - 1 - e + c - half)) : 0ll;
            if (SPREAD) { const long long t = q >> (8 * S - 16); sq += (unsigned long long)(t * t); }
            d[i] = digit_bytes<S>(q);
        }
#pragma unroll
        for (int s = 0; s < S; ++s) {
            uint32_t p = 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) p |= (uint32_t)((d[i] >> (8 * (S - 1 - s))) & 0xff) << (8 * i);
            w[s][q4] = p;
        }
    }
    if (SPREAD) {                                  // eight neighbouring threads share a column
        for (int o = 4; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
        if (n < N && kg == 0) atomicAdd(&spread[n], sq);
        if (n >= N || k0 + kg >= ldk) return;
    }
#pragma unroll
    for (int s = 0; s < S; ++s)
        *reinterpret_cast<uint4*>(planes + s * plane + n * ldk + k0 + kg) = make_uint4(w[s][0], w[s][1], w[s][2], w[s][3]);
}

// K-major operand tile, SWIZZLE_128B: rows of 128 bytes, 8-row atoms 1024 bytes apart.
__device__ __forceinline__ uint64_t i8_desc(uint32_t saddr) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}
__device__ __forceinline__ void umma_i8(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accum) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n\t}"
                 ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accum) : "memory");
}

struct I8Maps { CUtensorMap a, b; };
struct I8Epi {
    const double *sa, *sb;        // scales of the rows of A and of the columns of B
    double alpha, beta;
    const float *C0, *C0sub; int64_t ldc0;      // EPI_DOT: rows of C0 - C0sub (or of C0)
    void* C; int64_t ldc;         // EPI_F32: float, EPI_F64: double, EPI_DOT: partial sums [row][2 * TN]
    int identity, vec;
    int64_t row0, col0;           // position of this panel in the whole product (identity)
};

// Which tiles and k-ranges a launch covers.  tri = 1 + k-blocks left of this column panel: a tile reads only the k-range down
// to its own diagonal block (0: the whole range).  upper: only tiles that reach the diagonal or lie above it.  ksplit > 1
// (EPI_F32 only): the k-range of a tile is dealt to that many CTAs, slice s writes to C + s * slice_stride.
struct I8Cover { int tri, upper, ksplit; int64_t slice_stride; };

// TNC columns per tile; digit products up to order OM.
template <int S, int TNC, int EPI, int OM = S + 1>
__global__ void __launch_bounds__(I8_THREADS, 1)
k_mma_i8(const __grid_constant__ I8Maps maps, int M, int N, int K, const __grid_constant__ I8Epi ep, const I8Cover cov, int num_ids,
         SearchCtl* __restrict__ ctl, const int32_t* __restrict__ done)
{
    constexpr int B_BYTES = TNC * I8_BK, STAGE = I8_A_BYTES + B_BYTES, STAGES = I8_RING / STAGE;
    constexpr int HALF = TNC / 2, TMEM_COLS = 2 * TNC;
    constexpr uint32_t kIdesc = (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(TNC >> 3) << 17) | ((uint32_t)(I8_TM >> 4) << 24);
    if (done && *done) return;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t tiles_base = (raw + 1023u) & ~1023u;
    uint8_t* bar_ptr = smem_raw + (tiles_base - raw) + I8_RING;
    const uint32_t bars = tiles_base + I8_RING;
    auto full_bar = [&](int s) { return bars + 8u * s; };
    auto empty_bar = [&](int s) { return bars + 8u * (STAGES + s); };
    auto tfull_bar = [&](int b) { return bars + 8u * (2 * STAGES + b); };
    auto tempty_bar = [&](int b) { return bars + 8u * (2 * STAGES + 2 + b); };
    const uint32_t drain_bar = bars + 8u * (2 * STAGES + 4);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bar_ptr + 8 * (2 * STAGES + 5));
    volatile int* abort_flag = reinterpret_cast<volatile int*>(bar_ptr + 8 * (2 * STAGES + 5) + 8);
    const long long wl = ctl->wait_limit;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int TM = (M + I8_TM - 1) / I8_TM, TN = (N + TNC - 1) / TNC;
    const int nkb_all = (K + I8_BK - 1) / I8_BK;
    auto tile_of = [&](int id, int* tm, int* tn, int* kb0, int* kb1) {
        int slice = 0;
        if (cov.ksplit > 1) { slice = id % cov.ksplit; id /= cov.ksplit; }
        *kb0 = 0; *kb1 = nkb_all;
        if (cov.tri) {                   // longest columns first, so that the persistent CTAs end together
            *tn = TN - 1 - id / TM; *tm = id % TM;
            *kb1 = min(nkb_all, cov.tri - 1 + (*tn + 1) * (TNC / I8_BK));
        } else if (cov.upper) {          // row by row of tiles
            constexpr int kPer = TNC / I8_TM;
            int r = 0;
            while (id >= TN - r / kPer) { id -= TN - r / kPer; ++r; }
            *tm = r; *tn = r / kPer + id;
        } else {
            const int per_band = I8_BAND * TN, b = id / per_band, r = id % per_band, rows = min(I8_BAND, TM - b * I8_BAND);
            *tn = r / rows; *tm = b * I8_BAND + r % rows;
        }
        if (cov.ksplit > 1) { *kb1 = (int)((int64_t)nkb_all * (slice + 1) / cov.ksplit); *kb0 = (int)((int64_t)nkb_all * slice / cov.ksplit); }
        return slice;
    };

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(tfull_bar(b), 1); mbar_init(tempty_bar(b), 8); }
        mbar_init(drain_bar, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "n"(TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = *tmem_slot;

    // 384 x 168 registers at launch = 128 x 72 + 256 x 216: the accumulate warps hold 128 sums each, which spilled within 168
    if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
    if (warp == 0) {
        if (lane == 0) {
            uint32_t it = 0;
            bool ok = true;
            for (int id = blockIdx.x; id < num_ids && ok; id += gridDim.x) {
                int tm, tn, kb0, kb1;
                tile_of(id, &tm, &tn, &kb0, &kb1);
                for (int o = OM; o >= 2 && ok; o -= 2) {
                    const int sum = min(o, S + 1), n = sum - 1;          // step i: digit i of A, digit sum - i of B
                    for (int kb = kb0; kb < kb1 && ok; ++kb)
                        for (int i = 1; i <= n; ++i, ++it) {
                            const int s = it % STAGES;
                            if (!mbar_wait(empty_bar(s), ((it / STAGES) & 1) ^ 1, abort_flag, wl)) { ok = false; break; }
                            mbar_expect_tx(full_bar(s), STAGE);
                            const uint32_t a_dst = tiles_base + s * STAGE;
                            // the planes of an operand are stacked: rows past its end are another plane's and only feed
                            // rows or columns of the tile that are never written
                            tma_load_2d(a_dst, &maps.a, full_bar(s), kb * I8_BK, (i - 1) * M + tm * I8_TM);
                            tma_load_2d(a_dst + I8_A_BYTES, &maps.b, full_bar(s), kb * I8_BK, (sum - i - 1) * N + tn * TNC);
                        }
                }
            }
            if (*abort_flag) {                    // the copies still in flight must land before the CTA exits
                const uint32_t first = it > STAGES ? it - STAGES : 0;
                for (uint32_t j = first; j < it; ++j) mbar_drain(full_bar(j % STAGES), (j / STAGES) & 1);
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            uint32_t it = 0, fl = 0;
            bool ok = true;
            for (int id = blockIdx.x; id < num_ids && ok; id += gridDim.x) {
                int tm, tn, kb0, kb1;
                tile_of(id, &tm, &tn, &kb0, &kb1);
                for (int o = OM; o >= 2 && ok; o -= 2) {
                    const int sum = min(o, S + 1), n = sum - 1, pair = o > 2 ? 2 : 1;
                    for (int b = 0; b < pair && ok; ++b) ok = mbar_wait(tempty_bar((fl + b) & 1), (((fl + b) >> 1) & 1) ^ 1, abort_flag, wl);
                    if (!ok) break;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t d_hi = tmem_base + (uint32_t)((fl & 1) * TNC), d_lo = tmem_base + (uint32_t)(((fl + 1) & 1) * TNC);
                    const bool wide = o > S + 1;            // step i belongs to the lower order of the pair
                    for (int kb = kb0; kb < kb1 && ok; ++kb)
                        for (int i = 1; i <= n; ++i, ++it) {
                            const int s = it % STAGES, s1 = (it + 1) % STAGES;
                            // of the k-block's steps only the first is not waited for by the step before it
                            if (i == 1 && !mbar_wait(full_bar(s), (it / STAGES) & 1, abort_flag, wl)) { ok = false; break; }
                            if (i < n && !mbar_wait(full_bar(s1), ((it + 1) / STAGES) & 1, abort_flag, wl)) { ok = false; break; }
                            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                            const uint32_t a_src = tiles_base + s * STAGE, b_src = a_src + I8_A_BYTES;
                            const uint32_t a_next = tiles_base + s1 * STAGE, b_next = a_next + I8_A_BYTES;
                            const uint32_t go_on = kb > kb0 || i > 1 ? 1u : 0u;
#pragma unroll
                            for (int j = 0; j < I8_BK / I8_UK; ++j)
                                umma_i8(wide ? d_lo : d_hi, i8_desc(a_src + j * I8_UK), i8_desc(b_src + j * I8_UK), kIdesc, go_on | (j ? 1u : 0u));
                            if (i < n)
#pragma unroll
                                for (int j = 0; j < I8_BK / I8_UK; ++j)
                                    umma_i8(wide ? d_hi : d_lo, i8_desc((wide ? a_next : a_src) + j * I8_UK), i8_desc((wide ? b_src : b_next) + j * I8_UK),
                                            kIdesc, go_on | (j ? 1u : 0u));
                            umma_commit(empty_bar(s));
                        }
                    if (ok)
                        for (int b = 0; b < pair; ++b) umma_commit(tfull_bar((fl + b) & 1));
                    fl += pair;
                }
            }
            if (!ok) {            // MMAs already issued keep running: they must finish before TMEM and the tiles are released
                umma_commit(drain_bar);
                mbar_drain(drain_bar, 0);
            }
        }
    }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 216;");
        const int lg = warp & 3, half = (warp - 4) >> 2;
        const int rsub = lane >> 2, c4 = (lane & 3) * 4;
        // staging block: entry (row, j) at row * 16 + (j ^ (row & 15)).  This lane writes row `lane` and reads rows q * 8 + rsub, columns c4 ...
        const uint32_t stg = bars + 256 + (warp - 4) * I8_STG;
        const uint32_t st_w = stg + lane * 128 + (lane & 15) * 8;
        const uint32_t st_r[2] = { stg + rsub * 128 + ((rsub ^ c4) * 8), stg + (rsub + 8) * 128 + (((rsub + 8) ^ c4) * 8) };
        uint32_t fl = 0;
        bool ok = true;
        for (int id = blockIdx.x; id < num_ids && ok; id += gridDim.x) {
            int tm, tn, kb0, kb1;
            const int slice = tile_of(id, &tm, &tn, &kb0, &kb1);
            const int64_t grow0 = (int64_t)tm * I8_TM + lg * 32;
            const int64_t gcol0 = (int64_t)tn * TNC + half * HALF;
            const bool with_c0 = EPI == EPI_DOT || (EPI == EPI_F32 && !ep.identity && ep.beta != 0.0);
            if (with_c0 && grow0 + lane < M)          // the tile's part of C0 comes to L2 while its products run
                for (int64_t gc = gcol0; gc < gcol0 + HALF && gc < N; gc += 32) {
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(ep.C0 + (grow0 + lane) * ep.ldc0 + gc));
                    if (EPI == EPI_DOT && ep.C0sub) asm volatile("prefetch.global.L2 [%0];" ::"l"(ep.C0sub + (grow0 + lane) * ep.ldc0 + gc));
                }
            float lo[HALF];               // orders above 3, in units of order 4
#pragma unroll
            for (int j = 0; j < HALF; ++j) lo[j] = 0.f;
            for (int o = OM; o >= 4 && ok; --o, ++fl) {
                const int buf = fl & 1;
                if (!mbar_wait(tfull_bar(buf), (fl >> 1) & 1, abort_flag, wl)) { ok = false; break; }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                for (int c = 0; c < HALF / 32; ++c) {
                    uint32_t r[32];
                    tmem_ld32(tmem_base + ((uint32_t)(lg * 32) << 16) + (uint32_t)(buf * TNC + half * HALF + c * 32), r);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                    for (int j = 0; j < 32; ++j) lo[c * 32 + j] = fmaf(lo[c * 32 + j], 0.00390625f, (float)(int)r[j]);
                }
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(tempty_bar(buf));
            }
            if (!ok) break;
            // whole pieces of C0 are requested a chunk ahead: the two TMEM buffers are held until the last chunk has been read out
            float4 pre[4], pre_sub[4];
            auto request = [&](int c) {
                const int64_t gc = gcol0 + c * 16 + c4;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int64_t gr = grow0 + q * 8 + rsub;
                    if (with_c0 && ep.vec && gr < M && gcol0 + c * 16 + 16 <= N) {
                        pre[q] = *reinterpret_cast<const float4*>(ep.C0 + gr * ep.ldc0 + gc);
                        if (EPI == EPI_DOT && ep.C0sub) pre_sub[q] = *reinterpret_cast<const float4*>(ep.C0sub + gr * ep.ldc0 + gc);
                    }
                }
            };
            if (EPI != EPI_F64) request(0);
            const int b3 = fl & 1, b2 = b3 ^ 1;       // orders 3 and 2 wait in the two buffers
            if (!mbar_wait(tfull_bar(b3), (fl >> 1) & 1, abort_flag, wl)) break;
            if (!mbar_wait(tfull_bar(b2), ((fl + 1) >> 1) & 1, abort_flag, wl)) break;
            fl += 2;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            double sa[4], dot[4];
            bool row_in[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int64_t gr = grow0 + q * 8 + rsub;
                row_in[q] = gr < M;
                sa[q] = row_in[q] ? ep.alpha * ep.sa[gr] : 0.0;
                dot[q] = 0.0;
            }
            int sbx[HALF / 32];               // column scales, one column in 32 per lane: powers of two (or NaN), their low word is zero
#pragma unroll
            for (int i = 0; i < HALF / 32; ++i) {
                const int64_t gc = gcol0 + i * 32 + lane;
                sbx[i] = gc < N ? __double2hiint(ep.sb[gc] * (1.0 / 1073741824.0)) : 0;            // 2^-30: weight of order 4
            }
            float* const out = (float*)ep.C + (int64_t)slice * cov.slice_stride + (grow0 + rsub) * ep.ldc + gcol0 + c4;       // EPI_F32
            const int64_t step8 = 8 * ep.ldc;
            // A loop that is not unrolled, with the sums moved down by sixteen registers after each chunk: as straight code (60 KB,
            // run once per tile) it spent its time on instruction fetches, 55000 to 75000 cycles per tile.
#pragma unroll 1
            for (int c = 0; c < HALF / 16; ++c) {
                if (c > 0) {
#pragma unroll
                    for (int j = 0; j < HALF - 16; ++j) lo[j] = lo[j + 16];
                    if (!(c & 1)) {
#pragma unroll
                        for (int i = 0; i < HALF / 32 - 1; ++i) sbx[i] = sbx[i + 1];
                    }
                }
                uint32_t r3[16], r2[16];
                const uint32_t ta = tmem_base + ((uint32_t)(lg * 32) << 16) + (uint32_t)(half * HALF + c * 16);
                tmem_ld16(ta + b3 * TNC, r3);
                tmem_ld16(ta + b2 * TNC, r2);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                if (c == HALF / 16 - 1) {             // TMEM is read out: the next tile may start
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) { mbar_arrive(tempty_bar(b3)); mbar_arrive(tempty_bar(b2)); }
                }
                const int64_t gc = gcol0 + c * 16 + c4;
                if (gcol0 + c * 16 >= N) continue;                    // the same in the whole warp
                const bool whole = ep.vec && gcol0 + c * 16 + 16 <= N;
                __syncwarp();
#pragma unroll
                for (int j = 0; j < 16; ++j)          // order 2 + order 3 / 256 + ..., an exact integer part and a small fp32 tail
                    sts64(st_w ^ (j * 8), fma(whole_double((long long)(int)r2[j] * 256 + (int)r3[j]), 256.0, (double)lo[j]));
                __syncwarp();
                float4 cur[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) cur[q] = pre[q];
                if (EPI == EPI_F32 && c + 1 < HALF / 16) request(c + 1);
                double sb[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) sb[i] = __hiloint2double(__shfl_sync(0xffffffffu, sbx[0], (c & 1) * 16 + c4 + i), 0);
                const bool diagonal = EPI == EPI_F32 && ep.identity && ep.row0 + grow0 < ep.col0 + gcol0 + c * 16 + 16 && ep.col0 + gcol0 + c * 16 < ep.row0 + grow0 + 32;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    double v[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) v[i] = lds64((st_r[q & 1] + (q >> 1) * 2048) ^ (i * 8)) * (EPI == EPI_DOT ? sb[i] : sa[q] * sb[i]);
                    const int64_t gr = grow0 + q * 8 + rsub;
                    if (EPI == EPI_DOT) {
                        if (!row_in[q]) continue;
                        if (whole) {
                            float4 x = cur[q];
                            if (ep.C0sub) { const float4 y = pre_sub[q]; x.x -= y.x; x.y -= y.y; x.z -= y.z; x.w -= y.w; }
                            dot[q] += (v[0] * (double)x.x + v[1] * (double)x.y) + (v[2] * (double)x.z + v[3] * (double)x.w);
                        } else {
                            const float* h = ep.C0 + gr * ep.ldc0 + gc;
                            const float* hs = ep.C0sub + gr * ep.ldc0 + gc;
#pragma unroll
                            for (int i = 0; i < 4; ++i) if (gc + i < N) dot[q] += v[i] * (double)(ep.C0sub ? h[i] - hs[i] : h[i]);
                        }
                    } else if (EPI == EPI_F64) {
                        if (!row_in[q]) continue;
                        double* cp = (double*)ep.C + gr * ep.ldc + gc;
#pragma unroll
                        for (int i = 0; i < 4; ++i) if (gc + i < N) cp[i] = v[i];
                    } else {
                        if (diagonal) {
#pragma unroll
                            for (int i = 0; i < 4; ++i) v[i] += ep.row0 + gr == ep.col0 + gc + i ? 1.0 : 0.0;
                        }
                        if (!row_in[q]) continue;
                        float* cp = out + q * step8 + c * 16;
                        if (whole) {
                            if (with_c0) {
                                const float4 x = cur[q];
                                v[0] += ep.beta * (double)x.x; v[1] += ep.beta * (double)x.y;
                                v[2] += ep.beta * (double)x.z; v[3] += ep.beta * (double)x.w;
                            }
                            *reinterpret_cast<float4*>(cp) = make_float4((float)v[0], (float)v[1], (float)v[2], (float)v[3]);
                        } else {
                            const float* c0 = ep.C0 + gr * ep.ldc0 + gc;
#pragma unroll
                            for (int i = 0; i < 4; ++i) if (gc + i < N) cp[i] = (float)(with_c0 ? v[i] + ep.beta * (double)c0[i] : v[i]);
                        }
                    }
                }
                if (EPI == EPI_DOT && c + 1 < HALF / 16) request(c + 1);       // two matrices: no room for a second set of registers
            }
            if (EPI == EPI_DOT) {                 // partial sum of this tile half for each of the warp's rows
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    double v = dot[q];
                    v += __shfl_xor_sync(0xffffffffu, v, 1);
                    v += __shfl_xor_sync(0xffffffffu, v, 2);
                    const int64_t gr = grow0 + q * 8 + rsub;
                    if ((lane & 3) == 0 && gr < M) ((double*)ep.C)[gr * ep.ldc + 2 * tn + half] = sa[q] * v;
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "n"(TMEM_COLS) : "memory");
    }
    if (threadIdx.x == 0 && *abort_flag) ctl->status = OSSCAR_E_TIMEOUT;
}

bool encode_planes(PFN_encodeTiled enc, CUtensorMap* map, const void* base, uint64_t K, uint64_t rows, uint64_t ldk, uint32_t box_rows)
{
    const cuuint64_t dims[2] = {K, rows};
    const cuuint64_t strides[1] = {ldk};
    const cuuint32_t box[2] = {(cuuint32_t)I8_BK, box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

inline size_t up256(size_t x) { return (x + 255) / 256 * 256; }

// Panel sizes of one product: `mp` rows of A and `np` columns of B at a time.
struct I8Panels { int64_t mp, np, ldk; bool ok; };
I8Panels plan_stride(int64_t M, int64_t N, int64_t K, int S, size_t a_bytes, size_t b_bytes, int tn, int sms, int64_t ldk)
{
    I8Panels p;
    p.ldk = ldk;
    const size_t per_a = (size_t)S * p.ldk + sizeof(double), per_b = (size_t)S * p.ldk + sizeof(double) + sizeof(unsigned long long);
    const size_t fix_a = 1024, fix_b = 4 * (size_t)K + 2048;
    int64_t mp = a_bytes > fix_a ? (int64_t)((a_bytes - fix_a) / per_a) : 0;
    int64_t np = b_bytes > fix_b ? (int64_t)((b_bytes - fix_b) / per_b) : 0;
    // whole tiles; planes are addressed with 32-bit coordinates
    p.mp = mp >= M ? M : mp / I8_TM * I8_TM;
    p.np = np >= N ? N : np / tn * tn;
    if (p.mp < M && p.np > 0) {          // row panels of the size that takes the fewest rounds over the SMs in all
        const int64_t TN = (p.np + tn - 1) / tn, TM = (M + I8_TM - 1) / I8_TM;
        int64_t best = 0, best_cost = 0;
        for (int64_t t = p.mp / I8_TM; t >= 1; --t) {
            const int64_t cost = (TM / t) * ((t * TN + sms - 1) / sms) + ((TM % t) * TN + sms - 1) / sms;
            if (best == 0 || cost < best_cost) { best = t; best_cost = cost; }
        }
        if (best > 0) p.mp = best * I8_TM;
    }
    p.ok = p.mp > 0 && p.np > 0 && K > 0 && K <= max_k(S) && M < (1 << 28) && N < (1 << 28);
    return p;
}
// Rows of digits start on cache lines where that costs no panel: the 128 bytes of a row in a tile are then one line in L2 instead
// of two, and requests to L2 are what the loads of large products wait for: two tiles of K = 5000 took 566000 cycles with rows of 5008 bytes,
// 486000 with 5120.
I8Panels plan(int64_t M, int64_t N, int64_t K, int S, size_t a_bytes, size_t b_bytes, int tn, int sms = 148)
{
    const I8Panels p = plan_stride(M, N, K, S, a_bytes, b_bytes, tn, sms, digit_stride(K));
    return p.ok && p.mp >= M && p.np >= N ? p : plan_stride(M, N, K, S, a_bytes, b_bytes, tn, sms, round_up(K, 16));
}

template <int S, int TNC, int EPI, int OM = S + 1>
cudaError_t launch_mma(cudaStream_t st, const I8Maps& maps, int64_t M, int64_t N, int64_t K, const I8Epi& ep, const I8Cover& cov, int sms,
                       SearchCtl* ctl, const int32_t* done)
{
    const cudaError_t e = cudaFuncSetAttribute(k_mma_i8<S, TNC, EPI, OM>, cudaFuncAttributeMaxDynamicSharedMemorySize, I8_SMEM);
    if (e != cudaSuccess) return e;
    const int64_t TM = (M + I8_TM - 1) / I8_TM, TN = (N + TNC - 1) / TNC;
    int64_t ids = TM * TN;
    if (cov.upper) { ids = 0; for (int64_t r = 0; r < TM; ++r) ids += TN - r / (TNC / I8_TM); }
    ids *= cov.ksplit > 1 ? cov.ksplit : 1;
    k_mma_i8<S, TNC, EPI, OM><<<(unsigned)(ids < sms ? ids : sms), I8_THREADS, I8_SMEM, st>>>(maps, (int)M, (int)N, (int)K, ep, cov, (int)ids, ctl, done);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace

// Whether the product is worth its digits and fits the scratch.  The fp64 pipe keeps products of less than 2^29 multiply-adds
// (its tiles are smaller, and it needs one launch instead of six) and contractions longer than max_k.
bool gemm_i8_usable(int64_t M, int64_t N, int64_t K, int S, const I8Scratch& sc)
{
    if (!sc.a || !sc.b || ((uintptr_t)sc.a & 255) || ((uintptr_t)sc.b & 255)) return false;
    if (M <= 0 || N <= 0 || K < 256) return false;
    if ((double)M * (double)N * (double)K < 536870912.0) return false;
    return plan(M, N, K, S, sc.a_bytes, sc.b_bytes, 256).ok;
}

template <int S>
static cudaError_t gemm_i8_run(cudaStream_t st, const I8Gemm& p, I8Scratch& sc, SearchCtl* ctl, const int32_t* done)
{
    PFN_encodeTiled enc = get_encode();
    if (!enc) return cudaErrorNotSupported;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int64_t M = p.M, N = p.N, K = p.K;
    // 128-column tiles where the 256-column ones of a panel would leave half of the SMs without work (with more of those, twice as
    // many half tiles take two rounds: G = H W of 96 tiles, 3072 x 1024, 0.281 ms in halves, 0.225 whole)
    int tn = 256;
    I8Panels pl = plan(M, N, K, S, sc.a_bytes, sc.b_bytes, tn, sms);
    if (pl.ok && ((pl.mp + I8_TM - 1) / I8_TM) * ((pl.np + 255) / 256) * 2 <= sms) {
        tn = 128;
        pl = plan(M, N, K, S, sc.a_bytes, sc.b_bytes, tn, sms);
    }
    if (!pl.ok) return cudaErrorInvalidValue;
    char* b = (char*)sc.b;
    int32_t* ck = (int32_t*)b;                                 b += up256(4 * (size_t)K);
    unsigned long long* cmax = (unsigned long long*)b;         b += up256(8 * (size_t)pl.np);
    double* sb = (double*)b;                                   b += up256(8 * (size_t)pl.np);
    int8_t* bp = (int8_t*)b;
    char* a = (char*)sc.a;
    double* sa = (double*)a;                                   a += up256(8 * (size_t)pl.mp);
    int8_t* ap = (int8_t*)a;
    const int vecA = (((uintptr_t)p.A & 15) == 0 && (p.lda % 4) == 0) ? 1 : 0;
    if (p.diag) {
        k_i8_balance<<<(unsigned)((K + 255) / 256), 256, 0, st>>>(p.diag, p.diag_stride, K, p.inverse_scale ? 1 : 0, ck);
        count_launches(1);
    } else if (p.pivots) {
        k_i8_balance_pivots<<<(unsigned)((K + 255) / 256), 256, 0, st>>>(p.pivots, K, ck);
        count_launches(1);
    } else {
        e = cudaMemsetAsync(ck, 0, sizeof(int32_t) * (size_t)K, st);
        if (e != cudaSuccess) return e;
    }
    for (int64_t n0 = 0; n0 < N; n0 += pl.np) {
        const int64_t nw = N - n0 < pl.np ? N - n0 : pl.np;
        if (!p.BT) {
            e = cudaMemsetAsync(cmax, 0, 8 * (size_t)nw, st);
            if (e != cudaSuccess) return e;
        }
        const dim3 gm((unsigned)((nw + 63) / 64), (unsigned)((K + 255) / 256)), gs((unsigned)((nw + 31) / 32), (unsigned)((pl.ldk + 127) / 128));
        const int tri_block = p.tri ? tn : 0;
        const float* sub = p.Bsub ? p.Bsub + n0 : nullptr;
        if (p.BT) {
            const float* bt = p.BT + n0 * p.ldb;
            k_i8_slice_rows<S><<<(unsigned)nw, 256, 0, st>>>(bt, p.ldb, K, ck, bp, nw * pl.ldk, pl.ldk, sb,
                                                             ((uintptr_t)bt & 15) == 0 && (p.ldb % 4) == 0 ? 1 : 0, done);
        } else if (p.Bd) {
            k_i8_colmax<double><<<gm, 256, 0, st>>>(p.Bd + n0, nullptr, p.ldb, K, nw, ck, cmax, done);
            k_i8_slice_cols<S, double><<<gs, 256, 0, st>>>(p.Bd + n0, nullptr, p.ldb, K, nw, ck, cmax, bp, nw * pl.ldk, pl.ldk, sb, tri_block, n0, done);
        } else {
            k_i8_colmax<float><<<gm, 256, 0, st>>>(p.B + n0, sub, p.ldb, K, nw, ck, cmax, done);
            k_i8_slice_cols<S, float><<<gs, 256, 0, st>>>(p.B + n0, sub, p.ldb, K, nw, ck, cmax, bp, nw * pl.ldk, pl.ldk, sb, tri_block, n0, done);
        }
        count_launches(2);
        for (int64_t m0 = 0; m0 < M; m0 += pl.mp) {
            const int64_t mw = M - m0 < pl.mp ? M - m0 : pl.mp;
            // the digits of A from the product before serve again when the whole of A is there, in rows of the same length: that
            // depends on the scratch left for B too (plan())
            const bool have = pl.mp >= M && sc.have_A == p.A && sc.have_rows == M && sc.have_K == K && sc.have_S == S && sc.have_ldk == pl.ldk;
            if (!have) {
                sc.have_A = nullptr;
                k_i8_slice_rows<S><<<(unsigned)mw, 256, 0, st>>>(p.A + m0 * p.lda, p.lda, K, ck, ap, mw * pl.ldk, pl.ldk, sa, vecA, done);
                count_launches(1);
                if (pl.mp >= M) { sc.have_A = p.A; sc.have_rows = M; sc.have_K = K; sc.have_S = S; sc.have_ldk = pl.ldk; }
            }
            e = cudaGetLastError();
            if (e != cudaSuccess) return e;
            I8Maps maps;
            if (!encode_planes(enc, &maps.a, ap, (uint64_t)K, (uint64_t)(S * mw), (uint64_t)pl.ldk, I8_TM)) return cudaErrorInvalidValue;
            if (!encode_planes(enc, &maps.b, bp, (uint64_t)K, (uint64_t)(S * nw), (uint64_t)pl.ldk, (uint32_t)tn)) return cudaErrorInvalidValue;
            I8Epi ep = {};
            ep.sa = sa; ep.sb = sb; ep.alpha = p.alpha; ep.beta = p.beta; ep.identity = p.identity ? 1 : 0;
            ep.row0 = m0; ep.col0 = p.identity_col0 + n0; ep.ldc0 = p.ldc0; ep.ldc = p.ldc;
            ep.C0 = p.C0 ? p.C0 + m0 * p.ldc0 + n0 : nullptr;
            ep.C0sub = p.C0sub ? p.C0sub + m0 * p.ldc0 + n0 : nullptr;
            if (p.dot) {
                ep.ldc = p.ldc;
                ep.C = (double*)p.C + m0 * p.ldc + 2 * (n0 / tn);
            } else if (p.out64) ep.C = (double*)p.C + m0 * p.ldc + n0;
            else ep.C = (float*)p.C + m0 * p.ldc + n0;
            ep.vec = (!ep.C0 || ((((uintptr_t)ep.C0 | (uintptr_t)ep.C0sub) & 15) == 0 && (p.ldc0 % 4) == 0)) && (p.dot || p.out64 || (((uintptr_t)ep.C & 15) == 0 && (p.ldc % 4) == 0)) ? 1 : 0;
            const I8Cover cov = { p.tri ? 1 + (int)(n0 / I8_BK) : 0, 0, 1, 0 };
            // the combinations of digits and epilogues that the callers use
            if constexpr (S == 4 || S == 5) {
                if (p.dot) e = tn == 256 ? launch_mma<S, 256, EPI_DOT>(st, maps, mw, nw, K, ep, cov, sms, ctl, done)
                                         : launch_mma<S, 128, EPI_DOT>(st, maps, mw, nw, K, ep, cov, sms, ctl, done);
            }
            if constexpr (S == 6) {
                if (p.out64) e = tn == 256 ? launch_mma<S, 256, EPI_F64>(st, maps, mw, nw, K, ep, cov, sms, ctl, done)
                                           : launch_mma<S, 128, EPI_F64>(st, maps, mw, nw, K, ep, cov, sms, ctl, done);
            }
            if (p.dot ? (S != 4 && S != 5) : (p.out64 && S != 6)) return cudaErrorInvalidValue;
            if (!p.dot && !p.out64)
                e = tn == 256 ? launch_mma<S, 256, EPI_F32>(st, maps, mw, nw, K, ep, cov, sms, ctl, done)
                              : launch_mma<S, 128, EPI_F32>(st, maps, mw, nw, K, ep, cov, sms, ctl, done);
            if (e != cudaSuccess) return e;
        }
    }
    return cudaSuccess;
}

cudaError_t gemm_i8(cudaStream_t st, const I8Gemm& p, int S, I8Scratch& sc, SearchCtl* ctl, const int32_t* done)
{
    switch (S) {
        case 3: return gemm_i8_run<3>(st, p, sc, ctl, done);
        case 4: return gemm_i8_run<4>(st, p, sc, ctl, done);
        case 5: return gemm_i8_run<5>(st, p, sc, ctl, done);
        case 6: return gemm_i8_run<6>(st, p, sc, ctl, done);
        default: return cudaErrorInvalidValue;
    }
}

int64_t gemm_i8_row_bytes(int64_t K) { return digit_stride(K); }
size_t gemm_i8_operand_bytes(int64_t rows, int64_t K, int S)
{
    return (size_t)rows * ((size_t)S * digit_stride(K) + 16) + 4 * (size_t)K + 2048;
}

// Whether some column of a panel of `rows` rows has its scale above 16 times its root mean square (see gram_i8): skip[0] = 1 and
// skip[1] = 0 then, the other way round otherwise.  Columns of zeros or with entries that are not finite do not count.
__global__ void __launch_bounds__(1024) k_i8_outliers(const unsigned long long* __restrict__ cmax, const unsigned long long* __restrict__ spread,
                                                      int64_t rows, int64_t d1, int32_t* __restrict__ skip)
{
    bool out = false;
    for (int64_t j = threadIdx.x; j < d1; j += 1024) out |= cmax[j] != 0 && finite_bits(cmax[j]) && spread[j] < ((unsigned long long)rows << 22);
    const int any = __syncthreads_or(out);
    if (threadIdx.x == 0) { skip[0] = any ? 1 : 0; skip[1] = any ? 0 : 1; }
}

// C (upper-triangle tiles) = beta C + sum of `slices` partial products, in slice order; block rows of tiles as in the product.
__global__ void __launch_bounds__(256) k_i8_add_slices(float* __restrict__ C, int64_t d1, const float* __restrict__ part, int slices, int64_t stride, int add, int per,
                                                       const int32_t* __restrict__ done)
{
    if (*done) return;
    const int64_t row = blockIdx.y;
    const int64_t c0 = (row / I8_TM / per) * (I8_TM * per);
    for (int64_t c = c0 + (int64_t)blockIdx.x * 256 + threadIdx.x; c < d1; c += (int64_t)gridDim.x * 256) {
        float s = add ? C[row * d1 + c] : 0.f;
        for (int i = 0; i < slices; ++i) s += part[(int64_t)i * stride + row * d1 + c];
        C[row * d1 + c] = s;
    }
}

// H (+)= Xc^T Xc over the upper-triangle tiles for fp32 Xc (n_rows x d1): three digits per entry, the eight digit products of orders
// 2 to 5 at twice the bf16 rate.  Both operands are the same transposed digits.  A layer with fewer tiles than SMs splits the
// rows of a panel over CTAs, whose fp32 partial sums are added in order.
// Digits are fixed-point below the scale s_j of a column (a power of two, less than 2.1 times its largest entry): an entry is rounded
// by up to 2^-24 s_j, and values that repeat (pixels, padding) add that up with one sign.  Where the scale is at most 16 times
// the column's root mean square it stays below 2^-19 sqrt(H_ii H_jj) in the worst case (1e-7 measured on pixels and on
// rectified Gaussians), less than the truncating sums of the bf16 terms lose.  A panel with a column beyond it (single large
// entries) goes through the bf16 terms, whose bits are relative to every entry: both paths are enqueued, one returns at once.
// (Six products without this test left 2e-5 of sqrt(H_ii H_jj), and 1e-3 of an entry, where one entry of a column was 300 times
// the rest; four digits, ten products, 0.74 ms at 6272 x 4608.)
// One chunk, ms, bf16 terms -> digits: 0.171 -> 0.108 at 4900 x 256, 0.187 -> 0.117 at 4900 x 1024, 0.087 -> 0.087 at 2048 x 1024, 0.80 -> 0.62
// at 6272 x 4608, 0.22 -> 0.23 at 4900 x 2048; before the row thresholds 0.034 -> 0.056 at 512 x 1024 and 0.072 -> 0.081 at 1500 x 2304: short
// chunks stay on the terms.
// cudaErrorMemoryAllocation where the scratch is too small or the product too small to pay: the caller takes another path.
cudaError_t gram_i8(cudaStream_t st, const float* X, int64_t n_rows, int64_t d1, float* C, bool accumulate,
                    void* scratch, size_t scratch_bytes, SearchCtl* ctl_dev)
{
    constexpr int S = 3;
    if (n_rows <= 0) return cudaSuccess;
    if (!scratch || ((uintptr_t)scratch & 255) || d1 >= (1 << 28)) return cudaErrorMemoryAllocation;
    if (n_rows < (d1 < 1536 ? 2048 : 4096) || (double)n_rows * (double)d1 * (double)d1 < 268435456.0) return cudaErrorMemoryAllocation;
    PFN_encodeTiled enc = get_encode();
    if (!enc) return cudaErrorNotSupported;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int64_t TM = (d1 + I8_TM - 1) / I8_TM;
    constexpr int tn = 256;
    int64_t tiles = 0;
    for (int64_t r = 0; r < TM; ++r) tiles += (d1 + tn - 1) / tn - r / (tn / I8_TM);
    // rows of a panel: digits, balance exponents, column scales and sums
    const size_t fixed = 24 * (size_t)d1 + 4096;
    if (scratch_bytes <= fixed) return cudaErrorMemoryAllocation;
    auto panel_rows = [&](size_t bytes) {
        int64_t r = (int64_t)(bytes / ((size_t)S * d1 + 4)) / 16 * 16 - 16;
        if (r > max_k(S) / 16 * 16) r = max_k(S) / 16 * 16;
        return r;
    };
    int64_t panel = panel_rows(scratch_bytes - fixed);
    if (panel > n_rows) panel = n_rows;
    // CTAs per tile: fill the SMs once, at least eight k-blocks each, if the partial products fit beside the panel
    int ksplit = 1;
    if (tiles < sms) {
        int64_t ks = sms / tiles;
        const int64_t most = (panel < n_rows ? panel : n_rows) / (8 * I8_BK);
        if (ks > most) ks = most;
        const size_t pb = up256(sizeof(float) * (size_t)d1 * d1);
        for (; ks > 1; --ks) {
            const int64_t left = fixed + pb * (size_t)ks < scratch_bytes ? panel_rows(scratch_bytes - fixed - pb * (size_t)ks) : 0;
            if (left < n_rows && left < 1024) continue;
            ksplit = (int)ks;
            if (panel > left) panel = left;
            break;
        }
    }
    if (panel < n_rows) {                // panels of equal height
        if (panel < 1024) return cudaErrorMemoryAllocation;
        const int64_t np = (n_rows + panel - 1) / panel;
        panel = round_up((n_rows + np - 1) / np, 16);
    }
    char* b = (char*)scratch;
    float* part = (float*)b;                                   if (ksplit > 1) b += up256(sizeof(float) * (size_t)d1 * d1) * ksplit;
    int32_t* ck = (int32_t*)b;                                 b += up256(4 * (size_t)round_up(panel, 16));
    unsigned long long* cmax = (unsigned long long*)b;         b += up256(8 * (size_t)d1);
    unsigned long long* spread = (unsigned long long*)b;       b += up256(8 * (size_t)d1);
    double* sc = (double*)b;                                   b += up256(8 * (size_t)d1);
    int8_t* planes = (int8_t*)b;
    const int32_t *skip_digits = &ctl_dev->gram_skip[0], *skip_terms = &ctl_dev->gram_skip[1];
    for (int64_t r0 = 0; r0 < n_rows; r0 += panel) {
        const int64_t rows = n_rows - r0 < panel ? n_rows - r0 : panel;
        const bool lines = (size_t)S * d1 * digit_stride(rows) <= scratch_bytes - (size_t)((char*)planes - (char*)scratch);       // see plan()
        const int64_t ldk = lines ? digit_stride(rows) : round_up(rows, 16);
        e = cudaMemsetAsync(ck, 0, (size_t)((char*)sc - (char*)ck), st);           // and the column maxima and sums behind it
        if (e != cudaSuccess) return e;
        k_i8_colmax<float><<<dim3((unsigned)((d1 + 63) / 64), (unsigned)((rows + 255) / 256)), 256, 0, st>>>(X + r0 * d1, nullptr, d1, rows, d1, ck, cmax, nullptr);
        k_i8_slice_cols<S, float, true><<<dim3((unsigned)((d1 + 31) / 32), (unsigned)((ldk + 127) / 128)), 256, 0, st>>>(
            X + r0 * d1, nullptr, d1, rows, d1, ck, cmax, planes, d1 * ldk, ldk, sc, 0, 0, nullptr, spread);
        k_i8_outliers<<<1, 1024, 0, st>>>(cmax, spread, rows, d1, ctl_dev->gram_skip);
        count_launches(3);
        I8Maps maps;
        if (!encode_planes(enc, &maps.a, planes, (uint64_t)rows, (uint64_t)(S * d1), (uint64_t)ldk, I8_TM)) return cudaErrorInvalidValue;
        if (!encode_planes(enc, &maps.b, planes, (uint64_t)rows, (uint64_t)(S * d1), (uint64_t)ldk, (uint32_t)tn)) return cudaErrorInvalidValue;
        const bool add = accumulate || r0 > 0;
        const int ks = rows >= (int64_t)ksplit * I8_BK ? ksplit : 1;          // a short last panel is not worth splitting
        I8Epi ep = {};
        ep.sa = sc; ep.sb = sc; ep.alpha = 1.0; ep.ldc = ep.ldc0 = d1;
        ep.C = ks > 1 ? part : C; ep.C0 = C; ep.beta = ks == 1 && add ? 1.0 : 0.0;
        ep.vec = ((uintptr_t)ep.C & 15) == 0 && ((uintptr_t)C & 15) == 0 && (d1 % 4) == 0 ? 1 : 0;
        const I8Cover cov = { 0, 1, ks, (int64_t)(up256(sizeof(float) * (size_t)d1 * d1) / sizeof(float)) };
        e = launch_mma<S, 256, EPI_F32, S + 2>(st, maps, d1, d1, rows, ep, cov, sms, ctl_dev, skip_digits);
        if (e != cudaSuccess) return e;
        if (ks > 1) {
            k_i8_add_slices<<<dim3((unsigned)((d1 + 1023) / 1024), (unsigned)d1), 256, 0, st>>>(C, d1, part, ks, cov.slice_stride, add ? 1 : 0, tn / I8_TM, skip_digits);
            count_launches(1);
        }
        e = gram_tc3(st, X + r0 * d1, rows, d1, C, add, scratch, scratch_bytes, ctl_dev, skip_terms);
        if (e != cudaSuccess) return e;
    }
    return cudaGetLastError();
}

// G = H W.  Ten products of four digits at twice the bf16 rate against six of bf16 terms, and 31 bits of every row and column
// instead of the 24 of an fp32 product summed by a truncating accumulator: 65 -> 50 ms with the mirroring at d1 = 28672, m = 7168.
cudaError_t cross_term_tc(cudaStream_t st, const float* H, int64_t d1, const float* W, int64_t m, float* G,
                          void* scratch, size_t scratch_bytes, SearchCtl* ctl_dev)
{
    constexpr int S = 4;
    if ((double)d1 * (double)d1 * (double)m <= kTinyProduct)
        return gemm_f64acc(st, d1, m, d1, 1.0, H, d1, W, m, 0.0, nullptr, 0, G, m, false, nullptr);
    I8Scratch sc;
    const size_t room = scratch_bytes / 256 * 256;
    size_t need_b = up256(gemm_i8_operand_bytes(m, d1, S));
    if (need_b > room / 2) need_b = room / 2 / 256 * 256;
    sc.b = scratch; sc.b_bytes = need_b;
    sc.a = (char*)scratch + need_b; sc.a_bytes = room - need_b;
    if (!gemm_i8_usable(d1, m, d1, S, sc)) return gemm_tc(st, d1, m, d1, 1.f, H, d1, W, m, 0.f, G, m, scratch, scratch_bytes, ctl_dev);
    I8Gemm p = {};
    p.M = d1; p.N = m; p.K = d1; p.alpha = 1.0;
    p.A = H; p.lda = d1; p.B = W; p.ldb = m; p.C = G; p.ldc = m;
    p.diag = H; p.diag_stride = d1 + 1;
    return gemm_i8(st, p, S, sc, ctl_dev, nullptr);
}

// Fixed-order sum of n doubles in two stages, the first over 256 blocks (added to what the blocks already have, if `add`).
__global__ void __launch_bounds__(256) k_i8_sum(const double* __restrict__ x, int64_t n, double* __restrict__ part, int add)
{
    __shared__ double red[8];
    double s = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) s += x[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 1; i < 8; ++i) s += red[i];
        part[blockIdx.x] = add ? part[blockIdx.x] + s : s;
    }
}

// *out = sum of D o (H D), D = W - Wt (fp32 differences), as digit products with the sum in their epilogue: neither D nor H D
// is ever stored.  Four digits (ten products): 1e-9 of the result, least-squares refits and columns with single large
// weights included.  (Three digits left up to 5e-7 there, the fp32 pipes 9e-8.)
// The scratch takes one partial sum per row and half tile and the digits of a slab of the contraction: some columns of H
// and as many rows of D, whose sums add up.  A slab has all tiles of the result, whatever m is.
// A call takes 1.64 ms at d1 = 8192, m = 2048 and 0.24 ms at 2048, 512, on the fp32 pipes 6.99 and 0.32 ms.  Bound: the int8 tensor pipe (1.3 of the 1.64 ms),
// then the slicing of H.  Narrow results stay on the fp32 pipes: the scratch shrinks with m, and every slab costs its launches and the
// slicing of d1 rows (about 90 us at d1 = 8192).  Pipes against digits, ms: 3.15 / 3.78 at 12288, 384, 4.68 / 2.96 at 12288, 512, 1.28 / 1.92
// at 8192, 256, 2.11 / 1.34 at 8192, 512, 0.32 / 0.38 at 2048, 256, 0.33 / 0.24 at 2048, 512.
cudaError_t objective_i8(cudaStream_t st, const float* H, const float* W, const float* Wt, int64_t d1, int64_t m,
                         void* scratch, size_t scratch_bytes, double* partials, double* out_dev, SearchCtl* ctl_dev)
{
    constexpr int S = 4;
    const int64_t pc = gemm_i8_dot_cols(m);
    const size_t part_bytes = up256(sizeof(double) * (size_t)d1 * pc);
    if (!scratch || ((uintptr_t)scratch & 255) || m <= 384 || (double)d1 * (double)d1 * (double)m < 536870912.0) return cudaErrorMemoryAllocation;
    auto b_bytes = [&](int64_t w) { return up256(gemm_i8_operand_bytes(m, w, S)); };
    auto a_bytes = [&](int64_t w) { return up256(gemm_i8_operand_bytes(d1, w, S)); };
    int64_t w = round_up(d1, I8_BK) < max_k(S) ? round_up(d1, I8_BK) : max_k(S) / I8_BK * I8_BK;
    while (w >= 256 && part_bytes + a_bytes(w) + b_bytes(w) > scratch_bytes) w -= I8_BK;
    if (w < 256) return cudaErrorMemoryAllocation;
    const int64_t slabs = (d1 + w - 1) / w;
    w = round_up((d1 + slabs - 1) / slabs, I8_BK);
    double* part = (double*)scratch;
    cudaError_t e = cudaMemsetAsync(part, 0, sizeof(double) * (size_t)d1 * pc, st);       // 256-column tiles fill half of the columns
    if (e != cudaSuccess) return e;
    for (int64_t k0 = 0; k0 < d1; k0 += w) {
        I8Scratch sc;
        sc.b = (char*)scratch + part_bytes; sc.b_bytes = b_bytes(w);
        sc.a = (char*)sc.b + sc.b_bytes; sc.a_bytes = a_bytes(w);
        I8Gemm p = {};
        p.M = d1; p.N = m; p.K = d1 - k0 < w ? d1 - k0 : w; p.alpha = 1.0; p.dot = true;
        p.A = H + k0; p.lda = d1; p.B = W + k0 * m; p.Bsub = Wt + k0 * m; p.ldb = m;
        p.C0 = W; p.C0sub = Wt; p.ldc0 = m; p.C = part; p.ldc = pc;
        p.diag = H + k0 * (d1 + 1); p.diag_stride = d1 + 1;
        e = gemm_i8(st, p, S, sc, ctl_dev, nullptr);
        if (e != cudaSuccess) return e;
        k_i8_sum<<<256, 256, 0, st>>>(part, d1 * pc, partials, k0 > 0 ? 1 : 0);
        count_launches(1);
    }
    return sum_partials(st, partials, 256, out_dev);
}

// columns of partial sums a `dot` product leaves per row
int64_t gemm_i8_dot_cols(int64_t N) { return 2 * ((N + 127) / 128); }

}  // namespace osscar
