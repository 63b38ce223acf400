// FP64 products dX/dT(q) = c_X A(q) L(q) A(q) for large M (multi-orbital bond sets, M > 64) on the tensor cores
// (Eq. RGE_spin, c_P = 1, and the orbital form of Eq. rge_Dmat, c_C = 2).
//
// This GPU's FP64 pipe gives 1.2 TFLOP/s, its BF16 tensor cores 1.9 PFLOP/s, so the FP64 product is formed from exact
// integer products (the scheme of Ozaki, Ogita, Oishi and Rump, "Error-free transformations of matrix multiplication by
// using fast routines of matrix multiplication and its applications", Numer. Algorithms 59, 2012): every row of the
// left and every column of the right operand is scaled by a power of two to a 62-bit fixed-point number and cut into
// nine signed digits of seven bits, |d| <= 64, exact in BF16.  The digit matrices' products are sums of integers,
//   sum_k d_i(r,k) d'_j(k,c),  |.| <= 4096 per term,
// accumulated in FP32 in tensor memory for every level i + j <= 8: the L + 1 pairs of a level and the two real products of
// a complex one stay below 2^24, hence exact, for 224 values of k; longer sums are drained in between.  The digits carry
// their weights 2^{-7 i} (exact in BF16), so that the pairs of level 9 add to level 8's sum as its fraction.  The levels'
// integers are then joined in FP64.
//
// Fixed point holds an entry to its row's (column's) scale, not to its own, so the result is off by at most
// 2^-60.9 2^(Er + Ec) per term (rounding of both operands 2^-61, the levels above 9 2^-65; 2^Er, 2^Ec: the scales), while an
// FP64 sum of complex terms is off by up to 2^-52 times its sum of magnitudes S(r,c) = sum_k |a(r,k)| |b(k,c)| per term.
// The first is the smaller where S >= 2^-8.9 2^(Er + Ec).  S comes from one more MMA per step, of the operands' magnitudes
// in BF16; the entries with 0 < S < 2^-8 2^(Er + Ec) (small ones that only meet zeros or small ones), and those of rows and
// columns that hold an infinity or NaN, are summed in FP64 over the row's nonzero entries by a second kernel.  So every
// entry is at least as good as an FP64 sum's bound, and not finite exactly where an FP64 sum is.
//
// Per chunk of matrices (channel, momentum): the exponents, the digits of A (rows) and L (columns, gathered from the
// compact loops through the bond-pair table), T = A L, the digits of T and of A (columns), and c T A.  The GEMM kernel: one
// CTA per 128 x 48 tile and part (real or imaginary), all nine levels' accumulators and S in its tensor memory, so
// that each 16 values of k are loaded once (105 KB by two bulk copies, two stages).  The levels' accumulators lie
// side by side, and so do the digits of the right operand, so one MMA multiplies a digit of the left operand by up to five
// digits of the right one (N = 240, level by level).  Warp 0 copies, warp 1 issues, warps 2-5 join the levels.
// Products of the 8 x 8 three-orbital representatives (30 matrices, two products each, M = 324): 1.53 ms at T = 0.1, where
// one or two entries of a hundred take FP64 sums, 2.44 ms at T = 3 (a third; many entries of a hot, symmetric state are tiny),
// 21.6 ms on the FP64 pipe alone; general states of all 64 momenta 5.6 ms.  Eight digits without the FP64 sums take 1.31,
// 1.31 and 5.1 ms, but keep an entry 1e-9 of its row's largest to 25 bits.  A GEMM of 30 matrices takes 0.61 ms: the tensor
// pipe is busy 41% of the cycles (MMAs of K = 16 with their fixed cost, one accumulator set, so that joining the levels is
// not overlapped).
#include <cuda_bf16.h>

#include <algorithm>

#include "tc_common.cuh"
#include "tufrg_internal.cuh"

namespace tufrg {
namespace {

constexpr int NSL = 9;                     // digits (slices) per value
constexpr int TM = 128, TN = 48, KS = 16;  // tile, k values per stage (nine levels and S: 480 tensor-memory columns)
constexpr int KCHUNK = 224 / KS;           // stages whose sums stay exact in FP32
constexpr unsigned A_BLK = TM * KS * 2;    // bytes of one slice and part of the left operand
constexpr int BR = NSL * TN;               // rows (slice, column) of one part of the right operand
constexpr unsigned B_PART = BR * KS * 2;   // its bytes
// a stage: the digits, then the magnitudes
constexpr unsigned A_MAG = NSL * 2 * A_BLK, B_MAG = 2 * B_PART;
constexpr unsigned A_STAGE = A_MAG + A_BLK, B_STAGE = B_MAG + TN * KS * 2, STAGE = A_STAGE + B_STAGE;
constexpr int FRAC = 62;                   // fraction bits of the scaled values
constexpr float S_MIN = 1.f / 256;         // entries of smaller S (and not 0) are summed in FP64
static_assert((NSL + 1) * TN <= 512 && NSL * 2 * 4096 * KCHUNK * KS < (1 << 24), "tensor memory; exact sums");
constexpr int NTHREADS = 192;
constexpr size_t CHUNK_BYTES = size_t(1) << 30;   // digit buffers of one chunk of matrices, at most

struct Dims {
    int M, ks, m_tiles, n_tiles;
    __host__ __device__ size_t a_bytes() const { return (size_t)m_tiles * ks * A_STAGE; }
    __host__ __device__ size_t b_bytes() const { return (size_t)n_tiles * ks * B_STAGE; }
};

Dims dims_of(int M)
{
    Dims d{};
    d.M = M;
    d.ks = (M + KS - 1) / KS;
    d.m_tiles = (M + TM - 1) / TM;
    d.n_tiles = (M + TN - 1) / TN;
    return d;
}

// the matrices of a call: channels of the mask, then listed momenta
struct Mats {
    const int *qlist;
    int nl, Nq, ch0, m0;    // momenta per channel, first channel, first matrix of the chunk
    __device__ size_t row(int local, int &ch) const   // (channel, momentum) row of matrix m0 + local
    {
        const int mat = m0 + local, p = mat % nl;
        ch = ch0 + mat / nl;
        return (size_t)ch * Nq + (qlist ? qlist[p] : p);
    }
};

__device__ __forceinline__ unsigned mag_hi(double2 v)   // the larger magnitude's high word
{
    const unsigned a = (unsigned)__double2hiint(v.x) & 0x7fffffffu, b = (unsigned)__double2hiint(v.y) & 0x7fffffffu;
    return a > b ? a : b;
}

// Row and column maxima of A (high words of the magnitudes): one CTA per 32 rows of a matrix, a warp per row, four rows
// per warp; the columns through shared memory.
__global__ void __launch_bounds__(256) oz_scale_kernel(const double2 *A, Mats mt, int M, unsigned *rmax, unsigned *cmax)
{
    extern __shared__ unsigned s_c[];
    int ch;
    const double2 *a = A + mt.row(blockIdx.y, ch) * (size_t)M * M;
    for (int c = threadIdx.x; c < M; c += 256) s_c[c] = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = 0; i < 4; i++) {
        const int r = blockIdx.x * 32 + warp * 4 + i;
        if (r >= M) break;
        unsigned m = 0;
        for (int c = lane; c < M; c += 32) {
            const unsigned h = mag_hi(a[(size_t)r * M + c]);
            m = max(m, h);
            atomicMax(&s_c[c], h);
        }
        for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (lane == 0) rmax[(size_t)blockIdx.y * M + r] = m;
    }
    __syncthreads();
    for (int c = threadIdx.x; c < M; c += 256) atomicMax(cmax + (size_t)blockIdx.y * M + c, s_c[c]);
}

// Column maxima of the gathered loop matrix: thread = column (R2, b); blockIdx.y splits the rows' pair index a.
__global__ void oz_scale_loop_kernel(const double2 *Lc, const int *dij, Mats mt, int M, int nff, int ns2, int nd, unsigned *cmax)
{
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= M) return;
    int ch;
    const double2 *lc = Lc + mt.row(blockIdx.z, ch) * (size_t)nd * ns2 * ns2;
    const int r2 = n / ns2, b = n - r2 * ns2;
    unsigned m = 0;
    for (int r1 = 0; r1 < nff; r1++) {
        const double2 *p = lc + (size_t)dij[r1 * nff + r2] * ns2 * ns2 + b;
        for (int a = blockIdx.y; a < ns2; a += gridDim.y) m = max(m, mag_hi(p[(size_t)a * ns2]));
    }
    atomicMax(cmax + (size_t)blockIdx.z * M + n, m);
}

// x scaled by 2^(62 - E) and rounded to an integer, |x| < 2^E, E = (biased exponent of the largest magnitude) - 1022
__device__ __forceinline__ long long to_fixed(double x, int E)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int e = (int)((b >> 52) & 0x7ffu);
    if (e == 0x7ff) return 0;   // (this row's or column's results are summed in FP64)
    unsigned long long m = (b & 0xfffffffffffffull) | (e ? 1ull << 52 : 0ull);
    const int sh = (e ? e : 1) - 1075 + FRAC - E;   // at most 9
    if (sh >= 0) m <<= sh;
    else if (sh > -64) m = (m + (1ull << (-sh - 1))) >> -sh;
    else m = 0;
    return (b >> 63) ? -(long long)m : (long long)m;
}

__device__ __forceinline__ int exp_of_hi(unsigned hi) { return max((int)(hi >> 20), 1) - 1022; }

// The digits of eight complex values (k0 .. k0 + 7 of one row) into their places of the nine slices, real then
// imaginary parts: slice i and part p at dst + i slice + p part bytes; the values' magnitudes |Re| + |Im| in units of 2^E
// at mag, rounded down to BF16 (at least 2^-31 where the value is not zero).
__device__ __forceinline__ void put_digits(const double2 (&v)[8], int E, unsigned char *dst, unsigned slice, unsigned part, unsigned char *mag)
{
    unsigned top[8];
#pragma unroll
    for (int k = 0; k < 8; k++) top[k] = v[k].x != 0.0 || v[k].y != 0.0;
#pragma unroll
    for (int p = 0; p < 2; p++) {
        int hi[8], mid[8], lo[8];   // digits 0-3 (28 bits), 4 and 5-8 (28 bits)
#pragma unroll
        for (int k = 0; k < 8; k++) {
            const long long x = to_fixed(p ? v[k].y : v[k].x, E);
            const unsigned t = (unsigned)((unsigned long long)(x < 0 ? -x : x) >> 31);
            top[k] = p ? top[k] + (t & ~1u) : top[k] | t;   // (the sum of two: below 2^32 + 1, kept below 2^32)
            const long long h = (x + (1ll << 34)) >> 35, r = x - h * (1ll << 35), m = (r + (1ll << 27)) >> 28;
            hi[k] = (int)h;
            mid[k] = (int)m;
            lo[k] = (int)(r - m * (1ll << 28));
        }
#pragma unroll
        for (int i = 0; i < NSL; i++) {
            int (&w)[8] = i < 4 ? hi : i == 4 ? mid : lo;
            const int sh = i < 4 ? 21 - 7 * i : i == 4 ? 0 : 21 - 7 * (i - 5);
            float d[8];
#pragma unroll
            for (int k = 0; k < 8; k++) {
                const int g = sh ? (w[k] + (1 << sh >> 1)) >> sh : w[k];
                w[k] -= g * (1 << sh);
                d[k] = (float)g * __uint_as_float((unsigned)(127 - 7 * i) << 23);   // 2^(-7 i)
            }
            __align__(16) __nv_bfloat162 q[4];
#pragma unroll
            for (int k = 0; k < 4; k++) q[k] = __floats2bfloat162_rn(d[2 * k], d[2 * k + 1]);
            *reinterpret_cast<uint4 *>(dst + (size_t)i * slice + (size_t)p * part) = *reinterpret_cast<const uint4 *>(q);
        }
    }
    unsigned w[4];
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const unsigned a = __float_as_uint(__uint2float_rz(top[2 * k]) * 0x1p-31f), b = __float_as_uint(__uint2float_rz(top[2 * k + 1]) * 0x1p-31f);
        w[k] = (a >> 16) | (b & 0xffff0000u);
    }
    *reinterpret_cast<uint4 *>(mag) = make_uint4(w[0], w[1], w[2], w[3]);
}

// Digits of a left operand, [matrix][row tile][stage][slice][part][128 x 16 in core matrices], and its magnitudes [128 x 16]
// after them: thread = row, one CTA per
// (row tile, eight k values) and matrix.  src: the call's A matrices (mt), or T, the chunk's own matrices in order.
template <bool OWN>
__global__ void __launch_bounds__(TM) oz_left_kernel(const double2 *src, Mats mt, Dims d, const unsigned *rmax, unsigned char *out)
{
    const int tile = blockIdx.x / (2 * d.ks), kc = blockIdx.x - tile * 2 * d.ks, r = tile * TM + threadIdx.x, M = d.M;
    int ch;
    const double2 *a = src + (OWN ? (size_t)blockIdx.y : mt.row(blockIdx.y, ch)) * M * M + (size_t)r * M;
    double2 v[8];
#pragma unroll
    for (int k = 0; k < 8; k++) v[k] = r < M && kc * 8 + k < M ? a[kc * 8 + k] : make_double2(0.0, 0.0);
    const int E = r < M ? exp_of_hi(rmax[(size_t)blockIdx.y * M + r]) : 1;
    unsigned char *dst = out + (size_t)blockIdx.y * d.a_bytes() + ((size_t)tile * d.ks + (kc >> 1)) * A_STAGE +
                         ((size_t)(kc & 1) * TM + threadIdx.x) * 16;
    put_digits(v, E, dst, 2 * A_BLK, A_BLK, dst + A_MAG);
}

// Digits of a right operand, [matrix][column tile][stage][part][(slice, column) x 16], and its magnitudes [column x 16]: thread = column, one CTA per (128
// columns, eight k values) and matrix.  LOOP: the loop matrix gathered from the compact loops, else the matrices of src.
template <bool LOOP>
__global__ void __launch_bounds__(128) oz_right_kernel(const double2 *src, const int *dij, int nff, int ns2, int nd, Mats mt, Dims d,
                                                       const unsigned *cmax, unsigned char *out)
{
    const int cb = blockIdx.x / (2 * d.ks), kc = blockIdx.x - cb * 2 * d.ks, n = cb * 128 + threadIdx.x, M = d.M;
    const int tile = n / TN;
    if (tile >= d.n_tiles) return;
    int ch;
    const size_t row = mt.row(blockIdx.y, ch);
    double2 v[8];
#pragma unroll
    for (int k = 0; k < 8; k++) {
        const int kk = kc * 8 + k;
        v[k] = make_double2(0.0, 0.0);
        if (n < M && kk < M) {
            if (LOOP) {
                const int r1 = kk / ns2, r2 = n / ns2;
                v[k] = src[((row * nd + dij[r1 * nff + r2]) * ns2 + kk - r1 * ns2) * ns2 + n - r2 * ns2];
            } else {
                v[k] = src[row * M * M + (size_t)kk * M + n];
            }
        }
    }
    const int E = n < M ? exp_of_hi(cmax[(size_t)blockIdx.y * M + n]) : 1;
    unsigned char *stage = out + (size_t)blockIdx.y * d.b_bytes() + ((size_t)tile * d.ks + (kc >> 1)) * B_STAGE;
    const int c = n - tile * TN;
    put_digits(v, E, stage + ((size_t)(kc & 1) * BR + c) * 16, TN * 16, B_PART, stage + B_MAG + ((size_t)(kc & 1) * TN + c) * 16);
}

struct GemmArgs {
    const unsigned char *PA, *PB;
    const unsigned *ea, *eb;     // row maxima of the left, column maxima of the right operands (high words)
    double2 *out;
    unsigned *rmax_out;          // T: its row maxima (zeroed), or null
    unsigned long long *exact;   // [matrix][row][column tile] bit j: column j of the tile is left to oz_exact_kernel
    Mats mt;
    Dims d;
    const double *scal;          // output scale (null: 1, the chunk's own matrices in order)
    int *err;
};

// instruction descriptor: D = F32, A = B = BF16, both K-major, M x N; bit 13 negates A
__device__ __forceinline__ unsigned idesc_bf16(int n, bool neg_a)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | (neg_a ? (1u << 13) : 0u) | ((unsigned)(n >> 3) << 17) | ((unsigned)(TM >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(unsigned d, unsigned long long da, unsigned long long db, unsigned id, unsigned acc)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d), "l"(da), "l"(db), "r"(id),
                 "r"(acc) : "memory");
}

__device__ __forceinline__ void tmem_ld4(unsigned addr, unsigned (&v)[4])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "r"(addr));
}

// an integer below 2^51 in magnitude as a double
__device__ __forceinline__ double int_double(long long v)
{
    return __longlong_as_double(0x4338000000000000ll + v) - 6755399441055744.0;   // 2^52 + 2^51
}

// sum_L S_L 2^(56 - 7 L) of the nine levels' sums S_L 2^(-7 L)
__device__ __forceinline__ double join(const unsigned (&v)[NSL][4], int j)
{
    int s[NSL];
#pragma unroll
    for (int L = 0; L < NSL; L++) s[L] = __float2int_rn(__uint_as_float(v[L][j]) * __uint_as_float((unsigned)(127 + 7 * L) << 23));
    // |S_L| <= (L + 1) 1.84e6: two levels fit 31 bits, five levels 49, four 45
    const long long hi = ((long long)(s[0] * 128 + s[1]) * 16384 + (s[2] * 128 + s[3])) * 128 + s[4];
    const long long lo = (long long)(s[5] * 128 + s[6]) * 16384 + (s[7] * 128 + s[8]);
    return fma(int_double(hi), 268435456.0, int_double(lo));
}

__global__ void __launch_bounds__(NTHREADS, 1) oz_gemm_kernel(const __grid_constant__ GemmArgs g)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) unsigned long long full[2], empty[2], accf, acce, done;
    __shared__ unsigned tmem_base;
    __shared__ int abort_flag, last_issued[2];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const Dims d = g.d;
    const int part = blockIdx.x & 1, tile = blockIdx.x >> 1;
    const int nt = tile % d.n_tiles, mt = (tile / d.n_tiles) % d.m_tiles, mat = tile / (d.n_tiles * d.m_tiles);
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(tc::smem_u32(&tmem_base)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int b = 0; b < 2; b++) {
            tc::mbar_init(tc::smem_u32(&full[b]), 1);
            tc::mbar_init(tc::smem_u32(&empty[b]), 1);
            last_issued[b] = -1;
        }
        tc::mbar_init(tc::smem_u32(&accf), 1);
        tc::mbar_init(tc::smem_u32(&acce), 128);
        tc::mbar_init(tc::smem_u32(&done), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        abort_flag = 0;
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const unsigned tmem = tmem_base;
    const int n_chunks = (d.ks + KCHUNK - 1) / KCHUNK, per = (d.ks + n_chunks - 1) / n_chunks;   // stages per exact sum
    if (tid == 0) {
        const unsigned char *pa = g.PA + (size_t)mat * d.a_bytes() + (size_t)mt * d.ks * A_STAGE;
        const unsigned char *pb = g.PB + (size_t)mat * d.b_bytes() + (size_t)nt * d.ks * B_STAGE;
        for (int s = 0; s < d.ks; s++) {
            const int b = s & 1;
            if (s >= 2 && !tc::mbar_wait_or_abort(tc::smem_u32(&empty[b]), ((s >> 1) - 1) & 1, &abort_flag)) {
                atomicExch(&abort_flag, 1);
                break;
            }
            const unsigned bar = tc::smem_u32(&full[b]), dst = tc::smem_u32(smem + b * STAGE);
            asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n\t}" ::"r"(bar), "r"(STAGE) : "memory");
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                         "l"(pa + (size_t)s * A_STAGE), "r"(A_STAGE), "r"(bar) : "memory");
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst + A_STAGE),
                         "l"(pb + (size_t)s * B_STAGE), "r"(B_STAGE), "r"(bar) : "memory");
            last_issued[b] = s;
        }
    } else if (tid == 32) {
        bool ok = true;
        for (int s = 0; s < d.ks && ok; s++) {
            const int b = s & 1, in = s % per;
            // the accumulators of the previous chunk must have been read
            if (s > 0 && in == 0) ok = tc::mbar_wait_or_abort(tc::smem_u32(&acce), (s / per - 1) & 1, &abort_flag);
            if (ok) ok = tc::mbar_wait_or_abort(tc::smem_u32(&full[b]), (s >> 1) & 1, &abort_flag);
            if (!ok) break;
            tc::fence_after();
            const unsigned sa = tc::smem_u32(smem + b * STAGE), sb = sa + A_STAGE;
            mma_bf16(tmem + (unsigned)(NSL * TN), tc::smem_desc(sa + A_MAG, TM), tc::smem_desc(sb + B_MAG, TN), idesc_bf16(TN, false), s ? 1u : 0u);   // S
            // Re: Ar Br - Ai Bi; Im: Ar Bi + Ai Br
#pragma unroll
            for (int i = 0; i < NSL; i++)
#pragma unroll
                for (int p = 0; p < 2; p++) {
                    const unsigned long long da = tc::smem_desc(sa + (2 * i + p) * A_BLK, TM);
                    const unsigned pb = sb + (p ^ part) * B_PART;
                    const bool neg = p == 1 && part == 0;
                    const unsigned first = in == 0 && i == 0 && p == 0 ? 0u : 1u;   // (slice 0 reaches every level)
                    constexpr int NM = 256 / TN;                                      // digits of B per MMA, at most
#pragma unroll
                    for (int j = 0; j < NSL - i; j += NM) {
                        const int nj = NSL - i - j < NM ? NSL - i - j : NM;
                        mma_bf16(tmem + (unsigned)((i + j) * TN), da, tc::smem_desc(pb + j * TN * 16, BR), idesc_bf16(nj * TN, neg), first);
                    }
                    if (i > 0)   // level 9: to level 8's sum
                        mma_bf16(tmem + (unsigned)((NSL - 1) * TN), da, tc::smem_desc(pb + (NSL - i) * TN * 16, BR), idesc_bf16(TN, neg), 1u);
                }
            tc::commit(tc::smem_u32(&empty[b]));
            if (in == per - 1 || s == d.ks - 1) tc::commit(tc::smem_u32(&accf));
        }
        if (!ok) atomicExch(&abort_flag, 1);
        tc::commit(tc::smem_u32(&done));
    } else if (warp >= 2) {
        const int qw = warp & 3, r = mt * TM + qw * 32 + lane;
        const unsigned base = tmem + ((unsigned)(qw * 32) << 16);
        double acc[TN];
#pragma unroll
        for (int c = 0; c < TN; c++) acc[c] = 0.0;
        int ok = 1;
        for (int ck = 0; ck < n_chunks; ck++) {
            if (lane == 0) ok = tc::mbar_wait_or_abort(tc::smem_u32(&accf), ck & 1, &abort_flag) ? 1 : 0;
            ok = __shfl_sync(0xffffffffu, ok, 0);
            if (!ok) break;
            tc::fence_after();
#pragma unroll
            for (int c0 = 0; c0 < TN; c0 += 4) {
                unsigned v[NSL][4];
#pragma unroll
                for (int i = 0; i < NSL; i++) tmem_ld4(base + (unsigned)(i * TN + c0), v[i]);
                tc::tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 4; j++) acc[c0 + j] += join(v, j);
            }
            tc::fence_before();
            tc::mbar_arrive(tc::smem_u32(&acce));
        }
        unsigned long long exact = 0;
        if (ok) {
#pragma unroll
            for (int c0 = 0; c0 < TN; c0 += 4) {
                unsigned v[4];
                tmem_ld4(base + (unsigned)(NSL * TN + c0), v);
                tc::tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    const float S = __uint_as_float(v[j]);
                    if (S > 0.f && S < S_MIN) exact |= 1ull << (c0 + j);
                }
            }
        }
        if (!ok) {
            if (lane == 0) atomicExch(&abort_flag, 1);
        } else if (r < d.M) {
            int ch;
            const size_t row = g.mt.row(mat, ch);
            const double c = g.scal ? (ch == 0 ? 1.0 : 2.0) * g.scal[1] : 1.0;   // c_P = 1, c_C = 2, times the output scale
            double *o = reinterpret_cast<double *>(g.out + (g.scal ? row : (size_t)mat) * d.M * d.M + (size_t)r * d.M) + part;
            const unsigned ha = g.ea[(size_t)mat * d.M + r];
            unsigned top = 0;
#pragma unroll
            for (int j = 0; j < TN; j++) {
                const int n = nt * TN + j;
                if (n >= d.M) break;
                const unsigned hb = g.eb[(size_t)mat * d.M + n];
                if (ha >= 0x7ff00000u || hb >= 0x7ff00000u) exact |= 1ull << j;
                if ((exact >> j) & 1) continue;
                const int e = exp_of_hi(ha) + exp_of_hi(hb) - 68;   // value = sum 2^e
                const double v = e > -900 && e < 900 ? acc[j] * (c * __hiloint2double((e + 1023) << 20, 0)) : c * scalbn(acc[j], e);
                o[2 * n] = v;
                top = max(top, (unsigned)__double2hiint(v) & 0x7fffffffu);
            }
            if (part == 0) g.exact[((size_t)mat * d.M + r) * d.n_tiles + nt] = exact;
            if (g.rmax_out) atomicMax(g.rmax_out + (size_t)mat * d.M + r, top);
        }
    }
    __syncwarp();
    __syncthreads();
    if (tid == 32) (void)tc::mbar_wait(tc::smem_u32(&done), 0);   // bounded; the MMAs read shared memory
    if (tid == 0 && abort_flag) {
        atomicExch(g.err, 1);
        for (int b = 0; b < 2; b++)   // copies still in flight into this CTA's shared memory
            if (last_issued[b] >= 0) (void)tc::mbar_wait(tc::smem_u32(&full[b]), (last_issued[b] >> 1) & 1);
    }
    tc::fence_before();
    __syncthreads();
    if (warp == 0) {
        tc::fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
    }
}

// The entries that oz_gemm_kernel leaves out, summed in FP64: one CTA per row, its nonzero values of k in a list (all of
// them where a column holds an infinity or NaN, which zeros do not hide), lanes over the listed columns, the four warps over k.
constexpr int EX_WARPS = 4;
struct ExactArgs {
    const double2 *left, *right;   // left: the call's A (own_left = 0) or the chunk's T; right: the compact loops or A
    const int *dij;
    int own_left, nff, ns2, nd;
    GemmArgs g;
};
template <bool LOOP>
__global__ void __launch_bounds__(32 * EX_WARPS) oz_exact_kernel(const __grid_constant__ ExactArgs x)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const GemmArgs &g = x.g;
    const int M = g.d.M, r = blockIdx.x, mat = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned long long *words = g.exact + ((size_t)mat * M + r) * g.d.n_tiles;
    bool any = false;
    for (int t = tid; t < g.d.n_tiles; t += 32 * EX_WARPS) any |= words[t] != 0;
    if (!__syncthreads_or(any)) return;
    double2 *a = reinterpret_cast<double2 *>(smem);      // [M] the row's listed values
    int2 *at = reinterpret_cast<int2 *>(a + M);          // [M] places of their row of the right operand
    int *cols = reinterpret_cast<int *>(at + M);         // [M] the listed columns
    __shared__ int count[EX_WARPS];
    __shared__ double2 part[EX_WARPS][32];
    // place of this thread's element in a list that keeps the order of the threads; n: the list's length
    auto place = [&](bool in, int &n) {
        const unsigned b = __ballot_sync(0xffffffffu, in);
        if (lane == 0) count[warp] = __popc(b);
        __syncthreads();
        int p = n + __popc(b & ((1u << lane) - 1));
        for (int w = 0; w < EX_WARPS; w++) {
            if (w < warp) p += count[w];
            n += count[w];
        }
        __syncthreads();
        return p;
    };
    int n_cols = 0, n_k = 0;
    bool open = false;   // a listed column that is not finite
    for (int c0 = 0; c0 < M; c0 += 32 * EX_WARPS) {
        const int c = c0 + tid;
        const bool in = c < M && ((words[c / TN] >> (c % TN)) & 1);
        const int p = place(in, n_cols);
        if (in) cols[p] = c;
        open |= in && g.eb[(size_t)mat * M + c] >= 0x7ff00000u;
    }
    open = __syncthreads_or(open);
    int ch;
    const size_t row = g.mt.row(mat, ch);
    const double2 *left = x.left + ((x.own_left ? (size_t)mat : row) * M + r) * M;
    for (int k0 = 0; k0 < M; k0 += 32 * EX_WARPS) {
        const int k = k0 + tid;
        const double2 v = k < M ? left[k] : make_double2(0.0, 0.0);
        const bool in = k < M && (open || v.x != 0.0 || v.y != 0.0);
        const int p = place(in, n_k);
        if (in) {
            a[p] = v;
            at[p] = LOOP ? make_int2(k / x.ns2 * x.nff, k % x.ns2 * x.ns2) : make_int2(0, k * M);
        }
    }
    __syncthreads();
    const double2 *right = x.right + row * (LOOP ? (size_t)x.nd * x.ns2 * x.ns2 : (size_t)M * M);
    const double scale = g.scal ? (ch == 0 ? 1.0 : 2.0) * g.scal[1] : 1.0;
    double2 *out = g.out + ((g.scal ? row : (size_t)mat) * M + r) * M;
    unsigned top = 0;
    for (int c0 = 0; c0 < n_cols; c0 += 32) {
        const int c = cols[min(c0 + lane, n_cols - 1)], r2 = LOOP ? c / x.ns2 : 0, off = LOOP ? c % x.ns2 : c;
        double re = 0.0, im = 0.0;
#pragma unroll 4
        for (int i = warp; i < n_k; i += EX_WARPS) {
            const int2 p = at[i];
            const double2 u = a[i], v = right[LOOP ? (size_t)x.dij[p.x + r2] * x.ns2 * x.ns2 + p.y + off : (size_t)p.y + off];
            re = fma(-u.y, v.y, fma(u.x, v.x, re));
            im = fma(u.y, v.x, fma(u.x, v.y, im));
        }
        part[warp][lane] = make_double2(re, im);
        __syncthreads();
        if (warp == 0 && c0 + lane < n_cols) {
            double2 v = part[0][lane];
            for (int w = 1; w < EX_WARPS; w++) {
                v.x += part[w][lane].x;
                v.y += part[w][lane].y;
            }
            v.x *= scale;
            v.y *= scale;
            out[c] = v;
            top = max(top, mag_hi(v));
        }
        __syncthreads();
    }
    if (g.rmax_out && warp == 0 && top) atomicMax(g.rmax_out + (size_t)mat * M + r, top);
}

// scratch of one matrix of a chunk: T, left and right digits, the bits of the entries left to FP64 sums, row and column
// maxima of A, column maxima of L, row maxima of T
size_t mat_bytes(const Dims &d)
{
    return (size_t)d.M * d.M * sizeof(double2) + d.a_bytes() + d.b_bytes() +
           (size_t)d.M * (d.n_tiles * sizeof(unsigned long long) + 4 * sizeof(unsigned));
}

}  // namespace

// The scratch of a chunk of matrices, as many as fit 1 GiB and a sixteenth of the free memory (112 matrices of M = 324 fill
// the GPU many times over; the chunk does not change results), fewer where the allocation fails, one at least.
cudaError_t vlv64_alloc(tufrg_model *m)
{
    const size_t per = mat_bytes(dims_of(m->M));
    size_t free_bytes = 0, total = 0;
    TUFRG_CUDA_TRY(cudaMemGetInfo(&free_bytes, &total));
    size_t n = std::max<size_t>(1, std::min<size_t>((size_t)m->Nq, std::min(CHUNK_BYTES, free_bytes / 16) / per));
    cudaError_t e;
    while ((e = cudaMalloc(&m->d_oz, n * per)) == cudaErrorMemoryAllocation && n > 1) {
        (void)cudaGetLastError();
        n /= 2;
    }
    m->oz_mats = (int)n;
    return e;
}

cudaError_t launch_vlv64(tufrg_model *m, const double2 *d_A, int channel_mask, double2 *d_out, const int *qlist, int nlist)
{
    const int M = m->M, ns2 = m->ns * m->ns, nl = qlist ? nlist : m->Nq;
    const size_t M2 = (size_t)M * M;
    for (int ch = 0; ch < 2; ch++)
        if (!((channel_mask >> ch) & 1))
            TUFRG_CUDA_TRY(cudaMemsetAsync(d_out + (size_t)ch * m->Nq * M2, 0, sizeof(double2) * m->Nq * M2, m->stream));
    if (!(channel_mask & 3)) return cudaSuccess;
    const Dims d = dims_of(M);
    const int cap = m->oz_mats, total = nl * (channel_mask == 3 ? 2 : 1);
    double2 *T = static_cast<double2 *>(m->d_oz);
    unsigned char *pa = reinterpret_cast<unsigned char *>(T + (size_t)cap * M2), *pb = pa + (size_t)cap * d.a_bytes();
    unsigned long long *ex = reinterpret_cast<unsigned long long *>(pb + (size_t)cap * d.b_bytes());
    unsigned *mx = reinterpret_cast<unsigned *>(ex + (size_t)cap * M * d.n_tiles);
    unsigned *ra = mx, *ca = ra + (size_t)cap * M, *cl = ca + (size_t)cap * M, *rt = cl + (size_t)cap * M;
    const size_t smem = 2 * (size_t)STAGE;
    TUFRG_CUDA_TRY(cudaFuncSetAttribute(oz_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    for (int m0 = 0; m0 < total; m0 += cap) {
        const int n = std::min(cap, total - m0);
        const Mats mt{qlist, nl, m->Nq, (channel_mask & 1) ? 0 : 1, m0};
        PhaseScope ps(m, PH_VLV, 10);
        TUFRG_CUDA_TRY(cudaMemsetAsync(mx, 0, 4 * (size_t)cap * M * sizeof(unsigned), m->stream));
        oz_scale_kernel<<<dim3((M + 31) / 32, n), 256, sizeof(unsigned) * M, m->stream>>>(d_A, mt, M, ra, ca);
        oz_scale_loop_kernel<<<dim3((M + 127) / 128, 4, n), 128, 0, m->stream>>>(m->d_Lc, m->d_dij, mt, M, m->nff, ns2, m->nd, cl);
        oz_left_kernel<false><<<dim3(d.m_tiles * d.ks * 2, n), TM, 0, m->stream>>>(d_A, mt, d, ra, pa);
        const dim3 gr((d.n_tiles * TN + 127) / 128 * d.ks * 2, n), rows(M, n);
        const size_t ex_smem = (size_t)M * (sizeof(double2) + sizeof(int2) + sizeof(int));
        oz_right_kernel<true><<<gr, 128, 0, m->stream>>>(m->d_Lc, m->d_dij, m->nff, ns2, m->nd, mt, d, cl, pb);
        GemmArgs g{pa, pb, ra, cl, T, rt, ex, mt, d, nullptr, m->d_err};
        const unsigned tiles = (unsigned)((size_t)n * d.m_tiles * d.n_tiles * 2);   // two parts
        oz_gemm_kernel<<<tiles, NTHREADS, smem, m->stream>>>(g);
        oz_exact_kernel<true><<<rows, 32 * EX_WARPS, ex_smem, m->stream>>>(ExactArgs{d_A, m->d_Lc, m->d_dij, 0, m->nff, ns2, m->nd, g});
        oz_left_kernel<true><<<dim3(d.m_tiles * d.ks * 2, n), TM, 0, m->stream>>>(T, mt, d, rt, pa);
        oz_right_kernel<false><<<gr, 128, 0, m->stream>>>(d_A, nullptr, 0, 1, 0, mt, d, ca, pb);
        g = GemmArgs{pa, pb, rt, ca, d_out, nullptr, ex, mt, d, m->d_scal, m->d_err};
        oz_gemm_kernel<<<tiles, NTHREADS, smem, m->stream>>>(g);
        oz_exact_kernel<false><<<rows, 32 * EX_WARPS, ex_smem, m->stream>>>(ExactArgs{T, d_A, nullptr, 1, 0, 1, 0, g});
        TUFRG_CUDA_TRY(cudaGetLastError());
    }
    return cudaSuccess;
}

}  // namespace tufrg
