// Tensor-core V.L.V products for the split path: dX/dT(q) = c_X A(q) L(q) A(q) (Eq. RGE_spin and the
// orbital form of Eq. rge_Dmat) on 5th-generation tensor cores (tcgen05, sm_103a).
//
// Two persistent launches per right-hand side, each over the work list (channel, momentum, 128-row tile, NB-column
// tile) of every requested channel and momentum:
//   first:   T = A L    with L[k][n] gathered from the compact loops through the bond-pair table, FP32 scratch;
//   second:  dX = c T A in FP64 (exact widening on the integer pipe).
// Complex GEMM as two real MMA streams into one tensor-memory accumulator [Cr | Ci] of twice the columns:
//   [Cr | Ci] += Ar [Br | Bi],   [Cr | Ci] += Ai [-Bi | Br];
// the right operand is stored as [-Bi | Br | Bi], whose two windows are the two right-hand factors.  An MMA of 128 x N x 8
// takes about 34 cycles plus half a cycle per column, so half as many of twice the width are faster than four streams
// into two accumulators.
// Both products of 225 momenta, two channels, M = 324: 1.45 ms with four streams, one row per lane and a shared-memory
// tile for the epilogue; 1.15 ms now (its MMAs alone about 0.95 ms, its producers alone 0.88 ms).  The tensor pipe is busy
// 78% of the cycles in the first product and 62% in the second, which writes FP64 (45 representatives).
// Precision: 3xTF32 - every FP32 operand x is split into hi = x with the 13 low mantissa bits cleared and lo = x - hi
// (exact), and each real product is hi*hi + hi*lo + lo*hi accumulated in FP32 in tensor memory.
//
// The operands are read in FP32 straight from the matrices and split inside the kernel (no packing launches).  Warp
// roles of the 640-thread CTA (one per SM):
//   warps 0-15  producers, two groups of eight that take the K stages of 16 columns in turn (the waits, fences and
//               arrivals of a stage are paid half as often per warp): each thread loads 8 complex values of the left
//               operand and 8 of the right operand of its group's next stage into registers while it splits the
//               current one.  Left operand: warp (quarter w % 4 of the rows, columns 8 (w / 4 % 2)), a thread two
//               neighbouring columns of rows lane / 4 + 8 i, so that a load covers 64 contiguous bytes of 8 rows (one
//               row per lane, 32 lines per load, kept the L1 tags busy for half of a stage); its four TF32 planes
//               (Re hi, Re lo, Im hi, Im lo) go to tensor memory (tcgen05.st 16x256b: that same arrangement).  Right
//               operand: thread (K half, column tid % 128), to shared memory in the K-major core-matrix layout;
//   warp 16     tensor-memory allocation and the MMA issuer (one thread): 12 MMAs per stage (2 K-steps x 2 real
//               streams x 3 TF32 passes), the left operand read from tensor memory; then its quarter of the
//               epilogue (20 warps leave every thread 96 registers, 21 would leave 80);
//   warps 16-19 epilogue: tensor memory (16x256b: a thread holds two neighbouring columns of a row, four threads 8)
//               -> T (FP32) or c dX (FP64, one 32-byte store per thread) in global memory.
// Four stage buffers (mbarriers full / empty), one accumulator (mbarriers accf / acce).  Every wait is
// bounded; on time-out the kernel raises the error flag, every role stops, the MMAs in flight are waited for
// (bounded) and the tensor memory is freed.
#include "tc_common.cuh"
#include "tufrg_internal.cuh"

namespace tufrg {
namespace {

constexpr int TM = 128;             // MMA M: rows per tile
constexpr int KS = 16;              // K per stage (two MMA K-steps of 8)
constexpr int NSTAGE = 4;           // stage buffers (a multiple of the producer groups: each buffer belongs to one)
constexpr int NPROD = 512;          // producer threads (warps 0-15)
constexpr int MMA_WARP = 16;        // it and warps 17-19: epilogue
constexpr int NTHREADS = 20 * 32;
constexpr int NB_MAX = 112;         // columns per tile (complex), a multiple of 16
// tensor memory: accumulator Re at [0, NB), Im at [NB, 2 NB); left operand of stage b at 256 + 64 b, plane p at + 16 p
// (K = 16 columns)
constexpr unsigned A_COL0 = 256, A_STAGE_COLS = 64, A_PLANE_COLS = 16;
constexpr unsigned TMEM_COLS = 512;
static_assert(A_COL0 + NSTAGE * A_STAGE_COLS <= TMEM_COLS, "tensor memory budget");

struct Dims {
    int M;          // complex matrix order (a multiple of 4)
    int nks;        // K stages covering M
    int nb;         // complex columns per tile (multiple of 16, <= 112)
    int m_tiles;    // 128-row tiles covering M
    int n_tiles;    // nb-column tiles covering M
};

// n_tiles column tiles (0: the fewest that keep NB <= 112), NB the smallest multiple of 16 covering M with them
Dims dims_of(int M, int n_tiles)
{
    Dims d{};
    d.M = M;
    d.nks = (M + KS - 1) / KS;
    d.m_tiles = (M + TM - 1) / TM;
    d.n_tiles = std::max(n_tiles, (M + NB_MAX - 1) / NB_MAX);
    d.nb = ((M + d.n_tiles - 1) / d.n_tiles + 15) / 16 * 16;
    return d;
}

struct VlvArgs {
    const float2 *A;        // [2][Nq][M][M] projections (FP32, row-major)
    const float2 *Lc;       // [2][Nq][lper] compact loops (first product)
    const int *dij;         // [nff][nff] bond pair -> bond-difference index of the compact loops
    float2 *T;              // [2][nz][M][M] first product (written by the first launch, read by the second)
    double2 *out;           // [2][Nq][M][M] second product
    int out32B;             // out lies on a 32-byte boundary
    const int *qlist;       // slot z -> transfer momentum (null: the slot is the momentum)
    const double *scal;     // scal[1]: the flow-scale factor of the right-hand side
    int *err;
    Dims d;
    int nff, lper, Nq, nz;
    int ch0, nch;           // channels ch0 .. ch0 + nch - 1
    int n_items;
};

// the stage's values of one producer thread: left-operand rows ra + 8 i at two K (a[2 i], a[2 i + 1]), and right-operand
// row r (an output column) at eight K
struct Vals {
    float2 a[8], b[8];
};

// one producer thread's sources for one item: the left operand's row (A in the first product, T in the second) and
// the right operand's column (the compact loops of the momentum, or A), null when the row / column is padding
struct Src {
    const float2 *a;    // row ra of the left operand
    int rows;           // rows from ra on that exist
    const float2 *b;    // first product: the momentum's compact loops + (n % NS2); second: column n of A
    int nj;             // first product: n / NS2 (the column's bond index)
};

template <int PH, int NS2>
__device__ __forceinline__ Src item_src(const VlvArgs &p, int ch, int z, int mt, int nt, int ra, int r)
{
    const int M = p.d.M, n = nt * p.d.nb + r;
    const size_t M2 = (size_t)M * M;
    const int qs = p.qlist ? p.qlist[z] : z;
    Src s{};
    const int m = mt * TM + ra;
    s.a = (PH == 0 ? p.A + ((size_t)ch * p.Nq + qs) * M2 : p.T + ((size_t)ch * p.nz + z) * M2) + (size_t)m * M;
    s.rows = M - m;
    if (r < p.d.nb && n < M) {
        if (PH == 0) {
            s.b = p.Lc + ((size_t)ch * p.Nq + qs) * p.lper + n % NS2;
            s.nj = n / NS2;
        } else {
            s.b = p.A + ((size_t)ch * p.Nq + qs) * M2 + n;
        }
    }
    return s;
}

// K = ka, ka + 1 of the left operand (ka even, M a multiple of 4) and k0 .. k0 + 7 of the right operand (k0 a multiple
// of 4; M and NS2 are multiples of 4, so each four of them lie in one bond block)
template <int PH, int NS2>
__device__ __forceinline__ void load_stage(const Src &src, const int *sdij, int nff, int M, int ka, int k0, Vals &v)
{
#pragma unroll
    for (int i = 0; i < 4; i++) {
        float4 u = make_float4(0.f, 0.f, 0.f, 0.f);
        if (8 * i < src.rows && ka < M) u = __ldg(reinterpret_cast<const float4 *>(src.a + (size_t)(8 * i) * M + ka));
        v.a[2 * i] = make_float2(u.x, u.y);
        v.a[2 * i + 1] = make_float2(u.z, u.w);
    }
#pragma unroll
    for (int i = 0; i < 8; i += 4) {
        const int k = k0 + i;
        if (src.b && k < M) {
            if (PH == 0) {
                // L[k][n] = Lc[(d(k / NS2, n / NS2) NS2 + k % NS2) NS2 + n % NS2]
                const float2 *b = src.b + ((size_t)sdij[(k / NS2) * nff + src.nj] * NS2 + k % NS2) * NS2;
#pragma unroll
                for (int j = 0; j < 4; j++) v.b[i + j] = __ldg(b + j * NS2);
            } else {
                const float2 *b = src.b + (size_t)k * M;
#pragma unroll
                for (int j = 0; j < 4; j++) v.b[i + j] = __ldg(b + (size_t)j * M);
            }
        } else {
#pragma unroll
            for (int j = 0; j < 4; j++) v.b[i + j] = make_float2(0.f, 0.f);
        }
    }
}

// exact FP32 -> FP64 by the two formats' bit layouts with selects only (the library's widen_f also handles
// subnormals, through a call that costs the epilogue's store loop its throughput); FP32 subnormals become signed
// zeros here (products below 1.2e-38 in magnitude)
__device__ __forceinline__ double f32_to_f64(float x)
{
    const unsigned u = __float_as_uint(x), e = (u >> 23) & 0xffu, sign = u & 0x80000000u;
    const unsigned e64 = e == 0xffu ? 0x7ffu : e + 896u;
    const unsigned hi = e == 0 ? sign : sign | (e64 << 20) | ((u & 0x7fffffu) >> 3);
    const unsigned lo = e == 0 ? 0u : u << 29;
    return __hiloint2double((int)hi, (int)lo);
}

// two neighbouring entries: one 32-byte store where the output starts on a 32-byte boundary (its rows then do)
__device__ __forceinline__ void store_pair(double2 *o, int aligned32, double a, double b, double c, double d)
{
    if (aligned32) {
        asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(o), "d"(a), "d"(b), "d"(c), "d"(d) : "memory");
    } else {
        o[0] = make_double2(a, b);
        o[1] = make_double2(c, d);
    }
}

__device__ __forceinline__ float tf32_trunc(float x) { return __uint_as_float(__float_as_uint(x) & 0xffffe000u); }

template <int PH, int NS2>
__global__ void __launch_bounds__(NTHREADS, 1) vlv_tc_kernel(VlvArgs p)
{
    // dynamic shared memory: NSTAGE right-operand stages, the bond table
    extern __shared__ __align__(1024) unsigned char smem[];
    const int NB = p.d.nb, nks = p.d.nks;
    const unsigned b_plane = 3u * NB * KS * 4, b_stage = 2 * b_plane;   // bytes; planes hi, lo of [-Bi | Br | Bi]
    int *sdij = reinterpret_cast<int *>(smem + NSTAGE * (size_t)b_stage);
    __shared__ __align__(8) unsigned long long full[NSTAGE], empty[NSTAGE], accf, acce, done;
    __shared__ unsigned tmem_base;
    __shared__ int abort_flag;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (warp == MMA_WARP) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc::smem_u32(&tmem_base)),
                     "r"(TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int b = 0; b < NSTAGE; b++) {
            tc::mbar_init(tc::smem_u32(&full[b]), NPROD / 2);
            tc::mbar_init(tc::smem_u32(&empty[b]), 1);
        }
        tc::mbar_init(tc::smem_u32(&accf), 1);
        tc::mbar_init(tc::smem_u32(&acce), 96);   // (warp 16 itself issues the next MMAs)
        tc::mbar_init(tc::smem_u32(&done), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        abort_flag = 0;
    }
    if (PH == 0)
        for (int i = tid; i < p.nff * p.nff; i += NTHREADS) sdij[i] = p.dij[i];
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const unsigned tmem = tmem_base;
    const int G = (int)gridDim.x;
    const int my_items = p.n_items > (int)blockIdx.x ? (p.n_items - 1 - (int)blockIdx.x) / G + 1 : 0;
    // item -> (channel, slot, row tile, column tile); column tiles fastest so that neighbouring CTAs share rows
    auto decode = [&](int item, int &ch, int &z, int &mt, int &nt) {
        nt = item % p.d.n_tiles;
        int t = item / p.d.n_tiles;
        mt = t % p.d.m_tiles;
        t /= p.d.m_tiles;
        z = t % p.nz;
        ch = p.ch0 + t / p.nz;
    };

    if (warp < MMA_WARP) {
        // ------------------------------------------------------------------ producers
        const int grp = warp >> 3, r = tid & 127, kh = (tid >> 7) & 1;
        // left operand: the 32 rows of the warp's quarter, columns 8 kh of the stage
        const int ra = (warp & 3) * 32 + (lane >> 2), ca0 = 8 * kh + 2 * (lane & 3);
        const unsigned a_base = ((unsigned)((warp & 3) * 32) << 16) + A_COL0 + (unsigned)(8 * kh);
        const int n_stages = my_items * nks;
        const int M = p.d.M, nff = p.nff;
        int li = 0, st = grp;   // item (local index) and its stage of the loads in flight
        Src src;
        auto settle = [&]() {   // the item that stage st of item li falls into
            while (st >= nks) {
                st -= nks;
                li++;
            }
        };
        auto locate = [&]() {
            int ch, z, mt, nt;
            decode((int)blockIdx.x + li * G, ch, z, mt, nt);
            src = item_src<PH, NS2>(p, ch, z, mt, nt, ra, r);
        };
        Vals cur, nxt;
        settle();
        if (grp < n_stages) {
            locate();
            load_stage<PH, NS2>(src, sdij, nff, M, st * KS + ca0, st * KS + 8 * kh, nxt);
        }
        for (int n = grp; n < n_stages; n += 2) {
            cur = nxt;
            // issue the loads of the group's next stage (they land while this stage is split and stored)
            if (n + 2 < n_stages) {
                const int before = li;
                st += 2;
                settle();
                if (li != before) locate();
                load_stage<PH, NS2>(src, sdij, nff, M, st * KS + ca0, st * KS + 8 * kh, nxt);
            }
            const int b = n % NSTAGE;
            // the MMAs that read this stage buffer NSTAGE stages ago must be complete
            int ok = 1;
            if (lane == 0) {
                if (*(volatile int *)&abort_flag) ok = 0;
                else if (n >= NSTAGE) ok = tc::mbar_wait_or_abort(tc::smem_u32(&empty[b]), ((n / NSTAGE) - 1) & 1, &abort_flag) ? 1 : 0;
            }
            ok = __shfl_sync(0xffffffffu, ok, 0);
            if (!ok) {
                if (lane == 0) {
                    atomicExch(&abort_flag, 1);
                    atomicExch(p.err, 1);
                }
                break;   // the whole warp leaves (the MMA thread's waits then run out or see the flag)
            }
            tc::fence_after();
            // left operand: four planes x two blocks of 16 rows x 8 columns into tensor memory
            const unsigned ca = tmem + a_base + b * A_STAGE_COLS;
#pragma unroll
            for (int g = 0; g < 2; g++) {
                const unsigned cg = ca + ((unsigned)(16 * g) << 16);
                float h[4], l[4];
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    h[j] = tf32_trunc(cur.a[4 * g + j].x);
                    l[j] = cur.a[4 * g + j].x - h[j];
                }
                tc::tmem_st_16x8(cg + 0 * A_PLANE_COLS, h[0], h[1], h[2], h[3]);
                tc::tmem_st_16x8(cg + 1 * A_PLANE_COLS, l[0], l[1], l[2], l[3]);
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    h[j] = tf32_trunc(cur.a[4 * g + j].y);
                    l[j] = cur.a[4 * g + j].y - h[j];
                }
                tc::tmem_st_16x8(cg + 2 * A_PLANE_COLS, h[0], h[1], h[2], h[3]);
                tc::tmem_st_16x8(cg + 3 * A_PLANE_COLS, l[0], l[1], l[2], l[3]);
            }
            // right operand: row r of the stage's four planes in shared memory
            if (r < NB) {
                float *pb = reinterpret_cast<float *>(smem + (size_t)b * b_stage);
#pragma unroll
                for (int i = 0; i < 8; i += 4) {
                    const int o = tc::core_off(r, 8 * kh + i, 3 * NB), bo = NB * 4;   // (rows + NB: 4 NB floats on)
                    const float2 *v = cur.b + i;
                    float4 hv, lv;
                    hv = make_float4(tf32_trunc(v[0].x), tf32_trunc(v[1].x), tf32_trunc(v[2].x), tf32_trunc(v[3].x));
                    lv = make_float4(v[0].x - hv.x, v[1].x - hv.y, v[2].x - hv.z, v[3].x - hv.w);
                    *reinterpret_cast<float4 *>(pb + o + bo) = hv;
                    *reinterpret_cast<float4 *>(pb + b_plane / 4 + o + bo) = lv;
                    hv = make_float4(tf32_trunc(v[0].y), tf32_trunc(v[1].y), tf32_trunc(v[2].y), tf32_trunc(v[3].y));
                    lv = make_float4(v[0].y - hv.x, v[1].y - hv.y, v[2].y - hv.z, v[3].y - hv.w);
                    *reinterpret_cast<float4 *>(pb + o + 2 * bo) = hv;
                    *reinterpret_cast<float4 *>(pb + b_plane / 4 + o + 2 * bo) = lv;
                    *reinterpret_cast<float4 *>(pb + o) = make_float4(-hv.x, -hv.y, -hv.z, -hv.w);
                    *reinterpret_cast<float4 *>(pb + b_plane / 4 + o) = make_float4(-lv.x, -lv.y, -lv.z, -lv.w);
                }
            }
            tc::tmem_wait_st();
            tc::fence_smem_async();
            tc::fence_before();
            tc::mbar_arrive(tc::smem_u32(&full[b]));
        }
    } else {
        // ------------------------------------------------------------------ MMA issuer (warp 16) and epilogue
        const int qw = warp & 3, M = p.d.M;
        const unsigned lane_off = (unsigned)(qw * 32) << 16;
        const size_t M2 = (size_t)M * M;
        const unsigned id = tc::idesc_tf32(TM, 2 * NB, false);
        int n = 0;
        // a wait of the warp's first lane, its outcome for the whole warp
        auto wait_all = [&](unsigned long long *bar, int parity) {
            int ok = 1;
            if (lane == 0) ok = tc::mbar_wait_or_abort(tc::smem_u32(bar), parity, &abort_flag) ? 1 : 0;
            return __shfl_sync(0xffffffffu, ok, 0) != 0;
        };
        bool ok = true;
        for (int it = 0; it < my_items; it++) {
            if (warp == MMA_WARP) {
                int issued = 1;
                // the accumulator must have been read by the other warps' epilogue of the previous item
                if (lane == 0) {
                    if (it >= 1 && !tc::mbar_wait_or_abort(tc::smem_u32(&acce), (it - 1) & 1, &abort_flag)) issued = 0;
                    tc::fence_after();
                    for (int s = 0; s < nks && issued; s++, n++) {
                        const int b = n % NSTAGE;
                        if (!tc::mbar_wait_or_abort(tc::smem_u32(&full[b]), (n / NSTAGE) & 1, &abort_flag)) { issued = 0; break; }
                        tc::fence_after();
                        const unsigned sb = tc::smem_u32(smem + (size_t)b * b_stage), ta = tmem + A_COL0 + b * A_STAGE_COLS;
#pragma unroll
                        for (int kk = 0; kk < KS / 8; kk++) {
                            const unsigned bo = sb + kk * 2 * (3 * NB / 8) * 128, win = (NB / 8) * 128;   // [-Bi | Br], [Br | Bi] at + win
                            const unsigned arh = ta + 0 * A_PLANE_COLS + 8 * kk, arl = ta + 1 * A_PLANE_COLS + 8 * kk;
                            const unsigned aih = ta + 2 * A_PLANE_COLS + 8 * kk, ail = ta + 3 * A_PLANE_COLS + 8 * kk;
                            const unsigned long long rh = tc::smem_desc(bo + win, 3 * NB), rl = tc::smem_desc(bo + b_plane + win, 3 * NB);
                            const unsigned long long ih = tc::smem_desc(bo, 3 * NB), il = tc::smem_desc(bo + b_plane, 3 * NB);
                            const unsigned first = (s == 0 && kk == 0) ? 0u : 1u;
                            tc::mma_tf32_ta(tmem, arh, rh, id, first); tc::mma_tf32_ta(tmem, arh, rl, id, 1u); tc::mma_tf32_ta(tmem, arl, rh, id, 1u);
                            tc::mma_tf32_ta(tmem, aih, ih, id, 1u);    tc::mma_tf32_ta(tmem, aih, il, id, 1u); tc::mma_tf32_ta(tmem, ail, ih, id, 1u);
                        }
                        tc::commit(tc::smem_u32(&empty[b]));
                    }
                    if (issued) tc::commit(tc::smem_u32(&accf));
                }
                ok = __shfl_sync(0xffffffffu, issued, 0) != 0;
                if (!ok) break;
            }
            // the item's MMAs are complete
            ok = wait_all(&accf, it & 1);
            if (!ok) break;
            tc::fence_after();
            int ch, z, mt, nt;
            decode((int)blockIdx.x + it * G, ch, z, mt, nt);
            const int qs = p.qlist ? p.qlist[z] : z;
            const int n0 = nt * NB, m0 = mt * TM + qw * 32 + (lane >> 2), cl = n0 + 2 * (lane & 3);
            const int nlim = min(n0 + NB, M);
            // c_X times the flow-scale factor, applied in FP32 (the products carry FP32 accuracy)
            const float c = PH == 1 ? (float)((ch == 0 ? 1.0 : 2.0) * (p.scal ? p.scal[1] : 1.0)) : 1.f;
            float2 *dT = p.T + ((size_t)ch * p.nz + z) * M2;
            double2 *dX = p.out + ((size_t)ch * p.Nq + qs) * M2;
            for (int c0 = 0; c0 < NB; c0 += 8) {
                unsigned vr[2][4], vi[2][4];   // rows lane / 4 + 16 g (0, 1) and + 8 (2, 3), two columns each
#pragma unroll
                for (int g = 0; g < 2; g++) {
                    tc::tmem_ld_16x8(tmem + lane_off + ((unsigned)(16 * g) << 16) + (unsigned)c0, vr[g]);
                    tc::tmem_ld_16x8(tmem + lane_off + ((unsigned)(16 * g) << 16) + (unsigned)(NB + c0), vi[g]);
                }
                tc::tmem_wait_ld();
                const int n = cl + c0;   // (even, as is M: the second column exists with the first)
#pragma unroll
                for (int g = 0; g < 4; g++) {
                    const int m = m0 + 8 * g, h = 2 * (g & 1);
                    if (n >= nlim || m >= M) continue;
                    const float r0 = __uint_as_float(vr[g >> 1][h]), r1 = __uint_as_float(vr[g >> 1][h + 1]);
                    const float i0 = __uint_as_float(vi[g >> 1][h]), i1 = __uint_as_float(vi[g >> 1][h + 1]);
                    const size_t o = (size_t)m * M + n;
                    if (PH == 0) *reinterpret_cast<float4 *>(dT + o) = make_float4(r0, i0, r1, i1);
                    else store_pair(dX + o, p.out32B, f32_to_f64(c * r0), f32_to_f64(c * i0), f32_to_f64(c * r1), f32_to_f64(c * i1));
                }
                __syncwarp();   // (the loads are warp-collective)
            }
            tc::fence_before();
            if (warp == MMA_WARP) __syncwarp();   // (its own reads are complete before it issues the next item's MMAs)
            else tc::mbar_arrive(tc::smem_u32(&acce));
        }
        if (!ok && lane == 0) {
            atomicExch(&abort_flag, 1);
            atomicExch(p.err, 1);
        }
        if (warp == MMA_WARP && lane == 0) tc::commit(tc::smem_u32(&done));   // completion of every MMA issued above
        __syncwarp();
    }
    __syncthreads();
    if (tid == MMA_WARP * 32) (void)tc::mbar_wait(tc::smem_u32(&done), 0);   // bounded; the MMAs read shared memory
    tc::fence_before();
    __syncthreads();
    if (warp == MMA_WARP) {
        tc::fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    }
}

template <int PH>
cudaError_t launch_phase(tufrg_model *m, const VlvArgs &a)
{
    const size_t smem = NSTAGE * 6 * (size_t)a.d.nb * KS * 4 + sizeof(int) * (size_t)a.nff * a.nff;
    void (*k)(VlvArgs) = nullptr;
    switch (m->ns * m->ns) {
    case 4: k = vlv_tc_kernel<PH, 4>; break;
    case 16: k = vlv_tc_kernel<PH, 16>; break;
    case 36: k = vlv_tc_kernel<PH, 36>; break;
    default: return cudaErrorInvalidValue;
    }
    TUFRG_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    k<<<std::min(a.n_items, m->sm_count), NTHREADS, smem, m->stream>>>(a);
    return cudaGetLastError();
}

}  // namespace

// the column-tile counts the products autotuner times: the fewest (widest tiles) and one more; the second only when it
// changes the tile width and keeps it at least 16
std::vector<int> tc_tile_candidates(const tufrg_model *m)
{
    const Dims a = dims_of(m->M, 0), b = dims_of(m->M, a.n_tiles + 1);
    std::vector<int> v{a.n_tiles};
    if (b.nb != a.nb && b.nb >= 16) v.push_back(b.n_tiles);
    return v;
}

int tc_tile_width(const tufrg_model *m) { return dims_of(m->M, m->tc_ntiles).nb; }

bool tc_supported(const tufrg_model *m)
{
    const int ns2 = m->ns * m->ns;
    return m->precision == TUFRG_SPLIT32 && m->products == TUFRG_PRODUCTS_TC && (ns2 == 4 || ns2 == 16 || ns2 == 36) &&
           m->M % 4 == 0;
}

cudaError_t launch_vlv_tc(tufrg_model *m, int channel_mask, double2 *d_out, const int *qlist, int nlist)
{
    if (!m->d_T) return cudaErrorNotReady;
    const int M = m->M, ns2 = m->ns * m->ns;
    const size_t M2 = (size_t)M * M;
    PhaseScope ps(m, PH_VLV, 2);
    for (int ch = 0; ch < 2; ch++)
        if (!((channel_mask >> ch) & 1))
            TUFRG_CUDA_TRY(cudaMemsetAsync(d_out + (size_t)ch * m->Nq * M2, 0, sizeof(double2) * m->Nq * M2, m->stream));
    if (!(channel_mask & 3)) return cudaSuccess;
    VlvArgs a{};
    a.A = m->d_A32;
    a.Lc = m->d_Lc32;
    a.dij = m->d_dij;
    a.T = reinterpret_cast<float2 *>(m->d_T);
    a.out = d_out;
    a.out32B = (reinterpret_cast<uintptr_t>(d_out) & 31) == 0;
    a.qlist = qlist;
    a.scal = m->d_scal;
    a.err = m->d_err;
    a.d = dims_of(M, m->tc_ntiles);
    a.nff = m->nff;
    a.lper = m->nd * ns2 * ns2;
    a.Nq = m->Nq;
    a.nz = qlist ? nlist : m->Nq;
    a.ch0 = (channel_mask & 1) ? 0 : 1;
    a.nch = (channel_mask & 3) == 3 ? 2 : 1;
    a.n_items = a.nch * a.nz * a.d.m_tiles * a.d.n_tiles;
    if (a.n_items == 0) return cudaSuccess;
    TUFRG_CUDA_TRY(launch_phase<0>(m, a));
    return launch_phase<1>(m, a);
}

}  // namespace tufrg
