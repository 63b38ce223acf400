// Tensor-core GEMMs of the loop surrogate's network (5th-generation tensor cores, tcgen05, sm_103a).
//
//   C[M][N] = op(A)[M][K] op(B)[K][N] (+ bias[N]),  FP32 accumulation in tensor memory.
//
// Training passes multiply BF16 activations by BF16 weights: kind::f16 with BF16 operands, one MMA per K-step.
// Inference keeps the activations in FP32: kind::tf32, the activations split into a TF32 part and its FP32
// remainder (a = hi + lo exactly), the BF16 weights exact in TF32, two MMAs per K-step (hi B + lo B), which keeps
// the products at FP32 accuracy.  Operands (either orientation, any size) are first packed into the K-major,
// no-swizzle core-matrix layout of the MMA, zero-padded to whole tiles, so that one pipeline stage of one operand
// is one contiguous block: [tile][K stage][plane][rows x stage K].
//
// A pass over this network (1024 x 256-wide layers) is a chain of small dependent steps, so launches and their gaps
// count as much as the arithmetic.  Each layer is two launches: one packs every operand of the layer, forming the
// element-wise functions on the way (GELU of the previous pre-activations, dZ = dA GELU'(Z), the loss gradient
// 2 (Y - T) / n, and the partial sums of the bias gradients and of the loss), one runs the layer's GEMMs (backward: the
// weight and the input gradient together).   One training
// step's gradients at batch 1024 (20 -> 4 x 256 -> 1600): 195 us (4.0 ms with one kernel per function, a
// one-block loss and one thread per bias column).
//
// The GEMM kernel (one CTA = 128 rows x NB columns, NB chosen so that the tiles cover the GPU) runs a bulk-copy pipeline
// of up to four stages (thread 0 issues the copies with mbarrier transaction counts, thread 32 the MMAs, committed to
// the stage's "empty" barrier); the epilogue reads the accumulator from tensor
// memory (lane = row) and writes C with the bias.  The K order of an output element's sum does not depend on the tiles
// or stages.  Every wait is bounded: on time-out the kernel raises the error
// flag, waits (bounded) for its MMAs and its copies, frees its tensor memory and returns.
#include <cuda_bf16.h>

#include <algorithm>

#include "tc_common.cuh"
#include "mlp.cuh"
#include "tufrg_internal.cuh"

namespace tufrg {
namespace {

constexpr int MT = 128;         // rows per CTA (MMA M)
constexpr int NMAX = 256;       // largest N tile
constexpr int NMIN = 32;        // smallest N tile worth a CTA
constexpr int MAXST = 4;        // pipeline stages
constexpr int KS_BYTES = 128;   // stage K in bytes per row: 64 BF16 or 32 FP32 values (8 core matrices)

template <int KIND> struct Kind;
template <> struct Kind<0> {   // BF16 x BF16 (kind::f16)
    using T = __nv_bfloat16;
    static constexpr int ELEM = 2, KSTEP = 16, A_PLANES = 1;
};
template <> struct Kind<1> {   // (FP32 hi + lo) x BF16-in-FP32 (kind::tf32)
    using T = float;
    static constexpr int ELEM = 4, KSTEP = 8, A_PLANES = 2;
};

struct Dims {
    int M, N, K;
    int m_tiles, n_tiles, nb, nks;   // nb: columns per N tile (multiple of 16), nks: K stages
};

__device__ __forceinline__ float gelu(float x) { return 0.5f * x * (1.f + erff(x * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_d(float x)
{
    return 0.5f * (1.f + erff(x * 0.70710678118654752f)) + x * 0.39894228040143268f * expf(-0.5f * x * x);
}

// value of an operand's source from its buffers' elements
__device__ __forceinline__ float src_value(const MlpSrc &s, float a, float b)
{
    switch (s.mode) {
    case MLP_GELU: return gelu(a);
    case MLP_DGELU: return a * gelu_d(b);
    case MLP_MSE: return 2.f * (a - b) * s.scale;
    default: return a;   // MLP_F32, MLP_BF16
    }
}
__device__ __forceinline__ float src_a(const MlpSrc &s, size_t i)
{
    return s.mode == MLP_BF16 ? __bfloat162float(static_cast<const __nv_bfloat16 *>(s.S)[i]) : static_cast<const float *>(s.S)[i];
}

struct PackJob {
    MlpSrc src;
    int rows, K, R, tiles, nks, planes;
    int vec;            // contiguous FP32 chunks on 16-byte boundaries
    void *dst;
    unsigned blocks;
};
constexpr int SUM_ROWS = 16;    // rows per partial column sum
struct PackJobs {
    PackJob job[4];
    int n;
    MlpSrc sum;                 // column sums of this source, rows x cols (blocks past the packing ones), or mode < 0
    int sum_rows, sum_cols;
    float *sum_part;            // [rows / SUM_ROWS][cols]
    double *loss_part;          // [rows / SUM_ROWS][cols / 256] partial sums of (Y - T)^2 (MLP_MSE)
    const int *skip;
};

// Packs op(S) (rows x K, element (r, k) = S[r * ld + k], or S[k * ld + r] when transposed) into tiles of R rows:
// dst [tile][stage][plane][R x stage K] in the core-matrix layout; planes: the value (BF16 or FP32), or for an
// FP32 split operand its TF32 part and remainder.  One thread per 16-byte chunk (8 BF16 or 4 FP32 values); consecutive
// threads take consecutive chunks along K, or consecutive rows of a transposed source, so that their reads are
// coalesced.  The blocks past the jobs' add SUM_ROWS rows of a column per thread.
template <typename TD>
__global__ void __launch_bounds__(256) pack_kernel(const __grid_constant__ PackJobs a)
{
    grid_release();
    grid_wait();
    if (a.skip && *a.skip) return;
    constexpr int EPC = 16 / (int)sizeof(TD);                  // elements per chunk
    constexpr int KSE = KS_BYTES / (int)sizeof(TD);            // stage K in elements
    constexpr int CPR = KSE / EPC;                             // chunks per row and stage
    unsigned b = blockIdx.x;
    int ji = 0;
    while (ji < a.n && b >= a.job[ji].blocks) b -= a.job[ji++].blocks;
    if (ji < a.n) {
        const PackJob &j = a.job[ji];
        const size_t t = (size_t)b * 256 + threadIdx.x;
        if (t >= (size_t)j.tiles * j.nks * j.R * CPR) return;
        int c, r;
        size_t rest;
        if (j.src.trans) {
            r = (int)(t % j.R);
            rest = t / j.R;
            c = (int)(rest % CPR);
            rest /= CPR;
        } else {
            c = (int)(t % CPR);
            rest = t / CPR;
            r = (int)(rest % j.R);
            rest /= j.R;
        }
        const int s = (int)(rest % j.nks), tile = (int)(rest / j.nks);
        const int row = tile * j.R + r, k0 = s * KSE + c * EPC;
        // all loads of the chunk, then its values
        float v[EPC], w[EPC];
        const size_t o = j.src.trans ? (size_t)k0 * j.src.ld + row : (size_t)row * j.src.ld + k0, st = j.src.trans ? j.src.ld : 1;
        const bool two = j.src.S2 != nullptr;
        if (j.vec && row < j.rows && k0 + EPC <= j.K) {
            const float4 *p = reinterpret_cast<const float4 *>(static_cast<const float *>(j.src.S) + o), *p2 = reinterpret_cast<const float4 *>(j.src.S2 + o);
#pragma unroll
            for (int i = 0; i < EPC / 4; i++) {
                const float4 x = p[i], y = two ? p2[i] : x;
                v[4 * i] = x.x; v[4 * i + 1] = x.y; v[4 * i + 2] = x.z; v[4 * i + 3] = x.w;
                w[4 * i] = y.x; w[4 * i + 1] = y.y; w[4 * i + 2] = y.z; w[4 * i + 3] = y.w;
            }
        } else {
#pragma unroll
            for (int i = 0; i < EPC; i++) {
                const bool in = row < j.rows && k0 + i < j.K;
                v[i] = in ? src_a(j.src, o + i * st) : 0.f;
                w[i] = in && two ? j.src.S2[o + i * st] : 0.f;
            }
        }
#pragma unroll
        for (int i = 0; i < EPC; i++) v[i] = row < j.rows && k0 + i < j.K ? src_value(j.src, v[i], w[i]) : 0.f;
        // element (r, k) of a plane: core matrix (k / EPC, r / 8) at ((k / EPC) (R / 8) + r / 8) 8 EPC, row r % 8
        const size_t per_stage = (size_t)j.R * KSE;            // elements of one plane of one stage
        const size_t off = (((size_t)(c) * (j.R / 8) + r / 8) * 8 + (r % 8)) * EPC;
        TD *base = static_cast<TD *>(j.dst) + ((size_t)tile * j.nks + s) * j.planes * per_stage;
        if constexpr (sizeof(TD) == 2) {
            __align__(16) __nv_bfloat16 h[EPC];
#pragma unroll
            for (int i = 0; i < EPC; i++) h[i] = __float2bfloat16(v[i]);
            *reinterpret_cast<uint4 *>(base + off) = *reinterpret_cast<const uint4 *>(h);
        } else if (j.planes == 1) {
            *reinterpret_cast<float4 *>(base + off) = make_float4(v[0], v[1], v[2], v[3]);
        } else {
            const float4 hi = make_float4(tc::tf32_hi(v[0]), tc::tf32_hi(v[1]), tc::tf32_hi(v[2]), tc::tf32_hi(v[3]));
            *reinterpret_cast<float4 *>(base + off) = hi;
            *reinterpret_cast<float4 *>(base + per_stage + off) =
                make_float4(v[0] - hi.x, v[1] - hi.y, v[2] - hi.z, v[3] - hi.w);
        }
        return;
    }
    // column sums: block b = (row chunk, 256 columns)
    const unsigned cb = (a.sum_cols + 255) / 256, chunk = b / cb;
    const int col = (int)(b % cb) * 256 + threadIdx.x, r0 = (int)chunk * SUM_ROWS, r1 = min(a.sum_rows, r0 + SUM_ROWS);
    const bool mse = a.sum.mode == MLP_MSE;
    double e = 0.0;
    if (col < a.sum_cols) {
        float s = 0.f, v[SUM_ROWS], w[SUM_ROWS];
#pragma unroll
        for (int r = 0; r < SUM_ROWS; r++) {
            const size_t i = (size_t)(r0 + r) * a.sum_cols + col;
            const bool in = r0 + r < r1;
            v[r] = in ? static_cast<const float *>(a.sum.S)[i] : 0.f;
            w[r] = in ? a.sum.S2[i] : 0.f;
        }
#pragma unroll
        for (int r = 0; r < SUM_ROWS; r++) {   // (rows past the end add zeros)
            s += src_value(a.sum, v[r], w[r]);
            if (mse) {
                const float d = v[r] - w[r];
                e += (double)d * d;
            }
        }
        a.sum_part[(size_t)chunk * a.sum_cols + col] = s;
    }
    if (mse) {
        __shared__ double sh[256];
        sh[threadIdx.x] = e;
        __syncthreads();
        for (int w = 128; w > 0; w >>= 1) {
            if ((int)threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
            __syncthreads();
        }
        if (threadIdx.x == 0) a.loss_part[b] = sh[0];
    }
}

// The bias gradients of every layer and the loss from their partial sums (fixed order): blocks over the concatenated
// columns, the last block the loss.
struct FinishJobs {
    int n_layers, n_part, n_loss;
    int dout[16];
    const float *part[16];
    float *db[16];
    const double *loss_part;
    double inv_n;
    float *loss;
};
__global__ void __launch_bounds__(256) mlp_finish_kernel(const __grid_constant__ FinishJobs f)
{
    grid_release();
    grid_wait();
    if (blockIdx.x + 1 == gridDim.x) {
        __shared__ double sh[256];
        double s = 0.0;
        for (int i = threadIdx.x; i < f.n_loss; i += 256) s += f.loss_part[i];
        sh[threadIdx.x] = s;
        __syncthreads();
        for (int w = 128; w > 0; w >>= 1) {
            if ((int)threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
            __syncthreads();
        }
        if (threadIdx.x == 0) *f.loss = (float)(sh[0] * f.inv_n);
        return;
    }
    int c = blockIdx.x * 256 + threadIdx.x, l = 0;
    while (l < f.n_layers && c >= f.dout[l]) c -= f.dout[l++];
    if (l == f.n_layers) return;
    float s = 0.f;
#pragma unroll 16
    for (int p = 0; p < f.n_part; p++) s += f.part[l][(size_t)p * f.dout[l] + c];
    f.db[l][c] = s;
}

// instruction descriptor: D = F32; A, B = BF16 (kind::f16) or TF32 (kind::tf32); both K-major; M = 128, N = nb
template <int KIND> __device__ __forceinline__ unsigned idesc(int nb)
{
    const unsigned fmt = KIND == 0 ? 1u : 2u;
    return (1u << 4) | (fmt << 7) | (fmt << 10) | ((unsigned)(nb >> 3) << 17) | ((unsigned)(MT >> 4) << 24);
}

template <int KIND> __device__ __forceinline__ void mma(unsigned tmem, unsigned long long da, unsigned long long db,
                                                        unsigned id, unsigned acc)
{
    if (KIND == 0)
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                     "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem), "l"(da), "l"(db), "r"(id),
                     "r"(acc) : "memory");
    else
        tc::mma_tf32(tmem, da, db, id, acc);
}

// one GEMM of a launch: packed operands, output, tiles; a launch runs up to two, one after the other in its grid
template <typename T>
struct GemmJob {
    const T *PA, *PB;
    float *C;
    int ldc;
    Dims d;
    const float *bias;
    int vec;                // rows of C start on 16-byte boundaries
};
template <typename T>
struct GemmJobs {
    GemmJob<T> job[2];
    int n, nst;             // jobs, pipeline stages
    unsigned tmem_cols;     // tensor-memory columns allocated (a power of two, at least the widest tile)
    int *err;
    const int *skip;
};

template <int KIND>
__global__ void __launch_bounds__(128, 1) mlp_gemm_kernel(const __grid_constant__ GemmJobs<typename Kind<KIND>::T> jobs)
{
    grid_release();
    if (jobs.skip) {   // uniform over the grid
        grid_wait();
        if (*jobs.skip) return;
    }
    int tile = blockIdx.x;
    const int first = jobs.job[0].d.m_tiles * jobs.job[0].d.n_tiles;
    const GemmJob<typename Kind<KIND>::T> &job = tile < first ? jobs.job[0] : jobs.job[1];
    if (tile >= first) tile -= first;
    const Dims &d = job.d;
    const int nst = jobs.nst;
    using K_ = Kind<KIND>;
    extern __shared__ __align__(1024) unsigned char smem[];
    const unsigned a_bytes = K_::A_PLANES * MT * KS_BYTES, b_bytes = (unsigned)d.nb * KS_BYTES;
    __shared__ __align__(8) unsigned long long full[MAXST], empty[MAXST], done;
    __shared__ unsigned tmem_base;
    __shared__ int failed;
    __shared__ int last_issued[MAXST];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nt = tile % d.n_tiles, mt = tile / d.n_tiles;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc::smem_u32(&tmem_base)),
                     "r"(jobs.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int b = 0; b < nst; b++) {
            tc::mbar_init(tc::smem_u32(&full[b]), 1);
            tc::mbar_init(tc::smem_u32(&empty[b]), 1);
            last_issued[b] = -1;
        }
        tc::mbar_init(tc::smem_u32(&done), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        failed = 0;
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const unsigned tmem = tmem_base;
    auto stage = [&](int b) { return smem + (size_t)b * (a_bytes + b_bytes); };
    const unsigned char *asrc = reinterpret_cast<const unsigned char *>(job.PA) + (size_t)mt * d.nks * a_bytes;
    const unsigned char *bsrc = reinterpret_cast<const unsigned char *>(job.PB) + (size_t)nt * d.nks * b_bytes;
    grid_wait();   // the packed operands (and every earlier reader of C) are done
    if (tid == 0) {
        for (int s = 0; s < d.nks; s++) {
            const int b = s % nst;
            if (s >= nst && !tc::mbar_wait(tc::smem_u32(&empty[b]), (s / nst - 1) & 1)) { failed = 1; break; }
            unsigned long long st;
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 %0, [%1], %2;"
                         : "=l"(st) : "r"(tc::smem_u32(&full[b])), "r"(a_bytes + b_bytes) : "memory");
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                         ::"r"(tc::smem_u32(stage(b))), "l"(asrc + (size_t)s * a_bytes), "r"(a_bytes),
                         "r"(tc::smem_u32(&full[b])) : "memory");
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                         ::"r"(tc::smem_u32(stage(b) + a_bytes)), "l"(bsrc + (size_t)s * b_bytes), "r"(b_bytes),
                         "r"(tc::smem_u32(&full[b])) : "memory");
            last_issued[b] = s;
        }
    } else if (tid == 32) {
        const unsigned id = idesc<KIND>(d.nb);
        bool ok = true;
        for (int s = 0; s < d.nks && ok; s++) {
            const int b = s % nst;
            if (!tc::mbar_wait(tc::smem_u32(&full[b]), (s / nst) & 1)) { ok = false; break; }
            tc::fence_after();
            const unsigned sa = tc::smem_u32(stage(b)), sb = sa + a_bytes;
            constexpr int NSTEP = KS_BYTES / (K_::KSTEP * K_::ELEM);   // MMA K-steps per stage (4)
#pragma unroll
            for (int kk = 0; kk < NSTEP; kk++) {
                // one K-step spans two core matrices along K
                const unsigned ao = kk * 2 * (MT / 8) * 128, bo = kk * 2 * (d.nb / 8) * 128;
                const unsigned first = (s == 0 && kk == 0) ? 0u : 1u;
                const unsigned long long db = tc::smem_desc(sb + bo, d.nb);
                mma<KIND>(tmem, tc::smem_desc(sa + ao, MT), db, id, first);
                if (K_::A_PLANES == 2) mma<KIND>(tmem, tc::smem_desc(sa + MT * KS_BYTES + ao, MT), db, id, 1u);
            }
            tc::commit(tc::smem_u32(&empty[b]));
        }
        if (!ok) failed = 1;
        tc::commit(tc::smem_u32(&done));
    }
    __syncwarp();
    const bool fin = tc::mbar_wait(tc::smem_u32(&done), 0);
    tc::fence_after();
    __syncthreads();
    if (!fin || failed) {
        if (tid == 0) {
            atomicExch(jobs.err, 1);
            for (int b = 0; b < nst; b++)   // copies still in flight into this CTA's shared memory
                if (last_issued[b] >= 0) (void)tc::mbar_wait(tc::smem_u32(&full[b]), (last_issued[b] / nst) & 1);
        }
    } else {
        const int row = mt * MT + warp * 32 + lane;
        const unsigned lane_off = (unsigned)(warp * 32) << 16;
        for (int c0 = 0; c0 < d.nb; c0 += 8) {
            unsigned v[8];
            tc::tmem_ld8(tmem + lane_off + (unsigned)c0, v);
            tc::tmem_wait_ld();
            const int col0 = nt * d.nb + c0;
            if (row < d.M && job.vec && col0 + 8 <= d.N) {   // a whole 32-byte sector per lane
                float o[8];
#pragma unroll
                for (int j = 0; j < 8; j++) o[j] = __uint_as_float(v[j]) + (job.bias ? job.bias[col0 + j] : 0.f);
                float4 *p = reinterpret_cast<float4 *>(job.C + (size_t)row * job.ldc + col0);
                p[0] = make_float4(o[0], o[1], o[2], o[3]);
                p[1] = make_float4(o[4], o[5], o[6], o[7]);
            } else if (row < d.M) {
#pragma unroll
                for (int j = 0; j < 8; j++) {
                    const int col = col0 + j;
                    if (col < d.N) job.C[(size_t)row * job.ldc + col] = __uint_as_float(v[j]) + (job.bias ? job.bias[col] : 0.f);
                }
            }
        }
    }
    tc::fence_before();
    __syncthreads();
    if (warp == 0) {
        tc::fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(jobs.tmem_cols) : "memory");
    }
}

// tiles: enough columns per tile for the MMA to be efficient, few enough that the tiles cover the SMs
Dims dims(int M, int N, int K, int elem)
{
    Dims d{};
    d.M = M; d.N = N; d.K = K;
    d.m_tiles = (M + MT - 1) / MT;
    // column tiles for about 128 CTAs: fewer leave SMs without a tile, more make tiles too narrow to matter (gradients of a
    // 1024 batch with 64, 96, 128, 152, 304 CTAs: 187, 182, 180, 178, 178 us; of 256: 143, 140, 141, 141, 141; of 4096: 395,
    // 398, 387, 386, 381)
    const int want = std::max(1, (128 + d.m_tiles - 1) / d.m_tiles);
    d.nb = std::min(NMAX, std::max(NMIN, ((N + want - 1) / want + 15) / 16 * 16));
    d.n_tiles = (N + d.nb - 1) / d.nb;
    const int kse = KS_BYTES / elem;
    d.nks = (K + kse - 1) / kse;
    return d;
}

template <typename A>
cudaError_t launch(void (*k)(const A), unsigned grid, int threads, size_t smem, cudaStream_t s, bool overlap, const A &args)
{
    cudaLaunchConfig_t c{};
    c.gridDim = dim3(grid);
    c.blockDim = dim3(threads);
    c.dynamicSmemBytes = smem;
    c.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    c.attrs = &at;
    c.numAttrs = overlap ? 1 : 0;
    return cudaLaunchKernelEx(&c, k, args);
}

template <int KIND> size_t pa_elems(const Dims &d) { return (size_t)d.m_tiles * d.nks * Kind<KIND>::A_PLANES * MT * (KS_BYTES / Kind<KIND>::ELEM); }
template <int KIND> size_t pb_elems(const Dims &d) { return (size_t)d.n_tiles * d.nks * d.nb * (KS_BYTES / Kind<KIND>::ELEM); }

template <int KIND>
cudaError_t run_gemms(cudaStream_t s, const MlpGemm *g, int n, const MlpSums *sums, const int *skip, void *ws, size_t ws_bytes, int *err)
{
    using T = typename Kind<KIND>::T;
    constexpr int EPC = 16 / (int)sizeof(T), KSE = KS_BYTES / (int)sizeof(T);
    PackJobs pj{};
    GemmJobs<T> gj{};
    T *p = static_cast<T *>(ws);
    unsigned blocks = 0, tiles = 0;
    size_t stage = 0, used = 0;
    int nb_max = 0;
    for (int i = 0; i < n; i++) {
        const Dims d = dims(g[i].M, g[i].N, g[i].K, Kind<KIND>::ELEM);
        GemmJob<T> &j = gj.job[i];
        j.PA = p;
        j.PB = p + pa_elems<KIND>(d);
        j.C = g[i].C;
        j.ldc = g[i].N;
        j.d = d;
        j.bias = g[i].bias;
        j.vec = g[i].N % 4 == 0 && (reinterpret_cast<uintptr_t>(g[i].C) & 15) == 0;
        p += pa_elems<KIND>(d) + pb_elems<KIND>(d);
        used += (pa_elems<KIND>(d) + pb_elems<KIND>(d)) * sizeof(T);
        // A rows = M (K along a row unless transposed); B as rows n of op(B)^T: element (n, k) = op(B)[k][n]
        auto add = [&](const MlpSrc &src, int rows, int R, int nt, int planes, const T *dst) {
            PackJob &k = pj.job[pj.n++];
            k.src = src;
            k.rows = rows;
            k.K = d.K;
            k.R = R;
            k.tiles = nt;
            k.nks = d.nks;
            k.planes = planes;
            k.vec = src.mode != MLP_BF16 && !src.trans && src.ld % 4 == 0 && (reinterpret_cast<uintptr_t>(src.S) & 15) == 0 &&
                    (reinterpret_cast<uintptr_t>(src.S2) & 15) == 0;
            k.dst = const_cast<T *>(dst);
            k.blocks = (unsigned)(((size_t)nt * d.nks * R * (KSE / EPC) + 255) / 256);
            blocks += k.blocks;
        };
        add(g[i].A, g[i].M, MT, d.m_tiles, Kind<KIND>::A_PLANES, j.PA);
        add(g[i].B, g[i].N, d.nb, d.n_tiles, 1, j.PB);
        tiles += (unsigned)(d.m_tiles * d.n_tiles);
        stage = std::max(stage, (size_t)(Kind<KIND>::A_PLANES * MT + d.nb) * KS_BYTES);
        nb_max = std::max(nb_max, d.nb);
    }
    if (used > ws_bytes) return cudaErrorInvalidValue;   // sized by the caller (mlp_tc_scratch_bytes)
    pj.skip = skip;
    if (sums) {
        pj.sum = sums->src;
        pj.sum_rows = sums->rows;
        pj.sum_cols = sums->cols;
        pj.sum_part = sums->part;
        pj.loss_part = sums->loss_part;
        blocks += (unsigned)(mlp_sum_parts(sums->rows) * ((sums->cols + 255) / 256));
    }
    const bool overlap = skip == nullptr;   // (the surrogate's passes, inside captured flows, launch in order)
    TUFRG_CUDA_TRY(launch(pack_kernel<T>, blocks, 256, 0, s, overlap, pj));
    gj.n = n;
    gj.nst = (int)std::min<size_t>(MAXST, 200 * 1024 / stage);
    gj.tmem_cols = 32;
    while ((int)gj.tmem_cols < nb_max) gj.tmem_cols *= 2;
    gj.err = err;
    gj.skip = skip;
    const size_t smem = gj.nst * stage;
    auto k = mlp_gemm_kernel<KIND>;
    TUFRG_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    return launch(k, tiles, 128, smem, s, overlap, gj);
}

}  // namespace

size_t mlp_tc_scratch_bytes(int M, int N, int K)
{
    // both kinds, B padded to any tile width (the tiles depend on M, so that a smaller M may pad B more)
    const size_t m = (size_t)(M + MT - 1) / MT * MT, n = (size_t)N + NMAX;
    const size_t k0 = (K * 2 + KS_BYTES - 1) / KS_BYTES, k1 = (K * 4 + KS_BYTES - 1) / KS_BYTES;
    return std::max((m + n) * k0, (2 * m + n) * k1) * KS_BYTES;
}

int mlp_sum_parts(int rows) { return (rows + SUM_ROWS - 1) / SUM_ROWS; }
int mlp_loss_parts(int rows, int cols) { return mlp_sum_parts(rows) * ((cols + 255) / 256); }

cudaError_t mlp_gemms(cudaStream_t s, bool fp32, const MlpGemm *g, int n, const MlpSums *sums, const int *skip, void *ws,
                      size_t ws_bytes, int *err)
{
    return fp32 ? run_gemms<1>(s, g, n, sums, skip, ws, ws_bytes, err) : run_gemms<0>(s, g, n, sums, skip, ws, ws_bytes, err);
}

cudaError_t mlp_finish(cudaStream_t s, int n_layers, const int *dout, float *const *part, float *const *db, int n_part,
                       const double *loss_part, int n_loss, double inv_n, float *loss)
{
    FinishJobs f{};
    for (int l0 = 0; l0 < n_layers; l0 += 16) {   // sixteen layers per launch (the loss with the first)
        f.n_layers = std::min(16, n_layers - l0);
        int cols = 0;
        for (int l = 0; l < f.n_layers; l++) {
            f.dout[l] = dout[l0 + l];
            f.part[l] = part[l0 + l];
            f.db[l] = db[l0 + l];
            cols += dout[l0 + l];
        }
        f.n_part = n_part;
        f.n_loss = n_loss;
        f.loss_part = loss_part;
        f.inv_n = inv_n;
        f.loss = loss;
        TUFRG_CUDA_TRY(launch(mlp_finish_kernel, (unsigned)((cols + 255) / 256 + 1), 256, 0, s, true, f));
    }
    return cudaSuccess;
}

}  // namespace tufrg
