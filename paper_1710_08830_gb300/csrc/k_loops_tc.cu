// Multi-orbital loop k-sum on the 5th-generation tensor cores (split path, N_s = 6; Eqs. loopminus, loopplus,
// loop_orbital with the temperature or momentum-shell weights of Eqs. disc_2a, disc_2b, def_lmp).
//
// For a transfer momentum s the compact loop is
//   Lc[Delta][(t1 t3),(t2 t4)] = (1/Nk) sum_k e^{-+ i k.Delta} sum_l rho^l_{t1 t3}(k) T^l_{t2 t4}(s, k)
// with rho^l_{tt'} = U_{tl} U*_{t'l} at the summation point k and T^l = sum_{l2} w_{l l2} rho'^{l2} at its partner:
//   C (u = s):  partner k - u, rho' = conj(rho), phase e^{-i k.Delta};
//   P (s):      the sum runs over the first propagator's momentum k' = s - q (a relabelling of the fine mesh),
//               partner s - k', rho' = rho, phase e^{-i (s - k').Delta} = e^{-i s.Delta} e^{+i k'.Delta}.
// Written this way the summation point's projectors do not depend on s, so one operand serves several momenta.
// Three exact rewritings keep the contraction small:
//   * rho and T are Hermitian 6 x 6 matrices (the weights are real): each is 36 real numbers (Re and Im of the upper
//     triangle, the diagonal), so the sums are real; the orbital entries are put together from them at the end
//     (loops_gen_finish; for C the imaginary parts of rho' change sign there);
//   * the row phase e^{-+ i ky dy} is a cosine and a sine (dy = 0: one), so for dy >= 0 there are five real row
//     phases: per fine-mesh column kx the sum over ky is one real GEMM
//       W[(s_j, c')][(p, c)] = sum_{(ky, l)} T^l_{c'}(s_j; kx, ky) * phi_p(ky) rho^l_c(kx, ky)
//     with M = 3 momenta x 36 = 108 rows (of 128), N = 5 x 36 = 180 columns (of 192), K = Lf x 6;
//   * exchanging the two propagators maps k to s - k, so one point of every pair {k, s - k} suffices where the channel
//     allows it (P always, C with a symmetry that inverts the momentum; see k_loops2h.cu): columns
//     kx = hx + c, 2 hx = sx (mod Lf), c up to Lf / 2.  The momenta of a group share sx and hence their columns.
// It runs as 3xTF32 (hi*hi + hi*lo + lo*hi, FP32 accumulation in tensor memory).  The x phases e^{-+ i kx dx} are
// applied afterwards by loops_tc_xsum over the written columns.
// Why this shape: complex arithmetic on both sides needs 4 real products of 108 x 36 per (momentum, k, band), the real
// basis one of 180 x 36, 2.4 times less, and half of the operand values to form, split and store.  A launch over the 153
// orbit representatives of the 32 x 32 / 6 x 6 workload takes 2.81 ms per channel (7.25 ms in complex arithmetic over the
// whole mesh); the MMAs alone are about 1.0 ms of it.  The producers bound it: on the 16 x 16 / 12 x 12
// mesh the tensor pipe is busy 28% of the cycles, the issue slots 45%, L1 and shared memory 56%; the warps wait for fixed
// latencies, L2 loads and shared memory in turn.
//
// The left operand (T, two TF32 planes) lives in tensor memory: the producers write it with tcgen05.st, and the MMAs
// read it from there, so shared memory carries only the right operand.
// One persistent CTA per SM walks its (momentum group, column) items.  Warp roles:
//   warps 0-15  producers, thread (ky row kb of the stage's four, operand row r): every thread holds the next stage's
//               inputs in registers (projector values of its rows and the Fermi entries of one pair weight, loaded
//               straight from the L2-resident tables one stage ahead); per stage it forms its pair weight into shared
//               memory, then row r of T at its ky row (six bands from the weights of its pair of points) and its one or
//               two phased projector rows, and writes the TF32 hi / lo parts: T into tensor memory (lane = row), the
//               projectors into shared memory in the K-major core-matrix layout;
//   warp 16     TMEM allocation and the MMA issuer (one thread): 9 MMAs of 128 x 192 x 8 per stage; then its quarter of
//               the previous column's epilogue (20 warps leave every thread 96 registers, 21 would leave 80);
//   warps 17-19 epilogue: tensor memory -> W in global memory (coalesced, row index fastest).
// Two stage buffers (mbarriers full / empty) and two tensor-memory accumulators (acc_full / acc_empty).  Every wait is
// bounded; on time-out the kernel raises the error flag, every role stops, the MMAs in flight are waited for (bounded)
// and the tensor memory is freed.
#include <algorithm>
#include <cmath>

#include "tc_common.cuh"
#include "tufrg_internal.cuh"

namespace tufrg {
namespace {

constexpr int NS = 6, NS2 = 36;
constexpr int GRP = 3;                       // transfer momenta per item (row blocks of the left operand)
constexpr int NDYM = 3;                      // non-negative y components of the bond differences
constexpr int NPH = 2 * NDYM - 1;            // real row phases: 1, then cos and sin per dy > 0
constexpr int ROWS = GRP * NS2;              // 108 rows used
constexpr int COLS = NPH * NS2;              // 180 columns used
constexpr int TM = 128;                      // MMA M
constexpr int TN = 192;                      // MMA N: COLS padded to a multiple of 16
constexpr int KB = 4;                        // ky rows per stage
constexpr int KST = KB * NS;                 // K per stage: 24 = three MMA K-steps of 8
constexpr int NPROD = 512;                   // producer threads, warps 0-15: thread (ky row kb, operand row r)
constexpr int MMA_WARP = 16;                 // it and warps 17-19: epilogue
constexpr int NTHREADS = 20 * 32;
constexpr unsigned B_PLANE = TN * KST * 4;   // bytes per plane and stage of the right operand (shared memory)
constexpr unsigned STAGE_BYTES = 2 * B_PLANE;   // planes: hi, lo
// tensor memory: accumulator b at [TN b, TN b + TN); left operand of stage b at A_COL0 + 64 b, planes hi, lo at + 32 p
// (K = 24 columns used)
constexpr unsigned A_COL0 = 2 * TN, A_STAGE_COLS = 64, A_PLANE_COLS = 32, TMEM_COLS = 512;
static_assert(A_COL0 + 2 * A_STAGE_COLS <= TMEM_COLS, "tensor memory budget");
constexpr int NW = GRP * KB * NS2;           // pair weights per stage
static_assert(NW <= NPROD, "one pair weight per producer thread");

struct LtArgs {
    const float *rho;           // [Nk][36][6] real projector components (loop_comp), band fastest
    const FermiEntry32 *ft;     // [Nk][NS] (e, g, g') at the flow scale, or (e, f, h) with the momentum shell
    float *W;                   // [n_groups][ncol][COLS][ROWS] column sums
    const int *s_list;          // slot -> transfer momentum (null: the slot is the momentum)
    const int *grp;             // [n_groups][GRP] slots of a group, -1: none (null: slot g GRP + j)
    int n_slot, n_items;
    int Lq, nc, Lf, spc;        // spc: stages per column
    int ncol, half;             // columns per group; half: kx = hx + c, else kx = c
    int dy1, dy2;               // y differences of the phases 1..4, modulo Lf (0 where absent)
    const float2 *ptab;         // e^{-2 pi i n / Lf}
    const double *Tp;           // device flow scale
    float thr_factor, shell_T;
    int *err;
};

__device__ __forceinline__ int wrapm(int v, int L)
{
    v %= L;
    return v < 0 ? v + L : v;
}

// the loop weight of one band pair (gen_pair_weight) with the FP32 fast division of the split two-band kernel
template <int WHICH>
__device__ __forceinline__ float tc_pair_weight(float e1, float g1, float gp1, float e2, float g2, float gp2, float thr, float lam)
{
    if (lam > 0.f) return shell_weight<WHICH, float>(e1, g1, gp1, e2, g2, gp2, thr, lam);
    if (WHICH == 0) {
        const float s = e1 + e2;
        return fabsf(s) > thr ? -__fdividef(g1 + g2, s) : -0.5f * (gp1 + gp2);
    }
    const float d = e1 - e2;
    return fabsf(d) > thr ? __fdividef(g1 - g2, d) : 0.5f * (gp1 + gp2);
}

// TF32 part of x by truncation (the 13 low mantissa bits cleared; one logic operation): x - hi is exact and below
// 2^-10 |x|, so hi + lo keeps FP32 accuracy through the three products of 3xTF32
__device__ __forceinline__ float tf32_trunc(float x) { return __uint_as_float(__float_as_uint(x) & 0xffffe000u); }

// the six K values kb * 6 + l (l = 0..5) of row r of the right operand, hi and lo planes: 4 + 2 or 2 + 4 along the
// 4-wide groups
__device__ __forceinline__ void put6(float *planes, int r, int kb, const float (&v)[NS])
{
    const int k0 = 6 * kb;
    float h[NS], l[NS];
#pragma unroll
    for (int i = 0; i < NS; i++) {
        h[i] = tf32_trunc(v[i]);
        l[i] = v[i] - h[i];
    }
    float *p0 = planes, *p1 = planes + B_PLANE / 4;
    if ((kb & 1) == 0) {
        const int a = tc::core_off(r, k0, TN), b = tc::core_off(r, k0 + 4, TN);
        *reinterpret_cast<float4 *>(p0 + a) = make_float4(h[0], h[1], h[2], h[3]);
        *reinterpret_cast<float2 *>(p0 + b) = make_float2(h[4], h[5]);
        *reinterpret_cast<float4 *>(p1 + a) = make_float4(l[0], l[1], l[2], l[3]);
        *reinterpret_cast<float2 *>(p1 + b) = make_float2(l[4], l[5]);
    } else {
        const int a = tc::core_off(r, k0, TN), b = tc::core_off(r, k0 + 2, TN);
        *reinterpret_cast<float2 *>(p0 + a) = make_float2(h[0], h[1]);
        *reinterpret_cast<float4 *>(p0 + b) = make_float4(h[2], h[3], h[4], h[5]);
        *reinterpret_cast<float2 *>(p1 + a) = make_float2(l[0], l[1]);
        *reinterpret_cast<float4 *>(p1 + b) = make_float4(l[2], l[3], l[4], l[5]);
    }
}

// the six K values kb * 6 + l of this lane's row of the left operand into tensor memory, hi and lo planes, as a 4 + 2
// (kb even) or 2 + 4 (kb odd) column split so that every store starts at a multiple of its width; warp-collective
__device__ __forceinline__ void put6_tmem(unsigned col0, int kb, const float (&v)[NS])
{
    const unsigned c = col0 + 6 * kb;
#pragma unroll
    for (int p = 0; p < 2; p++) {
        float t[NS];
#pragma unroll
        for (int l = 0; l < NS; l++) t[l] = p ? v[l] - tf32_trunc(v[l]) : tf32_trunc(v[l]);
        const unsigned cp = c + p * A_PLANE_COLS;
        if ((kb & 1) == 0) {
            tc::tmem_st4(cp, t[0], t[1], t[2], t[3]);
            tc::tmem_st2(cp + 4u, t[4], t[5]);
        } else {
            tc::tmem_st2(cp, t[0], t[1]);
            tc::tmem_st4(cp + 2u, t[2], t[3], t[4], t[5]);
        }
    }
}

__device__ __forceinline__ void ld_six(const float *p, float (&v)[NS])   // six consecutive floats, 8-byte aligned
{
#pragma unroll
    for (int i = 0; i < 3; i++) {
        const float2 t = __ldg(reinterpret_cast<const float2 *>(p) + i);
        v[2 * i] = t.x;
        v[2 * i + 1] = t.y;
    }
}

__device__ __forceinline__ void bar_producers() { asm volatile("bar.sync 1, %0;" ::"n"(NPROD) : "memory"); }

inline size_t lt_smem_bytes(int Lf) { return 2 * (size_t)STAGE_BYTES + 2 * NW * sizeof(float) + 2 * sizeof(float) * Lf; }

template <int WHICH>
__global__ void __launch_bounds__(NTHREADS, 1) loops_tc_kernel(const __grid_constant__ LtArgs a)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    float *sW = reinterpret_cast<float *>(smem + 2 * STAGE_BYTES);   // [2][GRP][KB][l2][l1]
    float *ptab = sW + 2 * NW;                                       // [Lf] cos, [Lf] sin of 2 pi n / Lf
    __shared__ __align__(8) unsigned long long full[2], empty[2], accf[2], acce[2], done;
    __shared__ unsigned tmem_base;
    __shared__ int abort_flag, stop[2];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int Lf = a.Lf, spc = a.spc;

    if (warp == MMA_WARP) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc::smem_u32(&tmem_base)),
                     "r"(TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int b = 0; b < 2; b++) {
            tc::mbar_init(tc::smem_u32(&full[b]), NPROD);
            tc::mbar_init(tc::smem_u32(&empty[b]), 1);
            tc::mbar_init(tc::smem_u32(&accf[b]), 1);
            tc::mbar_init(tc::smem_u32(&acce[b]), 128);
            stop[b] = 0;
        }
        tc::mbar_init(tc::smem_u32(&done), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        abort_flag = 0;
    }
    for (int n = tid; n < Lf; n += NTHREADS) {
        const float2 p = a.ptab[n];
        ptab[n] = p.x;
        ptab[Lf + n] = -p.y;
    }
    // the padding columns of the right operand (rows 180..191 of its planes) are zero in both stage buffers for the whole
    // kernel (the padding lanes of the left operand are written as zeros with every stage)
    for (int i = tid; i < 4 * (TN - COLS) * KST; i += NTHREADS) {
        const int pl = i / ((TN - COLS) * KST), r = i % ((TN - COLS) * KST);
        reinterpret_cast<float *>(smem)[pl * (B_PLANE / 4) + tc::core_off(COLS + r / KST, r % KST, TN)] = 0.f;
    }
    tc::fence_smem_async();
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const unsigned tmem = tmem_base;
    const int my_items = a.n_items > (int)blockIdx.x ? (a.n_items - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    const int n_stages = my_items * spc;

    if (warp < MMA_WARP) {
        // ------------------------------------------------------------------ producers
        const bool shell = a.shell_T > 0.f;
        const float lam = shell ? (float)(*a.Tp) : 0.f;
        const float thr = a.thr_factor * (shell ? a.shell_T : (float)(*a.Tp));
        const int kb = tid >> 7, r = tid & 127;            // ky row of the stage (warp-uniform) and operand row
        const int rj = r / NS2, rc = r % NS2;              // left operand: momentum of the group, component
        const bool has_a = r < ROWS, has_b1 = r + 128 < COLS;   // right operand rows r and (r < 52) r + 128
        const int p0 = r / NS2, p1 = (r + 128) / NS2, c1 = (r + 128) % NS2;   // their phases and components
        const bool has_w = tid < NW;                       // this thread's pair weight (wj, wk, l2, l1)
        const int wj = tid / (KB * NS2), wk = (tid / NS2) % KB, wl2 = (tid % NS2) / NS, wl1 = tid % NS;
        // phase of a row: 0 -> 1 (the cosine of zero), 1 / 3 -> cos, 2 / 4 -> sin of ky dy
        const int step0 = p0 == 0 ? 0 : p0 < 3 ? a.dy1 : a.dy2, step1 = p1 < 3 ? a.dy1 : a.dy2;
        const int adv0 = (KB * step0) % Lf, adv1 = (KB * step1) % Lf, beg0 = (kb * step0) % Lf, beg1 = (kb * step1) % Lf;
        const float *tab0 = ptab + (p0 == 0 || (p0 & 1) ? 0 : Lf), *tab1 = ptab + ((p1 & 1) ? 0 : Lf);
        const float *w_a = sW + (rj * KB + kb) * NS2;
        // cursor of the stage that is loaded next (one stage ahead of the one being formed): table offsets of this
        // thread's points, stepping by KB rows (the partner's by -KB for P), with wrap
        constexpr unsigned ROW = NS2 * NS;                 // floats of one fine k
        const unsigned col_len = (unsigned)Lf * ROW, fcol_len = (unsigned)Lf * NS;
        int f_item = (int)blockIdx.x, f_st = 0, kyA = 0, kyW = 0, i0 = 0, i1 = 0;
        unsigned oA = 0, oB = 0, oF1 = 0, oF2 = 0;
        bool okW = false;
        auto slot_q = [&](int g, int j) {   // transfer momentum of group member j (-1 where there is none)
            const int slot = a.grp ? a.grp[g * GRP + j] : (g * GRP + j < a.n_slot ? g * GRP + j : -1);
            if (slot < 0) return -1;
            return a.s_list ? a.s_list[slot] : slot;
        };
        auto column = [&]() {   // the cursor's column: points of this thread's rows at its first ky rows
            const int g = f_item / a.ncol, c = f_item - g * a.ncol;
            const int q0 = slot_q(g, 0), qa = has_a ? slot_q(g, rj) : -1, qw = has_w ? slot_q(g, wj) : -1;
            const int sx0 = (q0 / a.Lq) * a.nc;
            const int hx = !(sx0 & 1) ? sx0 / 2 : (Lf & 1) ? (sx0 + Lf) / 2 : (sx0 + 1) / 2;
            int kx = a.half ? hx + c : c;
            if (kx >= Lf) kx -= Lf;
            const int ua = qa < 0 ? q0 : qa, uw = qw < 0 ? q0 : qw;
            const int xa = ua / a.Lq, xw = uw / a.Lq;
            const int sxa = xa * a.nc, sya = (ua - xa * a.Lq) * a.nc, sxw = xw * a.nc, syw = (uw - xw * a.Lq) * a.nc;
            int kxA = WHICH == 0 ? sxa - kx : kx - sxa, kxW = WHICH == 0 ? sxw - kx : kx - sxw;
            if (kxA < 0) kxA += Lf;
            if (kxW < 0) kxW += Lf;
            kyA = WHICH == 0 ? wrapm(sya - kb, Lf) : wrapm(kb - sya, Lf);
            kyW = WHICH == 0 ? wrapm(syw - wk, Lf) : wrapm(wk - syw, Lf);
            oA = ((unsigned)(kxA * Lf + kyA) * NS2 + rc) * NS;
            oB = ((unsigned)(kx * Lf + kb) * NS2) * NS;
            oF1 = (unsigned)(kx * Lf + wk) * NS + wl1;
            oF2 = (unsigned)(kxW * Lf + kyW) * NS + wl2;
            okW = qw >= 0;
            i0 = beg0;
            i1 = beg1;
        };
        struct In {
            float A[NS], B0[NS], B1[NS];
            float4 f1, f2;
            float ph0, ph1;
            bool ok;
        };
        const float4 *ft = reinterpret_cast<const float4 *>(a.ft);
        auto load = [&](In &x) {   // the cursor's stage into registers; then the cursor steps
            // (rows past the column in its last stage are read from the tables' padding or the next column: their
            // weights are zero, so T is)
            if (has_a) ld_six(a.rho + oA, x.A);
            ld_six(a.rho + oB + rc * NS, x.B0);
            if (has_b1) ld_six(a.rho + oB + c1 * NS, x.B1);
            if (has_w) {
                x.f1 = __ldg(ft + oF1);
                x.f2 = __ldg(ft + oF2);
            }
            x.ok = okW && f_st * KB + wk < Lf;   // the weights of a row or momentum that does not exist are zero
            x.ph0 = tab0[i0];
            x.ph1 = tab1[i1];
            if (++f_st == spc) {
                f_st = 0;
                f_item += (int)gridDim.x;
                if (f_item < a.n_items) column();
                return;
            }
            oB += KB * ROW;
            oF1 += KB * NS;
            if (WHICH == 0) {
                kyA -= KB;
                kyW -= KB;
                oA -= KB * ROW;
                oF2 -= KB * NS;
                while (kyA < 0) { kyA += Lf; oA += col_len; }
                while (kyW < 0) { kyW += Lf; oF2 += fcol_len; }
            } else {
                kyA += KB;
                kyW += KB;
                oA += KB * ROW;
                oF2 += KB * NS;
                while (kyA >= Lf) { kyA -= Lf; oA -= col_len; }
                while (kyW >= Lf) { kyW -= Lf; oF2 -= fcol_len; }
            }
            i0 += adv0;
            i1 += adv1;
            if (i0 >= Lf) i0 -= Lf;
            if (i1 >= Lf) i1 -= Lf;
        };
        // one stage in buffer buf (n & 1): weights, T and projector rows from x; the next stage's inputs into y
        auto form = [&](int n, const int buf, In &x, In &y) -> bool {
            if (has_w)
                sW[buf * NW + tid] = x.ok ? tc_pair_weight<WHICH>(x.f1.x, x.f1.y, x.f1.z, x.f2.x, x.f2.y, x.f2.z, thr, lam) : 0.f;
            if (tid == 0) stop[buf] = *(volatile int *)&abort_flag;
            // the stage's weights are complete; weights and stop flag have two buffers, so that the next stage's may be
            // written while this stage's are read (those of the stage after next come behind the next barrier)
            bar_producers();
            if (stop[buf]) return false;   // every producer reads the same value: they leave the loop together
            if (n + 1 < n_stages) load(y);
            // T row r = (s_j, component): T^{l1} = sum_l2 w_{l1 l2} rho'^{l2} (zero in the padding lanes)
            float2 t2[3] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
            if (has_a) {
                const float4 *wr = reinterpret_cast<const float4 *>(w_a + buf * NW);
#pragma unroll
                for (int h = 0; h < 3; h++) {   // two partner bands: weights (l2, l1 = 0..5), (l2 + 1, l1 = 0..5)
                    const float4 w0 = wr[3 * h], w1 = wr[3 * h + 1], w2 = wr[3 * h + 2];
                    const float2 u = make_float2(x.A[2 * h], x.A[2 * h]), v = make_float2(x.A[2 * h + 1], x.A[2 * h + 1]);
                    t2[0] = __ffma2_rn(make_float2(w0.x, w0.y), u, t2[0]);
                    t2[1] = __ffma2_rn(make_float2(w0.z, w0.w), u, t2[1]);
                    t2[2] = __ffma2_rn(make_float2(w1.x, w1.y), u, t2[2]);
                    t2[0] = __ffma2_rn(make_float2(w1.z, w1.w), v, t2[0]);
                    t2[1] = __ffma2_rn(make_float2(w2.x, w2.y), v, t2[1]);
                    t2[2] = __ffma2_rn(make_float2(w2.z, w2.w), v, t2[2]);
                }
            }
            const float t[NS] = {t2[0].x, t2[0].y, t2[1].x, t2[1].y, t2[2].x, t2[2].y};
            // phased projector rows
#pragma unroll
            for (int l = 0; l < NS; l++) {
                x.B0[l] *= x.ph0;
                x.B1[l] *= x.ph1;
            }
            // the MMAs that read this stage (tensor-memory A, shared-memory B) two stages ago must be complete before
            // it is overwritten
            int ok = 1;
            if (n >= 2 && lane == 0)
                ok = tc::mbar_wait_or_abort(tc::smem_u32(&empty[buf]), ((n >> 1) - 1) & 1, &abort_flag) ? 1 : 0;
            ok = __shfl_sync(0xffffffffu, ok, 0);
            if (!ok) {
                // raise the flag and keep the producers in step: all of them leave at the next stage's check
                if (lane == 0) {
                    atomicExch(&abort_flag, 1);
                    atomicExch(a.err, 1);
                }
                return true;
            }
            tc::fence_after();
            put6_tmem(tmem + ((unsigned)((warp & 3) * 32) << 16) + A_COL0 + buf * A_STAGE_COLS, kb, t);
            float *pb = reinterpret_cast<float *>(smem + buf * STAGE_BYTES);
            put6(pb, r, kb, x.B0);
            if (has_b1) put6(pb, r + 128, kb, x.B1);
            tc::tmem_wait_st();
            tc::fence_smem_async();
            tc::fence_before();
            tc::mbar_arrive(tc::smem_u32(&full[buf]));
            return true;
        };
        In in0, in1;
#pragma unroll
        for (int l = 0; l < NS; l++) in0.B1[l] = in1.B1[l] = 0.f;
        if (n_stages > 0) {
            column();
            load(in0);
        }
        for (int n = 0; n < n_stages; n += 2) {
            if (!form(n, 0, in0, in1)) break;
            if (n + 1 < n_stages && !form(n + 1, 1, in1, in0)) break;
        }
    } else {
        // ------------------------------------------------------------------ MMA issuer (warp 16) and epilogue
        const int qw = warp & 3, row = qw * 32 + lane;
        const unsigned lane_off = (unsigned)(qw * 32) << 16;
        auto fail = [&]() {
            if (lane == 0) {
                atomicExch(&abort_flag, 1);
                atomicExch(a.err, 1);
            }
        };
        // this warp's rows of a finished column: tensor memory -> W
        auto drain = [&](int col) -> bool {
            const int ab = col & 1;
            int ok = 1;
            if (lane == 0) ok = tc::mbar_wait_or_abort(tc::smem_u32(&accf[ab]), (col >> 1) & 1, &abort_flag) ? 1 : 0;
            ok = __shfl_sync(0xffffffffu, ok, 0);
            if (!ok) return false;
            tc::fence_after();
            const int item = (int)blockIdx.x + col * (int)gridDim.x;
            float *Wc = a.W + (size_t)item * COLS * ROWS + row;
            for (int c0 = 0; c0 < COLS; c0 += 8) {
                unsigned v[8];
                tc::tmem_ld8(tmem + ab * TN + lane_off + (unsigned)c0, v);
                tc::tmem_wait_ld();
                if (row < ROWS) {
#pragma unroll
                    for (int i = 0; i < 8; i++)
                        if (c0 + i < COLS) Wc[(size_t)(c0 + i) * ROWS] = __uint_as_float(v[i]);
                }
            }
            tc::fence_before();
            tc::mbar_arrive(tc::smem_u32(&acce[ab]));
            return true;
        };
        // the MMAs of one column (one thread)
        auto issue = [&](int col) -> bool {
            const int ab = col & 1;
            // the accumulator must have been read by the epilogue of the column before the previous one
            if (col >= 2 && !tc::mbar_wait_or_abort(tc::smem_u32(&acce[ab]), ((col >> 1) - 1) & 1, &abort_flag)) return false;
            tc::fence_after();
            const unsigned id = tc::idesc_tf32(TM, TN, false), d = tmem + ab * TN;
            int n = col * spc;
            for (int st = 0; st < spc; st++, n++) {
                const int b = n & 1;
                if (!tc::mbar_wait_or_abort(tc::smem_u32(&full[b]), (n >> 1) & 1, &abort_flag)) return false;
                tc::fence_after();
                const unsigned sb = tc::smem_u32(smem + b * STAGE_BYTES), ta = tmem + A_COL0 + b * A_STAGE_COLS;
#pragma unroll
                for (int kk = 0; kk < KST / 8; kk++) {
                    const unsigned bo = kk * 2 * (TN / 8) * 128;
                    const unsigned ah = ta + 8 * kk, al = ah + A_PLANE_COLS;   // K-step kk = 8 columns of each plane
                    const unsigned long long bh = tc::smem_desc(sb + bo, TN), bl = tc::smem_desc(sb + B_PLANE + bo, TN);
                    tc::mma_tf32_ta(d, ah, bh, id, (st == 0 && kk == 0) ? 0u : 1u);
                    tc::mma_tf32_ta(d, ah, bl, id, 1u);
                    tc::mma_tf32_ta(d, al, bh, id, 1u);
                }
                tc::commit(tc::smem_u32(&empty[b]));
            }
            tc::commit(tc::smem_u32(&accf[ab]));
            return true;
        };
        if (warp == MMA_WARP) {
            bool ok = true;
            for (int col = 0; col <= my_items && ok; col++) {
                if (col < my_items) {
                    int y = 1;
                    if (lane == 0) y = issue(col) ? 1 : 0;
                    ok = __shfl_sync(0xffffffffu, y, 0);
                }
                if (ok && col > 0) ok = drain(col - 1);
            }
            if (!ok) fail();
            if (lane == 0) tc::commit(tc::smem_u32(&done));   // completion of every MMA issued above
            __syncwarp();
        } else {
            for (int col = 0; col < my_items; col++)
                if (!drain(col)) {
                    fail();
                    break;
                }
        }
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

// Real projector components of every fine k and band, in the order of loop_comp: rho[k][c][l].
__global__ void loops_rho_kernel(const double2 *U, size_t n, float *rho)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;   // over Nk * 36 * 6
    if (i >= n) return;
    const int l = (int)(i % NS), c = (int)((i / NS) % NS2);
    const size_t k = i / (NS * NS2);
    int t, tp;
    bool im;
    loop_comp<NS>(c, t, tp, im);
    const double2 u = U[k * NS2 + t * NS + l], v = U[k * NS2 + tp * NS + l];
    rho[i] = (float)(im ? u.y * v.x - u.x * v.y : u.x * v.x + u.y * v.y);   // Im or Re of u conj(v)
}

struct XsArgs {
    const float *W;             // [n_groups][ncol][COLS][ROWS]
    float2 *acc;                // [n_slot][nd][36][36] half-plane entries written
    const int *s_list, *grp;
    int n_slot, n_groups, Lq, nc, Lf, nd, ndxh, ndyh, ncol, half;
    int dxm[4];                 // positive dx modulo Lf
    int dxs[5], dys[NDYM];      // non-negative dx and dy
    int dslot[9][NDYM];         // [4 + signed dx index][dy index] -> delta index of the half plane, or -1
    const float2 *ptab;
};

// x phases and the P-channel momentum phase: with C, S the column sums of the cosine and sine row phases,
//   F[d][c][c'] = sum_kx (cx C - sx S) +- i (sx C + cx S)   (upper sign P, lower sign C; times e^{-i s.Delta} for P),
// the sums of cx C, sx S, sx C, cx S serving dx and -dx; a column that is its own partner (half sums) enters with weight
// 1/2.  One thread per (group, dy, component c, row (j, c')), rows fastest; eight columns' loads in flight.
template <int WHICH>
__global__ void __launch_bounds__(256) loops_tc_xsum(const __grid_constant__ XsArgs x)
{
    extern __shared__ float2 ptab[];   // [Lf] e^{-2 pi i n / Lf}
    const int Lf = x.Lf;
    for (int n = threadIdx.x; n < Lf; n += blockDim.x) ptab[n] = x.ptab[n];
    __syncthreads();
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (size_t)x.n_groups * x.ndyh * NS2 * ROWS) return;
    const int r = (int)(idx % ROWS), c = (int)((idx / ROWS) % NS2), dyi = (int)((idx / (ROWS * NS2)) % x.ndyh);
    const int g = (int)(idx / ((size_t)ROWS * NS2 * x.ndyh));
    const int j = r / NS2, slot = x.grp ? x.grp[g * GRP + j] : (g * GRP + j < x.n_slot ? g * GRP + j : -1);
    if (slot < 0) return;
    const int s = x.s_list ? x.s_list[slot] : slot, sx = (s / x.Lq) * x.nc, sy = (s % x.Lq) * x.nc;
    const int hx = !x.half ? 0 : !(sx & 1) ? sx / 2 : (Lf & 1) ? (sx + Lf) / 2 : (sx + 1) / 2;
    const bool none = x.half && (sx & 1) && !(Lf & 1);   // no self-paired column, one column less
    const int ncol = none ? Lf / 2 : x.ncol;
    const int fix0 = x.half && !none ? 0 : -1, fix1 = x.half && !none && !(Lf & 1) ? Lf / 2 : -1;
    const size_t stride = (size_t)COLS * ROWS;
    const float *wc = x.W + (size_t)g * x.ncol * stride + (size_t)((dyi == 0 ? 0 : 2 * dyi - 1) * NS2 + c) * ROWS + r;
    const float *ws = wc + (size_t)NS2 * ROWS;   // the sine rows (dy > 0)
    float c0 = 0.f, s0 = 0.f, cC[4], sS[4], sC[4], cS[4];
    int ix[4];
#pragma unroll
    for (int i = 0; i < 4; i++) {
        cC[i] = sS[i] = sC[i] = cS[i] = 0.f;
        ix[i] = i + 1 < x.ndxh ? (int)(((long)hx * x.dxm[i]) % Lf) : 0;
    }
    constexpr int UB = 8;
    for (int k0 = 0; k0 < ncol; k0 += UB) {
        float vc[UB], vs[UB];
#pragma unroll
        for (int u = 0; u < UB; u++) {
            const bool in = k0 + u < ncol;
            vc[u] = in ? wc[(size_t)(k0 + u) * stride] : 0.f;
            vs[u] = in && dyi > 0 ? ws[(size_t)(k0 + u) * stride] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < UB; u++) {
            if (k0 + u >= ncol) break;
            const float f = k0 + u == fix0 || k0 + u == fix1 ? 0.5f : 1.f;
            const float C = f * vc[u], S = f * vs[u];
            c0 += C;
            s0 += S;
#pragma unroll
            for (int i = 0; i < 4; i++) {
                if (i + 1 >= x.ndxh) break;
                const float2 p = ptab[ix[i]];   // (cos, -sin)
                cC[i] = fmaf(p.x, C, cC[i]);
                sS[i] = fmaf(-p.y, S, sS[i]);
                sC[i] = fmaf(-p.y, C, sC[i]);
                cS[i] = fmaf(p.x, S, cS[i]);
                ix[i] += x.dxm[i];
                if (ix[i] >= Lf) ix[i] -= Lf;
            }
        }
    }
    auto put = [&](int xi, float re, float im) {   // xi: signed dx index
        const int d = x.dslot[4 + xi][dyi];
        if (d < 0) return;
        float2 v = make_float2(re, WHICH == 0 ? im : -im);
        if (WHICH == 0) {
            const int dx = xi < 0 ? -x.dxs[-xi] : x.dxs[xi];
            const float2 p = ptab[(int)(((long long)sx * dx + (long long)sy * x.dys[dyi]) % Lf + Lf) % Lf];
            v = make_float2(p.x * v.x - p.y * v.y, p.x * v.y + p.y * v.x);
        }
        x.acc[(((size_t)slot * x.nd + d) * NS2 + c) * NS2 + r % NS2] = v;
    };
    put(0, c0, s0);
#pragma unroll
    for (int i = 0; i < 4; i++) {
        if (i + 1 >= x.ndxh) break;
        put(i + 1, cC[i] - sS[i], sC[i] + cS[i]);
        put(-(i + 1), cC[i] + sS[i], cS[i] - sC[i]);
    }
}

}  // namespace

bool loops_tc_supported(const tufrg_model *m)
{
    int ndyh = 0;
    for (int v : m->dys) ndyh += v >= 0;
    return m->precision == TUFRG_SPLIT32 && m->ns == NS && ndyh <= NDYM && (int)m->dxs.size() <= 9 && m->Lf <= 4096;
}

// Groups of at most GRP list positions whose momenta share q_x (their half sums then run over the same columns).
std::vector<int> loops_tc_groups(const std::vector<int> &q_of_slot, int Lq)
{
    std::vector<std::vector<int>> by(Lq);
    for (size_t i = 0; i < q_of_slot.size(); i++) by[q_of_slot[i] / Lq].push_back((int)i);
    std::vector<int> g;
    for (auto &v : by)
        for (size_t i = 0; i < v.size(); i += GRP)
            for (size_t j = 0; j < GRP; j++) g.push_back(i + j < v.size() ? v[i + j] : -1);
    return g;
}

// columns of the sums: a list of momenta in any order (no groups) runs over the whole mesh
static int tc_cols(const tufrg_model *m, bool half) { return half ? m->Lf / 2 + 1 : m->Lf; }

size_t loops_tc_w_bytes(const tufrg_model *m)
{
    const size_t n_slot = m->sym ? m->n_loop_q : m->Nq;
    const size_t listed = (n_slot + GRP - 1) / GRP * m->Lf;                            // a shard's list: the whole mesh
    const size_t grouped = (size_t)m->n_tc_groups * tc_cols(m, m->sym_inv >= 0);       // (without inversion C is not halved)
    return std::max(listed, grouped) * COLS * ROWS * sizeof(float);
}

cudaError_t launch_loops_rho(tufrg_model *m)
{
    const size_t n = (size_t)m->Nk * NS2 * NS;
    loops_rho_kernel<<<(unsigned)((n + 255) / 256), 256, 0, m->stream>>>(m->d_U, n, m->d_rho);
    return cudaGetLastError();
}

// Loop column sums of one channel on the tensor cores, then the x phases into the accumulator slots of the
// multi-orbital path (one kx range): acc[slot][d][c][c'] for the half-plane d, real components (loop_comp).
cudaError_t launch_loops_tc(tufrg_model *m, int ch, bool half, float2 *acc)
{
    const int *grp = m->loop_list_is_reps ? m->d_tc_grp : nullptr;
    LtArgs a{};
    a.rho = m->d_rho;
    a.ft = m->d_ft32;
    a.W = reinterpret_cast<float *>(m->d_loop_w);
    a.s_list = m->sym ? m->d_loop_list : nullptr;
    a.grp = grp;
    a.n_slot = m->sym ? m->n_loop_q : m->Nq;
    const int n_groups = grp ? m->n_tc_groups : (a.n_slot + GRP - 1) / GRP;
    a.half = half ? 1 : 0;
    a.ncol = tc_cols(m, half);
    a.n_items = n_groups * a.ncol;
    a.Lq = m->Lq;
    a.nc = m->nc;
    a.Lf = m->Lf;
    a.spc = (m->Lf + KB - 1) / KB;
    XsArgs x{};
    std::vector<int> dxh;
    for (int v : m->dys)
        if (v >= 0) x.dys[x.ndyh++] = v;
    for (int v : m->dxs)
        if (v >= 0) dxh.push_back(v);
    a.dy1 = x.ndyh > 1 ? x.dys[1] % m->Lf : 0;
    a.dy2 = x.ndyh > 2 ? x.dys[2] % m->Lf : 0;
    a.ptab = m->d_lph32;
    a.Tp = m->d_scal;
    a.thr_factor = 1e-2f;
    a.shell_T = m->regulator == TUFRG_REG_MOMENTUM_SHELL ? (float)m->T_reg : 0.f;
    a.err = m->d_err;
    auto kern = ch == 0 ? loops_tc_kernel<0> : loops_tc_kernel<1>;
    const size_t smem_k = lt_smem_bytes(m->Lf);
    TUFRG_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_k));
    {
        PhaseScope ps(m, PH_LOOPS);
        kern<<<std::min(a.n_items, m->sm_count), NTHREADS, smem_k, m->stream>>>(a);
        TUFRG_CUDA_TRY(cudaGetLastError());
    }
    x.W = a.W;
    x.acc = acc;
    x.s_list = a.s_list;
    x.grp = grp;
    x.n_slot = a.n_slot;
    x.n_groups = n_groups;
    x.Lq = m->Lq;
    x.nc = m->nc;
    x.Lf = m->Lf;
    x.nd = m->nd;
    x.ncol = a.ncol;
    x.half = a.half;
    x.ptab = m->d_lph32;
    x.ndxh = (int)dxh.size();
    for (int i = 0; i < x.ndxh; i++) {
        x.dxs[i] = dxh[i];
        if (i > 0) x.dxm[i - 1] = dxh[i] % m->Lf;
    }
    for (int i = 0; i < 9; i++)
        for (int jy = 0; jy < NDYM; jy++) {
            x.dslot[i][jy] = -1;
            const int xi = i - 4;
            if (jy >= x.ndyh || std::abs(xi) >= x.ndxh) continue;
            const int dx = xi < 0 ? -dxh[-xi] : dxh[xi], dy = x.dys[jy];
            if (!(dy > 0 || dx >= 0)) continue;
            for (int d = 0; d < m->nd; d++)
                if (m->deltas[2 * d] == dx && m->deltas[2 * d + 1] == dy) x.dslot[i][jy] = d;
        }
    const size_t n = (size_t)n_groups * x.ndyh * NS2 * ROWS;
    const size_t smem = sizeof(float2) * (size_t)m->Lf;
    auto xk = ch == 0 ? loops_tc_xsum<0> : loops_tc_xsum<1>;
    if (smem > 48 * 1024) TUFRG_CUDA_TRY(cudaFuncSetAttribute(xk, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    PhaseScope ps(m, PH_LOOPRED);
    xk<<<(unsigned)((n + 255) / 256), 256, smem, m->stream>>>(x);
    return cudaGetLastError();
}

}  // namespace tufrg
