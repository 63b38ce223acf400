// Split-precision (FP32) loop k-sum for N_s = 2 over the whole fine mesh, as split-precision flows (and
// tufrg_loops_noalloc) take it; right-hand sides outside of flows, and FP64, take k_loops2h.cu, which sums half of the mesh
// and is faster.  Flows keep this order of summation: an adaptive flow that ends at a divergence turns a change of
// rounding in the loops (1e-7) into percents of its last state (and 1e-5 .. 1e-4 of the critical scale) through the
// steps it accepts, so a flow's results, and flows resumed from stored checkpoints, stay those they always were.
//
// Same sums as k_loops2h.cu (Eqs. loopminus / loopplus dressed by Eq. trafo), organised
// around the structure of the two-band problem:
//   * the band projectors are complete and rank one: rho^1 = 1 - rho^0 and
//     rho^0_00 + rho^0_11 = 1, so one 48-byte record per fine k holds
//     (rho^0_00, Re rho^0_01, Im rho^0_01) and the Fermi data (e_l, g_l = df/dT,
//     gp_l = dg/de), rewritten once per temperature;
//   * with D = T^0 - T^1, Y = 1 (x) T^1 + rho1^0 (x) D, where
//     T^{l1} = w_{l1 1} 1 + (w_{l1 0} - w_{l1 1}) rho2^0;  Y is Hermitian in the sense
//     Y[(t3 t1),(t4 t2)] = conj(Y[(t1 t3),(t2 t4)]), so only 4 real and 6 complex
//     entries are formed;
//   * the row sums W[dy] = sum_ky e^{-i ky dy} Y keep, for each complex pair
//     (Z, conj Z), the real sums of c Re Z, s Im Z, c Im Z, s Re Z, which give both
//     members; dy = 0 needs no phase;
//   * the records are stored as three float4 planes transposed to [ky][kx], so the
//     32 columns of a warp read 512 contiguous bytes per plane (coalesced), and each
//     thread loads the next row while it computes the current one; rows advance
//     without integer division.
// One thread per fine-mesh column, one CTA per (transfer momentum, 64 columns, row range).
// A warp's columns leave one partial sum; a deterministic reduction kernel finishes the sum.
#include <algorithm>
#include <cmath>

#include "tufrg_internal.cuh"

namespace tufrg {
namespace {

constexpr int MAXD = 9;
constexpr int WARPS = 2;

constexpr int RECF4 = 3;         // float4 planes per record
constexpr int RING = 4;          // rows of records in flight per thread (asynchronous copies into shared memory)

// Shared memory of one CTA: the phase table, then one region per warp that holds the warp's ring of
// record rows during the k-sum ([RING][2 sides x 3 planes][32 lanes] float4) and its flush buffer
// (32 x (2 NDYH 16 + 1) floats) after it.
__host__ __device__ constexpr size_t warp_region_bytes(int ndyh)
{
    return ((sizeof(float) * 32 * (2 * ndyh * 16 + 1) > sizeof(float4) * RING * 2 * RECF4 * 32
                 ? sizeof(float) * 32 * (2 * ndyh * 16 + 1)
                 : sizeof(float4) * RING * 2 * RECF4 * 32) + 15) & ~size_t(15);
}
inline size_t loops2_smem_bytes(int Lf, int ndyh)
{
    return ((sizeof(float2) * Lf + 15) & ~size_t(15)) + WARPS * warp_region_bytes(ndyh);
}

struct Args2 {
    const float4 *rec;       // [3][Lf][Lf] planes, index [j][ky][kx]:
                             //   (rho00, Re rho01, Im rho01, e0), (e1, g0, g1, gp0), (gp1, -, -, -)
    float2 *part;            // [Nq][n_part][ndx][ndyh][16]
    int Lq, nc, Lf, ndx, ndyh;
    int dxs[MAXD], dys[MAXD];
    unsigned needed[MAXD];
    int ky_chunks, ky_len;
    float thr;               // degenerate-pair switch, used when Tp is null
    const double *Tp;        // device flow scale (T, or Lambda with the momentum shell): switch = 1e-2 * T
    float shell_T;           // > 0: momentum-shell regulator at this fixed temperature (records hold f, h)
    const int *s_list;       // optional: CTA x evaluates transfer momentum s_list[x] (partials indexed by x)
    const int *skip;         // optional: the whole launch returns at once when *skip != 0
    const float2 *ptab;      // optional: e^{-2 pi i n / Lf}, n < Lf (computed in the kernel when null)
};

// (t1,t3,t2,t4) -> ab index of the compact loop (P: a=(t2,t1), b=(t4,t3); C: a=(t1,t2), b=(t3,t4))
template <int WHICH>
__host__ __device__ constexpr int abx(int t1, int t3, int t2, int t4)
{
    return WHICH == 0 ? ((t2 * 2 + t1) * 4 + t4 * 2 + t3) : ((t1 * 2 + t2) * 4 + t3 * 2 + t4);
}

template <int WHICH, bool SHELL>
__device__ __forceinline__ float pw(float e1, float g1, float gp1, float e2, float g2, float gp2, float thr, float lam)
{
    if (SHELL) return shell_weight<WHICH, float>(e1, g1, gp1, e2, g2, gp2, thr, lam);   // (g, gp) = (f, h)
    if (WHICH == 0) {
        const float s = e1 + e2;
        return fabsf(s) > thr ? -__fdividef(g1 + g2, s) : -0.5f * (gp1 + gp2);
    } else {
        const float d = e1 - e2;
        return fabsf(d) > thr ? __fdividef(g1 - g2, d) : 0.5f * (gp1 + gp2);
    }
}

// The sums of one CTA: row range kyc of a column block of one transfer momentum.
// SHELL: momentum-shell regulator (a separate instantiation, so that the temperature flow's code is unchanged)
template <int NDYH, int WHICH, bool SHELL>
__device__ __forceinline__ void loops2_body(const Args2 &a, const int kyc)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2 *ptab = reinterpret_cast<float2 *>(smem_raw);
    const int Lf = a.Lf;
    if (a.ptab) {
        for (int n = threadIdx.x; n < Lf; n += blockDim.x) ptab[n] = a.ptab[n];
    } else {
        for (int n = threadIdx.x; n < Lf; n += blockDim.x) {
            double sn, cs;
            sincospi(2.0 * (double)n / (double)Lf, &sn, &cs);
            ptab[n] = make_float2((float)cs, (float)-sn);   // e^{-2 pi i n / Lf}
        }
    }
    __syncthreads();

    constexpr int NT = 32 * WARPS;
    const int s = blockIdx.x;                                    // slot of the partial sums
    const int sq = a.s_list ? a.s_list[blockIdx.x] : blockIdx.x;  // transfer momentum
    const int sx = (sq / a.Lq) * a.nc, sy = (sq % a.Lq) * a.nc;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned char *region = smem_raw + ((sizeof(float2) * Lf + 15) & ~size_t(15)) + warp * warp_region_bytes(NDYH);
    float4 *ring = reinterpret_cast<float4 *>(region);   // [RING][6][32]: rows in flight of this warp's columns
    const int kx = blockIdx.y * NT + threadIdx.x;
    // temperature flow: the scale is T; momentum shell: the scale is Lambda and the temperature is fixed
    const float lam = SHELL ? (float)*a.Tp : 0.f;
    const float thr = SHELL ? 1e-2f * a.shell_T : (a.Tp ? (float)(1e-2 * *a.Tp) : a.thr);
    const bool valid = kx < Lf;
    const int ky0 = kyc * a.ky_len;
    const int ky1 = min(Lf, ky0 + a.ky_len);

    float R0[4], P0y[6], P0z[6];
    float Rc[NDYH > 1 ? NDYH - 1 : 1][4], Rs[NDYH > 1 ? NDYH - 1 : 1][4];
    float Pcy[NDYH > 1 ? NDYH - 1 : 1][6], Psz[NDYH > 1 ? NDYH - 1 : 1][6];
    float Pcz[NDYH > 1 ? NDYH - 1 : 1][6], Psy[NDYH > 1 ? NDYH - 1 : 1][6];
#pragma unroll
    for (int j = 0; j < 4; j++) R0[j] = 0.f;
#pragma unroll
    for (int j = 0; j < 6; j++) { P0y[j] = 0.f; P0z[j] = 0.f; }
#pragma unroll
    for (int i = 0; i < NDYH - 1; i++) {
#pragma unroll
        for (int j = 0; j < 4; j++) { Rc[i][j] = 0.f; Rs[i][j] = 0.f; }
#pragma unroll
        for (int j = 0; j < 6; j++) { Pcy[i][j] = 0.f; Psz[i][j] = 0.f; Pcz[i][j] = 0.f; Psy[i][j] = 0.f; }
    }

    if (valid && ky0 < ky1) {
        // columns of k1 and k2; rows step by +1 on the q side and by -1 on the s - q side
        const int k1x = WHICH == 0 ? (sx - kx + Lf) % Lf : kx;
        const int k2x = WHICH == 0 ? kx : (kx - sx + Lf) % Lf;
        int k1y = WHICH == 0 ? ((sy - ky0) % Lf + Lf) % Lf : ky0;
        int k2y = WHICH == 0 ? ky0 : ((ky0 - sy) % Lf + Lf) % Lf;
        const size_t plane = (size_t)Lf * Lf;
        int o1 = k1y * Lf + k1x, o2 = k2y * Lf + k2x;        // offsets of the next row to be copied
        const int wrap = (Lf - 1) * Lf;
        // copy one row (both sides, three planes) into ring slot sl, then step the offsets to the next
        // row: the q side moves by +Lf, the s - q side by -Lf (P), both +Lf (C), with wrap
        auto issue_row = [&](int sl) {
            float4 *r = ring + sl * 2 * RECF4 * 32 + lane;
#pragma unroll
            for (int pl = 0; pl < RECF4; pl++) {
                cp_async16(r + pl * 32, a.rec + pl * plane + o1);
                cp_async16(r + (RECF4 + pl) * 32, a.rec + pl * plane + o2);
            }
            if (WHICH == 0) { o1 = o1 >= Lf ? o1 - Lf : o1 + wrap; o2 = o2 < wrap ? o2 + Lf : o2 - wrap; }
            else            { o1 = o1 < wrap ? o1 + Lf : o1 - wrap; o2 = o2 < wrap ? o2 + Lf : o2 - wrap; }
        };
#pragma unroll
        for (int i = 0; i < RING - 1; i++) {   // rows ky0 .. ky0 + RING - 2 in flight
            if (ky0 + i < ky1) issue_row(i);
            cp_async_commit();
        }
        int pn[MAXD];
#pragma unroll
        for (int i = 1; i < NDYH; i++) pn[i] = (int)(((long)ky0 * a.dys[i]) % Lf);
        const float sgn = WHICH == 0 ? 1.f : -1.f;
        for (int ky = ky0; ky < ky1; ky++) {
            const int it = ky - ky0;
            if (ky + RING - 1 < ky1) issue_row((it + RING - 1) & (RING - 1));
            cp_async_commit();
            cp_async_wait<RING - 1>();   // this thread's copies of row ky have landed
            const float4 *r = ring + (it & (RING - 1)) * 2 * RECF4 * 32 + lane;
            const float4 a0 = r[0], a1 = r[32], a2 = r[64], b0 = r[96], b1 = r[128], b2 = r[160];
            // pair weights w[l1][l2]: l1 on k1, l2 on k2
            const float e1[2] = {a0.w, a1.x}, g1[2] = {a1.y, a1.z}, gp1[2] = {a1.w, a2.x};
            const float e2[2] = {b0.w, b1.x}, g2[2] = {b1.y, b1.z}, gp2[2] = {b1.w, b2.x};
            float w[2][2];
#pragma unroll
            for (int l1 = 0; l1 < 2; l1++)
#pragma unroll
                for (int l2 = 0; l2 < 2; l2++) w[l1][l2] = pw<WHICH, SHELL>(e1[l1], g1[l1], gp1[l1], e2[l2], g2[l2], gp2[l2], thr, lam);
            // T^{l1} = w_{l1 1} 1 + (w_{l1 0} - w_{l1 1}) rho2'^0 ;  D = T^0 - T^1
            const float A2 = b0.x, C2r = b0.y, C2i = sgn * b0.z;    // rho2' = rho2 (P) or conj(rho2) (C)
            const float dw0 = w[0][0] - w[0][1], dw1 = w[1][0] - w[1][1];
            const float T1_00 = fmaf(dw1, A2, w[1][1]), T1_11 = fmaf(dw1, 1.f - A2, w[1][1]);
            const float T1r = dw1 * C2r, T1i = dw1 * C2i;
            const float dd = dw0 - dw1, dd0 = w[0][1] - w[1][1];
            const float D00 = fmaf(dd, A2, dd0), D11 = fmaf(dd, 1.f - A2, dd0);
            const float Dr = dd * C2r, Di = dd * C2i;
            // Y = 1 (x) T^1 + rho1^0 (x) D: 4 real and 6 complex independent entries
            const float A1 = a0.x, B1 = 1.f - a0.x, C1r = a0.y, C1i = a0.z;
            float X[4], Zy[6], Zz[6];
            X[0] = fmaf(A1, D00, T1_00);    // Y[00][00]
            X[1] = fmaf(A1, D11, T1_11);    // Y[00][11]
            X[2] = fmaf(B1, D00, T1_00);    // Y[11][00]
            X[3] = fmaf(B1, D11, T1_11);    // Y[11][11]
            Zy[0] = fmaf(A1, Dr, T1r); Zz[0] = fmaf(A1, Di, T1i);   // Y[00][01]
            Zy[1] = fmaf(B1, Dr, T1r); Zz[1] = fmaf(B1, Di, T1i);   // Y[11][01]
            Zy[2] = C1r * D00; Zz[2] = C1i * D00;                   // Y[01][00]
            Zy[3] = C1r * D11; Zz[3] = C1i * D11;                   // Y[01][11]
            Zy[4] = C1r * Dr - C1i * Di; Zz[4] = C1r * Di + C1i * Dr;   // Y[01][01] = rho01 D01
            Zy[5] = C1r * Dr + C1i * Di; Zz[5] = C1i * Dr - C1r * Di;   // Y[01][10] = rho01 conj(D01)
            // row sums
#pragma unroll
            for (int j = 0; j < 4; j++) R0[j] += X[j];
#pragma unroll
            for (int j = 0; j < 6; j++) { P0y[j] += Zy[j]; P0z[j] += Zz[j]; }
#pragma unroll
            for (int i = 1; i < NDYH; i++) {
                const float2 ph = ptab[pn[i]];
                pn[i] += a.dys[i];
                if (pn[i] >= Lf) pn[i] -= Lf;
#pragma unroll
                for (int j = 0; j < 4; j++) { Rc[i - 1][j] = fmaf(ph.x, X[j], Rc[i - 1][j]); Rs[i - 1][j] = fmaf(ph.y, X[j], Rs[i - 1][j]); }
#pragma unroll
                for (int j = 0; j < 6; j++) {
                    Pcy[i - 1][j] = fmaf(ph.x, Zy[j], Pcy[i - 1][j]);
                    Psz[i - 1][j] = fmaf(ph.y, Zz[j], Psz[i - 1][j]);
                    Pcz[i - 1][j] = fmaf(ph.x, Zz[j], Pcz[i - 1][j]);
                    Psy[i - 1][j] = fmaf(ph.y, Zy[j], Psy[i - 1][j]);
                }
            }
        }
        cp_async_wait<0>();   // nothing in flight before the region is reused below (trailing groups are empty)
    }

    // ---- rebuild W[dy][ab] from the paired sums
    constexpr int XR[4] = {abx<WHICH>(0, 0, 0, 0), abx<WHICH>(0, 0, 1, 1), abx<WHICH>(1, 1, 0, 0), abx<WHICH>(1, 1, 1, 1)};
    constexpr int ZA[6] = {abx<WHICH>(0, 0, 0, 1), abx<WHICH>(1, 1, 0, 1), abx<WHICH>(0, 1, 0, 0),
                           abx<WHICH>(0, 1, 1, 1), abx<WHICH>(0, 1, 0, 1), abx<WHICH>(0, 1, 1, 0)};
    constexpr int ZB[6] = {abx<WHICH>(0, 0, 1, 0), abx<WHICH>(1, 1, 1, 0), abx<WHICH>(1, 0, 0, 0),
                           abx<WHICH>(1, 0, 1, 1), abx<WHICH>(1, 0, 1, 0), abx<WHICH>(1, 0, 0, 1)};
    float2 W[NDYH][16];
#pragma unroll
    for (int j = 0; j < 4; j++) W[0][XR[j]] = make_float2(R0[j], 0.f);
#pragma unroll
    for (int j = 0; j < 6; j++) {
        W[0][ZA[j]] = make_float2(P0y[j], P0z[j]);
        W[0][ZB[j]] = make_float2(P0y[j], -P0z[j]);
    }
#pragma unroll
    for (int i = 1; i < NDYH; i++) {
#pragma unroll
        for (int j = 0; j < 4; j++) W[i][XR[j]] = make_float2(Rc[i - 1][j], Rs[i - 1][j]);
#pragma unroll
        for (int j = 0; j < 6; j++) {
            W[i][ZA[j]] = make_float2(Pcy[i - 1][j] - Psz[i - 1][j], Pcz[i - 1][j] + Psy[i - 1][j]);
            W[i][ZB[j]] = make_float2(Pcy[i - 1][j] + Psz[i - 1][j], Psy[i - 1][j] - Pcz[i - 1][j]);
        }
    }

    // ---- flush: per distinct dx, multiply by e^{-i kx dx}, sum the warp through smem
    constexpr int NV = 2 * NDYH * 16;
    constexpr int PITCH = NV + 1;
    float *buf = reinterpret_cast<float *>(region);
    __syncwarp();   // every lane of the warp is done with its ring entries (lanes past Lf skipped the k-sum)
    const int n_part = gridDim.y * WARPS * a.ky_chunks;
    const int p = (blockIdx.y * WARPS + warp) * a.ky_chunks + kyc;
    for (int dxi = 0; dxi < a.ndx; dxi++) {
        if (a.needed[dxi] == 0) continue;
        const int n = (int)((((long)kx * a.dxs[dxi]) % Lf + Lf) % Lf);
        const float2 phx = valid ? ptab[n] : make_float2(0.f, 0.f);
#pragma unroll
        for (int i = 0; i < NDYH; i++)
#pragma unroll
            for (int j = 0; j < 16; j++) {
                buf[lane * PITCH + 2 * (i * 16 + j)] = phx.x * W[i][j].x - phx.y * W[i][j].y;
                buf[lane * PITCH + 2 * (i * 16 + j) + 1] = phx.x * W[i][j].y + phx.y * W[i][j].x;
            }
        __syncwarp();
        for (int v = lane; v < NV; v += 32) {
            float acc = 0.f;
#pragma unroll 8
            for (int r = 0; r < 32; r++) acc += buf[r * PITCH + v];
            const int i = v / 32, j = (v / 2) % 16, re = v & 1;
            if ((a.needed[dxi] >> i) & 1u) {
                const size_t o = ((((size_t)s * n_part + p) * a.ndx + dxi) * a.ndyh + i) * 16 + j;
                reinterpret_cast<float *>(a.part)[2 * o + re] = acc;
            }
        }
        __syncwarp();
    }
}

constexpr int NS2 = 4, NS4 = 16;

// Sum the partials of list position s in a fixed order and scale by 1/Nk; the half-plane partials
// give both Hermitian halves.  The sum runs in the partials' own precision (FP32 on the split path:
// this GPU's FP64 rate would make the reduction, not the memory traffic, its bound), with 16 loads
// in flight per thread (the additions keep their sequential order).
template <typename R>
__device__ __forceinline__ typename cpx<R>::t reduce_one(const typename cpx<R>::t *__restrict__ part, int n_part,
                                                         int ndx, int ndyh, const int *dslot, const int *deltas, int s,
                                                         int d, int ab, R inv_nk)
{
    using C2 = typename cpx<R>::t;
    const int dx = deltas[2 * d], dy = deltas[2 * d + 1];
    const bool half = dy > 0 || (dy == 0 && dx >= 0);
    const int ia = ab / NS2, ib = ab % NS2;
    const int src_ab = half ? ab : ib * NS2 + ia;
    const int slot = dslot[d];   // dxi * ndyh + dyi of the half-plane representative of +-delta
    const size_t stride = (size_t)ndx * ndyh * NS4;
    const C2 *src = part + (size_t)s * n_part * stride + (size_t)slot * NS4 + src_ab;
    R re = 0, im = 0;
    constexpr int UB = 16;
    int p = 0;
    for (; p + UB <= n_part; p += UB) {
        C2 v[UB];
#pragma unroll
        for (int j = 0; j < UB; j++) v[j] = src[(size_t)(p + j) * stride];
#pragma unroll
        for (int j = 0; j < UB; j++) {
            re += v[j].x;
            im += v[j].y;
        }
    }
    for (; p < n_part; p++) {
        const C2 v = src[(size_t)p * stride];
        re += v.x;
        im += v.y;
    }
    return mk(re * inv_nk, (half ? im : -im) * inv_nk);
}

__device__ __forceinline__ double2 to64(float2 v) { return make_double2(widen_f(v.x), widen_f(v.y)); }

// Grid: blockIdx.y = transfer momentum (list position), blockIdx.z = channel (skipped when not in chmask;
// its partials and outputs are offset by part_cs and out_cs), threads over (d, ab) = t (t >> 4, t & 15):
// no runtime integer division (this GPU issues its conversions to the slow FP64 pipe).  List position s
// is written at momentum qout[s] (orbit representatives only) or at s.
template <typename R>
__global__ void loops_reduce_kernel(const typename cpx<R>::t *__restrict__ part, int n_part, int ndx, int ndyh,
                                    const int *dslot, const int *deltas, int nd, double inv_nk, const int *qout,
                                    double2 *out64, typename cpx<R>::t *out32, const int *skip, int chmask,
                                    size_t part_cs, size_t out_cs)
{
    grid_wait();
    if (skip && *skip) return;
    const int ch = blockIdx.z;
    if (!((chmask >> ch) & 1)) return;
    part += ch * part_cs;
    if (out64) out64 += ch * out_cs;
    if (out32) out32 += ch * out_cs;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nd * NS4) return;
    const int s = blockIdx.y, d = t / NS4, ab = t % NS4;
    const auto v = reduce_one<R>(part, n_part, ndx, ndyh, dslot, deltas, s, d, ab, R(inv_nk));
    const size_t idx = (size_t)(qout ? qout[s] : s) * nd * NS4 + t;
    if (out64) out64[idx] = to64(v);
    if (out32) out32[idx] = v;
}

// Symmetry variant (two bands), gather form: blockIdx.y = output momentum q'; qmap[q'] = (list
// position i of its orbit representative, group element e).  Thread (d', a'b') reads the representative's
// partial sums of d = dinv[e][d'], a = src[a'], b = src[b'] (L2 resident) and writes
// Lc(q')[d'][a'][b'] = i^(qt[a'] - qt[b']) (conj ? conj(v) : v) coalesced (see SymElem).
template <typename C2>
__device__ __forceinline__ C2 quarter_turn(C2 v, int k)
{
    switch (k & 3) {
    case 0: return v;
    case 1: return mk(-v.y, v.x);
    case 2: return mk(-v.x, -v.y);
    default: return mk(v.y, -v.x);
    }
}

template <typename R>
__global__ void loops_reduce_sym_kernel(const typename cpx<R>::t *__restrict__ part, int n_part, int ndx, int ndyh,
                                        const int *dslot, const int *deltas, int nd, const int2 *qmap,
                                        const SymElem *elem, const int *dinv, double inv_nk, double2 *out64,
                                        typename cpx<R>::t *out32, const int *skip, int chmask, size_t part_cs,
                                        size_t out_cs)
{
    if (skip && *skip) return;
    const int ch = blockIdx.z;   // as in loops_reduce_kernel
    if (!((chmask >> ch) & 1)) return;
    part += ch * part_cs;
    if (out64) out64 += ch * out_cs;
    if (out32) out32 += ch * out_cs;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nd * NS4) return;
    const int q2 = blockIdx.y, d2 = t / NS4, a2 = (t / NS2) % NS2, b2 = t % NS2;
    const int2 ie = qmap[q2];
    const SymElem &e = elem[ie.y];
    const int d = dinv[ie.y * nd + d2], a = e.src[ch][a2], b = e.src[ch][b2];
    auto v = reduce_one<R>(part, n_part, ndx, ndyh, dslot, deltas, ie.x, d, a * NS2 + b, R(inv_nk));
    if (e.conj) v.y = -v.y;
    const auto w = quarter_turn(v, e.qt[ch][a2] - e.qt[ch][b2]);
    const size_t o = (size_t)q2 * nd * NS4 + t;
    if (out64) out64[o] = to64(w);
    if (out32) out32[o] = w;
}

// one channel
template <int NDYH, int WHICH, bool SHELL = false>
__global__ void __launch_bounds__(32 * WARPS) loops2_kernel(Args2 a)
{
    grid_release();
    if (a.skip && *a.skip) return;   // uniform over the grid
    loops2_body<NDYH, WHICH, SHELL>(a, blockIdx.z);
}

// both channels (blockIdx.z: channel, row range): the C channel's CTAs run beside the P channel's, which on small meshes
// fill a fraction of the SMs (8 x 8 transfer, 128 x 128 fine mesh, 15 representatives, 3 row ranges: 180 CTAs of two
// warps for both).  Latency bound there, 22 us for both channels.
template <int NDYH, bool SHELL>
__global__ void __launch_bounds__(32 * WARPS) loops2_both_kernel(Args2 a, size_t part_cs)
{
    grid_release();
    grid_wait();
    if (a.skip && *a.skip) return;
    if ((int)blockIdx.z < a.ky_chunks) {
        loops2_body<NDYH, 0, SHELL>(a, blockIdx.z);
    } else {
        a.part += part_cs;
        loops2_body<NDYH, 1, SHELL>(a, blockIdx.z - a.ky_chunks);
    }
}

template <int NDYH>
cudaError_t launch2_both(tufrg_model *m, const Args2 &a, int n_s, size_t part_cs)
{
    const dim3 grid(n_s, (m->Lf + 32 * WARPS - 1) / (32 * WARPS), 2 * a.ky_chunks);
    const size_t smem = loops2_smem_bytes(m->Lf, NDYH);
    auto kern = a.shell_T > 0.f ? loops2_both_kernel<NDYH, true> : loops2_both_kernel<NDYH, false>;
    if (smem > 48 * 1024) TUFRG_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    PhaseScope ps(m, PH_LOOPS);
    return launch_chained(kern, grid, 32 * WARPS, smem, m->stream, loops_chained(m), a, part_cs);
}

template <int NDYH, int WHICH>
cudaError_t launch2(tufrg_model *m, const Args2 &a, int n_s)
{
    dim3 grid(n_s, (m->Lf + 32 * WARPS - 1) / (32 * WARPS), a.ky_chunks);
    const size_t smem = loops2_smem_bytes(m->Lf, NDYH);
    auto kern = a.shell_T > 0.f ? loops2_kernel<NDYH, WHICH, true> : loops2_kernel<NDYH, WHICH, false>;
    if (smem > 48 * 1024) TUFRG_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    PhaseScope ps(m, PH_LOOPS);
    kern<<<grid, 32 * WARPS, smem, m->stream>>>(a);
    return cudaGetLastError();
}

}  // namespace

// Resident CTAs per SM of the instantiation this model launches (occupancy API).
int loops2_blocks_per_sm(const tufrg_model *m)
{
    int ndyh = 0;
    for (int v : m->dys) ndyh += v >= 0;
    const size_t smem = loops2_smem_bytes(m->Lf, ndyh);
    switch (ndyh) {
    case 1: return resident_ctas(loops2_kernel<1, 0>, 32 * WARPS, smem);
    case 2: return resident_ctas(loops2_kernel<2, 0>, 32 * WARPS, smem);
    case 3: return resident_ctas(loops2_kernel<3, 0>, 32 * WARPS, smem);
    case 4: return resident_ctas(loops2_kernel<4, 0>, 32 * WARPS, smem);
    case 5: return resident_ctas(loops2_kernel<5, 0>, 32 * WARPS, smem);
    default: return 0;
    }
}

static Args2 loops2_args(const tufrg_model *m, const int *s_list, float2 *part, const int *skip)
{
    const LoopPlan &pl = m->plan;
    Args2 a{};
    a.rec = static_cast<const float4 *>(m->d_rec);
    a.part = part;
    a.s_list = s_list;
    a.skip = skip;
    a.Lq = m->Lq; a.nc = m->nc; a.Lf = m->Lf;
    a.ndx = (int)m->dxs.size();
    int ndyh = 0;
    for (int v : m->dys)
        if (v >= 0) a.dys[ndyh++] = v;
    a.ndyh = ndyh;
    for (int i = 0; i < a.ndx; i++) {
        a.dxs[i] = m->dxs[i];
        a.needed[i] = 0;
        for (int j = 0; j < ndyh; j++) {
            const int dx = m->dxs[i], dy = a.dys[j];
            bool in = false;
            for (int d = 0; d < m->nd; d++) in |= (m->deltas[2 * d] == dx && m->deltas[2 * d + 1] == dy);
            if (in && (dy > 0 || dx >= 0)) a.needed[i] |= 1u << j;
        }
    }
    a.ky_chunks = pl.ky_chunks;
    a.ky_len = (m->Lf + pl.ky_chunks - 1) / pl.ky_chunks;
    a.thr = 0.f;
    a.Tp = m->d_scal;
    a.shell_T = m->regulator == TUFRG_REG_MOMENTUM_SHELL ? (float)m->T_reg : 0.f;
    a.ptab = m->d_lph32;
    return a;
}

// Loop sums of channel ch into the partial buffer (no reduction).  With s_list, only the
// listed transfer momenta (n_list of them) are evaluated, into partial slots 0..n_list-1 of part.
cudaError_t launch_loops2_ex(tufrg_model *m, int ch, const int *s_list, int n_list, float2 *part, const int *skip)
{
    const Args2 a = loops2_args(m, s_list, part, skip);
    const int n_s = s_list ? n_list : m->Nq;
    switch (a.ndyh) {
    case 1: return ch == 0 ? launch2<1, 0>(m, a, n_s) : launch2<1, 1>(m, a, n_s);
    case 2: return ch == 0 ? launch2<2, 0>(m, a, n_s) : launch2<2, 1>(m, a, n_s);
    case 3: return ch == 0 ? launch2<3, 0>(m, a, n_s) : launch2<3, 1>(m, a, n_s);
    case 4: return ch == 0 ? launch2<4, 0>(m, a, n_s) : launch2<4, 1>(m, a, n_s);
    case 5: return ch == 0 ? launch2<5, 0>(m, a, n_s) : launch2<5, 1>(m, a, n_s);
    default: return cudaErrorNotSupported;
    }
}

cudaError_t launch_loops2(tufrg_model *m, int ch)
{
    // with loop symmetries only the orbit representatives are summed (partial slots = list positions)
    return launch_loops2_ex(m, ch, m->sym ? m->d_loop_list : nullptr, m->sym ? m->n_loop_q : 0,
                            reinterpret_cast<float2 *>(m->d_part), m->sur ? m->d_sur_flag : nullptr);
}

LoopPlan plan_loops(const tufrg_model *m)
{
    // Choose the number of ky ranges so that the grid fills whole waves of the
    // SMs; the per-column flush costs about 8 rows of work.
    LoopPlan p{};
    p.kx_per_cta = 32 * WARPS;
    const int ctas_x = (m->Lf + p.kx_per_cta - 1) / p.kx_per_cta;
    const int per_sm = loops2_blocks_per_sm(m);
    if (per_sm == 0) return p;
    const double slots = (double)m->sm_count * per_sm;
    double best = 1e300;
    int best_c = 1;
    for (int c = 1; c <= 16; c++) {
        const int len = (m->Lf + c - 1) / c;
        if (len < 8) break;
        const double ctas = (double)m->n_loop_q * ctas_x * c;
        const double waves = std::ceil(ctas / slots);
        const double cost = waves * (len + 8.0);
        if (cost < best * 0.999) { best = cost; best_c = c; }
    }
    p.ky_chunks = best_c;
    p.n_partials = ctas_x * WARPS * best_c;
    return p;
}

std::vector<LoopPlan> loop_plan_candidates(const tufrg_model *m)
{
    // every number of ky ranges per column from 1 to 16 whose ranges keep at least 8 rows
    std::vector<LoopPlan> v;
    const int kx_per_cta = 32 * WARPS, ctas_x = (m->Lf + kx_per_cta - 1) / kx_per_cta;
    for (int c = 1; c <= 16; c++) {
        if ((m->Lf + c - 1) / c < 8) break;
        LoopPlan p{};
        p.kx_per_cta = kx_per_cta;
        p.ky_chunks = c;
        p.n_partials = ctas_x * WARPS * c;
        v.push_back(p);
    }
    return v;
}

// launch shape of the reductions: one row of CTAs per momentum, threads over (d, ab)
static void reduce_shape(const tufrg_model *m, int n_s, dim3 &grid, int &thr)
{
    const int per = m->nd * NS4;
    thr = std::min(1024, (per + 31) / 32 * 32);
    grid = dim3((per + thr - 1) / thr, n_s);
}

cudaError_t launch_loops_reduce_f32(tufrg_model *m, const float2 *part, int n_s, double2 *out64, float2 *out32,
                                    const int *skip)
{
    int ndyh = 0;
    for (int v : m->dys) ndyh += v >= 0;
    dim3 grid;
    int thr;
    reduce_shape(m, n_s, grid, thr);
    PhaseScope ps(m, PH_LOOPRED);
    loops_reduce_kernel<float><<<grid, thr, 0, m->stream>>>(part, m->plan.n_partials, (int)m->dxs.size(), ndyh,
                                                          m->d_dslot, m->d_deltas, m->nd, 1.0 / (double)m->Nk, nullptr,
                                                          out64, out32, skip, 1, 0, 0);
    return cudaGetLastError();
}

long loops_flow_ctas(const tufrg_model *m)
{
    return 2L * (m->sym ? m->n_loop_q : m->Nq) * ((m->Lf + 32 * WARPS - 1) / (32 * WARPS)) * m->plan.ky_chunks;
}

// The loops of a split two-band flow (every stage of it and the surrogate's fallback): FP32 only, what its products read (two
// stages' loops may run at a time, each into its own FP32 buffer).
cudaError_t launch_loops_flow(tufrg_model *m, int channel_mask, bool reps_only)
{
    const LoopPlan &pl = m->plan;
    const int ndx = (int)m->dxs.size();
    int ndyh = 0;
    for (int v : m->dys) ndyh += v >= 0;
    // both channels' k-sums into their own halves of the partial buffer, then one reduction launch
    const int n_s = m->sym ? m->n_loop_q : m->Nq;
    const size_t part_cs = (size_t)n_s * pl.n_partials * ndx * ndyh * NS4, out_cs = (size_t)m->Nq * m->nd * NS4;
    float2 *part = reinterpret_cast<float2 *>(m->d_part);
    const int *skip = m->sur ? m->d_sur_flag : nullptr;
    const int *list = m->sym ? m->d_loop_list : nullptr;
    if (channel_mask == 3) {
        const Args2 a = loops2_args(m, list, part, skip);
        switch (a.ndyh) {
        case 1: TUFRG_CUDA_TRY(launch2_both<1>(m, a, n_s, part_cs)); break;
        case 2: TUFRG_CUDA_TRY(launch2_both<2>(m, a, n_s, part_cs)); break;
        case 3: TUFRG_CUDA_TRY(launch2_both<3>(m, a, n_s, part_cs)); break;
        case 4: TUFRG_CUDA_TRY(launch2_both<4>(m, a, n_s, part_cs)); break;
        default: TUFRG_CUDA_TRY(launch2_both<5>(m, a, n_s, part_cs)); break;   // (loops2_supported)
        }
    } else {
        for (int ch = 0; ch < 2; ch++)
            if ((channel_mask >> ch) & 1) TUFRG_CUDA_TRY(launch_loops2_ex(m, ch, list, n_s, part + ch * part_cs, skip));
    }
    dim3 grid;
    int thr;
    reduce_shape(m, reps_only ? m->n_loop_q : m->Nq, grid, thr);
    grid.z = 2;
    const double inv_nk = 1.0 / (double)m->Nk;
    PhaseScope ps(m, PH_LOOPRED);
    if (reps_only)   // the representatives' FP32 loops at their own momenta (what their products read)
        return launch_chained(loops_reduce_kernel<float>, grid, thr, 0, m->stream, true, part, pl.n_partials, ndx, ndyh, m->d_dslot,
                              m->d_deltas, m->nd, inv_nk, m->d_loop_list, nullptr, m->d_Lc32, skip, channel_mask, part_cs, out_cs);
    if (m->sym)
        loops_reduce_sym_kernel<float><<<grid, thr, 0, m->stream>>>(
            part, pl.n_partials, ndx, ndyh, m->d_dslot, m->d_deltas, m->nd, m->d_qmap, m->d_sym_elem, m->d_sym_dinv,
            inv_nk, nullptr, m->d_Lc32, skip, channel_mask, part_cs, out_cs);
    else
        return launch_chained(loops_reduce_kernel<float>, grid, thr, 0, m->stream, true, part, pl.n_partials, ndx, ndyh, m->d_dslot,
                              m->d_deltas, m->nd, inv_nk, nullptr, nullptr, m->d_Lc32, skip, channel_mask, part_cs, out_cs);
    return cudaGetLastError();
}

}  // namespace tufrg

// ---------------------------------------------------------------------------------
// Loop k-sum without allocation: the same kernels with their scratch in a static array.
// ---------------------------------------------------------------------------------
#include <mutex>
#include <utility>
#include <vector>

namespace tufrg {
namespace {

// Records of one fine mesh plus the partial sums of one channel; see tufrg.h.
__device__ __align__(256) unsigned char g_noalloc_scratch[TUFRG_NOALLOC_SCRATCH_BYTES];

constexpr int NOALLOC_MAXND = 64;
constexpr int NOALLOC_MAXDEV = 64;

struct NoallocTables {
    int nd;
    int d[2 * NOALLOC_MAXND];      // sorted bond differences (dx, dy)
    int slot[NOALLOC_MAXND];       // dxi * ndyh + dyi of the half-plane representative
};

// Fixed-order sum of the partials, scaled by 1/Nk; writes both Hermitian halves (FP64).
__global__ void noalloc_reduce_kernel(const float2 *part, int n_part, int ndx, int ndyh, NoallocTables t, int Nq,
                                      double inv_nk, double2 *out)
{
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (size_t)Nq * t.nd * 16) return;
    const int ab = idx % 16;
    const int d = (idx / 16) % t.nd;
    const int s = (int)(idx / (16 * (size_t)t.nd));
    const int dx = t.d[2 * d], dy = t.d[2 * d + 1];
    const bool half = dy > 0 || (dy == 0 && dx >= 0);
    const int src_ab = half ? ab : (ab % 4) * 4 + ab / 4;
    double re = 0.0, im = 0.0;
    for (int p = 0; p < n_part; p++) {
        const float2 v = part[(((size_t)s * n_part + p) * ndx * ndyh + t.slot[d]) * 16 + src_ab];
        re += (double)v.x;
        im += (double)v.y;
    }
    out[idx] = make_double2(re * inv_nk, (half ? im : -im) * inv_nk);
}

std::mutex g_noalloc_mu;
void *g_noalloc_addr[NOALLOC_MAXDEV] = {};

}  // namespace
}  // namespace tufrg

extern "C" tufrg_status tufrg_loops_noalloc(int Lq, int nc, const double *d_E, const double *d_U, double mu, double T,
                                            int n_ff, const int *h_ffR, int channel_mask, void *d_loops,
                                            void *cuda_stream)
{
    using namespace tufrg;
    if (Lq < 2 || nc < 1 || (long)Lq * nc > 4096 || !d_E || !d_U || !h_ffR || !d_loops || n_ff < 1)
        return TUFRG_EINVAL;
    if (!(T > 0) || !std::isfinite(T) || !std::isfinite(mu) || (channel_mask & ~3)) return TUFRG_EINVAL;
    if (h_ffR[0] != 0 || h_ffR[1] != 0) return TUFRG_EINVAL;
    const int Lf = Lq * nc;
    const size_t Nk = (size_t)Lf * Lf;
    const int Nq = Lq * Lq;
    // bond differences (sorted) and their separable parts, as the model builds them
    std::vector<std::pair<int, int>> dl;
    for (int i = 0; i < n_ff; i++)
        for (int j = 0; j < n_ff; j++) dl.emplace_back(h_ffR[2 * i] - h_ffR[2 * j], h_ffR[2 * i + 1] - h_ffR[2 * j + 1]);
    std::sort(dl.begin(), dl.end());
    dl.erase(std::unique(dl.begin(), dl.end()), dl.end());
    std::vector<int> xs, ys;
    for (auto &p : dl) { xs.push_back(p.first); ys.push_back(p.second); }
    std::sort(xs.begin(), xs.end()); xs.erase(std::unique(xs.begin(), xs.end()), xs.end());
    std::sort(ys.begin(), ys.end()); ys.erase(std::unique(ys.begin(), ys.end()), ys.end());
    std::vector<int> dyh;
    for (int v : ys) if (v >= 0) dyh.push_back(v);
    const int ndx = (int)xs.size(), ndyh = (int)dyh.size(), nd = (int)dl.size();
    if (ndyh < 1 || ndyh > 3 || ndx > MAXD || nd > NOALLOC_MAXND) return TUFRG_ENOTSUP;
    // scratch budget: records, then the partials of one channel (one row range per column)
    const int ctas_x = (Lf + 32 * WARPS - 1) / (32 * WARPS);
    const int n_part = ctas_x * WARPS;
    const size_t rec_bytes = ((Nk * RECF4 * sizeof(float4)) + 255) & ~size_t(255);
    const size_t part_bytes = (size_t)Nq * n_part * ndx * ndyh * 16 * sizeof(float2);
    if (rec_bytes + part_bytes > (size_t)TUFRG_NOALLOC_SCRATCH_BYTES) return TUFRG_ETOOBIG;
    // device address of the static scratch (the device must be current).  Outside stream capture it is looked
    // up on every call, so that a device reset or a new primary context never leaves a stale address behind;
    // during capture the address of the last uncaptured call on this device is used.
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= NOALLOC_MAXDEV) return TUFRG_ECUDA;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(cuda_stream);
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    const bool capturing = cudaStreamIsCapturing(st, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone;
    if (capturing) (void)cudaGetLastError();   // clear the (non-sticky) error a refused capture query leaves
    void *base = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_noalloc_mu);
        if (!capturing) {
            void *p = nullptr;
            if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return TUFRG_ECUDA;
            g_noalloc_addr[dev] = p;
        }
        base = g_noalloc_addr[dev];
    }
    if (!base) return TUFRG_ECUDA;   // first call on this device inside a capture: nothing looked up yet
    float4 *rec = reinterpret_cast<float4 *>(base);
    float2 *part = reinterpret_cast<float2 *>(reinterpret_cast<unsigned char *>(base) + rec_bytes);

    if (launch_records_f32(d_E, reinterpret_cast<const double2 *>(d_U), (int)Nk, Lf, mu, T, rec, st) != cudaSuccess) return TUFRG_ECUDA;
    Args2 a{};
    a.rec = rec;
    a.part = part;
    a.Lq = Lq; a.nc = nc; a.Lf = Lf; a.ndx = ndx; a.ndyh = ndyh;
    for (int j = 0; j < ndyh; j++) a.dys[j] = dyh[j];
    for (int i = 0; i < ndx; i++) {
        a.dxs[i] = xs[i];
        a.needed[i] = 0;
        for (int j = 0; j < ndyh; j++) {
            const bool in = std::binary_search(dl.begin(), dl.end(), std::make_pair(xs[i], dyh[j]));
            if (in && (dyh[j] > 0 || xs[i] >= 0)) a.needed[i] |= 1u << j;
        }
    }
    a.ky_chunks = 1;
    a.ky_len = Lf;
    a.thr = (float)(1e-2 * T);
    a.Tp = nullptr;
    NoallocTables t{};
    t.nd = nd;
    for (int k = 0; k < nd; k++) {
        int dx = dl[k].first, dy = dl[k].second;
        t.d[2 * k] = dx;
        t.d[2 * k + 1] = dy;
        if (!(dy > 0 || (dy == 0 && dx >= 0))) { dx = -dx; dy = -dy; }
        const int xi = (int)(std::find(xs.begin(), xs.end(), dx) - xs.begin());
        const int yi = (int)(std::find(dyh.begin(), dyh.end(), dy) - dyh.begin());
        t.slot[k] = xi * ndyh + yi;
    }
    const size_t smem = loops2_smem_bytes(Lf, ndyh);
    const dim3 grid(Nq, ctas_x, 1);
    const size_t per = (size_t)Nq * nd * 16;
    for (int ch = 0; ch < 2; ch++) {
        if (!((channel_mask >> ch) & 1)) continue;
        void (*kern)(Args2) = nullptr;
        if (ndyh == 1) kern = ch == 0 ? loops2_kernel<1, 0> : loops2_kernel<1, 1>;
        if (ndyh == 2) kern = ch == 0 ? loops2_kernel<2, 0> : loops2_kernel<2, 1>;
        if (ndyh == 3) kern = ch == 0 ? loops2_kernel<3, 0> : loops2_kernel<3, 1>;
        if (smem > 48 * 1024 && cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
            return TUFRG_ECUDA;
        kern<<<grid, 32 * WARPS, smem, st>>>(a);
        if (cudaGetLastError() != cudaSuccess) return TUFRG_ECUDA;
        noalloc_reduce_kernel<<<(unsigned)((per + 255) / 256), 256, 0, st>>>(
            part, n_part, ndx, ndyh, t, Nq, 1.0 / (double)Nk, reinterpret_cast<double2 *>(d_loops) + ch * per);
        if (cudaGetLastError() != cudaSuccess) return TUFRG_ECUDA;
    }
    return TUFRG_OK;
}
