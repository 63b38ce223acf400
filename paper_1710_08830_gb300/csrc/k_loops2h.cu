// Loop k-sum for N_s = 2 over half of the fine mesh, in both precisions: the dominant kernel of a two-band right-hand
// side (split-precision flows take the kernel of k_loops2.cu, see there).
//
//   P:  [L^-_{t1t2t3t4}(s)]_{R1R2} = (1/Nk) sum_q e^{-iq.(R1-R2)} sum_{l1 l2}
//         U_{t1l1}(s-q) U*_{t3l1}(s-q) dF^-_{l1l2}/dT U_{t2l2}(q) U*_{t4l2}(q)
//   C:  [L^+_{t1t2t3t4}(u)]_{R1R2} = (1/Nk) sum_q e^{-iq.(R1-R2)} sum_{l1 l2}
//         U_{t1l1}(q) U*_{t3l1}(q) dF^+_{l1l2}/dT U*_{t2l2}(q-u) U_{t4l2}(q-u)
// (Eqs. loopminus / loopplus with the band loops of Eq. def_lmp dressed by Eq. trafo), organised around the
// structure of the two-band problem:
//   * the band projectors are complete and rank one: rho^1 = 1 - rho^0 and
//     rho^0_00 + rho^0_11 = 1, so one record per fine k holds
//     (rho^0_00, Re rho^0_01, Im rho^0_01) and the Fermi data (e_l, g_l = df/dT,
//     gp_l = dg/de), rewritten once per temperature;
//   * with D = T^0 - T^1, Y = 1 (x) T^1 + rho1^0 (x) D, where
//     T^{l1} = w_{l1 1} 1 + (w_{l1 0} - w_{l1 1}) rho2^0;  Y is Hermitian in the sense
//     Y[(t3 t1),(t4 t2)] = conj(Y[(t1 t3),(t2 t4)]), so only 4 real and 6 complex
//     entries are formed;
//   * the row sums W[dy] = sum_ky e^{-i ky dy} Y keep, for each complex pair
//     (Z, conj Z), the real sums of c Re Z, s Im Z, c Im Z, s Re Z, which give both
//     members; dy = 0 needs no phase;
//   * half of the fine mesh suffices: exchanging the two propagators maps q to s - q.  The pair weights are
//     symmetric, so Y at s - q is Y at q with the index pairs exchanged, and the sum S over one point of every pair
//     {q, s - q} gives
//       P:  L[Delta][a][b] = S[Delta][a][b] + e^{-is.Delta} conj(S[Delta][b~][a~]),   (t2,t1)~ = (t1,t2).
//     For C the exchange leads to -u, and a symmetry of the model with G = -1 (inversion or time reversal) leads
//     back: L = S + V [e^{iu.Delta} S[b~][a~]] V^dagger in the notation of SymElem (without such a symmetry the C sum
//     runs over the whole mesh).  One point of every pair: the rows ky = hy + j with 2 hy = sy (mod Lf), j up to
//     Lf / 2; a row that is its own partner (j = 0, and j = Lf / 2 on even meshes) enters with weight 1/2.  The
//     reduction kernel adds the second term;
//   * the records are stored as three planes of four values transposed to [ky][kx], so the 32 columns of a warp
//     read contiguous bytes per plane (coalesced), several rows in flight by cp.async; rows advance without
//     integer division.
// One thread per fine-mesh column, one CTA per (transfer momentum, 64 columns, channel and row range).  At the end of
// its rows the CTA writes its columns' sums to shared memory and every thread applies the x phases of all columns to
// its share of the 16 (ND + Z) values: the sums of c Re, s Im, c Im, s Re serve dx and -dx together.  One partial
// sum per CTA goes to global memory and loops2h_reduce_kernel adds the partials in a fixed order.
// FP64: bound by the FP64 pipe (two results per clock and SM), so the four pair weights share one division, and bond
// sets with more than three non-negative y differences split them over two groups of CTAs (registers).
// Measured, both channels (before: the whole mesh, one launch per channel; FP64 also every transfer momentum and the
// projectors from the eigenvectors at every point): 24 x 24 / 8 x 8 mesh, 9 bonds: split 90 -> 45 us, FP64 43.2 -> 1.1 ms;
// 8 x 8 / 16 x 16, 5 bonds: split 30 -> 14 us, FP64 2.5 ms -> 139 us; 48 x 48 / 8 x 8, 13 bonds: split 1.40 -> 0.63 ms.
// Split: bound by latency and issue (24 x 24: 11 warps per SM by registers, issue slots 58% busy, the FMA pipe 32%; reads
// the records from DRAM once, 1.8 MB); FP64: by the FP64 pipe.
#include <algorithm>
#include <cmath>
#include <vector>

#include "tufrg_internal.cuh"

namespace tufrg {
namespace {

constexpr int MAXD = 9;
constexpr int MAXDH = 5;         // non-negative x (y) differences
constexpr int WARPS = 2;
constexpr int NT = 32 * WARPS;   // threads (columns) per CTA

constexpr int RECF4 = 3;         // planes of four values per record

struct alignas(32) D4 {
    double x, y, z, w;
};
template <typename R> struct vec4;
template <> struct vec4<float> { using t = float4; };
template <> struct vec4<double> { using t = D4; };
__device__ __forceinline__ float4 mk4(float x, float y, float z, float w) { return make_float4(x, y, z, w); }
__device__ __forceinline__ D4 mk4(double x, double y, double z, double w) { return D4{x, y, z, w}; }

// rows of records in flight per thread (asynchronous copies into shared memory); the FP64 kernel computes long enough
// per row that one row ahead hides the copy
template <typename R> constexpr int RING = sizeof(R) == 4 ? 4 : 2;

// Shared memory of one CTA: the y phase table [Lf], the x phases [64 columns][MAXDH - 1], then one region that holds
// the warps' rings of record rows during the k-sum ([warp][RING][2 sides x 3 planes][32 lanes]) and the columns' sums
// ([64][NV + 1] complex, NV = 16 (ND + Z)) after it.
template <typename R>
size_t loops2h_smem_bytes(int Lf, int n_dy)
{
    const size_t c2 = 2 * sizeof(R);
    const size_t ring = 4 * sizeof(R) * RING<R> * 2 * RECF4 * NT, sums = c2 * NT * (16 * n_dy + 1);
    return ((c2 * Lf + 15) & ~size_t(15)) + c2 * NT * (MAXDH - 1) + std::max(ring, sums);
}

template <typename R>
struct Args2 {
    const typename vec4<R>::t *rec;   // [3][Lf][Lf] planes, index [j][ky][kx]:
                             //   (rho00, Re rho01, Im rho01, e0), (e1, g0, g1, gp0), (gp1, -, -, -)
    typename cpx<R>::t *part;         // [channel][slot][n_part][ndx][ndyh][16]
    size_t part_cs;          // partials of one channel
    int Lq, nc, Lf, ndx, ndyh, ndxh;
    int dyo;                 // first y difference of this launch's group
    int dys[MAXDH], dym[MAXDH];       // non-negative y differences, the same modulo Lf
    int dxm[MAXDH - 1];               // positive x differences modulo Lf
    int xip[MAXDH], xim[MAXDH];       // indices of +dx and -dx (xip[0] = xim[0]: dx = 0)
    unsigned needed[MAXD];   // bit dyi set if (dx, dy) is in the Hermitian half of the bond differences
    int ky_chunks, ky_len;
    int ch0, half;           // first channel; bit ch set: channel ch sums half of the mesh
    R thr_factor;            // degenerate-pair switch = thr_factor * T
    const double *Tp;        // device flow scale (T, or Lambda with the momentum shell)
    R shell_T;               // > 0: momentum-shell regulator at this fixed temperature (records hold f, h)
    const int *s_list;       // optional: CTA x evaluates transfer momentum s_list[x] (partials indexed by x)
    const int *skip;         // optional: the whole launch returns at once when *skip != 0
    const typename cpx<R>::t *ptab;   // e^{-2 pi i n / Lf}, n < Lf
};

// (t1,t3,t2,t4) -> ab index of the compact loop (P: a=(t2,t1), b=(t4,t3); C: a=(t1,t2), b=(t3,t4))
template <int WHICH>
__host__ __device__ constexpr int abx(int t1, int t3, int t2, int t4)
{
    return WHICH == 0 ? ((t2 * 2 + t1) * 4 + t4 * 2 + t3) : ((t1 * 2 + t2) * 4 + t3 * 2 + t4);
}

// the four pair weights w[l1][l2]: l1 on the first point, l2 on the second
template <int WHICH, bool SHELL>
__device__ __forceinline__ void pair_weights(const float (&e1)[2], const float (&g1)[2], const float (&gp1)[2], const float (&e2)[2],
                                             const float (&g2)[2], const float (&gp2)[2], float thr, float lam, float (&w)[2][2])
{
#pragma unroll
    for (int i = 0; i < 2; i++)
#pragma unroll
        for (int j = 0; j < 2; j++) {
            if (SHELL) {
                w[i][j] = shell_weight<WHICH, float>(e1[i], g1[i], gp1[i], e2[j], g2[j], gp2[j], thr, lam);   // (g, gp) = (f, h)
            } else if (WHICH == 0) {
                const float s = e1[i] + e2[j];
                w[i][j] = fabsf(s) > thr ? -__fdividef(g1[i] + g2[j], s) : -0.5f * (gp1[i] + gp2[j]);
            } else {
                const float d = e1[i] - e2[j];
                w[i][j] = fabsf(d) > thr ? __fdividef(g1[i] - g2[j], d) : 0.5f * (gp1[i] + gp2[j]);
            }
        }
}
// FP64: numerators over denominators (1 for the degenerate limit), all four by one division of 1 by the product
template <int WHICH, bool SHELL>
__device__ __forceinline__ void pair_weights(const double (&e1)[2], const double (&g1)[2], const double (&gp1)[2], const double (&e2)[2],
                                             const double (&g2)[2], const double (&gp2)[2], double thr, double lam, double (&w)[2][2])
{
    double n[2][2], d[2][2];
#pragma unroll
    for (int i = 0; i < 2; i++)
#pragma unroll
        for (int j = 0; j < 2; j++) {
            if (SHELL) {
                w[i][j] = shell_weight<WHICH, double>(e1[i], g1[i], gp1[i], e2[j], g2[j], gp2[j], thr, lam);
                continue;
            }
            const double den = WHICH == 0 ? e1[i] + e2[j] : e1[i] - e2[j];
            const bool far = fabs(den) > thr;
            n[i][j] = far ? (WHICH == 0 ? -(g1[i] + g2[j]) : g1[i] - g2[j]) : (WHICH == 0 ? -0.5 : 0.5) * (gp1[i] + gp2[j]);
            d[i][j] = far ? den : 1.0;
        }
    if (SHELL) return;
    const double p0 = d[0][0] * d[0][1], p1 = d[1][0] * d[1][1], r = 1.0 / (p0 * p1), r0 = r * p1, r1 = r * p0;
    w[0][0] = n[0][0] * (d[0][1] * r0);
    w[0][1] = n[0][1] * (d[0][0] * r0);
    w[1][0] = n[1][0] * (d[1][1] * r1);
    w[1][1] = n[1][1] * (d[1][0] * r1);
}

__device__ __forceinline__ void cp_rec(float4 *d, const float4 *s) { cp_async16(d, s); }
__device__ __forceinline__ void cp_rec(D4 *d, const D4 *s)
{
    cp_async16(d, s);
    cp_async16(reinterpret_cast<char *>(d) + 16, reinterpret_cast<const char *>(s) + 16);
}

// two multiply-adds at a time (one instruction in FP32)
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ double2 fma2(double2 a, double2 b, double2 c) { return make_double2(fma(a.x, b.x, c.x), fma(a.y, b.y, c.y)); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ double2 add2(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
template <typename C2, int N>
__device__ __forceinline__ auto item(const C2 (&p)[N], int i) { return i & 1 ? p[i >> 1].y : p[i >> 1].x; }

// ND y differences with a phase, and dy = 0 when Z; SHELL: momentum-shell regulator.
// The sums are kept in pairs of neighbouring entries: a row of ND = 4 spends 128 of about 220 FP32 instructions on its
// phased sums, half as many in pairs: 48 x 48 momenta, five y differences 689 -> 628 us, 24 x 24, three 47.4 -> 45.4.
template <typename R, int ND, int Z, int WHICH, bool SHELL>
__device__ __forceinline__ void loops2h_body(const Args2<R> &a, unsigned char *smem_raw)
{
    using C2 = typename cpx<R>::t;
    using V4 = typename vec4<R>::t;
    constexpr int NRING = RING<R>;
    const int Lf = a.Lf;
    C2 *ptab = reinterpret_cast<C2 *>(smem_raw);
    C2 *xph = reinterpret_cast<C2 *>(smem_raw + ((sizeof(C2) * Lf + 15) & ~size_t(15)));   // [64][MAXDH - 1] e^{-i kx dx}
    unsigned char *region = reinterpret_cast<unsigned char *>(xph + NT * (MAXDH - 1));
    for (int n = threadIdx.x; n < Lf; n += NT) ptab[n] = a.ptab[n];
    __syncthreads();

    const int s = blockIdx.x;                                    // slot of the partial sums
    const int sq = a.s_list ? a.s_list[blockIdx.x] : blockIdx.x;  // transfer momentum
    const int sx = (sq / a.Lq) * a.nc, sy = (sq % a.Lq) * a.nc;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    V4 *ring = reinterpret_cast<V4 *>(region) + warp * NRING * 2 * RECF4 * 32;   // [RING][6][32]: rows of this warp's columns
    const int kx = blockIdx.y * NT + threadIdx.x;
    // temperature flow: the scale is T; momentum shell: the scale is Lambda and the temperature is fixed
    const R lam = SHELL ? (R)*a.Tp : R(0);
    const R thr = SHELL ? a.thr_factor * a.shell_T : (R)(a.thr_factor * *a.Tp);
    const bool valid = kx < Lf;
    const int kyc = blockIdx.z % a.ky_chunks;
    // rows of this sum: the whole column, or hy .. hy + n_rows - 1 (mod Lf) with the self-paired rows fix0, fix1
    const bool half = (a.half >> WHICH) & 1;
    const bool odd_s = sy & 1, even_L = !(Lf & 1);
    const int hy = !half ? 0 : !odd_s ? sy / 2 : even_L ? (sy + 1) / 2 : (sy + Lf) / 2;
    const int n_rows = !half ? Lf : even_L ? Lf / 2 + (odd_s ? 0 : 1) : (Lf + 1) / 2;
    const int fix0 = half && !(even_L && odd_s) ? 0 : -1, fix1 = half && even_L && !odd_s ? Lf / 2 : -1;
    const int j0 = kyc * a.ky_len, j1 = min(n_rows, j0 + a.ky_len);

    constexpr int NDA = ND > 0 ? ND : 1;
    C2 R0[2], P0y[3], P0z[3], Rc[NDA][2], Rs[NDA][2], Pcy[NDA][3], Psz[NDA][3], Pcz[NDA][3], Psy[NDA][3];
#pragma unroll
    for (int j = 0; j < 3; j++) {
        P0y[j] = P0z[j] = mk(R(0), R(0));
        if (j < 2) R0[j] = P0y[j];
#pragma unroll
        for (int i = 0; i < ND; i++) {
            Pcy[i][j] = Psz[i][j] = Pcz[i][j] = Psy[i][j] = P0y[j];
            if (j < 2) Rc[i][j] = Rs[i][j] = P0y[j];
        }
    }

    if (valid && j0 < j1) {
        // columns of k1 and k2; rows step by +1 on the q side and by -1 on the s - q side
        const int ky0 = hy + j0 < Lf ? hy + j0 : hy + j0 - Lf;
        const int k1x = WHICH == 0 ? (sx - kx + Lf) % Lf : kx;
        const int k2x = WHICH == 0 ? kx : (kx - sx + Lf) % Lf;
        const int k1y = WHICH == 0 ? (sy - ky0 + Lf) % Lf : ky0;
        const int k2y = WHICH == 0 ? ky0 : (ky0 - sy + Lf) % Lf;
        const size_t plane = (size_t)Lf * Lf;
        int o1 = k1y * Lf + k1x, o2 = k2y * Lf + k2x;        // offsets of the next row to be copied
        const int wrap = (Lf - 1) * Lf;
        // copy one row (both sides, three planes) into ring slot sl, then step the offsets to the next
        // row: the q side moves by +Lf, the s - q side by -Lf (P), both +Lf (C), with wrap
        auto issue_row = [&](int sl) {
            V4 *r = ring + sl * 2 * RECF4 * 32 + lane;
#pragma unroll
            for (int pl = 0; pl < RECF4; pl++) {
                cp_rec(r + pl * 32, a.rec + pl * plane + o1);
                cp_rec(r + (RECF4 + pl) * 32, a.rec + pl * plane + o2);
            }
            if (WHICH == 0) { o1 = o1 >= Lf ? o1 - Lf : o1 + wrap; o2 = o2 < wrap ? o2 + Lf : o2 - wrap; }
            else            { o1 = o1 < wrap ? o1 + Lf : o1 - wrap; o2 = o2 < wrap ? o2 + Lf : o2 - wrap; }
        };
#pragma unroll
        for (int i = 0; i < NRING - 1; i++) {   // the first RING - 1 rows in flight
            if (j0 + i < j1) issue_row(i);
            cp_async_commit();
        }
        int pn[ND > 0 ? ND : 1];
#pragma unroll
        for (int i = 0; i < ND; i++) pn[i] = (int)(((long)ky0 * a.dys[a.dyo + Z + i]) % Lf);
        const R sgn = WHICH == 0 ? R(1) : R(-1);
        for (int j = j0; j < j1; j++) {
            const int it = j - j0;
            if (j + NRING - 1 < j1) issue_row((it + NRING - 1) & (NRING - 1));
            cp_async_commit();
            cp_async_wait<NRING - 1>();   // this thread's copies of row j have landed
            const V4 *r = ring + (it & (NRING - 1)) * 2 * RECF4 * 32 + lane;
            const V4 a0 = r[0], a1 = r[32], a2 = r[64], b0 = r[96], b1 = r[128], b2 = r[160];
            const R e1[2] = {a0.w, a1.x}, g1[2] = {a1.y, a1.z}, gp1[2] = {a1.w, a2.x};
            const R e2[2] = {b0.w, b1.x}, g2[2] = {b1.y, b1.z}, gp2[2] = {b1.w, b2.x};
            R w[2][2];
            pair_weights<WHICH, SHELL>(e1, g1, gp1, e2, g2, gp2, thr, lam, w);
            if (j == fix0 || j == fix1) {   // a self-paired row (uniform over the CTA)
#pragma unroll
                for (int i = 0; i < 4; i++) w[i >> 1][i & 1] *= R(0.5);
            }
            // T^{l1} = w_{l1 1} 1 + (w_{l1 0} - w_{l1 1}) rho2'^0 ;  D = T^0 - T^1
            const R A2 = b0.x, C2r = b0.y, C2i = sgn * b0.z;    // rho2' = rho2 (P) or conj(rho2) (C)
            const R dw0 = w[0][0] - w[0][1], dw1 = w[1][0] - w[1][1];
            const R T1_00 = fma(dw1, A2, w[1][1]), T1_11 = fma(dw1, R(1) - A2, w[1][1]);
            const R T1r = dw1 * C2r, T1i = dw1 * C2i;
            const R dd = dw0 - dw1, dd0 = w[0][1] - w[1][1];
            const R D00 = fma(dd, A2, dd0), D11 = fma(dd, R(1) - A2, dd0);
            const R Dr = dd * C2r, Di = dd * C2i;
            // Y = 1 (x) T^1 + rho1^0 (x) D: 4 real and 6 complex independent entries
            const R A1 = a0.x, B1 = R(1) - a0.x, C1r = a0.y, C1i = a0.z;
            C2 X[2], Zy[3], Zz[3];
            X[0] = mk(fma(A1, D00, T1_00), fma(A1, D11, T1_11));    // Y[00][00], Y[00][11]
            X[1] = mk(fma(B1, D00, T1_00), fma(B1, D11, T1_11));    // Y[11][00], Y[11][11]
            Zy[0] = mk(fma(A1, Dr, T1r), fma(B1, Dr, T1r));         // Y[00][01], Y[11][01]
            Zz[0] = mk(fma(A1, Di, T1i), fma(B1, Di, T1i));
            Zy[1] = mk(C1r * D00, C1r * D11);                       // Y[01][00], Y[01][11]
            Zz[1] = mk(C1i * D00, C1i * D11);
            Zy[2] = mk(C1r * Dr - C1i * Di, C1r * Dr + C1i * Di);   // Y[01][01] = rho01 D01, Y[01][10] = rho01 conj(D01)
            Zz[2] = mk(C1r * Di + C1i * Dr, C1i * Dr - C1r * Di);
            // row sums
            if (Z) {
#pragma unroll
                for (int i = 0; i < 3; i++) {
                    P0y[i] = add2(P0y[i], Zy[i]);
                    P0z[i] = add2(P0z[i], Zz[i]);
                    if (i < 2) R0[i] = add2(R0[i], X[i]);
                }
            }
#pragma unroll
            for (int i = 0; i < ND; i++) {
                const C2 ph = ptab[pn[i]], phc = mk(ph.x, ph.x), phs = mk(ph.y, ph.y);
                pn[i] += a.dym[a.dyo + Z + i];
                if (pn[i] >= Lf) pn[i] -= Lf;
#pragma unroll
                for (int v = 0; v < 2; v++) { Rc[i][v] = fma2(phc, X[v], Rc[i][v]); Rs[i][v] = fma2(phs, X[v], Rs[i][v]); }
#pragma unroll
                for (int v = 0; v < 3; v++) {
                    Pcy[i][v] = fma2(phc, Zy[v], Pcy[i][v]);
                    Psz[i][v] = fma2(phs, Zz[v], Psz[i][v]);
                    Pcz[i][v] = fma2(phc, Zz[v], Pcz[i][v]);
                    Psy[i][v] = fma2(phs, Zy[v], Psy[i][v]);
                }
            }
        }
        cp_async_wait<0>();   // nothing in flight before the region is reused below (trailing groups are empty)
    }

    // ---- W[dy][ab] of this column, rebuilt from the paired sums, to shared memory
    constexpr int XR[4] = {abx<WHICH>(0, 0, 0, 0), abx<WHICH>(0, 0, 1, 1), abx<WHICH>(1, 1, 0, 0), abx<WHICH>(1, 1, 1, 1)};
    constexpr int ZA[6] = {abx<WHICH>(0, 0, 0, 1), abx<WHICH>(1, 1, 0, 1), abx<WHICH>(0, 1, 0, 0),
                           abx<WHICH>(0, 1, 1, 1), abx<WHICH>(0, 1, 0, 1), abx<WHICH>(0, 1, 1, 0)};
    constexpr int ZB[6] = {abx<WHICH>(0, 0, 1, 0), abx<WHICH>(1, 1, 1, 0), abx<WHICH>(1, 0, 0, 0),
                           abx<WHICH>(1, 0, 1, 1), abx<WHICH>(1, 0, 1, 0), abx<WHICH>(1, 0, 0, 1)};
    constexpr int NV = 16 * (ND + Z);
    constexpr int PITCH = NV + 1;   // odd: the columns' stores fall on different banks
    C2 *buf = reinterpret_cast<C2 *>(region);
    __syncthreads();   // every thread is done with its ring entries
    C2 *mine = buf + threadIdx.x * PITCH;
    if (Z) {
#pragma unroll
        for (int j = 0; j < 4; j++) mine[XR[j]] = mk(item(R0, j), R(0));
#pragma unroll
        for (int j = 0; j < 6; j++) {
            mine[ZA[j]] = mk(item(P0y, j), item(P0z, j));
            mine[ZB[j]] = mk(item(P0y, j), -item(P0z, j));
        }
    }
#pragma unroll
    for (int i = 0; i < ND; i++) {
        C2 *mi = mine + 16 * (i + Z);
#pragma unroll
        for (int j = 0; j < 4; j++) mi[XR[j]] = mk(item(Rc[i], j), item(Rs[i], j));
#pragma unroll
        for (int j = 0; j < 6; j++) {
            mi[ZA[j]] = mk(item(Pcy[i], j) - item(Psz[i], j), item(Pcz[i], j) + item(Psy[i], j));
            mi[ZB[j]] = mk(item(Pcy[i], j) + item(Psz[i], j), item(Psy[i], j) - item(Pcz[i], j));
        }
    }
#pragma unroll
    for (int i = 0; i < MAXDH - 1; i++)   // x phases of this column (columns past the mesh hold zero sums)
        if (i + 1 < a.ndxh) xph[threadIdx.x * (MAXDH - 1) + i] = ptab[(int)(((long)kx * a.dxm[i]) % Lf)];
    __syncthreads();
    // ---- sums over the CTA's columns for every dx: one value (dy, ab) per thread and round
    // FP32: in blocks of columns, a chain of 64 additions cut to 16 and 4.  The exchanged half repeats the rounding of the
    // first, so the other roundings have to be fewer: error of the loops 1.52e-7 in one chain, 1.27e-7 in blocks, 1.38e-7 by
    // the whole mesh (20 x 20 / 9 x 9, 9 bonds), for half a percent of the right-hand side's time.
    constexpr int BLK = sizeof(R) == 4 ? 16 : NT;
    const int n_part = gridDim.y * a.ky_chunks, p = blockIdx.y * a.ky_chunks + kyc;
    C2 *out = a.part + WHICH * a.part_cs + ((size_t)s * n_part + p) * a.ndx * a.ndyh * 16;
    for (int v = threadIdx.x; v < NV; v += NT) {
        C2 z0 = mk(R(0), R(0));
        R cr[MAXDH - 1], si[MAXDH - 1], ci[MAXDH - 1], sr[MAXDH - 1];
#pragma unroll
        for (int i = 0; i < MAXDH - 1; i++) { cr[i] = 0; si[i] = 0; ci[i] = 0; sr[i] = 0; }
        for (int r0 = 0; r0 < NT; r0 += BLK) {
            C2 y0 = mk(R(0), R(0));
            R c[4][MAXDH - 1];
#pragma unroll
            for (int i = 0; i < MAXDH - 1; i++) c[0][i] = c[1][i] = c[2][i] = c[3][i] = 0;
#pragma unroll 4
            for (int r = r0; r < r0 + BLK; r++) {
                const C2 x = buf[r * PITCH + v];
                y0.x += x.x;
                y0.y += x.y;
#pragma unroll
                for (int i = 0; i < MAXDH - 1; i++) {
                    if (i + 1 >= a.ndxh) break;
                    const C2 ph = xph[r * (MAXDH - 1) + i];
                    c[0][i] = fma(ph.x, x.x, c[0][i]);
                    c[1][i] = fma(ph.y, x.y, c[1][i]);
                    c[2][i] = fma(ph.x, x.y, c[2][i]);
                    c[3][i] = fma(ph.y, x.x, c[3][i]);
                }
            }
            z0.x += y0.x;
            z0.y += y0.y;
#pragma unroll
            for (int i = 0; i < MAXDH - 1; i++) {
                if (i + 1 >= a.ndxh) break;
                cr[i] += c[0][i];
                si[i] += c[1][i];
                ci[i] += c[2][i];
                sr[i] += c[3][i];
            }
        }
        const int dyi = a.dyo + v / 16, ab = v & 15;
        if ((a.needed[a.xip[0]] >> dyi) & 1u) out[(a.xip[0] * a.ndyh + dyi) * 16 + ab] = z0;
#pragma unroll
        for (int i = 0; i < MAXDH - 1; i++) {
            if (i + 1 >= a.ndxh) break;
            const int xp = a.xip[i + 1], xm = a.xim[i + 1];
            if ((a.needed[xp] >> dyi) & 1u) out[(xp * a.ndyh + dyi) * 16 + ab] = mk(cr[i] - si[i], ci[i] + sr[i]);
            if ((a.needed[xm] >> dyi) & 1u) out[(xm * a.ndyh + dyi) * 16 + ab] = mk(cr[i] + si[i], ci[i] - sr[i]);
        }
    }
}

// blockIdx.z = channel index (from a.ch0) times ky_chunks plus the row range: both channels share one launch, so that
// the second fills the last wave of the first
template <typename R, int ND, int Z, bool SHELL>
__global__ void __launch_bounds__(NT) loops2h_kernel(const __grid_constant__ Args2<R> a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if (a.skip && *a.skip) return;   // uniform over the grid
    if (a.ch0 + (int)blockIdx.z / a.ky_chunks == 0) loops2h_body<R, ND, Z, 0, SHELL>(a, smem_raw);
    else loops2h_body<R, ND, Z, 1, SHELL>(a, smem_raw);
}

// Record of one fine k (three planes [j][ky][kx]): plane 0 = (rho00, Re rho01, Im rho01, e0),
// plane 1 = (e1, g0, g1, g'0), plane 2 = (g'1, 0, 0, 0), with e = E - mu, g = dF/dT-type weight
// derivative of the Fermi function and g' its derivative in e.  The projector and e do not depend on
// T and are written once per model; only g and g' are refreshed per evaluation.
template <typename R>
__global__ void rec_static_kernel(const double *E, const double2 *U, int Nk, int Lf, double mu, typename vec4<R>::t *rec)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= Nk) return;
    // rho^0 = U_{.0} U*_{.0}: rho00 = |U_00|^2, rho01 = U_00 conj(U_10)
    const double2 u0 = U[(size_t)k * 4 + 0], u1 = U[(size_t)k * 4 + 2];
    const int kx = k / Lf, ky = k % Lf;
    const size_t t = (size_t)ky * Lf + kx, plane = (size_t)Lf * Lf;
    rec[t] = mk4((R)(u0.x * u0.x + u0.y * u0.y), (R)(u0.x * u1.x + u0.y * u1.y), (R)(u0.y * u1.x - u0.x * u1.y), (R)(E[2 * k] - mu));
    rec[plane + t] = mk4((R)(E[2 * k + 1] - mu), R(0), R(0), R(0));
    rec[2 * plane + t] = mk4(R(0), R(0), R(0), R(0));
}

// g = -df/dT = (x / T) f (1 - f) and g' = dg/de with x = e / T, in the overflow-safe form with
// z = exp(-|x|): f (1 - f) = z / (1 + z)^2 and dg/de = f (1 - f) / T^2 (1 - |x| (1 - z) / (1 + z)).
// In the precision of the loop sums.
__device__ __forceinline__ float exp_of(float x) { return expf(x); }
__device__ __forceinline__ double exp_of(double x) { return exp(x); }
template <typename R>
__global__ void rec_T_kernel(int n, double T_value, const double *Tp, typename vec4<R>::t *rec)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    grid_release();   // (the k-sum of a flow waits for it)
    if (t >= n) return;
    const R invT = R(1) / (R)(Tp ? *Tp : T_value);   // device-resident temperature when given
    const R e[2] = {rec[t].w, rec[n + t].x};
    R g[2], gp[2];
#pragma unroll
    for (int l = 0; l < 2; l++) {
        const R x = e[l] * invT, ax = fabs(x);
        const R z = exp_of(-ax), opz = R(1) + z;
        const R h = z / (opz * opz);
        g[l] = x * invT * h;
        gp[l] = h * invT * invT * (R(1) - ax * (R(1) - z) / opz);
    }
    rec[n + t] = mk4(e[1], g[0], g[1], gp[0]);
    rec[2 * n + t] = mk4(gp[1], R(0), R(0), R(0));
}

// Momentum-shell records: (f, h) = (f(e), f (1 - f) / T) at the fixed temperature T in the slots of
// (g, g'), from the FP64 energies (written once per model; the shell weight needs no T-dependent data).
template <typename R>
__global__ void rec_shell_kernel(const double *E, int Nk, int Lf, double mu, double T, typename vec4<R>::t *rec)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= Nk) return;
    const int kx = k / Lf, ky = k % Lf;
    const size_t t = (size_t)ky * Lf + kx, plane = (size_t)Lf * Lf;
    double f[2], h[2];
    for (int l = 0; l < 2; l++) {
        const double e = E[2 * k + l] - mu, z = exp(-fabs(e) / T);
        f[l] = e > 0 ? z / (1.0 + z) : 1.0 / (1.0 + z);
        h[l] = z / ((1.0 + z) * (1.0 + z)) / T;
    }
    const R e1 = rec[plane + t].x;
    rec[plane + t] = mk4(e1, (R)f[0], (R)f[1], (R)h[0]);
    rec[2 * plane + t] = mk4((R)h[1], R(0), R(0), R(0));
}

// Sum of the partials in a fixed order, the exchanged half, both Hermitian halves of the bond differences and, with
// loop symmetries, the other momenta of an orbit.  Grid: (output momenta, channels); a CTA first adds the partials
// of its list position for every value of the Hermitian half (d, ab) into shared memory, in their own precision, 16
// loads in flight per thread, and then forms every output (d, ab) from those sums.
template <typename R>
struct Red2 {
    const typename cpx<R>::t *part;
    size_t part_cs, out_cs;
    int n_part, ndx, ndyh, nd, n_hp, chmask, half;
    const int *dslot, *deltas, *hp;              // hp[i]: i-th bond difference of the half plane; dslot: partial slot
    const int *hpos;                             // [nd] position in hp of d or of -d
    const int *slot_q;                           // momentum of a list position (null: the position)
    const int2 *qmap;                            // symmetric gather: output momentum -> (list position, element); or null
    const SymElem *elem;
    const int *dinv;
    int inv;                                     // element with G = -1 (C channel's exchanged half)
    int at_q;                                    // outputs at the position's momentum (else at the position)
    int Lq, nc, Lf;
    const typename cpx<R>::t *ptab;
    R inv_nk;
    double2 *out64;
    float2 *out32;
    const int *skip;
};

template <typename C2>
__device__ __forceinline__ C2 turn(C2 v, int k)
{
    switch (k & 3) {
    case 0: return v;
    case 1: return mk(-v.y, v.x);
    case 2: return mk(-v.x, -v.y);
    default: return mk(v.y, -v.x);
    }
}
__device__ __forceinline__ int swap2(int a) { return (a & 1) * 2 + (a >> 1); }   // (t1,t2) -> (t2,t1)
__device__ __forceinline__ double2 wide2(float2 v) { return make_double2(widen_f(v.x), widen_f(v.y)); }
__device__ __forceinline__ double2 wide2(double2 v) { return v; }
__device__ __forceinline__ void put_f32(float2 *p, float2 v) { *p = v; }
__device__ __forceinline__ void put_f32(float2 *, double2) {}

template <typename R>
__global__ void loops2h_reduce_kernel(const __grid_constant__ Red2<R> a)
{
    using C2 = typename cpx<R>::t;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C2 *sum = reinterpret_cast<C2 *>(smem_raw);   // [n_hp][16]
    if (a.skip && *a.skip) return;
    const int ch = blockIdx.y;
    if (!((a.chmask >> ch) & 1)) return;
    const int2 ie = a.qmap ? a.qmap[blockIdx.x] : make_int2(blockIdx.x, -1);
    const int s = ie.x;
    const size_t stride = (size_t)a.ndx * a.ndyh * 16;
    const C2 *part = a.part + ch * a.part_cs + (size_t)s * a.n_part * stride;
    for (int t = threadIdx.x; t < a.n_hp * 16; t += blockDim.x) {
        const C2 *src = part + (size_t)a.dslot[a.hp[t >> 4]] * 16 + (t & 15);
        R re = 0, im = 0;
        constexpr int UB = 16;
        int p = 0;
        for (; p + UB <= a.n_part; p += UB) {
            C2 v[UB];
#pragma unroll
            for (int j = 0; j < UB; j++) v[j] = src[(size_t)(p + j) * stride];
#pragma unroll
            for (int j = 0; j < UB; j++) {
                re += v[j].x;
                im += v[j].y;
            }
        }
        C2 v[UB];
#pragma unroll
        for (int j = 0; j < UB; j++) v[j] = p + j < a.n_part ? src[(size_t)(p + j) * stride] : mk(R(0), R(0));
#pragma unroll
        for (int j = 0; j < UB; j++) {
            re += v[j].x;
            im += v[j].y;
        }
        sum[t] = mk(re, im);
    }
    __syncthreads();
    const int q = a.slot_q ? a.slot_q[s] : s, qx = q / a.Lq, qy = q % a.Lq;
    // S[d][a][b] for any d from the half plane's sums
    auto S = [&](int d, int x, int y) {
        const int dx = a.deltas[2 * d], dy = a.deltas[2 * d + 1];
        const bool hp = dy > 0 || (dy == 0 && dx >= 0);
        C2 v = sum[a.hpos[d] * 16 + (hp ? x * 4 + y : y * 4 + x)];
        if (!hp) v.y = -v.y;
        return v;
    };
    // e^{-i q.Delta} v (sign = 1) or its conjugate phase (sign = -1)
    auto phased = [&](C2 v, int d, int sign) {
        const int n = ((qx * a.deltas[2 * d] + qy * a.deltas[2 * d + 1]) % a.Lq + a.Lq) % a.Lq * a.nc;
        C2 p = a.ptab[n];
        if (sign < 0) p.y = -p.y;
        return mk(p.x * v.x - p.y * v.y, p.x * v.y + p.y * v.x);
    };
    for (int t = threadIdx.x; t < a.nd * 16; t += blockDim.x) {
        int d = t >> 4, x = (t >> 2) & 3, y = t & 3, k = 0;
        bool conj = false;
        if (ie.y >= 0) {   // the source of this output in the representative's loops
            const SymElem &e = a.elem[ie.y];
            k = e.qt[ch][x] - e.qt[ch][y];
            conj = e.conj;
            x = e.src[ch][x];
            y = e.src[ch][y];
            d = a.dinv[ie.y * a.nd + d];
        }
        C2 v = S(d, x, y);
        if ((a.half >> ch) & 1) {
            C2 w;
            if (ch == 0) {
                w = S(d, swap2(y), swap2(x));
                w.y = -w.y;
                w = phased(w, d, 1);
            } else {
                const SymElem &e = a.elem[a.inv];
                const int d2 = a.dinv[a.inv * a.nd + d];
                w = phased(S(d2, swap2(e.src[1][y]), swap2(e.src[1][x])), d2, -1);
                if (e.conj) w.y = -w.y;
                w = turn(w, e.qt[1][x] - e.qt[1][y]);
            }
            v.x += w.x;
            v.y += w.y;
        }
        if (conj) v.y = -v.y;
        v = turn(mk(v.x * a.inv_nk, v.y * a.inv_nk), k);
        const size_t o = ch * a.out_cs + (size_t)(a.qmap ? (int)blockIdx.x : a.at_q ? q : s) * a.nd * 16 + t;
        if (a.out64) a.out64[o] = wide2(v);
        if (a.out32) put_f32(a.out32 + o, v);
    }
}

template <typename R, int ND, int Z>
cudaError_t launch2(tufrg_model *m, Args2<R> a, int n_s, int dyo, int n_ch)
{
    a.dyo = dyo;
    const dim3 grid(n_s, (m->Lf + NT - 1) / NT, a.ky_chunks * n_ch);
    const size_t smem = loops2h_smem_bytes<R>(m->Lf, ND + Z);
    auto kern = a.shell_T > R(0) ? loops2h_kernel<R, ND, Z, true> : loops2h_kernel<R, ND, Z, false>;
    if (smem > 48 * 1024) TUFRG_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    PhaseScope ps(m, PH_LOOPS);
    kern<<<grid, NT, smem, m->stream>>>(a);
    return cudaGetLastError();
}

int n_dyh(const tufrg_model *m)
{
    int n = 0;
    for (int v : m->dys) n += v >= 0;
    return n;
}

// the bond differences' separable parts and the Hermitian half, from the sorted distinct dx and the non-negative dy
template <typename R, typename In>
void fill_bonds(Args2<R> &a, int Lf, const std::vector<int> &dxs, const std::vector<int> &dyh, In in_set)
{
    a.ndx = (int)dxs.size();
    a.ndyh = (int)dyh.size();
    for (int j = 0; j < a.ndyh; j++) {
        a.dys[j] = dyh[j];
        a.dym[j] = dyh[j] % Lf;
    }
    a.ndxh = 0;
    for (int i = 0; i < a.ndx; i++) {
        a.needed[i] = 0;
        for (int j = 0; j < a.ndyh; j++)
            if (in_set(dxs[i], dyh[j]) && (dyh[j] > 0 || dxs[i] >= 0)) a.needed[i] |= 1u << j;
        if (dxs[i] < 0) continue;
        a.xip[a.ndxh] = i;
        a.xim[a.ndxh] = (int)(std::find(dxs.begin(), dxs.end(), -dxs[i]) - dxs.begin());
        if (a.ndxh > 0) a.dxm[a.ndxh - 1] = dxs[i] % Lf;
        a.ndxh++;
    }
}

template <typename R>
cudaError_t run2(tufrg_model *m, int channel_mask, const int *s_list, int n_list, void *part, size_t part_cs, const int *skip)
{
    const LoopPlan &pl = m->plan_h;
    Args2<R> a{};
    a.rec = reinterpret_cast<const typename vec4<R>::t *>(m->d_rec);
    a.part = reinterpret_cast<typename cpx<R>::t *>(part);
    a.part_cs = part_cs;
    a.s_list = s_list;
    a.skip = skip;
    a.Lq = m->Lq; a.nc = m->nc; a.Lf = m->Lf;
    std::vector<int> dyh;
    for (int v : m->dys)
        if (v >= 0) dyh.push_back(v);
    fill_bonds(a, m->Lf, m->dxs, dyh, [&](int dx, int dy) {
        for (int d = 0; d < m->nd; d++)
            if (m->deltas[2 * d] == dx && m->deltas[2 * d + 1] == dy) return true;
        return false;
    });
    a.half = loops2_half_mask(m);
    // row ranges of the longest sum of this launch
    const int rows = (a.half & channel_mask) == channel_mask ? m->Lf / 2 + 1 : m->Lf;
    a.ky_chunks = pl.ky_chunks;
    a.ky_len = (rows + pl.ky_chunks - 1) / pl.ky_chunks;
    a.thr_factor = sizeof(R) == 4 ? R(1e-2) : R(1e-5);
    a.Tp = m->d_scal;
    a.shell_T = m->regulator == TUFRG_REG_MOMENTUM_SHELL ? (R)m->T_reg : R(0);
    a.ptab = reinterpret_cast<const typename cpx<R>::t *>(sizeof(R) == 4 ? (const void *)m->d_lph32 : (const void *)m->d_lph);
    a.ch0 = (channel_mask & 1) ? 0 : 1;
    const int n_ch = channel_mask == 3 ? 2 : 1, n_s = s_list ? n_list : m->Nq;
    switch (a.ndyh) {
    case 1: return launch2<R, 0, 1>(m, a, n_s, 0, n_ch);
    case 2: return launch2<R, 1, 1>(m, a, n_s, 0, n_ch);
    case 3: return launch2<R, 2, 1>(m, a, n_s, 0, n_ch);
    default: break;
    }
    if (a.ndyh > MAXDH) return cudaErrorNotSupported;
    if constexpr (sizeof(R) == 8) {   // at most three y differences per launch (registers of the FP64 sums)
        TUFRG_CUDA_TRY((launch2<R, 2, 1>(m, a, n_s, 0, n_ch)));
        return a.ndyh == 4 ? launch2<R, 1, 0>(m, a, n_s, 3, n_ch) : launch2<R, 2, 0>(m, a, n_s, 3, n_ch);
    } else {
        return a.ndyh == 4 ? launch2<R, 3, 1>(m, a, n_s, 0, n_ch) : launch2<R, 4, 1>(m, a, n_s, 0, n_ch);
    }
}

template <typename R>
cudaError_t reduce2(tufrg_model *m, int channel_mask, const void *part, size_t part_cs, const int *slot_q, int n_s, bool gather,
                    bool at_q, double2 *out64, float2 *out32, size_t out_cs, const int *skip)
{
    Red2<R> a{};
    a.part = reinterpret_cast<const typename cpx<R>::t *>(part);
    a.part_cs = part_cs;
    a.out_cs = out_cs;
    a.n_part = m->plan_h.n_partials;
    a.ndx = (int)m->dxs.size();
    a.ndyh = n_dyh(m);
    a.nd = m->nd;
    a.n_hp = (m->nd + 1) / 2;
    a.chmask = channel_mask;
    a.half = loops2_half_mask(m);
    a.dslot = m->d_dslot;
    a.deltas = m->d_deltas;
    a.hp = m->d_hp;
    a.hpos = m->d_hp + a.n_hp;
    a.slot_q = slot_q;
    a.qmap = gather ? m->d_qmap : nullptr;
    a.elem = m->d_sym_elem;
    a.dinv = m->d_sym_dinv;
    a.inv = m->sym_inv;
    a.at_q = at_q;
    a.Lq = m->Lq; a.nc = m->nc; a.Lf = m->Lf;
    a.ptab = reinterpret_cast<const typename cpx<R>::t *>(sizeof(R) == 4 ? (const void *)m->d_lph32 : (const void *)m->d_lph);
    a.inv_nk = R(1.0 / (double)m->Nk);
    a.out64 = out64;
    a.out32 = out32;
    a.skip = skip;
    const int thr = std::min(1024, (m->nd * 16 + 31) / 32 * 32);
    PhaseScope ps(m, PH_LOOPRED);
    loops2h_reduce_kernel<R><<<dim3(n_s, 2), thr, sizeof(typename cpx<R>::t) * a.n_hp * 16, m->stream>>>(a);
    return cudaGetLastError();
}

}  // namespace

// Resident CTAs per SM of the instantiation this model launches (occupancy API).
int loops2h_blocks_per_sm(const tufrg_model *m)
{
    const int ndyh = n_dyh(m);
    if (m->precision == TUFRG_FP64) {
        const size_t smem = loops2h_smem_bytes<double>(m->Lf, std::min(ndyh, 3));
        switch (ndyh) {
        case 1: return resident_ctas(loops2h_kernel<double, 0, 1, false>, NT, smem);
        case 2: return resident_ctas(loops2h_kernel<double, 1, 1, false>, NT, smem);
        default: return resident_ctas(loops2h_kernel<double, 2, 1, false>, NT, smem);
        }
    }
    const size_t smem = loops2h_smem_bytes<float>(m->Lf, ndyh);
    switch (ndyh) {
    case 1: return resident_ctas(loops2h_kernel<float, 0, 1, false>, NT, smem);
    case 2: return resident_ctas(loops2h_kernel<float, 1, 1, false>, NT, smem);
    case 3: return resident_ctas(loops2h_kernel<float, 2, 1, false>, NT, smem);
    case 4: return resident_ctas(loops2h_kernel<float, 3, 1, false>, NT, smem);
    case 5: return resident_ctas(loops2h_kernel<float, 4, 1, false>, NT, smem);
    default: return 0;
    }
}

bool loops2_supported(const tufrg_model *m) { return m->ns == 2 && n_dyh(m) <= MAXDH && (int)m->dxs.size() <= MAXD; }

// channels whose k-sum runs over half of the fine mesh: P always, C with a symmetry that inverts the momentum
int loops2_half_mask(const tufrg_model *m) { return 1 | (m->sym_inv >= 0 ? 2 : 0); }

size_t loops2_rec_bytes(const tufrg_model *m)
{
    return (size_t)m->Nk * RECF4 * 4 * (m->precision == TUFRG_FP64 ? sizeof(double) : sizeof(float));
}

cudaError_t launch_loop_records_static(tufrg_model *m)
{
    const int g = (m->Nk + 255) / 256;
    if (m->precision == TUFRG_FP64)
        rec_static_kernel<double><<<g, 256, 0, m->stream>>>(m->d_E, m->d_U, m->Nk, m->Lf, m->mu, static_cast<D4 *>(m->d_rec));
    else
        rec_static_kernel<float><<<g, 256, 0, m->stream>>>(m->d_E, m->d_U, m->Nk, m->Lf, m->mu, static_cast<float4 *>(m->d_rec));
    return cudaGetLastError();
}

cudaError_t launch_loop_records_shell(tufrg_model *m)
{
    const int g = (m->Nk + 255) / 256;
    if (m->precision == TUFRG_FP64)
        rec_shell_kernel<double><<<g, 256, 0, m->stream>>>(m->d_E, m->Nk, m->Lf, m->mu, m->T_reg, static_cast<D4 *>(m->d_rec));
    else
        rec_shell_kernel<float><<<g, 256, 0, m->stream>>>(m->d_E, m->Nk, m->Lf, m->mu, m->T_reg, static_cast<float4 *>(m->d_rec));
    return cudaGetLastError();
}

cudaError_t launch_loop_records(tufrg_model *m)
{
    if (m->regulator == TUFRG_REG_MOMENTUM_SHELL) return cudaSuccess;   // the shell records do not depend on Lambda
    PhaseScope ps(m, PH_FERMI);
    const int g = (m->Nk + 255) / 256;
    if (m->precision == TUFRG_FP64) rec_T_kernel<double><<<g, 256, 0, m->stream>>>(m->Nk, 0.0, m->d_scal, static_cast<D4 *>(m->d_rec));
    else rec_T_kernel<float><<<g, 256, 0, m->stream>>>(m->Nk, 0.0, m->d_scal, static_cast<float4 *>(m->d_rec));
    return cudaGetLastError();
}

// the records of one temperature for a caller's bands (tufrg_loops_noalloc)
cudaError_t launch_records_f32(const double *E, const double2 *U, int Nk, int Lf, double mu, double T, float4 *rec, cudaStream_t s)
{
    const int g = (Nk + 255) / 256;
    rec_static_kernel<float><<<g, 256, 0, s>>>(E, U, Nk, Lf, mu, rec);
    rec_T_kernel<float><<<g, 256, 0, s>>>(Nk, T, nullptr, rec);
    return cudaGetLastError();
}

// Loop sums of the channels of the mask into the partial buffer (no reduction).  With s_list, only the
// listed transfer momenta (n_list of them) are evaluated, into partial slots 0..n_list-1 of part.
cudaError_t launch_loops2h_ex(tufrg_model *m, int channel_mask, const int *s_list, int n_list, void *part, size_t part_cs, const int *skip)
{
    return m->precision == TUFRG_FP64 ? run2<double>(m, channel_mask, s_list, n_list, part, part_cs, skip)
                                      : run2<float>(m, channel_mask, s_list, n_list, part, part_cs, skip);
}

cudaError_t launch_loops2h_sum(tufrg_model *m, int channel_mask)
{
    // with loop symmetries only the orbit representatives are summed (partial slots = list positions)
    const size_t n_s = m->sym ? m->n_loop_q : m->Nq;
    return launch_loops2h_ex(m, channel_mask, m->sym ? m->d_loop_list : nullptr, m->sym ? m->n_loop_q : 0, m->d_part,
                            n_s * m->plan_h.n_partials * m->dxs.size() * n_dyh(m) * 16, m->sur ? m->d_sur_flag : nullptr);
}

// The reduction of launch_loops2h_ex's partials: the loops of the n_s list positions (momenta slot_q, or all of them),
// written at the positions or (at_q) at their momenta; gather: at every momentum, from the orbit representatives.
cudaError_t launch_loops2h_reduce(tufrg_model *m, int channel_mask, const void *part, size_t part_cs, const int *slot_q, int n_s,
                                 bool gather, bool at_q, double2 *out64, float2 *out32, size_t out_cs, const int *skip)
{
    return m->precision == TUFRG_FP64
               ? reduce2<double>(m, channel_mask, part, part_cs, slot_q, n_s, gather, at_q, out64, out32, out_cs, skip)
               : reduce2<float>(m, channel_mask, part, part_cs, slot_q, n_s, gather, at_q, out64, out32, out_cs, skip);
}

LoopPlan plan_loops2h(const tufrg_model *m)
{
    // Choose the number of ky ranges so that the grid fills whole waves of the SMs; the flush of the columns' sums costs
    // about 0.45 rows of work per pair of bond differences (measured: 6 rows for 5 x 3 pairs, 23 for 9 x 5).  Fewer
    // ranges can be faster alone (24 x 24 momenta: one range 47 us, three 49), but not beside the state's transforms and
    // projections (124 against 106 us for the whole right-hand side; FP64 8 x 8 five ranges 273, nine 252 us).
    // 48 x 48, 13 form factors: two ranges 727 us, one 690 us, whole right-hand side 998 and 940 us.
    LoopPlan p{};
    const int ctas_x = (m->Lf + NT - 1) / NT;
    const int half = loops2_half_mask(m);
    const int rows = half == 3 ? m->Lf / 2 + 1 : m->Lf;
    const int per_sm = loops2h_blocks_per_sm(m);
    if (per_sm == 0) return p;
    const double slots = (double)m->sm_count * per_sm;
    const double flush = 0.45 * (double)m->dxs.size() * n_dyh(m);
    double best = 1e300;
    int best_c = 1;
    for (int c = 1; c <= 16; c++) {
        const int len = (rows + c - 1) / c;
        if (len < 8) break;
        const double ctas = (double)m->n_loop_q * ctas_x * c * 2;
        const double waves = std::ceil(ctas / slots);
        const double cost = waves * (len + flush);
        if (cost < best * 0.999) { best = cost; best_c = c; }
    }
    p.ky_chunks = best_c;
    p.n_partials = ctas_x * best_c;
    return p;
}

cudaError_t launch_loops(tufrg_model *m, int channel_mask, bool reps_only, bool flow, bool want64)
{
    if (m->sur) TUFRG_CUDA_TRY(launch_surrogate(m, channel_mask));
    reps_only = reps_only && m->sym;
    if (m->ns != 2) return loops_gen_supported(m) ? launch_loops_gen(m, channel_mask, reps_only, want64) : cudaErrorNotSupported;
    if (!loops2_supported(m)) return cudaErrorNotSupported;
    if (flow && m->precision != TUFRG_FP64) return launch_loops_flow(m, channel_mask, reps_only);
    if (!(channel_mask & 3)) return cudaSuccess;
    const int n_s = m->sym ? m->n_loop_q : m->Nq;
    const size_t part_cs = (size_t)n_s * m->plan_h.n_partials * m->dxs.size() * n_dyh(m) * 16, out_cs = (size_t)m->Nq * m->nd * 16;
    TUFRG_CUDA_TRY(launch_loops2h_sum(m, channel_mask));
    const bool fp64 = m->precision == TUFRG_FP64;
    // symmetric states: the representatives' loops at their own momenta, in the precision their products read
    return launch_loops2h_reduce(m, channel_mask, m->d_part, part_cs, m->sym ? m->d_loop_list : nullptr,
                                reps_only ? m->n_loop_q : m->Nq, m->sym && !reps_only, reps_only,
                                fp64 || (want64 && !reps_only) ? m->d_Lc : nullptr, fp64 ? nullptr : m->d_Lc32, out_cs,
                                m->sur ? m->d_sur_flag : nullptr);
}

}  // namespace tufrg

