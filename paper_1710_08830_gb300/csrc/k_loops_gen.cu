// Loop k-sum for any N_s (used for N_s = 4, 6; the two-band case has dedicated kernels).
//
//   P:  [L^-_{t1t2t3t4}(s)]_{R1R2} = (1/Nk) sum_q e^{-iq.(R1-R2)} sum_{l1} rho1^{l1}_{t1t3}(s-q) T^{l1}_{t2t4}
//   C:  [L^+_{t1t2t3t4}(u)]_{R1R2} = (1/Nk) sum_q e^{-iq.(R1-R2)} sum_{l1} rho1^{l1}_{t1t3}(q)   T^{l1}_{t2t4}
//   with rho^l_{tt'} = U_{tl} U*_{t'l},  T^{l1} = sum_{l2} w_{l1 l2} rho2'^{l2},  rho2' = rho2 (P) or conj (C),
//   w the d/dT of the bubbles of Eqs. disc_2a / disc_2b (Eqs. loopminus, loopplus, loop_orbital).
//
// rho1 and T are Hermitian N_s x N_s matrices, so each is N_s^2 real numbers (loop_comp: Re and Im of the upper triangle,
// the diagonal; for C the sign of rho2' imaginary parts is left to the end), and for fixed (s, q) the orbital dressing is
// the real rank-N_s product Y = A B with A[c][l] = rho1, B[l][c'] = T.  The row phase e^{-iqy dy} is a cosine and a sine
// for dy > 0, so a column's sums are W[p][c][c'] = sum_qy phi_p(qy) Y, p over 1, cos, sin, cos, sin, ...: N_s^5 +
// (2 n_dy - 1) N_s^4 real multiply-adds per (s, q), 3.3 times fewer than in complex arithmetic at N_s = 6 and n_dy = 3.
// Half of the fine mesh suffices where exchanging the propagators maps the sum onto itself (see k_loops2h.cu): columns
// qx = hx + j, 2 hx = sx (mod Lf), a column that is its own partner with weight 1/2.
//
// One CTA owns one transfer momentum and a range of columns; it walks the fine mesh column by column in batches of KB
// rows.  The raw eigenvectors and Fermi entries of a batch arrive in shared memory by cp.async while the batch before it
// is multiplied (two buffers); from them all threads form A and B of the batch (projectors, pair weights, T), then every
// thread updates its TA x TB tile of W (NG thread groups share the batch's rows where the tiles alone are too few
// threads; their sums meet in shared memory at the end of the column).  At the end of a column the thread adds
// e^{-iqx dx} W into the accumulator of its own entries (no other CTA touches them, so no atomics; the order is fixed).
// loops_gen_finish puts the orbital entries together from the real components, adds the exchanged half, writes both
// Hermitian halves, L(-d)[b][a] = conj(L(d)[a][b]), and scales by 1/Nk; loops_gen_gather writes the other momenta of
// the orbits.  From the ranges' accumulators on, the split path adds in FP32 pairs (in FP32 alone the 12 x 12 / 5 x 5 bilayer
// mesh's P loops are off by 1.9e-7 instead of 0.7e-7).
// FP64: bound by the FP64 pipe (two results per clock and SM); the 8 x 8 / 6 x 6 three-orbital sums of both channels
// take 1.66 ms (6.9 ms in complex arithmetic over the whole mesh).
#include <cmath>
#include <type_traits>

#include "tufrg_internal.cuh"

namespace tufrg {
namespace {

constexpr int GMAXD = 9;
constexpr int GMAXND = 96;
constexpr int KB = 8;          // rows staged per batch

template <typename R> struct FTg;
template <> struct FTg<double> { using t = FermiEntry; };
template <> struct FTg<float> { using t = FermiEntry32; };

template <typename R>
struct GenArgs {
    const typename cpx<R>::t *U;        // [Nk][NS][NS]
    const typename FTg<R>::t *ft;       // [Nk][NS]
    typename cpx<R>::t *acc;            // [kx range][slot][nd][NS^2][NS^2] accumulators, half plane filled (by the first
                                        // column of a range, the others added);
                                        // FP64 on the plain path, FP32 on the split path
    const typename cpx<R>::t *ptab;     // e^{-2 pi i n / Lf}
    int Lq, nc, Lf, nd, ndx, ndyh;
    int dxs[GMAXD], dys[GMAXD];
    int dslot[GMAXD][GMAXD];            // [dxi][dyi] -> delta index (half plane), or -1
    R thr_factor;                       // degenerate-pair switch = thr_factor * T
    const double *Tp;                   // device flow scale (T, or Lambda with the momentum shell)
    R shell_T;                          // > 0: momentum-shell regulator at this temperature (tables hold e, f, h)
    const int *s_list;                  // optional: CTA x sums transfer momentum s_list[x] into accumulator slot x
    int n_slot;                         // momenta per kx range (accumulator slots of one range)
    int kx_len;                         // columns per kx range; CTA y covers [y kx_len, (y + 1) kx_len)
    int half;                           // half of the mesh
};

__device__ __forceinline__ void ldft(const FermiEntry *p, double &e, double &g, double &gp) { e = p->e; g = p->g; gp = p->gp; }
__device__ __forceinline__ void ldft(const FermiEntry32 *p, float &e, float &g, float &gp) { e = p->e; g = p->g; gp = p->gp; }

// v in [0, 2 L) -> v mod L without a division
__device__ __forceinline__ int wrap1(int v, int L) { return v >= L ? v - L : v; }

// Shared memory of one CTA: two buffers of the raw eigenvectors [2 sides][KB][NS^2] and Fermi entries
// [2 sides][KB][NS] of a batch (side 0: k1, side 1: k2; filled by cp.async one batch ahead), then rho1 / T / rho2'
// [KB][NS][NS^2] each (16-byte aligned rows of rho1), batch phases [KB][NPH], pair weights [KB][NS][NS], and with several
// thread groups their column sums [NG - 1][NPH][NS^4].
template <typename R, int NS>
constexpr size_t gen_raw_bytes()
{
    return 2 * (sizeof(typename cpx<R>::t) * 2 * KB * NS * NS + sizeof(typename FTg<R>::t) * 2 * KB * NS);
}
template <typename R, int NS, int NDYH, int NG>
size_t gen_smem()
{
    constexpr int NPH = 2 * NDYH - 1;
    return gen_raw_bytes<R, NS>() +
           sizeof(R) * (3 * KB * NS * NS * NS + KB * NPH + KB * NS * NS + (size_t)(NG - 1) * NPH * NS * NS * NS * NS);
}

// TA consecutive values from shared memory (aligned to their size where that is 16 bytes)
__device__ __forceinline__ void ld_tile(const float *p, float (&v)[4])
{
    const float4 t = *reinterpret_cast<const float4 *>(p);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
template <typename R, int N> __device__ __forceinline__ void ld_tile(const R *p, R (&v)[N])
{
#pragma unroll
    for (int i = 0; i < N; i++) v[i] = p[i];
}

template <typename R, int NS, int TA, int TB, int NG, int NDYH, int WHICH>
__global__ void loops_gen_kernel(const __grid_constant__ GenArgs<R> a)
{
    using C2 = typename cpx<R>::t;
    constexpr int NS2 = NS * NS, NPH = 2 * NDYH - 1;
    constexpr int GA = NS2 / TA, GB = NS2 / TB;     // thread grid over the (c, c') tiles: rows ta TA + i, columns tb + j GB
    constexpr int NT = GA * GB;
    using FT = typename FTg<R>::t;
    constexpr int CU = NS2 * (int)sizeof(C2) / 16, CF = NS * (int)sizeof(FT) / 16, CK = CU + CF;
    static_assert(CU * 16 == NS2 * (int)sizeof(C2) && CF * 16 == NS * (int)sizeof(FT), "rows of 16-byte chunks");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C2 *sUr = reinterpret_cast<C2 *>(smem_raw);                     // [2 buffers][2 sides][KB][NS2]
    FT *sFr = reinterpret_cast<FT *>(sUr + 2 * 2 * KB * NS2);       // [2 buffers][2 sides][KB][NS]
    R *sA = reinterpret_cast<R *>(smem_raw + gen_raw_bytes<R, NS>());   // [KB][NS][NS2] rho1
    R *sB = sA + KB * NS * NS2;                                    // [KB][NS][NS2] T
    R *sR2 = sB + KB * NS * NS2;                                   // [KB][NS][NS2] rho2
    R *sPh = sR2 + KB * NS * NS2;                                  // [KB][NPH] row phases
    R *sW = sPh + KB * NPH;                                        // [KB][NS][NS] pair weights
    R *sG = sW + KB * NS * NS;                                     // [NG - 1][NPH][NS2][NS2]
    __shared__ int2 comp[NS2];                                     // (t NS + t', imaginary part) of a component
    const int Lf = a.Lf;
    if (threadIdx.x < NS2) {
        int t, tp;
        bool im;
        loop_comp<NS>(threadIdx.x, t, tp, im);
        comp[threadIdx.x] = make_int2(t * NS + tp, im);
    }
    const int s = a.s_list ? a.s_list[blockIdx.x] : blockIdx.x;
    const int sx = (s / a.Lq) * a.nc, sy = (s % a.Lq) * a.nc;
    const int grp = threadIdx.x / NT, tt = threadIdx.x - grp * NT, ta = tt / GB, tb = tt - ta * GB;
    const bool shell = a.shell_T > R(0);
    const R lam = shell ? (R)(*a.Tp) : R(0);
    const R thr = a.thr_factor * (shell ? a.shell_T : (R)(*a.Tp));
    const bool active = threadIdx.x < NT * NG;
    // columns hx .. hx + ncol - 1 (mod Lf), fix0 and fix1 their own partners; or the whole mesh
    const bool even_L = !(Lf & 1), odd_s = sx & 1;
    const int hx = !a.half ? 0 : !odd_s ? sx / 2 : even_L ? (sx + 1) / 2 : (sx + Lf) / 2;
    const int ncol = !a.half ? Lf : even_L ? Lf / 2 + (odd_s ? 0 : 1) : (Lf + 1) / 2;
    const int fix0 = a.half && !(even_L && odd_s) ? 0 : -1, fix1 = a.half && even_L && !odd_s ? Lf / 2 : -1;
    C2 *acc = a.acc + ((size_t)blockIdx.y * a.n_slot + blockIdx.x) * a.nd * NS2 * NS2;
    const int j_end = min(ncol, (int)(blockIdx.y + 1) * a.kx_len);
    // fine-mesh indices of row ky of column kx: k1 = s - k, k2 = k (P); k1 = k, k2 = k - s (C)
    auto k_of = [&](int side, int kx, int ky) {
        if (side == (WHICH == 0 ? 1 : 0)) return kx * Lf + ky;                      // the point k itself
        return WHICH == 0 ? wrap1(sx - kx + Lf, Lf) * Lf + wrap1(sy - ky + Lf, Lf)  // s - k
                          : wrap1(kx - sx + Lf, Lf) * Lf + wrap1(ky - sy + Lf, Lf); // k - s
    };
    // copies of the raw eigenvectors and Fermi entries of the rows [ky0, ky0 + KB) of column j into buffer buf
    auto stage_raw = [&](int j, int ky0, int buf) {
        const int kx = wrap1(hx + j, Lf), nb = min(KB, Lf - ky0), per_side = nb * CK;
        for (int idx = threadIdx.x; idx < 2 * per_side; idx += blockDim.x) {
            const int side = idx >= per_side, r = idx - side * per_side, kb = r / CK, c = r % CK;
            const int k = k_of(side, kx, ky0 + kb);
            const int slot = (buf * 2 + side) * KB + kb;
            if (c < CU)
                cp_async16(reinterpret_cast<char *>(sUr + (size_t)slot * NS2) + 16 * c,
                           reinterpret_cast<const char *>(a.U + (size_t)k * NS2) + 16 * c);
            else
                cp_async16(reinterpret_cast<char *>(sFr + (size_t)slot * NS) + 16 * (c - CU),
                           reinterpret_cast<const char *>(a.ft + (size_t)k * NS) + 16 * (c - CU));
        }
        cp_async_commit();
    };
    int buf = 0;
    const int j_beg = blockIdx.y * a.kx_len;
    if (j_beg < j_end) stage_raw(j_beg, 0, 0);

    for (int j = j_beg; j < j_end; j++) {
        R W[NPH][TA][TB];
#pragma unroll
        for (int p = 0; p < NPH; p++)
#pragma unroll
            for (int i = 0; i < TA; i++)
#pragma unroll
                for (int k = 0; k < TB; k++) W[p][i][k] = R(0);
        for (int ky0 = 0; ky0 < Lf; ky0 += KB, buf ^= 1) {
            const int nb = min(KB, Lf - ky0);
            // copies of the next batch (this column's next rows, else the next column's first) go out before
            // this batch is used; the raw buffer they fill was last read before the previous batch's products
            if (ky0 + KB < Lf) stage_raw(j, ky0 + KB, buf ^ 1);
            else if (j + 1 < j_end) stage_raw(j + 1, 0, buf ^ 1);
            else cp_async_commit();   // an empty group keeps the count of one group in flight
            cp_async_wait<1>();        // this thread's copies of the current batch have landed
            __syncthreads();           // everyone's copies landed; previous batch fully consumed
            const C2 *rU1 = sUr + (size_t)(buf * 2 + 0) * KB * NS2, *rU2 = sUr + (size_t)(buf * 2 + 1) * KB * NS2;
            const FT *rF1 = sFr + (size_t)(buf * 2 + 0) * KB * NS, *rF2 = sFr + (size_t)(buf * 2 + 1) * KB * NS;
            for (int idx = threadIdx.x; idx < nb * NDYH; idx += blockDim.x) {
                const int kb = idx / NDYH, d = idx % NDYH;
                if (d >= a.ndyh) continue;
                const C2 ph = a.ptab[(int)(((long)(ky0 + kb) * a.dys[d]) % Lf)];   // (cos, -sin)
                if (d == 0) sPh[kb * NPH] = R(1);
                else {
                    sPh[kb * NPH + 2 * d - 1] = ph.x;
                    sPh[kb * NPH + 2 * d] = -ph.y;
                }
            }
            // projector components of the batch: rho1 (k1 side) into sA, rho2 (k2 side) into sR2
            for (int idx = threadIdx.x; idx < nb * NS * NS2; idx += blockDim.x) {
                const int kb = idx / (NS * NS2), r = idx % (NS * NS2), l = r / NS2;
                const int2 cc = comp[r % NS2];
                const int o1 = kb * NS2 + (cc.x / NS) * NS + l, o2 = kb * NS2 + (cc.x % NS) * NS + l;
                const C2 u = rU1[o1], v = rU1[o2], x = rU2[o1], y = rU2[o2];
                sA[idx] = cc.y ? u.y * v.x - u.x * v.y : u.x * v.x + u.y * v.y;   // u conj(v)
                sR2[idx] = cc.y ? x.y * y.x - x.x * y.y : x.x * y.x + x.y * y.y;
            }
            for (int idx = threadIdx.x; idx < nb * NS * NS; idx += blockDim.x) {
                const int kb = idx / (NS * NS), l1 = (idx / NS) % NS, l2 = idx % NS;
                R e1, g1, gp1, e2, g2, gp2;
                ldft(&rF1[kb * NS + l1], e1, g1, gp1);
                ldft(&rF2[kb * NS + l2], e2, g2, gp2);
                sW[idx] = gen_pair_weight<WHICH, R>(e1, g1, gp1, e2, g2, gp2, thr, lam);
            }
            __syncthreads();
            // T^{l1}_{c'} = sum_l2 w_{l1 l2} rho2^{l2}_{c'}
            for (int idx = threadIdx.x; idx < nb * NS * NS2; idx += blockDim.x) {
                const int kb = idx / (NS * NS2), l1 = (idx / NS2) % NS, p = idx % NS2;
                R t = R(0);
#pragma unroll
                for (int l2 = 0; l2 < NS; l2++) t = fma(sW[(kb * NS + l1) * NS + l2], sR2[(kb * NS + l2) * NS2 + p], t);
                sB[idx] = t;
            }
            __syncthreads();
            if (active) {
                for (int kb = grp; kb < nb; kb += NG) {
                    R Y[TA][TB];
#pragma unroll
                    for (int i = 0; i < TA; i++)
#pragma unroll
                        for (int k = 0; k < TB; k++) Y[i][k] = R(0);
#pragma unroll
                    for (int l = 0; l < NS; l++) {
                        R av[TA], bv[TB];
                        ld_tile(sA + (kb * NS + l) * NS2 + ta * TA, av);
#pragma unroll
                        for (int k = 0; k < TB; k++) bv[k] = sB[(kb * NS + l) * NS2 + tb + k * GB];
#pragma unroll
                        for (int i = 0; i < TA; i++)
#pragma unroll
                            for (int k = 0; k < TB; k++) Y[i][k] = fma(av[i], bv[k], Y[i][k]);
                    }
#pragma unroll
                    for (int i = 0; i < TA; i++)
#pragma unroll
                        for (int k = 0; k < TB; k++) W[0][i][k] += Y[i][k];
#pragma unroll
                    for (int d = 1; d < NDYH; d++) {
                        if (d >= a.ndyh) break;
                        const R c = sPh[kb * NPH + 2 * d - 1], sn = sPh[kb * NPH + 2 * d];
#pragma unroll
                        for (int i = 0; i < TA; i++)
#pragma unroll
                            for (int k = 0; k < TB; k++) {
                                W[2 * d - 1][i][k] = fma(c, Y[i][k], W[2 * d - 1][i][k]);
                                W[2 * d][i][k] = fma(sn, Y[i][k], W[2 * d][i][k]);
                            }
                    }
                }
            }
        }
        if (NG > 1) {   // the other groups' sums of this column
            __syncthreads();
            if (active && grp > 0) {
#pragma unroll
                for (int p = 0; p < NPH; p++)
#pragma unroll
                    for (int i = 0; i < TA; i++)
#pragma unroll
                        for (int k = 0; k < TB; k++) sG[(((grp - 1) * NPH + p) * NS2 + ta * TA + i) * NS2 + tb + k * GB] = W[p][i][k];
            }
            __syncthreads();
            if (active && grp == 0) {
#pragma unroll
                for (int g = 0; g < NG - 1; g++)
#pragma unroll
                    for (int p = 0; p < NPH; p++)
#pragma unroll
                        for (int i = 0; i < TA; i++)
#pragma unroll
                            for (int k = 0; k < TB; k++) W[p][i][k] += sG[((g * NPH + p) * NS2 + ta * TA + i) * NS2 + tb + k * GB];
            }
        }
        // add e^{-i kx dx} W into this thread's accumulators (fixed order, no other writer)
        if (active && grp == 0) {
            const int kx = wrap1(hx + j, Lf);
            const R f = j == fix0 || j == fix1 ? R(0.5) : R(1);
            for (int xi = 0; xi < a.ndx; xi++) {
                C2 ph = a.ptab[(int)((((long)kx * a.dxs[xi]) % Lf + Lf) % Lf)];   // (cos, -sin)
                ph.x *= f;
                ph.y *= f;
#pragma unroll
                for (int d = 0; d < NDYH; d++) {
                    if (d >= a.ndyh) break;
                    const int di = a.dslot[xi][d];
                    if (di < 0) continue;
                    C2 *o = acc + ((size_t)di * NS2 + ta * TA) * NS2 + tb;
                    C2 v[TA][TB];   // all loads before the additions
#pragma unroll
                    for (int i = 0; i < TA; i++)
#pragma unroll
                        for (int k = 0; k < TB; k++) v[i][k] = j == j_beg ? mk(R(0), R(0)) : o[i * NS2 + k * GB];
#pragma unroll
                    for (int i = 0; i < TA; i++)
#pragma unroll
                        for (int k = 0; k < TB; k++) {
                            // (C - i S) (cos - i sin)
                            const R C = W[d == 0 ? 0 : 2 * d - 1][i][k], S = d == 0 ? R(0) : W[d == 0 ? 0 : 2 * d][i][k];
                            v[i][k].x += ph.x * C + ph.y * S;
                            v[i][k].y += ph.y * C - ph.x * S;
                            o[i * NS2 + k * GB] = v[i][k];
                        }
                }
            }
        }
    }
    cp_async_wait<0>();   // nothing in flight at exit (the last group is empty)
    if (j_beg >= j_end)   // a range without columns
        for (size_t i = threadIdx.x; i < (size_t)a.nd * NS2 * NS2; i += blockDim.x) acc[i] = mk(R(0), R(0));
}

// Numbers of the sums after the k-sum: FP64, or on the split path an unevaluated FP32 pair h + l (l the rounding errors of
// h), good to about 2^-46.  The pairs take FP32 operations only: FP64 ones have one 64th of their rate, and with the
// conversions the 153 representatives of the 32 x 32 three-orbital mesh took 0.24 ms more per channel (10.07 against 9.60 ms
// for the right-hand side).
struct Pair {
    float h, l;
};
__device__ __forceinline__ double plus(double a, double b) { return a + b; }
__device__ __forceinline__ Pair plus(Pair a, Pair b)   // Knuth's two-sum of the leading parts
{
    const float t = __fadd_rn(a.h, b.h), u = __fsub_rn(t, a.h);
    const float e = __fadd_rn(__fsub_rn(a.h, __fsub_rn(t, u)), __fsub_rn(b.h, u));
    return Pair{t, __fadd_rn(e, __fadd_rn(a.l, b.l))};
}
__device__ __forceinline__ double times(double a, double b) { return a * b; }
__device__ __forceinline__ Pair times(Pair a, Pair b)
{
    const float t = __fmul_rn(a.h, b.h);
    return Pair{t, fmaf(a.l, b.h, fmaf(a.h, b.l, fmaf(a.h, b.h, -t)))};
}
__device__ __forceinline__ double minus(double a) { return -a; }
__device__ __forceinline__ Pair minus(Pair a) { return Pair{-a.h, -a.l}; }
// (an infinite leading part leaves a NaN in the other)
__device__ __forceinline__ float as_f32(Pair a) { return isfinite(a.h) ? __fadd_rn(a.h, a.l) : a.h; }
__device__ __forceinline__ float as_f32(double a) { return narrow_f(a); }
__device__ __forceinline__ double as_f64(Pair a) { return isfinite(a.h) ? widen_f(a.h) + widen_f(a.l) : widen_f(a.h); }
__device__ __forceinline__ double as_f64(double a) { return a; }

template <typename V>
struct Cx {
    V x, y;
};
template <typename V> __device__ __forceinline__ Cx<V> add(Cx<V> a, Cx<V> b) { return Cx<V>{plus(a.x, b.x), plus(a.y, b.y)}; }
template <typename V> __device__ __forceinline__ Cx<V> times(Cx<V> a, Cx<V> b)
{
    return Cx<V>{plus(times(a.x, b.x), minus(times(a.y, b.y))), plus(times(a.x, b.y), times(a.y, b.x))};
}
template <typename V> __device__ __forceinline__ Cx<V> turn(Cx<V> v, int k)   // i^k v
{
    switch (k & 3) {
    case 0: return v;
    case 1: return Cx<V>{minus(v.y), v.x};
    case 2: return Cx<V>{minus(v.x), minus(v.y)};
    default: return Cx<V>{v.y, minus(v.x)};
    }
}
// complex values as they lie in memory: FP64, FP32 accumulators, FP32 pairs (h, h, l, l)
__device__ __forceinline__ Cx<double> ld_cx(double2 v) { return Cx<double>{v.x, v.y}; }
__device__ __forceinline__ Cx<Pair> ld_cx(float2 v) { return Cx<Pair>{Pair{v.x, 0.f}, Pair{v.y, 0.f}}; }
__device__ __forceinline__ Cx<Pair> ld_cx(float4 v) { return Cx<Pair>{Pair{v.x, v.z}, Pair{v.y, v.w}}; }
__device__ __forceinline__ double2 st_cx(Cx<double> v) { return make_double2(v.x, v.y); }
__device__ __forceinline__ float4 st_cx(Cx<Pair> v) { return make_float4(v.x.h, v.y.h, v.x.l, v.y.l); }
template <typename S> using val_t = decltype(ld_cx(S{}).x);                    // its number
template <typename S> using wide_t = decltype(st_cx(ld_cx(S{})));               // a sum of such values in memory

// the kx ranges' accumulators added (fixed order, eight loads in flight): FP64 over the first range's accumulators, FP32
// into pairs; the half-plane differences hp only, which alone the k-sum writes.  Grid: (n_hp entries / 256, slots); n: values
// of one range.
template <int NS, typename S>
__global__ void __launch_bounds__(256) loops_gen_chunk_sum(const S *acc, int nchunk, size_t n, const int *hp, int n_hp, int nd, wide_t<S> *sum)
{
    constexpr int NS4 = NS * NS * NS * NS;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_hp * NS4) return;
    const size_t t = ((size_t)blockIdx.y * nd + hp[i / NS4]) * NS4 + i % NS4;
    constexpr int UB = 8;
    auto s = ld_cx(acc[t]);
    for (int c = 1; c < nchunk; c += UB) {
        S w[UB];
#pragma unroll
        for (int j = 0; j < UB; j++)
            if (c + j < nchunk) w[j] = acc[(size_t)(c + j) * n + t];
#pragma unroll
        for (int j = 0; j < UB; j++)
            if (c + j < nchunk) s = add(s, ld_cx(w[j]));
    }
    sum[t] = st_cx(s);
}

template <typename S>
struct FinArgs {
    const S *acc;                // [slot][nd][NS2][NS2] half-plane sums in real components
    const wide_t<S> *ptab;       // e^{-2 pi i n / Lf}
    const int *deltas, *partner, *slot_q;   // slot_q: momentum of a slot (null: the slot)
    const SymElem *elem;         // the element inv inverts the momentum (C channel's exchanged half)
    const int *dinv;
    int nd, Lq, nc, half, inv;
    val_t<S> inv_nk;
    double2 *out64;
    float2 *out32;
};

// orbital entry S[d][ia][ib] of one slot's half-plane sums
template <int NS, int CH, typename S>
__device__ __forceinline__ auto gen_entry(const S *acc, const FinArgs<S> &f, int d, int ia, int ib)
{
    constexpr int NS2 = NS * NS;
    const int dx = f.deltas[2 * d], dy = f.deltas[2 * d + 1];
    const bool hp = dy > 0 || (dy == 0 && dx >= 0);
    if (!hp) {   // L(-d)[b][a] = conj(L(d)[a][b])
        d = f.partner[d];
        const int t = ia;
        ia = ib;
        ib = t;
    }
    // compact pairs -> (t1 t3), (t2 t4)
    const int ax = ia / NS, ay = ia % NS, bx = ib / NS, by = ib % NS;
    const int t1 = CH == 0 ? ay : ax, t2 = CH == 0 ? ax : ay, t3 = CH == 0 ? by : bx, t4 = CH == 0 ? bx : by;
    const int lr = loop_comp_index<NS>(t1, t3), rr = loop_comp_index<NS>(t2, t4);
    const int ls = t1 == t3 ? 0 : t1 < t3 ? 1 : -1, rs0 = t2 == t4 ? 0 : t2 < t4 ? 1 : -1, rs = CH == 0 ? rs0 : -rs0;
    const S *o = acc + (size_t)d * NS2 * NS2;
    auto v = ld_cx(o[lr * NS2 + rr]);
    if (ls) v = add(v, turn(ld_cx(o[(lr + 1) * NS2 + rr]), ls));        // + i ls w
    if (rs) v = add(v, turn(ld_cx(o[lr * NS2 + rr + 1]), rs));
    if (ls && rs) v = add(v, turn(ld_cx(o[(lr + 1) * NS2 + rr + 1]), ls + rs));
    if (!hp) v.y = minus(v.y);
    return v;
}

// Every entry of every slot's loops at the slot's momentum: the sums, the exchanged half, 1/Nk, rounded once for the FP32
// loops.  Grid: (entries / 256, slots).
template <int NS, int CH, typename S>
__global__ void __launch_bounds__(256) loops_gen_finish(const __grid_constant__ FinArgs<S> f)
{
    constexpr int NS2 = NS * NS, NS4 = NS2 * NS2;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= f.nd * NS4) return;
    const int s = blockIdx.y, d = t / NS4, ia = (t / NS2) % NS2, ib = t % NS2;
    const int q = f.slot_q ? f.slot_q[s] : s;
    const S *acc = f.acc + (size_t)s * f.nd * NS4;
    auto v = gen_entry<NS, CH>(acc, f, d, ia, ib);
    if (f.half) {
        auto swp = [](int a) { return (a % NS) * NS + a / NS; };
        int d2 = d, k = 0;
        decltype(v) w;
        if (CH == 0) {   // e^{-is.Delta} conj(S[b~][a~])
            w = gen_entry<NS, CH>(acc, f, d, swp(ib), swp(ia));
            w.y = minus(w.y);
        } else {         // V [e^{iu.Delta} S[b~][a~]] V^dagger
            const SymElem &e = f.elem[f.inv];
            d2 = f.dinv[f.inv * f.nd + d];
            w = gen_entry<NS, CH>(acc, f, d2, swp(e.src[1][ib]), swp(e.src[1][ia]));
            k = e.qt[1][ia] - e.qt[1][ib];
        }
        const int n = (((q / f.Lq) * f.deltas[2 * d2] + (q % f.Lq) * f.deltas[2 * d2 + 1]) % f.Lq + f.Lq) % f.Lq * f.nc;
        auto p = ld_cx(f.ptab[n]);
        if (CH == 1) p.y = minus(p.y);
        w = times(p, w);
        if (CH == 1) {
            if (f.elem[f.inv].conj) w.y = minus(w.y);
            w = turn(w, k);
        }
        v = add(v, w);
    }
    v.x = times(v.x, f.inv_nk);
    v.y = times(v.y, f.inv_nk);
    const size_t o = (size_t)q * f.nd * NS4 + t;
    if (f.out64) f.out64[o] = make_double2(as_f64(v.x), as_f64(v.y));
    if (f.out32) f.out32[o] = make_float2(as_f32(v.x), as_f32(v.y));
}

// The momenta that are not orbit representatives: entry (d', a', b') of q' from the representative's (d, src a', src b'),
// i^(qt[a'] - qt[b']) (conj ? conj(v) : v).  Grid: (entries / 256, momenta).  Reads and writes the same buffers (the
// representatives' rows are only read).
template <int NS>
__global__ void __launch_bounds__(256) loops_gen_gather(double2 *L64, float2 *L32, int nd, const int2 *qmap, const int *list,
                                                        const SymElem *elem, const int *dinv, int ch)
{
    constexpr int NS2 = NS * NS, NS4 = NS2 * NS2;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nd * NS4) return;
    const int q2 = blockIdx.y;
    const int2 ie = qmap[q2];
    const int q = list[ie.x];
    if (q == q2) return;
    const int d2 = t / NS4, a2 = (t / NS2) % NS2, b2 = t % NS2;
    const SymElem &e = elem[ie.y];
    const size_t i = (size_t)q * nd * NS4 + ((size_t)dinv[ie.y * nd + d2] * NS2 + e.src[ch][a2]) * NS2 + e.src[ch][b2];
    const size_t o = (size_t)q2 * nd * NS4 + t;
    const int k = e.qt[ch][a2] - e.qt[ch][b2], conj = e.conj;
    auto image = [&](auto v) {
        Cx<decltype(v.x)> w{v.x, conj ? -v.y : v.y};
        switch (k & 3) {
        case 0: return mk(w.x, w.y);
        case 1: return mk(-w.y, w.x);
        case 2: return mk(-w.x, -w.y);
        default: return mk(w.y, -w.x);
        }
    };
    if (L64) L64[o] = image(L64[i]);
    if (L32) L32[o] = image(L32[i]);
}

// per instantiation: tile and thread groups.  FP64 tiles are sized for the registers of the column sums; the FP32
// N_s = 4 case (256 entries) takes 4 x 2 tiles, one warp, and four warps that share the rows.
template <typename R, int NS> struct Tile;
template <> struct Tile<double, 6> { static constexpr int A = 3, B = 3, G = 1; };
template <> struct Tile<double, 4> { static constexpr int A = 2, B = 2, G = 1; };
template <> struct Tile<float, 6> { static constexpr int A = 4, B = 3, G = 1; };
template <> struct Tile<float, 4> { static constexpr int A = 4, B = 2, G = 4; };

template <typename R, int NS> constexpr int gen_threads()
{
    using T = Tile<R, NS>;
    return ((NS * NS / T::A) * (NS * NS / T::B) * T::G + 31) / 32 * 32;
}
template <typename R, int NS, int NDYH, int WHICH>
auto gen_kernel() { return loops_gen_kernel<R, NS, Tile<R, NS>::A, Tile<R, NS>::B, Tile<R, NS>::G, NDYH, WHICH>; }

template <typename R, int NS, int NDYH, int WHICH>
cudaError_t launch_gen(tufrg_model *m, const GenArgs<R> &a)
{
    const size_t smem = gen_smem<R, NS, NDYH, Tile<R, NS>::G>();
    auto kern = gen_kernel<R, NS, NDYH, WHICH>();
    if (smem > 48 * 1024) TUFRG_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    PhaseScope ps(m, PH_LOOPS);
    kern<<<dim3(a.n_slot, m->gen_chunks), gen_threads<R, NS>(), smem, m->stream>>>(a);
    return cudaGetLastError();
}

template <typename R, int NS>
cudaError_t dispatch_gen(tufrg_model *m, const GenArgs<R> &a, int ch)
{
    if (a.ndyh <= 3) return ch == 0 ? launch_gen<R, NS, 3, 0>(m, a) : launch_gen<R, NS, 3, 1>(m, a);
    if (a.ndyh <= 5) return ch == 0 ? launch_gen<R, NS, 5, 0>(m, a) : launch_gen<R, NS, 5, 1>(m, a);
    return cudaErrorNotSupported;
}

// where the sums over several kx ranges lie: behind FP32 accumulators, over the first range's FP64 ones
size_t gen_acc_bytes(const tufrg_model *m)
{
    const size_t ns2 = (size_t)m->ns * m->ns, values = (size_t)m->gen_chunks * m->n_loop_q * m->nd * ns2 * ns2;
    return (values * (m->precision == TUFRG_FP64 ? sizeof(double2) : sizeof(float2)) + 15) & ~size_t(15);
}
template <typename S> wide_t<S> *gen_sums(tufrg_model *m)   // S: the accumulators
{
    return reinterpret_cast<wide_t<S> *>(static_cast<char *>(m->d_part) + (sizeof(S) == sizeof(double2) ? 0 : gen_acc_bytes(m)));
}

template <typename R>
cudaError_t run_gen(tufrg_model *m, int ch, bool half, const typename cpx<R>::t *U, const typename FTg<R>::t *ft,
                    const typename cpx<R>::t *ptab)
{
    using C2 = typename cpx<R>::t;
    GenArgs<R> a{};
    a.U = U; a.ft = ft; a.ptab = ptab;
    a.acc = reinterpret_cast<C2 *>(m->d_part);
    a.thr_factor = sizeof(R) == 4 ? R(1e-2) : R(1e-5);
    a.Tp = m->d_scal;
    a.shell_T = m->regulator == TUFRG_REG_MOMENTUM_SHELL ? (R)m->T_reg : R(0);
    a.Lq = m->Lq; a.nc = m->nc; a.Lf = m->Lf; a.nd = m->nd;
    a.ndx = (int)m->dxs.size();
    for (int v : m->dys)
        if (v >= 0) a.dys[a.ndyh++] = v;
    for (int i = 0; i < a.ndx; i++) {
        a.dxs[i] = m->dxs[i];
        for (int j = 0; j < GMAXD; j++) {
            a.dslot[i][j] = -1;
            if (j >= a.ndyh) continue;
            const int dx = a.dxs[i], dy = a.dys[j];
            if (!(dy > 0 || dx >= 0)) continue;
            for (int d = 0; d < m->nd; d++)
                if (m->deltas[2 * d] == dx && m->deltas[2 * d + 1] == dy) a.dslot[i][j] = d;
        }
    }
    a.s_list = m->sym ? m->d_loop_list : nullptr;
    a.n_slot = m->sym ? m->n_loop_q : m->Nq;
    a.half = half ? 1 : 0;
    const int ncol = half ? m->Lf / 2 + 1 : m->Lf;
    a.kx_len = (ncol + m->gen_chunks - 1) / m->gen_chunks;
    const size_t n = (size_t)a.n_slot * m->nd * m->ns * m->ns * m->ns * m->ns;
    TUFRG_CUDA_TRY((m->ns == 6 ? dispatch_gen<R, 6>(m, a, ch) : dispatch_gen<R, 4>(m, a, ch)));
    if (m->gen_chunks > 1) {
        PhaseScope ps(m, PH_LOOPRED);
        const int n_hp = (m->nd + 1) / 2;
        const dim3 grid((n_hp * m->ns * m->ns * m->ns * m->ns + 255) / 256, a.n_slot);
        auto k = m->ns == 6 ? loops_gen_chunk_sum<6, C2> : loops_gen_chunk_sum<4, C2>;
        k<<<grid, 256, 0, m->stream>>>(a.acc, m->gen_chunks, n, m->d_hp, n_hp, m->nd, gen_sums<C2>(m));
    }
    return cudaGetLastError();
}

template <int NS, typename S>
cudaError_t finish(tufrg_model *m, int ch, int n_slot, const FinArgs<S> &f, bool gather)
{
    constexpr int NS4 = NS * NS * NS * NS;
    const unsigned gx = (unsigned)((m->nd * NS4 + 255) / 256);
    PhaseScope ps(m, PH_LOOPRED, gather ? 2 : 1);
    if (ch == 0) loops_gen_finish<NS, 0><<<dim3(gx, n_slot), 256, 0, m->stream>>>(f);
    else loops_gen_finish<NS, 1><<<dim3(gx, n_slot), 256, 0, m->stream>>>(f);
    TUFRG_CUDA_TRY(cudaGetLastError());
    if (gather)
        loops_gen_gather<NS><<<dim3(gx, m->Nq), 256, 0, m->stream>>>(f.out64, f.out32, m->nd, m->d_qmap, m->d_loop_list,
                                                                    m->d_sym_elem, m->d_sym_dinv, ch);
    return cudaGetLastError();
}

int gen_ndyh(const tufrg_model *m)
{
    int n = 0;
    for (int v : m->dys) n += v >= 0;
    return n;
}

// Resident CTAs per SM of the instantiation the model launches
template <typename R, int NS>
int gen_blocks_per_sm(int ndyh)
{
    return ndyh <= 3 ? resident_ctas(gen_kernel<R, NS, 3, 0>(), gen_threads<R, NS>(), gen_smem<R, NS, 3, Tile<R, NS>::G>())
                     : resident_ctas(gen_kernel<R, NS, 5, 0>(), gen_threads<R, NS>(), gen_smem<R, NS, 5, Tile<R, NS>::G>());
}

}  // namespace

bool loops_gen_supported(const tufrg_model *m)
{
    return (m->ns == 4 || m->ns == 6) && (int)m->dxs.size() <= GMAXD && gen_ndyh(m) <= 5 && m->nd <= GMAXND;
}

size_t gen_part_bytes(const tufrg_model *m)
{
    const size_t ns2 = (size_t)m->ns * m->ns, sums = (size_t)m->n_loop_q * m->nd * ns2 * ns2 * sizeof(float4);
    return gen_acc_bytes(m) + (m->precision != TUFRG_FP64 && m->gen_chunks > 1 ? sums : 0);
}

// The kx ranges per momentum that fill the GPU best: the fewest waves of CTAs times columns per range (plus about one
// column's time of start and end per CTA), up to one column per range within MAX_RANGES accumulators.  With few
// momenta the short ranges are what fills the SMs: the sums of 28 momenta of the 12 x 12 / 5 x 5 bilayer mesh take 76 us
// per evaluation, 206 us with at least four columns per range.  The FP64 sums of six states fill the FP64 pipe to nine
// tenths with one CTA (0.60 ms per column; two side by side 0.54 each), so their waves are counted over the SMs: 15 momenta
// of 25 columns take 1.81 ms in 9 ranges, 2.16 in 13 (195 CTAs, two on some SMs), 1.66 in 25; 10 of 22 1.08 in 11, 0.97 in 22.
int plan_gen_chunks(const tufrg_model *m)
{
    constexpr int MAX_RANGES = 64;
    const int ndyh = gen_ndyh(m);
    int per_sm;
    if (m->precision == TUFRG_FP64) per_sm = m->ns == 6 ? gen_blocks_per_sm<double, 6>(ndyh) : gen_blocks_per_sm<double, 4>(ndyh);
    else per_sm = m->ns == 6 ? gen_blocks_per_sm<float, 6>(ndyh) : gen_blocks_per_sm<float, 4>(ndyh);
    if (per_sm == 0) return 0;
    const bool pipe = m->precision == TUFRG_FP64 && m->ns == 6;
    const long slots = (long)m->sm_count * (pipe ? 1 : per_sm);
    const int ncol = loops2_half_mask(m) == 3 ? m->Lf / 2 + 1 : m->Lf;
    int best = 1;
    double best_cost = 1e300;
    for (int c = 1; c <= std::min(MAX_RANGES, ncol); c++) {
        const double waves = std::ceil((double)m->n_loop_q * c / (double)slots);
        const double cost = waves * (std::ceil((double)ncol / c) + (pipe ? 0.05 : 1.0)) * (pipe && waves > 1.0 ? 0.9 : 1.0);
        if (cost < best_cost * 0.999) { best_cost = cost; best = c; }
    }
    return best;
}

cudaError_t launch_loops_gen(tufrg_model *m, int channel_mask, bool reps_only, bool want64)
{
    const size_t ns4 = (size_t)m->ns * m->ns * m->ns * m->ns, per = (size_t)m->Nq * m->nd * ns4;
    const int n_slot = m->sym ? m->n_loop_q : m->Nq;
    const bool fp64 = m->precision == TUFRG_FP64;
    for (int ch = 0; ch < 2; ch++) {
        if (!((channel_mask >> ch) & 1)) continue;
        // the tensor-core kernel's half sums need the init-time list (its groups share their columns)
        const bool half = ((loops2_half_mask(m) >> ch) & 1) && (!m->loops_tc || m->loop_list_is_reps);
        if (m->loops_tc) TUFRG_CUDA_TRY(launch_loops_tc(m, ch, half, reinterpret_cast<float2 *>(m->d_part)));
        else if (fp64) TUFRG_CUDA_TRY(run_gen<double>(m, ch, half, m->d_U, m->d_ft, m->d_lph));
        else TUFRG_CUDA_TRY(run_gen<float>(m, ch, half, m->d_U32, m->d_ft32, m->d_lph32));
        auto run = [&](auto *acc) {
            FinArgs<std::remove_pointer_t<decltype(acc)>> f{};
            f.acc = acc;
            f.ptab = reinterpret_cast<decltype(f.ptab)>(fp64 ? (const void *)m->d_lph : (const void *)m->d_lph_pair);
            f.deltas = m->d_deltas;
            f.partner = m->d_dpartner;
            f.slot_q = m->sym ? m->d_loop_list : nullptr;
            f.elem = m->d_sym_elem;
            f.dinv = m->d_sym_dinv;
            f.nd = m->nd;
            f.Lq = m->Lq;
            f.nc = m->nc;
            f.half = half ? 1 : 0;
            f.inv = m->sym_inv;
            const double inv_nk = 1.0 / (double)m->Nk;
            if constexpr (sizeof(f.inv_nk) == sizeof(double) && std::is_floating_point_v<decltype(f.inv_nk)>) f.inv_nk = inv_nk;
            else f.inv_nk = Pair{(float)inv_nk, (float)(inv_nk - (double)(float)inv_nk)};
            f.out64 = fp64 || (want64 && !reps_only) ? m->d_Lc + ch * per : nullptr;
            f.out32 = fp64 ? nullptr : m->d_Lc32 + ch * per;
            const bool gather = m->sym && !reps_only;
            return m->ns == 6 ? finish<6>(m, ch, n_slot, f, gather) : finish<4>(m, ch, n_slot, f, gather);
        };
        if (fp64) TUFRG_CUDA_TRY(run(reinterpret_cast<double2 *>(m->d_part)));
        else if (m->gen_chunks > 1) TUFRG_CUDA_TRY(run(gen_sums<float2>(m)));
        else TUFRG_CUDA_TRY(run(reinterpret_cast<float2 *>(m->d_part)));
    }
    return cudaSuccess;
}

}  // namespace tufrg
