// Associated-Legendre part of the spherical-harmonic basis change (the
// expensive half of "change the basis" in Sect. 2.1; O(nside lmax^2) per
// transform, Sect. 3) and the harmonic-space blend of Eq. (4), fused into
// the analysis epilogue.
//
//   synthesis  G_m(theta_r) = sum_{l=m..L} a_lm lambda_lm(cos theta_r)
//   analysis   b_lm = sum_r lambda_lm(cos theta_r) F_m(theta_r)
//              a_new = S_l / (S_l + lambda tau Omega) * Omega b_lm   (Eq. 4)
//
// North/south ring pairs share lambda up to (-1)^(l-m): synthesis keeps an
// even and an odd partial sum per pair, analysis folds F_N +- F_S before the
// sum.  The recurrence runs in "mu form" (wf_internal.cuh) from per-(m, pair)
// seeds at the first l where |lambda_lm| exceeds 2^-80 (computed in FP64 with
// an explicit binary exponent, since sin^m(theta) underflows FP64 near the
// poles at large m); below that l every term is < 2^-80 and is dropped.
//
// Two precisions:
//   FP64     k_legsyn<TG>, k_legana<TF, NP>: one ring pair per lane, two in large analyses.
//   mixed    k_legsyn_mx<NP>, k_legana_mx<NP>: FP32 recurrence and
//            contraction, NP ring pairs per thread (synthesis) or per lane
//            (analysis) in packed f32x2 lanes (__ffma2_rn), in the two-step
//            forms of the belt and the polar cap described above MxTables below.
//            The block l < l_c, where the messenger iteration's contraction
//            margin tau_h / S_l is below the FP32 error, runs through the FP64
//            kernels instead (the FP32 recurrence restarts at l_c from FP64
//            seeds), so the mixed iteration keeps the FP64 iteration's
//            stability on the modes that converge slowest.
#include <climits>
#include <cmath>
#include <cstdio>
#include <type_traits>

#include "wf_internal.cuh"

namespace wf {

namespace {

constexpr double SEED_LOG2_THRESHOLD = -80.0;
constexpr int BIG = INT_MAX / 2;

__host__ __device__ inline long long mbase(int lmax, int m) { return (long long)m * (2 * lmax + 3 - m) / 2; }

// first l of the FP32 range for m < lc: l_c rounded up to the parity of m
__host__ __device__ inline int lcm_of(int lc, int m) { return m + 2 * ((lc - m + 1) / 2); }

// ---------------------------------------------------------------------------
// seeds: one thread per (m, pair), FP64 with a carried binary exponent
// ---------------------------------------------------------------------------
__global__ void k_seeds(int lmax, int npairs, const double *__restrict__ xp, const double *__restrict__ stp,
                        const double *__restrict__ log2c, const double *__restrict__ A,
                        const double *__restrict__ c, int *__restrict__ ls_out, double *__restrict__ s0_out,
                        double *__restrict__ s1_out)
{
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long long)(lmax + 1) * npairs) return;
    const int m = (int)(idx / npairs);
    const int p = (int)(idx % npairs);
    const double x = xp[p], st = stp[p];
    const long long base = mbase(lmax, m);
    const double lg2 = log2c[m] + (m > 0 ? m * log2(st) : 0.0);
    int E = (int)floor(lg2);
    double u = exp2(lg2 - E);  // mu_m * 2^-E (c_m = 1)
    if (m & 1) u = -u;
    double up = 0.0;           // mu_{l-1} * 2^-E
    double thr = ldexp(1.0, (int)(SEED_LOG2_THRESHOLD) - E);
    int l = m;
    for (;;) {
        if (fabs(c[base + (l - m)] * u) >= thr) break;
        if (l >= lmax) { l = lmax + 1; break; }
        const double un = A[base + (l + 1 - m)] * x * u - up;
        up = u;
        u = un;
        ++l;
        if (fabs(u) > 0x1p+500) {
            u *= 0x1p-500;
            up *= 0x1p-500;
            E += 500;
            thr = ldexp(1.0, (int)(SEED_LOG2_THRESHOLD) - E);
        }
    }
    int ls;
    double s0 = 0.0, s1 = 0.0;
    if (l > lmax) {
        ls = lmax + 1;
    } else if (((l - m) & 1) == 0) {
        ls = l;
        s0 = ldexp(u, E);
        s1 = (l < lmax) ? ldexp(A[base + (l + 1 - m)] * x * u - up, E) : 0.0;
    } else {
        ls = l - 1;
        s0 = ldexp(up, E);
        s1 = ldexp(u, E);
    }
    ls_out[idx] = ls;
    s0_out[idx] = s0;
    s1_out[idx] = s1;
}

// first entry of m in the tables per (m, k), k = (l - m) / 2: at least (lmax - m + 1)/2 + 1
// entries before the next m's
__host__ __device__ inline long long kbase(int lmax, int m) { return (mbase(lmax, m) + 4 * (long long)m) >> 1; }

// Starting states of the mixed kernels for a given FP64 block l < lc.
//
// Two-step kernels: k0 (k = (l - m) / 2) is the first kept k rounded up to a multiple of four,
// so that a pair starts between two blocks of four steps (the terms between, at most
// three k after |lambda| first exceeds 2^-80, stay below 2^-50); k0 = lmax where nothing is
// kept.  For m < lc the FP64-accurate values of l_c's multiple of four below start a ring
// that has begun by then; the kernels leave out what lies below l_c.
// seed, belt (p >= ncap): (mu_l, x mu_{l+1}); cap: (E, D) = (mu_l / e_k, mu_{l+2} / e_{k+1} - mu_l / e_k).
//
// Tensor-core synthesis (ls_out not null): the recurrence starts at l = max(l_s, lcm) from
// s0, s1 = (mu_l, mu_{l+1}).
__global__ void k_restart_seeds(int lmax, int npairs, int lc, int ncap, const double *__restrict__ xp,
                                const double *__restrict__ A, const double *__restrict__ Atop,
                                const double4 *__restrict__ kd, const int *__restrict__ ls_in,
                                const double *__restrict__ s0_in, const double *__restrict__ s1_in,
                                int *__restrict__ k0_out, float2 *__restrict__ seed, int *__restrict__ ls_out,
                                float *__restrict__ s0_out, float *__restrict__ s1_out)
{
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long long)(lmax + 1) * npairs) return;
    const int m = (int)(idx / npairs);
    const int p = (int)(idx % npairs);
    const double *Am = A + mbase(lmax, m) - m;  // A_l = Am[l]
    const double x = xp[p];
    const int ls = ls_in[idx];
    const int l1 = m < lc ? lcm_of(lc, m) : m;  // the FP64 block's end
    // (mu_l, mu_{l+1}) from the seeds at ls up to l = la <= lmax (mu_{lmax+1} = 0 where la = lmax)
    auto at = [&](int la, double &a, double &b) {
        a = s0_in[idx];
        b = s1_in[idx];
        for (int l = ls; l < la; ++l) {
            const double c = l + 2 <= lmax ? Am[l + 2] * x * b - a : 0.0;
            a = b;
            b = c;
        }
    };
    double a = 0.0, b = 0.0;
    if (ls_out) {
        const int l = ls > lmax ? ls : l1 > ls ? (l1 > lmax ? lmax + 1 : l1) : ls;
        if (l <= lmax) at(l, a, b);
        ls_out[idx] = l;
        s0_out[idx] = (float)a;
        s1_out[idx] = (float)b;
    }
    int k0 = lmax;
    float2 sd = make_float2(0.f, 0.f);
    if (ls <= lmax) {
        const int kn = (ls - m) >> 1, k1 = ((l1 - m) >> 1) & ~3;
        const int k = kn <= k1 ? k1 : (kn + 3) & ~3, l = m + 2 * k;
        if (l <= lmax && l1 <= lmax) {
            k0 = k;
            at(l, a, b);
            sd = make_float2((float)a, (float)(x * b));
            if (p < ncap) {
                const long long kk = kbase(lmax, m) + k;
                const double e0 = a * kd[kk].w;
                double e1 = 0.0;
                if (l + 2 <= lmax + 1) e1 = ((l + 2 <= lmax ? Am[l + 2] : Atop[m]) * x * b - a) * kd[kk + 1].w;
                sd = make_float2((float)e0, (float)(e1 - e0));
            }
        }
    }
    k0_out[idx] = k0;
    seed[idx] = sd;
}

// ---------------------------------------------------------------------------
// FP64 transforms.  FP64 runs at 1/64 of the FP32 rate (two lanes per clock and SM), so what
// counts is the FP64 operations per (l, ring pair) and that all SMs have work.
//
// Both directions take one warp per (group of 32 ring pairs, m) and advance two l at once
// (k = (l - m)/2) with the odd values carried as x mu, which saves the product A_l x on the
// way from odd to even:
//     E_k = mu_{m+2k},  O_k = x mu_{m+2k+1},
//     E_{k+1} = A_{2k+2} O_k - E_k,  O_{k+1} = (A_{2k+3} X) E_{k+1} - O_k,
// with X = x^2 rounded; X's rounding error d, which would move the ring, is made up for in
// every fourth step by O += 4 (2 d) E, with the limit 2 of A.  3.6 operations per (l, pair)
// with the contraction (4 before).  The odd sum is divided by x at the end (analysis: its
// input is).  A, c and a_lm pass through shared memory in blocks of 32 l, the next block's
// loads in flight over the present one.
//
// One CTA per m before: the SMs waited for those that had m = 0 and its neighbours where the
// ring pairs are few.  Synthesis at nside 256, lmax 512
// 0.606 -> 0.390 ms (its FP64 operations take 0.38); at nside 100, lmax 200, 46 -> 35 us and the
// analysis 87 -> 60 + 6 us.
//
// lcut > 0: the FP64 block of the mixed path, l < lcm_of(lcut, m), output into G with row
// stride gstride.
// ---------------------------------------------------------------------------
constexpr int F64_BLK = 32;  // l per block of the tables

struct F64Pair {
    int k0, kmin, kmaxs;  // first k of this lane's pair; the warp's least and largest first k
    double s0, s1;        // mu_{m+2k0}, x mu_{m+2k0+1}
    double4 xw;           // X, 8 (x^2 - X), x, 1/x (0 for x = 0)
};

__device__ __forceinline__ F64Pair f64_pair(int m, int Lm, int npairs, int p, const int *__restrict__ ls_tab,
                                            const double *__restrict__ s0_tab, const double *__restrict__ s1_tab,
                                            const double4 *__restrict__ xw)
{
    F64Pair P{BIG, 0, -1, 0.0, 0.0, make_double4(0.0, 0.0, 0.0, 0.0)};
    if (p < npairs) {
        const size_t sidx = (size_t)m * npairs + p;
        const int ls = ls_tab[sidx];
        if (ls <= Lm) {
            P.k0 = (ls - m) >> 1;
            P.xw = xw[p];
            P.s0 = s0_tab[sidx];
            P.s1 = P.xw.z * s1_tab[sidx];
        }
    }
    P.kmin = __reduce_min_sync(0xffffffffu, P.k0);
    P.kmaxs = __reduce_max_sync(0xffffffffu, P.k0 == BIG ? -1 : P.k0);
    return P;
}

// (E_k, O_k) to k + 1; FIX: with the correction of X, in every fourth step
template <bool FIX>
__device__ __forceinline__ void f64_advance(double2 A /* A_{2k+2}, A_{2k+3} */, const double4 &xw, double &E, double &O)
{
    E = fma(A.x, O, -E);
    O = fma(A.y * xw.x, E, -O);
    if (FIX) O = fma(xw.y, E, O);
}

// TG: element type of the output (FP32 for the FP64 block of the mixed path,
// whose ring pass adds it to the FP32 coefficients in FP32 anyway: converting
// here keeps the 1/64-rate conversions off the ring kernel).
template <typename TG>
__global__ void __launch_bounds__(32) k_legsyn(int lmax, int L, int npairs, int lcut, const double2 *__restrict__ alm,
                                               const double *__restrict__ A, const double *__restrict__ c64,
                                               const int *__restrict__ ls_tab, const double *__restrict__ s0_tab,
                                               const double *__restrict__ s1_tab, const double4 *__restrict__ xw,
                                               cx<TG> *__restrict__ G, int gstride)
{
    __shared__ double2 sac[F64_BLK];    // c a_lm
    __shared__ double2 sA[F64_BLK / 2];
    const int m = blockIdx.y, lane = threadIdx.x;
    const int p = (gridDim.x - 1 - blockIdx.x) * 32 + lane;  // the equator (most work) first
    const int Lm = lcut > 0 ? min(L, lcm_of(lcut, m) - 1) : L;
    const int nl = Lm - m + 1;
    const long long base = mbase(lmax, m);
    const F64Pair P = f64_pair(m, Lm, npairs, p, ls_tab, s0_tab, s1_tab, xw);
    double er = 0.0, ei = 0.0, orr = 0.0, oi = 0.0;
    double E = 0.0, O = 0.0;
    double2 na;
    double nc, nA;
    auto fetch = [&](int j) {
        na = j < nl ? alm[base + j] : make_double2(0.0, 0.0);
        nc = j < nl ? c64[base + j] : 0.0;
        nA = j + 2 < nl ? A[base + j + 2] : 0.0;
    };
    int kc = P.kmin & ~3;
    const int nk = (nl + 1) >> 1;
    if (P.kmin != BIG) fetch(2 * kc + lane);
    auto block4 = [&](int k, bool start) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (start && kc + k + i == P.k0) {
                E = P.s0;
                O = P.s1;
            }
            const double2 a0 = sac[2 * (k + i)], a1 = sac[2 * (k + i) + 1], c = sA[k + i];
            er = fma(a0.x, E, er);
            ei = fma(a0.y, E, ei);
            orr = fma(a1.x, O, orr);
            oi = fma(a1.y, O, oi);
            if (i == 3) f64_advance<true>(c, P.xw, E, O);
            else f64_advance<false>(c, P.xw, E, O);
        }
    };
    if (P.kmin != BIG)
        for (; kc < nk; kc += F64_BLK / 2) {
            __syncwarp();
            sac[lane] = cscale(na, nc);
            reinterpret_cast<double *>(sA)[lane] = nA;
            __syncwarp();
            fetch(2 * (kc + F64_BLK / 2) + lane);
            const int kn = min(F64_BLK / 2, nk - kc);  // (a block of four runs up to three k past the end, on zeros)
            for (int k = 0; k < kn; k += 4) {
                if (kc + k <= P.kmaxs) block4(k, true);
                else block4(k, false);
            }
        }
    if (p < npairs) {
        orr *= P.xw.w;
        oi *= P.xw.w;
        cx<TG> *g = G + ((size_t)p * gstride + m) * 2;
        g[0] = mk<TG>((TG)(er + orr), (TG)(ei + oi));
        g[1] = mk<TG>((TG)(er - orr), (TG)(ei - oi));
    }
}

// ---------------------------------------------------------------------------
// warp reduce-scatter of CH complex values: lane i ends with the sum over the
// warp of value (i >> (5 - log2 CH)).
// ---------------------------------------------------------------------------
template <typename T, int CH>
__device__ __forceinline__ void warp_reduce_scatter(T (&vr)[CH], T (&vi)[CH], int lane)
{
#pragma unroll
    for (int r = 0; r < 5; ++r) {
        const int off = 16 >> r;
        const int n = CH >> r;
        if (n >= 2) {
            const int half = n / 2;
            const bool up = (lane & off) != 0;
#pragma unroll
            for (int i = 0; i < half; ++i) {
                const T sr = up ? vr[i] : vr[i + half];
                const T kr = up ? vr[i + half] : vr[i];
                const T si = up ? vi[i] : vi[i + half];
                const T ki = up ? vi[i + half] : vi[i];
                vr[i] = kr + __shfl_xor_sync(0xffffffffu, sr, off);
                vi[i] = ki + __shfl_xor_sync(0xffffffffu, si, off);
            }
        } else {
            vr[0] += __shfl_xor_sync(0xffffffffu, vr[0], off);
            vi[0] += __shfl_xor_sync(0xffffffffu, vi[0], off);
        }
    }
}

// Eq. (4) epilogue shared by both precisions: t_hat = Omega (c acc + low),
// a_new = S/(S + lam tau_h) t_hat, chi^2 of a_old, lambda = 1 residual.
__global__ void k_epi_table(EpiArgs a)
{
    epi_entry(a, blockIdx.x * blockDim.x + threadIdx.x);
}

// sums of one thread over its a_lm: chi^2 of a_old, residual^2, x^T S^-1 x and x^T S^-2 x of a_new
struct BlendSums {
    double chi2 = 0.0, res2 = 0.0, hnew = 0.0, qnew = 0.0;
};

// one a_lm: b = c_lm times its ring sum, or 0 (l > L); the sums leave out the weight 2 of m > 0.
// (Every FP64 operation counts here: at 1/64 of the FP32 rate the epilogue of the mixed analysis
// is bound by the FP64 pipe.)
__device__ __forceinline__ void blend_one(int l, int L, long long idx, int mode, const BlendArgs &ba, double2 b,
                                          const double2 *__restrict__ a_old, double2 *__restrict__ out, BlendSums &v)
{
    if (mode == LEG_ADJOINT) {
        out[idx] = b;
        return;
    }
    // per-l factors tabulated once per launch (no FP64 division per a_lm)
    const double4 e = ba.epi[l];
    const bool on = __double2hiint(e.w) != 0;  // 1 or 0
    const double2 ao = a_old[idx];
    double2 an = make_double2(0.0, 0.0);
    if (l <= L && on) {
        an.x = e.x * b.x;
        an.y = e.x * b.y;
    }
    if (on) {
        v.chi2 += (ao.x * ao.x + ao.y * ao.y) * e.y;
        if (ba.want_norms) {
            const double an2 = (an.x * an.x + an.y * an.y) * e.y;
            v.hnew += an2;
            v.qnew += an2 * e.y;
        }
        if (ba.want_resid) {
            const double dx = e.z * (ao.x - an.x), dy = e.z * (ao.y - an.y);
            v.res2 = fma(dx, dx, fma(dy, dy, v.res2));
        }
    }
    out[idx] = an;
}

// the CTA's sums into part[4 m ..]: a warp per sum that is wanted (128 threads); the last CTA adds
// up the partials of all (fixed order).  Every warp reducing all four by shuffles took more FP64
// operations than the blend itself at lmax 1024.  Totals by a launch of its own: 25 iterations at
// nside 128 1.55 ms, 1.51 here; 16 at nside 512 (with a sweep) 7.56 and 7.49 ms.
constexpr int EPI_THREADS = 128;

__device__ __forceinline__ void blend_sums(const BlendSums &s, int m, const BlendArgs &ba, double *__restrict__ part,
                                           double (*red)[EPI_THREADS])
{
    __shared__ int last;
    const int t = threadIdx.x, w = t >> 5, lane = t & 31;
    auto wanted = [&](int k) { return k == 0 || (k == 1 ? ba.want_resid : ba.want_norms); };
    // the sum of row k, in every lane of the warp that asks
    auto row_sum = [&](int k) {
        double x = red[k][lane];
#pragma unroll
        for (int i = 32; i < EPI_THREADS; i += 32) x += red[k][i + lane];
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        return x;
    };
    red[0][t] = s.chi2;
    if (ba.want_resid) red[1][t] = s.res2;
    if (ba.want_norms) {
        red[2][t] = s.hnew;
        red[3][t] = s.qnew;
    }
    __syncthreads();
    const double x = wanted(w) ? row_sum(w) : 0.0;
    if (lane == 0) {
        __stcg(&part[4 * m + w], m ? 2.0 * x : x);
        __threadfence();
    }
    if (!ba.sums_out) return;
    __syncthreads();
    if (t == 0) last = atomicAdd(ba.sums_count, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    for (int k = 0; k < 4; ++k) {
        if (!wanted(k)) continue;
        double v = 0.0;
#pragma unroll 4
        for (int i = t; i < (int)gridDim.x; i += EPI_THREADS) v += __ldcg(&part[4 * i + k]);
        red[k][t] = v;
    }
    double v = 0.0;
#pragma unroll 4
    for (int i = t; i < ba.npix; i += EPI_THREADS) v += __ldcg(&ba.pix[i]);
    red[4][t] = v;
    __syncthreads();
    for (int k = w; k < 5; k += EPI_THREADS / 32) {
        const double y = k == 4 || wanted(k) ? row_sum(k) : 0.0;
        if (lane == 0) ba.sums_out[k == 4 ? 0 : 1 + k] = y;
    }
    if (t == 0) *ba.sums_count = 0;
}

// val(j): c_lm times the ring sum at l = m + j
template <typename VAL>
__device__ __forceinline__ void blend_epilogue(int lmax, int L, int m, long long base, int mode, const BlendArgs &ba,
                                               VAL val, const double2 *__restrict__ a_old, double2 *__restrict__ out,
                                               double *__restrict__ part, double (*red)[EPI_THREADS])
{
    BlendSums v;
    for (int j = threadIdx.x; j <= lmax - m; j += blockDim.x)
        blend_one(m + j, L, base + j, mode, ba, m + j <= L ? val(j) : make_double2(0.0, 0.0), a_old, out, v);
    if (mode == LEG_BLEND) blend_sums(v, m, ba, part, red);
}

// FP64 analysis: chunks of 16 l in registers, summed over a lane's NP ring pairs, reduced across
// the warp (one addition per value), times c_l added to acc (zero before).  Two pairs per lane
// halve the reduction per pair, 3.6 + 2/NP operations per (l, pair), where there are ring pairs
// for it (ANA64_MIN_PAIRS).  TF is the storage type of F (FP64 plans: double; FP64 block of the
// mixed path: float).
template <typename TF, int NP>
__global__ void __launch_bounds__(32) k_legana(int lmax, int L, int npairs, int lcut, const cx<TF> *__restrict__ F,
                                               const double *__restrict__ A, const int *__restrict__ ls_tab,
                                               const double *__restrict__ s0_tab, const double *__restrict__ s1_tab,
                                               const double4 *__restrict__ xw, const double *__restrict__ c64,
                                               double2 *__restrict__ acc)
{
    constexpr int CH = 16;
    __shared__ double2 sA[F64_BLK / 2];
    const int m = blockIdx.y, lane = threadIdx.x;
    const int p0 = (gridDim.x - 1 - blockIdx.x) * 32 * NP + lane;
    const int Lm = lcut > 0 ? min(L, lcm_of(lcut, m) - 1) : L;
    const int nl = Lm - m + 1;
    const long long base = mbase(lmax, m);
    F64Pair P[NP];
    double2 FE[NP], FO[NP];
    double E[NP], O[NP];
    int kmin = BIG, kmaxs = -1;
#pragma unroll
    for (int q = 0; q < NP; ++q) {
        const int p = p0 + 32 * q;
        P[q] = f64_pair(m, Lm, npairs, p, ls_tab, s0_tab, s1_tab, xw);
        kmin = min(kmin, P[q].kmin);
        kmaxs = max(kmaxs, P[q].kmaxs);
        E[q] = O[q] = 0.0;
        FE[q] = FO[q] = make_double2(0.0, 0.0);
        if (P[q].k0 != BIG) {
            const cx<TF> *f = F + ((size_t)p * (lmax + 1) + m) * 2;
            const cx<TF> fn = f[0], fs = f[1];
            FE[q] = make_double2((double)fn.x + (double)fs.x, (double)fn.y + (double)fs.y);
            FO[q] = make_double2(((double)fn.x - (double)fs.x) * P[q].xw.w, ((double)fn.y - (double)fs.y) * P[q].xw.w);
        }
    }
    if (kmin == BIG) return;
    int kc = kmin & ~3;
    const int nk = (nl + 1) >> 1;
    double nA = 2 * kc + lane + 2 < nl ? A[base + 2 * kc + lane + 2] : 0.0;
    for (; kc < nk; kc += F64_BLK / 2) {
        __syncwarp();
        reinterpret_cast<double *>(sA)[lane] = nA;
        __syncwarp();
        const int jn = 2 * kc + F64_BLK + lane + 2;
        nA = jn < nl ? A[base + jn] : 0.0;
        for (int k = 0; k < min(F64_BLK / 2, nk - kc); k += CH / 2) {
            double vr[CH], vi[CH];
            const bool start = kc + k <= kmaxs;
#pragma unroll
            for (int i = 0; i < CH / 2; ++i) {
#pragma unroll
                for (int q = 0; q < NP; ++q) {
                    if (start && kc + k + i == P[q].k0) {
                        E[q] = P[q].s0;
                        O[q] = P[q].s1;
                    }
                    vr[2 * i] = q ? fma(E[q], FE[q].x, vr[2 * i]) : E[q] * FE[q].x;
                    vi[2 * i] = q ? fma(E[q], FE[q].y, vi[2 * i]) : E[q] * FE[q].y;
                    vr[2 * i + 1] = q ? fma(O[q], FO[q].x, vr[2 * i + 1]) : O[q] * FO[q].x;
                    vi[2 * i + 1] = q ? fma(O[q], FO[q].y, vi[2 * i + 1]) : O[q] * FO[q].y;
                    if ((i & 3) == 3) f64_advance<true>(sA[k + i], P[q].xw, E[q], O[q]);
                    else f64_advance<false>(sA[k + i], P[q].xw, E[q], O[q]);
                }
            }
            // c_l for this lane's l, in flight over the reduction
            const int j = 2 * (kc + k) + (lane >> 1);
            const double cc = j < nl ? c64[base + j] : 0.0;
            warp_reduce_scatter<double, CH>(vr, vi, lane);
            if (j < nl) atomicAdd(lane & 1 ? &acc[base + j].y : &acc[base + j].x, cc * (lane & 1 ? vi[0] : vr[0]));
        }
    }
}

// Eq. (4) epilogue of the FP64 analysis, a CTA per m; clears the sums for the next launch
__global__ void __launch_bounds__(EPI_THREADS) k_ana64_epilogue(int lmax, int L, int mode, BlendArgs ba,
                                                        const double2 *__restrict__ a_old, double2 *__restrict__ out,
                                                        double *__restrict__ part, double2 *__restrict__ acc)
{
    __shared__ double red[5][EPI_THREADS];
    const int m = blockIdx.x;
    const long long base = mbase(lmax, m);
    auto val = [&](int j) {
        const double2 v = acc[base + j];
        acc[base + j] = make_double2(0.0, 0.0);
        return v;
    };
    blend_epilogue(lmax, L, m, base, mode, ba, val, a_old, out, part, red);
}

// ---------------------------------------------------------------------------
// FP64 block of the mixed path from a table.  The block (m < l_c,
// m <= l < lcm(l_c, m)) holds few (l, m) but every ring pair, and GB300 runs
// FP64 at 1/64 of the FP32 rate, so the FP64 recurrence kernels above spend
// more time on it than the FP32 kernels spend on a far larger share of the
// band.  Here lambda_lm(x_p) is computed once per l_c by the FP64 recurrence
// and stored as a pair of FP32 numbers (hi, lo) with hi + lo = lambda to 48
// significant bits; both directions then stream the table and accumulate in
// double-float arithmetic on the FP32 pipe: products split exactly with an
// FMA (Dekker's product) and sums with Knuth's two-sum, so each term carries
// about 2^-46 relative error against 2^-53 in FP64, far below the FP32
// operator error the block exists to avoid.
// Layout: row r = rowoff[m] + (l - m), column p (ring pair), row stride
// np_pad (npairs rounded up to 32; padding columns hold zeros).
// ---------------------------------------------------------------------------
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e)
{
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// (shi, slo) += (xh + xl)(yh + yl), dropping only the xl yl term (2^-48 relative)
__device__ __forceinline__ void df_fma(float &shi, float &slo, float xh, float xl, float yh, float yl)
{
    const float p = __fmul_rn(xh, yh);
    float e = __fmaf_rn(xh, yh, -p);  // xh yh - p exactly
    e = __fmaf_rn(xh, yl, e);
    e = __fmaf_rn(xl, yh, e);
    float s, t;
    two_sum(shi, p, s, t);
    shi = s;
    slo = __fadd_rn(slo, __fadd_rn(t, e));
}

// (ahi, alo) += (bhi, blo)
__device__ __forceinline__ void df_add(float &ahi, float &alo, float bhi, float blo)
{
    float s, e;
    two_sum(ahi, bhi, s, e);
    ahi = s;
    alo = __fadd_rn(alo, __fadd_rn(e, blo));
}

// FP64 value split into (hi, lo) floats
__device__ __forceinline__ float2 df_split(double v)
{
    const float hi = narrow(v);
    return make_float2(hi, narrow(v - widen(hi)));
}

__host__ __device__ inline int low_rows(int lmax, int lc, int m) { return min(lcm_of(lc, m), lmax + 1) - m; }

// one thread per (m, column): the FP64 recurrence from the plan's FP64 seeds
__global__ void k_lowtab_build(int lmax, int npairs, int np_pad, int lc, const long long *__restrict__ rowoff,
                               const double *__restrict__ A, const double *__restrict__ c,
                               const int *__restrict__ ls_tab, const double *__restrict__ s0_tab,
                               const double *__restrict__ s1_tab, const double *__restrict__ xp,
                               float2 *__restrict__ tab)
{
    const int m = blockIdx.y;
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= np_pad) return;
    const int nr = low_rows(lmax, lc, m);
    const long long base = mbase(lmax, m);
    const size_t sidx = (size_t)m * npairs + p;
    const int ls = (p < npairs) ? ls_tab[sidx] : BIG;
    const double x = (p < npairs) ? xp[p] : 0.0;
    float2 *col = tab + (size_t)rowoff[m] * np_pad + p;
    double mu2 = 0.0, mu1 = 0.0;  // mu_{l-2}, mu_{l-1}
    for (int i = 0; i < nr; ++i) {
        const int l = m + i;
        double mu = 0.0;
        if (l == ls) mu = s0_tab[sidx];
        else if (l == ls + 1) mu = s1_tab[sidx];
        else if (l > ls + 1) mu = A[base + i] * x * mu1 - mu2;
        mu2 = mu1;
        mu1 = mu;
        col[(size_t)i * np_pad] = df_split(c[base + i] * mu);
    }
}

// synthesis: G_m(theta_p) = sum over the block's l <= L of a_lm lambda_lm, as even and
// odd partial sums (north = E + O, south = E - O), rounded to FP32 into the block's
// [pair][m][hemisphere] layout (row stride gstride)
__global__ void __launch_bounds__(LEG_THREADS) k_lowsyn_df(int lmax, int L, int npairs, int np_pad, int lc,
                                                           const long long *__restrict__ rowoff,
                                                           const float2 *__restrict__ tab,
                                                           const double2 *__restrict__ alm, float2 *__restrict__ G,
                                                           int gstride)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float4 *sa = reinterpret_cast<float4 *>(smem_raw);  // a_lm as (re hi, re lo, im hi, im lo)
    const int m = blockIdx.y;
    const int nr = min(low_rows(lmax, lc, m), L - m + 1);
    const long long base = mbase(lmax, m);
    for (int i = threadIdx.x; i < nr + 1; i += blockDim.x) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i < nr) {
            const double2 a = alm[base + i];
            const float2 re = df_split(a.x), im = df_split(a.y);
            v = make_float4(re.x, re.y, im.x, im.y);
        }
        sa[i] = v;
    }
    __syncthreads();
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < npairs; p += gridDim.x * blockDim.x) {
        const float2 *col = tab + (size_t)rowoff[m] * np_pad + p;
        float erh = 0.f, erl = 0.f, eih = 0.f, eil = 0.f, orh = 0.f, orl = 0.f, oih = 0.f, oil = 0.f;
        for (int i = 0; i < nr; i += 2) {  // sa[nr] is zero, so an odd nr needs no tail
            const float2 t0 = col[(size_t)i * np_pad];
            const float2 t1 = (i + 1 < nr) ? col[(size_t)(i + 1) * np_pad] : make_float2(0.f, 0.f);
            const float4 a0 = sa[i], a1 = sa[i + 1];
            df_fma(erh, erl, t0.x, t0.y, a0.x, a0.y);
            df_fma(eih, eil, t0.x, t0.y, a0.z, a0.w);
            df_fma(orh, orl, t1.x, t1.y, a1.x, a1.y);
            df_fma(oih, oil, t1.x, t1.y, a1.z, a1.w);
        }
        float nrh = erh, nrl = erl, nih = eih, nil = eil;  // E + O
        df_add(nrh, nrl, orh, orl);
        df_add(nih, nil, oih, oil);
        float srh = erh, srl = erl, sih = eih, sil = eil;  // E - O
        df_add(srh, srl, -orh, -orl);
        df_add(sih, sil, -oih, -oil);
        float2 *g = G + ((size_t)p * gstride + m) * 2;
        g[0] = make_float2(nrh + nrl, nih + nil);
        g[1] = make_float2(srh + srl, sih + sil);
    }
}

// analysis: b_lm = sum_p lambda_lm(x_p) (F_N +- F_S)(p) for the block's l <= L (sign
// + for even l - m).  CTA = (rows of one parity of one m, LOWANA_ROWS at most): it
// stages F_N +- F_S exactly as double-float for every pair in shared memory, each
// warp then takes LOWANA_RW rows at a time, lanes over pairs, and reduces across
// the warp.
constexpr int LOWANA_ROWS = 32, LOWANA_RW = 4;

__global__ void __launch_bounds__(LEG_THREADS) k_lowana_df(int lmax, int L, int npairs, int np_pad, int lc,
                                                           const long long *__restrict__ rowoff,
                                                           const float2 *__restrict__ tab,
                                                           const float2 *__restrict__ F, double2 *__restrict__ out)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float4 *sf = reinterpret_cast<float4 *>(smem_raw);  // F_N +- F_S as (re hi, re lo, im hi, im lo)
    const int m = blockIdx.z, parity = blockIdx.y;
    const int nr = min(low_rows(lmax, lc, m), L - m + 1);
    const int npar = (nr - parity + 1) / 2;  // rows i = parity + 2 k, k < npar
    const int k0 = blockIdx.x * LOWANA_ROWS;
    if (k0 >= npar) return;
    const int k1 = min(npar, k0 + LOWANA_ROWS);
    const size_t pstride = (size_t)(lmax + 1) * 2;
    const float sg = parity ? -1.f : 1.f;
#pragma unroll 4
    for (int p = threadIdx.x; p < np_pad; p += blockDim.x) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (p < npairs) {
            const float2 *f = F + (size_t)p * pstride + 2 * (size_t)m;
            const float2 fn = f[0], fs = f[1];
            float rh, rl, ih, il;
            two_sum(fn.x, sg * fs.x, rh, rl);
            two_sum(fn.y, sg * fs.y, ih, il);
            v = make_float4(rh, rl, ih, il);
        }
        sf[p] = v;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const long long base = mbase(lmax, m);
    const float2 *rows = tab + (size_t)rowoff[m] * np_pad;
    // LOWANA_RW rows of this parity per warp and pass: one shared F value feeds all of
    // them, and the unrolled pair loop keeps several table loads in flight per lane
    for (int k = k0 + LOWANA_RW * warp; k < k1; k += LOWANA_RW * nwarps) {
        const float2 *r[LOWANA_RW];
        float acc[LOWANA_RW][4];
#pragma unroll
        for (int q = 0; q < LOWANA_RW; ++q) {
            const int kq = min(k + q, k1 - 1);  // rows past k1 repeat the last one, unwritten
            r[q] = rows + (size_t)(parity + 2 * kq) * np_pad;
            acc[q][0] = acc[q][1] = acc[q][2] = acc[q][3] = 0.f;
        }
#pragma unroll 4
        for (int p = lane; p < np_pad; p += 32) {
            const float4 f = sf[p];
#pragma unroll
            for (int q = 0; q < LOWANA_RW; ++q) {
                const float2 t = r[q][p];
                df_fma(acc[q][0], acc[q][1], t.x, t.y, f.x, f.y);
                df_fma(acc[q][2], acc[q][3], t.x, t.y, f.z, f.w);
            }
        }
#pragma unroll
        for (int q = 0; q < LOWANA_RW; ++q) {
#pragma unroll
            for (int o = 16; o >= 1; o >>= 1) {
                const float a = __shfl_xor_sync(0xffffffffu, acc[q][0], o), b = __shfl_xor_sync(0xffffffffu, acc[q][1], o);
                const float c = __shfl_xor_sync(0xffffffffu, acc[q][2], o), d = __shfl_xor_sync(0xffffffffu, acc[q][3], o);
                df_add(acc[q][0], acc[q][1], a, b);
                df_add(acc[q][2], acc[q][3], c, d);
            }
            if (lane == 0 && k + q < k1)
                out[base + parity + 2 * (k + q)] =
                    make_double2((double)acc[q][0] + (double)acc[q][1], (double)acc[q][2] + (double)acc[q][3]);
        }
    }
}

// ---------------------------------------------------------------------------
// Double-float transforms for the FP64 correction sweeps of mixed plans.  The
// sweeps' FP64 plan ran these transforms at the FP64 rate (1/64 of FP32 on
// GB300): three FP64 synthesis/analysis pairs per solve cost about a tenth of
// a 1000-iteration benchmark solve.  Here the recurrence, the seeds, x, A and
// c a_lm are (hi, lo) float pairs and every product and sum is an error-free
// FP32 transformation (Dekker's product via FMA, Knuth's two-sum): about 48
// significant bits, against the 24 of the mixed kernels that the sweeps
// correct.  Near the poles the plain recurrence loses ~log2(1/sin theta) bits
// in any precision (12 at nside 2048), so the sweeps stay ~10 digits accurate.
// ---------------------------------------------------------------------------
// Cross-lane sum of one chunk (CH = 8) through shared memory: lane w stores its
// (AR.x, AR.y, AI.x, AI.y) for each row i of the chunk; lane (i, q) = (lane / 4,
// lane % 4) then adds the eight stores of lanes 8q..8q+7 for row i, and two shuffles
// combine the four quarters.  Per chunk that is 8 stores, 8 loads, 16 packed adds
// and 4 shuffles per lane against 16 adds, 18 shuffles, 18 adds and 28 selects for
// the shuffle reduce-scatter.  Slots are XOR-swizzled so that both the stores (8
// lanes of one q) and the loads (8 lanes over two rows and four q) of each
// 128-byte phase hit distinct bank groups.
__device__ __forceinline__ int stage_slot(int i, int w)
{
    const int q = w >> 3, j = w & 7;
    return 32 * i + 8 * q + (j ^ (q + 4 * (i & 1)));
}

// (ph, pl) ~ (ah + al)(bh + bl), unnormalised (|pl| ~ 2^-23 |ph|)
__device__ __forceinline__ void df_mul(float ah, float al, float bh, float bl, float &ph, float &pl)
{
    ph = __fmul_rn(ah, bh);
    float e = __fmaf_rn(ah, bh, -ph);
    e = __fmaf_rn(ah, bl, e);
    pl = __fmaf_rn(al, bh, e);
}

// (sh, sl) = (ah + al) - (bh + bl), normalised
__device__ __forceinline__ void df_sub(float ah, float al, float bh, float bl, float &sh, float &sl)
{
    float s, e;
    two_sum(ah, -bh, s, e);
    e = __fadd_rn(e, __fsub_rn(al, bl));
    sh = __fadd_rn(s, e);
    sl = __fsub_rn(e, __fsub_rn(sh, s));
}

// (E_k, O_k) to k + 1 in double-float, odd values carried as x mu as in the FP64 kernels
// (A = (A_{2k+2} hi, lo, A_{2k+3} hi, lo), X = x^2): 17 operations per l, 19 with x in each step
__device__ __forceinline__ void df_advance(float4 A, float2 X, float2 &E, float2 &O)
{
    float uh, ul, ch, cl;
    df_mul(A.x, A.y, O.x, O.y, uh, ul);
    df_sub(uh, ul, E.x, E.y, E.x, E.y);
    df_mul(A.z, A.w, X.x, X.y, ch, cl);
    df_mul(ch, cl, E.x, E.y, uh, ul);
    df_sub(uh, ul, O.x, O.y, O.x, O.y);
}

__device__ __forceinline__ double df_val(float h, float l) { return widen(h) + widen(l); }

// synthesis: CTA per (m, block of pairs, the equator first), thread per pair.  nside 512, lmax 1024
// 0.927 -> 0.697 ms: a CTA that took four blocks of an m in turn left all CTAs resident at once and
// the SMs unevenly loaded; the two-step form and conversions on the bits are the rest.
__global__ void __launch_bounds__(LEG_THREADS) k_legsyn_df(int lmax, int L, int npairs,
                                                           const double2 *__restrict__ alm, const double *__restrict__ A,
                                                           const double *__restrict__ c64,
                                                           const int *__restrict__ ls_tab,
                                                           const double *__restrict__ s0_tab,
                                                           const double *__restrict__ s1_tab,
                                                           const double4 *__restrict__ xw, double2 *__restrict__ G)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int m = blockIdx.y;
    const int nl = L - m + 1, nk = (nl + 1) >> 1;
    const long long base = mbase(lmax, m);
    float4 *sac = reinterpret_cast<float4 *>(smem_raw);  // c a_lm as (re hi, re lo, im hi, im lo)
    float4 *sA = sac + 2 * nk;                           // per k: A_{2k+2} and A_{2k+3} as (hi, lo)
    for (int i = threadIdx.x; i < 2 * nk; i += blockDim.x) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i < nl) {
            const double2 q = cscale(alm[base + i], c64[base + i]);
            const float2 re = df_split(q.x), im = df_split(q.y);
            v = make_float4(re.x, re.y, im.x, im.y);
        }
        sac[i] = v;
        reinterpret_cast<float2 *>(sA)[i] = i + 2 < nl ? df_split(A[base + i + 2]) : make_float2(0.f, 0.f);
    }
    __syncthreads();
    const int p = (gridDim.x - 1 - blockIdx.x) * LEG_THREADS + threadIdx.x;
    if (p >= npairs) return;
    const size_t sidx = (size_t)m * npairs + p;
    const int ls = ls_tab[sidx];
    float erh = 0.f, erl = 0.f, eih = 0.f, eil = 0.f, orh = 0.f, orl = 0.f, oih = 0.f, oil = 0.f;
    const double4 x = xw[p];
    if (ls <= L) {
        const float2 X = df_split(x.x);
        float2 E = df_split(s0_tab[sidx]), O = df_split(x.z * s1_tab[sidx]);
        for (int k = (ls - m) >> 1; k < nk; ++k) {
            const float4 a0 = sac[2 * k], a1 = sac[2 * k + 1];
            df_fma(erh, erl, a0.x, a0.y, E.x, E.y);
            df_fma(eih, eil, a0.z, a0.w, E.x, E.y);
            df_fma(orh, orl, a1.x, a1.y, O.x, O.y);
            df_fma(oih, oil, a1.z, a1.w, O.x, O.y);
            df_advance(sA[k], X, E, O);
        }
    }
    const double er = df_val(erh, erl), ei = df_val(eih, eil);
    const double orr = x.w * df_val(orh, orl), oi = x.w * df_val(oih, oil);
    double2 *g = G + ((size_t)p * (lmax + 1) + m) * 2;
    g[0] = make_double2(er + orr, ei + oi);
    g[1] = make_double2(er - orr, ei - oi);
}

// analysis: one warp per (group of 32 x DFP ring pairs, m); chunks of 8 values of l are summed
// over the lane's pairs in double-float, across the warp through a swizzled shared stage (with
// (hi, lo) of the real and imaginary parts per slot and double-float additions), and times c_l
// added in FP64 to acc (zero before).  nside 512, lmax 1024 0.888 -> 0.818 ms (a CTA per m before:
// warps without a group waited at the barrier before the epilogue).  Bound by FP32 issue, four
// warps per scheduler.  The loop over k stays rolled: unrolled four times with a second copy for
// the starting steps it took 1.03 ms (instruction fetch).  Twenty warps per SM at 96 registers:
// 0.91 ms; two pairs per lane: 0.98.
constexpr int DFP = 4;

__global__ void __launch_bounds__(32, 16) k_legana_df(int lmax, int L, int npairs, const double2 *__restrict__ F,
                                                      const double *__restrict__ A, const int *__restrict__ ls_tab,
                                                      const double *__restrict__ s0_tab,
                                                      const double *__restrict__ s1_tab,
                                                      const double4 *__restrict__ xw, const double *__restrict__ c64,
                                                      double2 *__restrict__ acc)
{
    constexpr int CH = 8;
    __shared__ float4 sA[F64_BLK / 2];  // per k: A_{2k+2} and A_{2k+3} as (hi, lo)
    __shared__ float4 wst[CH * 32];     // 8 rows x 32 lanes of (re hi, lo, im hi, lo)
    const int m = blockIdx.y, lane = threadIdx.x;
    const int nl = L - m + 1;
    const long long base = mbase(lmax, m);
    const int p0 = (gridDim.x - 1 - blockIdx.x) * 32 * DFP + lane * DFP;  // the equator (most work) first
    int k0[DFP], kmin = BIG, kmaxs = -1;
    float2 s0[DFP], s1[DFP], X[DFP], E[DFP], O[DFP], fer[DFP], fei[DFP], forr[DFP], foi[DFP];
#pragma unroll
    for (int i = 0; i < DFP; ++i) {
        const int p = p0 + i;
        k0[i] = BIG;
        s0[i] = s1[i] = X[i] = E[i] = O[i] = make_float2(0.f, 0.f);
        fer[i] = fei[i] = forr[i] = foi[i] = make_float2(0.f, 0.f);
        if (p < npairs) {
            const size_t sidx = (size_t)m * npairs + p;
            const int ls = ls_tab[sidx];
            if (ls <= L) {
                const double4 x = xw[p];
                k0[i] = (ls - m) >> 1;
                s0[i] = df_split(s0_tab[sidx]);
                s1[i] = df_split(x.z * s1_tab[sidx]);
                X[i] = df_split(x.x);
                const double2 *f = F + ((size_t)p * (lmax + 1) + m) * 2;
                const double2 fn = f[0], fs = f[1];
                fer[i] = df_split(fn.x + fs.x);
                fei[i] = df_split(fn.y + fs.y);
                forr[i] = df_split((fn.x - fs.x) * x.w);
                foi[i] = df_split((fn.y - fs.y) * x.w);
                kmin = min(kmin, k0[i]);
                kmaxs = max(kmaxs, k0[i]);
            }
        }
    }
    kmin = __reduce_min_sync(0xffffffffu, kmin);
    kmaxs = __reduce_max_sync(0xffffffffu, kmaxs);
    if (kmin == BIG) return;
    const int nk = (nl + 1) >> 1;
    int k = kmin & ~(CH / 2 - 1);
    auto fetch = [&](int kb) { return 2 * kb + lane + 2 < nl ? A[base + 2 * kb + lane + 2] : 0.0; };
    double nA = fetch(k & ~(F64_BLK / 2 - 1));
    while (k < nk) {
        if ((k & (F64_BLK / 2 - 1)) == 0 || k == (kmin & ~(CH / 2 - 1))) {
            __syncwarp();
            reinterpret_cast<float2 *>(sA)[lane] = df_split(nA);
            __syncwarp();
            nA = fetch((k & ~(F64_BLK / 2 - 1)) + F64_BLK / 2);
        }
#pragma unroll 1
        for (int j = 0; j < CH / 2; ++j) {
            if (k + j <= kmaxs) {
#pragma unroll
                for (int i = 0; i < DFP; ++i)
                    if (k + j == k0[i]) {
                        E[i] = s0[i];
                        O[i] = s1[i];
                    }
            }
            const float4 a = sA[(k & (F64_BLK / 2 - 1)) + j];
            float r0h = 0.f, r0l = 0.f, i0h = 0.f, i0l = 0.f, r1h = 0.f, r1l = 0.f, i1h = 0.f, i1l = 0.f;
#pragma unroll
            for (int i = 0; i < DFP; ++i) {
                df_fma(r0h, r0l, fer[i].x, fer[i].y, E[i].x, E[i].y);
                df_fma(i0h, i0l, fei[i].x, fei[i].y, E[i].x, E[i].y);
                df_fma(r1h, r1l, forr[i].x, forr[i].y, O[i].x, O[i].y);
                df_fma(i1h, i1l, foi[i].x, foi[i].y, O[i].x, O[i].y);
                df_advance(a, X[i], E[i], O[i]);
            }
            wst[stage_slot(2 * j, lane)] = make_float4(r0h, r0l, i0h, i0l);
            wst[stage_slot(2 * j + 1, lane)] = make_float4(r1h, r1l, i1h, i1l);
        }
        __syncwarp();
        const int i = lane >> 2, q = lane & 3;
        const float4 *row = wst + 32 * i + 8 * q;
        const int c = q + 4 * (i & 1);
        float4 v = row[c];
        float rh = v.x, rl = v.y, ih = v.z, il = v.w;
#pragma unroll
        for (int j = 1; j < 8; ++j) {
            v = row[j ^ c];
            df_add(rh, rl, v.x, v.y);
            df_add(ih, il, v.z, v.w);
        }
#pragma unroll
        for (int o = 1; o <= 2; o <<= 1) {
            const float a = __shfl_xor_sync(0xffffffffu, rh, o), b = __shfl_xor_sync(0xffffffffu, rl, o);
            const float cc = __shfl_xor_sync(0xffffffffu, ih, o), d = __shfl_xor_sync(0xffffffffu, il, o);
            df_add(rh, rl, a, b);
            df_add(ih, il, cc, d);
        }
        const int j = 2 * k + i;
        if (q < 2 && j < nl) atomicAdd(q ? &acc[base + j].y : &acc[base + j].x, c64[base + j] * (q ? df_val(ih, il) : df_val(rh, rl)));
        __syncwarp();
        k += CH / 2;
    }
}

// ---------------------------------------------------------------------------
// Mixed precision: FP32 kernels, NP ring pairs per thread (synthesis) or lane
// (analysis) in NP/2 f32x2 packs.
//
// Both kernels are bound by the FP32 FMA pipe, so what counts is the operations
// per (l, m, ring pair): two for the complex contraction with lambda_lm and as
// few as possible for the recurrence.  The ring pairs fall into two parts with
// a form each, both of which advance two l at once (k = (l - m)/2) with three
// operations:
//
//  belt (rings of 4 nside pixels below x = 2/3): the one-step recurrence
//  mu_l = A_l x mu_{l-1} - mu_{l-2} with the odd values carried as x mu, so that
//  the step from odd to even needs no product A_l x:
//      E_k = mu_{m+2k},  O_k = x mu_{m+2k+1}
//      E_{k+1} = A_{2k+2} O_k - E_k,  O_{k+1} = (A_{2k+3} x^2) E_{k+1} - O_k.
//  The odd sum is divided by x at the end (analysis: its input is).  On the
//  belt x = 2j / (3 nside), so x^2 enters as the integer j^2 (exact in FP32)
//  with 4 / (9 nside^2) in the tabulated A_{2k+3}.
//
//  polar cap (x >= 2/3): the even values alone, by the recurrence in x^2 that
//  follows from eliminating O (Ishioka, J. Met. Soc. Japan 96, 2018, has one
//  recurrence of this kind), rescaled (mu_{m+2k} = e_k E_k) so that the
//  coefficient of E_{k-1} is one, in difference form (Reinsch's modification,
//  with w2 = 1 - x^2 = sin^2 theta, small near the pole):
//      D_{k+1} = D_k + (gamma_k - alpha_k w2) E_k,  E_{k+1} = E_k + D_{k+1}.
//  An odd value is the neighbouring even ones' sum over x,
//      x mu_{m+2k+1} = (mu_{m+2k+2} + mu_{m+2k}) / A_{2k+2},
//  so the odd coefficients fold into coefficients of the E_k once per m (FP64)
//  and the contraction costs the same two operations.  1/x <= 1.5 here.
//
// 3.5 operations per (l, pair) (cap 3.6, see below), against 5 (difference form, x > 0.4)
// and 4 of the one-step forms before.
//
// Accuracy.  A rounding of a ring's variable (x, w2) moves the ring: a phase error that
// grows with l, the same in both directions.  The round trip of a smooth signal keeps of it
// what does not average out over the rings, so the variable has to be better than one FP32
// rounding: the belt's is exact; the cap's rounding error dw is made up for in every fourth
// step (k = 3 mod 4) by D += -4 (4 dw) E, with the limit 4 of alpha (a quarter operation per k).
// FP32 emulation against extended precision, nside 1024, one m, relative error of G and of
// the analysis of a smooth exact G: belt 1.0 to 2.9e-6 and 6 to 10e-7 (one-step forms
// 1.2e-5 and 14 to 33e-7); cap 0.8 to 3.1e-6 and 7 to 16e-7 (4 to 8e-6 and 14 to 25e-7; without
// the correction 4 to 9e-6 and 26 to 50e-7).
// ---------------------------------------------------------------------------
__device__ __forceinline__ float2 dup(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float get(const float2 &v, int k) { return k ? v.y : v.x; }
__device__ __forceinline__ void put(float2 &v, int k, float a)
{
    if (k) v.y = a;
    else v.x = a;
}

struct MxTables {
    int lmax, L, npairs, ncap, lc;
    const int *k0;            // per (m, pair): first k, a multiple of four
    const float2 *seed;       // per (m, pair): state of the part's form at k0
    const float4 *xw;         // per pair: belt (j^2, 0, 1/x), cap (w2, -16 times its rounding error, 1/x); 1/x = 0 for x = 0
    const float2 *tb, *tp;    // per (m, k): (A_{2k+2}, A_{2k+3} 4 / (9 nside^2)); (-alpha_{k+1}, gamma_{k+1})
    const double *c64;        // per a_lm: lambda = c mu
    const double4 *kd;        // per (m, k): (c_2k e_k, c_{2k+1} e_k / A_{2k+2}, c_{2k-1} e_k / A_{2k}, 1 / e_k)
};

// the pairs of one thread: first k and starting state (needed until the last of the warp's
// pairs has started), ring variable and the cap's correction of its rounding
template <int NP> struct MxPairs {
    int k0[NP];
    float2 sd[NP];
    float2 X[NP / 2], C[NP / 2];
    int kmin, kmaxs;
};

template <int NP>
__device__ __forceinline__ void mx_load_pairs(MxPairs<NP> &P, const MxTables &t, int m, int nk, int p0, int pend)
{
    P.kmin = BIG;
    P.kmaxs = -1;
#pragma unroll
    for (int i = 0; i < NP; ++i) {
        const int p = p0 + i;
        int k0 = BIG;
        float2 sd = make_float2(0.f, 0.f);
        float4 X = make_float4(0.f, 0.f, 0.f, 0.f);
        if (p < pend) {
            const size_t idx = (size_t)m * t.npairs + p;
            k0 = t.k0[idx];
            if (k0 < nk) sd = t.seed[idx];
            else k0 = BIG;
            X = t.xw[p];
        }
        P.k0[i] = k0;
        P.sd[i] = sd;
        put(P.X[i >> 1], i & 1, X.x);
        put(P.C[i >> 1], i & 1, X.y);
        P.kmin = min(P.kmin, k0);
        if (k0 != BIG) P.kmaxs = max(P.kmaxs, k0);
    }
}

// advance from k to k + 1 with the table entry of k (CAP: O holds D_{k+1}); FIX: k = 3 mod 4.
// (The two copies of a scalar operand and the signs cost nothing: with every value stored twice
// in shared memory and the signs moved into the tables the synthesis ran 12 % longer.)
template <bool CAP, bool FIX, int NPK>
__device__ __forceinline__ void mx_advance(float2 t, const float2 (&X)[NPK], const float2 (&C)[NPK], float2 (&E)[NPK],
                                           float2 (&O)[NPK])
{
#pragma unroll
    for (int i = 0; i < NPK; ++i) {
        if (CAP) {
            E[i] = __fadd2_rn(E[i], O[i]);
            O[i] = __ffma2_rn(__ffma2_rn(dup(t.x), X[i], dup(t.y)), E[i], O[i]);
            if (FIX) O[i] = __ffma2_rn(C[i], E[i], O[i]);
        } else {
            E[i] = __ffma2_rn(dup(t.x), O[i], neg2(E[i]));
            O[i] = __ffma2_rn(__fmul2_rn(dup(t.y), X[i]), E[i], neg2(O[i]));
        }
    }
}

// Measured (nside 1024, one map): 0.608 ms with the one-step forms, 0.442 ms with these, the FMA
// pipe 71 % busy; mean over the syntheses of an nside 2048 solve 2.93 -> 2.11 ms.
// Synthesis of one (m, part): blockDim.x threads, NP pairs each, per pass.  Shared staging per
// k: st[k] the recurrence entry, sac[k] = coefficients of E (re, im) and of O or folded odd
// (re, im).  Control flow is warp-uniform: one first k and one seeding range per warp (lanes
// not yet started add zeros).
template <int NP, bool CAP>
__device__ __forceinline__ void mx_synthesis(const MxTables &t, int m, const double2 *__restrict__ alm,
                                             float2 *__restrict__ G, float4 *sac, float2 *st)
{
    constexpr int NPK = NP / 2;
    const int nl = t.L - m + 1, nk = (nl >> 1) + 1;  // k with 2k <= L - m + 1
    const long long base = mbase(t.lmax, m), kb = kbase(t.lmax, m);
    const int i_lo = m < t.lc ? lcm_of(t.lc, m) - m : 0;  // coefficients below the FP64 block's end stay out
    for (int k = threadIdx.x; k < nk + 3; k += blockDim.x) {  // steps run in fours: zeros past the end
        const int i0 = 2 * k, i1 = 2 * k + 1;
        double2 e = make_double2(0.0, 0.0), o = e;
        if (k >= nk) {
        } else if (CAP) {
            const double4 d = t.kd[kb + k];
            if (i0 >= i_lo && i0 < nl) e = cscale(alm[base + i0], d.x);
            if (i1 >= i_lo && i1 < nl) o = cscale(alm[base + i1], d.y);
            if (k > 0 && i0 - 1 >= i_lo) o = cadd(o, cscale(alm[base + i0 - 1], d.z));  // i0 - 1 < nl: k < nk
        } else {
            if (i0 >= i_lo && i0 < nl) e = cscale(alm[base + i0], t.c64[base + i0]);
            if (i1 >= i_lo && i1 < nl) o = cscale(alm[base + i1], t.c64[base + i1]);
        }
        sac[k] = make_float4((float)e.x, (float)e.y, (float)o.x, (float)o.y);
        st[k] = k < nk ? (CAP ? t.tp : t.tb)[kb + k] : make_float2(0.f, 0.f);
    }
    __syncthreads();
    const int pbeg = CAP ? 0 : t.ncap, pend = CAP ? t.ncap : t.npairs;
    const size_t pstride = (size_t)(t.lmax + 1) * 2;
    for (int w0 = (blockIdx.x * blockDim.x + (threadIdx.x & ~31)) * NP; pbeg + w0 < pend; w0 += gridDim.x * blockDim.x * NP) {
        const int p0 = pbeg + w0 + (threadIdx.x & 31) * NP;
        MxPairs<NP> P;
        mx_load_pairs<NP>(P, t, m, nk, p0, pend);
        float2 ER[NPK], EI[NPK], OR[NPK], OI[NPK], E[NPK], O[NPK];
#pragma unroll
        for (int i = 0; i < NPK; ++i) ER[i] = EI[i] = OR[i] = OI[i] = E[i] = O[i] = dup(0.f);
        int k = __reduce_min_sync(0xffffffffu, P.kmin);
        const int kmaxs = __reduce_max_sync(0xffffffffu, P.kmaxs);
        auto step = [&](int kk, auto fix) {
            const float4 ac = sac[kk];
            const float2 tt = st[kk];
#pragma unroll
            for (int i = 0; i < NPK; ++i) {
                ER[i] = __ffma2_rn(dup(ac.x), E[i], ER[i]);
                EI[i] = __ffma2_rn(dup(ac.y), E[i], EI[i]);
                OR[i] = __ffma2_rn(dup(ac.z), CAP ? E[i] : O[i], OR[i]);
                OI[i] = __ffma2_rn(dup(ac.w), CAP ? E[i] : O[i], OI[i]);
            }
            mx_advance<CAP, decltype(fix)::value, NPK>(tt, P.X, P.C, E, O);
        };
        auto four = [&]() {
            step(k, std::false_type{});
            step(k + 1, std::false_type{});
            step(k + 2, std::false_type{});
            step(k + 3, std::true_type{});
        };
        for (; k < nk && k <= kmaxs; k += 4) {
#pragma unroll
            for (int i = 0; i < NP; ++i)
                if (k == P.k0[i]) {
                    put(E[i >> 1], i & 1, P.sd[i].x);
                    put(O[i >> 1], i & 1, P.sd[i].y);
                }
            four();
        }
        for (; k < nk; k += 4) four();
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            const int p = p0 + i;
            if (p >= pend) break;
            const int pk = i >> 1, h = i & 1;
            const float ix = t.xw[p].z;
            const float er = get(ER[pk], h), ei = get(EI[pk], h), orr = get(OR[pk], h) * ix, oi = get(OI[pk], h) * ix;
            *reinterpret_cast<float4 *>(G + (size_t)p * pstride + 2 * (size_t)m) =
                make_float4(er + orr, ei + oi, er - orr, ei - oi);
        }
    }
}

// grid: (CTAs of a part, m, part), the belt's (more work per pair) first
template <int NP>
__global__ void __launch_bounds__(LEG_THREADS) k_legsyn_mx(const MxTables t, const double2 *__restrict__ alm,
                                                           float2 *__restrict__ G)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int m = blockIdx.y, nk = ((t.L - m + 1) >> 1) + 1;
    float4 *sac = reinterpret_cast<float4 *>(smem_raw);
    float2 *st = reinterpret_cast<float2 *>(sac + nk + 3);
    if (blockIdx.z) mx_synthesis<NP, true>(t, m, alm, G, sac, st);
    else mx_synthesis<NP, false>(t, m, alm, G, sac, st);
}

constexpr int MX_TBLK = 64;  // table entries a warp stages at a time

// shared memory of an analysis warp: two stages of the cross-lane sum (per lane and k of a block
// E re, im, O re, im), table entries, and the pairs' first k (two to a word) and starting
// states, read while pairs start
template <int NP> struct __align__(16) MxAnaShared {
    float4 stage[2][4 * 32];
    float2 tab[MX_TBLK];
    unsigned k0[NP / 2][32];
    float2 sd[NP][32];
};

// Analysis of one (m, part, group of 32 NP pairs) by one warp: blocks of four k (eight l) are
// summed over the packs in registers, across the warp through a shared stage, and added to
// sum[4 k + (0, 1)] (E re, im), sum[4 k + (2, 3)] (O, or the folded odd values' E / x) in global
// memory.  The stage of one block is read while the next block's FMAs run (two stages), one
// row per step, so that its latency is not waited for.
//
// What bounds it: the FMA pipe (about 270 cycles per block and warp) and, four warps to a
// shared-memory port, the stage: with both halves of each packed sum staged (64 wavefronts per
// block and 16 more additions when read) the cross-lane sum took 38 % of the time, the
// port being busy as long as the pipe.  Adding the halves first leaves 32.
template <int NP, bool CAP>
__device__ __forceinline__ void mx_analysis(const MxTables &t, int m, int grp, const float2 *__restrict__ F,
                                            float *sum, MxAnaShared<NP> &S, int nk)
{
    constexpr int NPK = NP / 2;
    const int lane = threadIdx.x;
    const int pend = CAP ? t.ncap : t.npairs;
    const int p0 = (CAP ? 0 : t.ncap) + grp * 32 * NP + lane * NP;
    const size_t pstride = (size_t)(t.lmax + 1) * 2;
    const float2 *tab = (CAP ? t.tp : t.tb) + kbase(t.lmax, m);
    float2 X[NPK], C[NPK], FEr[NPK], FEi[NPK], FOr[NPK], FOi[NPK], E[NPK], O[NPK];
    int kmin, kmaxs, knext;  // first and last starting k of the warp; next one of this lane
    {
        MxPairs<NP> P;
        mx_load_pairs<NP>(P, t, m, nk, p0, pend);
        knext = P.kmin;
        kmin = __reduce_min_sync(0xffffffffu, P.kmin);
        kmaxs = __reduce_max_sync(0xffffffffu, P.kmaxs);
        if (kmin >= nk) return;
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
            float ix = 0.f;
            if (P.k0[i] != BIG) {
                f = *reinterpret_cast<const float4 *>(F + (size_t)(p0 + i) * pstride + 2 * (size_t)m);
                ix = t.xw[p0 + i].z;
            }
            put(FEr[i >> 1], i & 1, f.x + f.z);
            put(FEi[i >> 1], i & 1, f.y + f.w);
            put(FOr[i >> 1], i & 1, (f.x - f.z) * ix);
            put(FOi[i >> 1], i & 1, (f.y - f.w) * ix);
            S.sd[i][lane] = P.sd[i];
        }
#pragma unroll
        for (int i = 0; i < NPK; ++i) {
            X[i] = P.X[i];
            C[i] = P.C[i];
            S.k0[i][lane] = (unsigned)(P.k0[2 * i] & 0xffff) | (unsigned)P.k0[2 * i + 1] << 16;  // BIG: 0xffff, no k
            E[i] = O[i] = dup(0.f);
        }
    }
    auto load_table = [&](int k0) {
        __syncwarp();
#pragma unroll
        for (int i = 0; i < MX_TBLK / 32; ++i) {
            const int k = k0 + i * 32 + lane;
            S.tab[i * 32 + lane] = k < nk ? tab[k] : make_float2(0.f, 0.f);  // blocks run up to three k past the end
        }
        __syncwarp();
    };
    load_table(kmin & ~(MX_TBLK - 1));
    // lane (r, q) = (lane / 8, lane % 8) reads k = r of a block, lanes 4q .. 4q + 3 (in an order that
    // keeps the eight lanes of a phase on distinct banks); three shuffles' exchange then leaves
    // component q & 3 summed over the warp
    const int rr = lane >> 3, rq = lane & 7, rc = rq >> 1, rrow = 32 * rr + 4 * rq;
    float *dst = sum + 4 * rr + (rq & 3);
    auto finish = [&](int kc, float4 v) {
        const bool odd = rq & 2, im = rq & 1;
        float a = odd ? v.z : v.x, b = odd ? v.w : v.y;
        a += __shfl_xor_sync(0xffffffffu, odd ? v.x : v.z, 2);
        b += __shfl_xor_sync(0xffffffffu, odd ? v.y : v.w, 2);
        float c = im ? b : a;
        c += __shfl_xor_sync(0xffffffffu, im ? a : b, 1);
        c += __shfl_xor_sync(0xffffffffu, c, 4);
        if (rq < 4 && kc + rr < nk) atomicAdd(dst + 4 * kc, c);  // no value used: a native reduction in L2
    };
    int buf = 0, kc = kmin;
    auto block = [&]() {
        if ((kc & (MX_TBLK - 1)) == 0 && kc != kmin) load_table(kc);
        const float2 *tk = S.tab + (kc & (MX_TBLK - 1));
        float4 *stage = S.stage[buf] + lane;
        const float4 *prev = S.stage[buf ^ 1] + rrow;
        float4 v;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float4 w = prev[i ^ rc];
            float2 er = __fmul2_rn(FEr[0], E[0]), ei = __fmul2_rn(FEi[0], E[0]);
            float2 orr = __fmul2_rn(FOr[0], CAP ? E[0] : O[0]), oi = __fmul2_rn(FOi[0], CAP ? E[0] : O[0]);
#pragma unroll
            for (int q = 1; q < NPK; ++q) {
                er = __ffma2_rn(FEr[q], E[q], er);
                ei = __ffma2_rn(FEi[q], E[q], ei);
                orr = __ffma2_rn(FOr[q], CAP ? E[q] : O[q], orr);
                oi = __ffma2_rn(FOi[q], CAP ? E[q] : O[q], oi);
            }
            stage[32 * i] = make_float4(er.x + er.y, ei.x + ei.y, orr.x + orr.y, oi.x + oi.y);
            if (i == 3) mx_advance<CAP, true, NPK>(tk[i], X, C, E, O);
            else mx_advance<CAP, false, NPK>(tk[i], X, C, E, O);
            v = i ? make_float4(v.x + w.x, v.y + w.y, v.z + w.z, v.w + w.w) : w;
        }
        if (kc != kmin) finish(kc - 4, v);
        __syncwarp();
        buf ^= 1;
        kc += 4;
    };
    // two loops: the starting states' writes into halves of packed registers stay out of the second
    while (kc < nk && kc <= kmaxs) {
        if (knext == kc) {
            knext = BIG;
#pragma unroll
            for (int i = 0; i < NPK; ++i) {
                const unsigned w = S.k0[i][lane];
                const int ka = (int)(w & 0xffff), kb = (int)(w >> 16);
                if (ka == kc) {
                    const float2 s = S.sd[2 * i][lane];
                    E[i].x = s.x;
                    O[i].x = s.y;
                } else if (ka > kc) {
                    knext = min(knext, ka);
                }
                if (kb == kc) {
                    const float2 s = S.sd[2 * i + 1][lane];
                    E[i].y = s.x;
                    O[i].y = s.y;
                } else if (kb > kc) {
                    knext = min(knext, kb);
                }
            }
        }
        __syncwarp();
        block();
    }
    while (kc < nk) block();
    const float4 *prev = S.stage[buf ^ 1] + rrow;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float4 w = prev[i ^ rc];
        v.x += w.x;
        v.y += w.y;
        v.z += w.z;
        v.w += w.w;
    }
    finish(kmin + ((nk - 1 - kmin) & ~3), v);
}

// Measured with the epilogue below: nside 768 adjoint 0.443 -> 0.262 + 0.031 ms, mean over the
// analyses of a solve at nside 2048 3.90 -> 2.72 + 0.30 ms, at nside 512 0.138 -> 0.068 + 0.031 ms,
// at nside 128 0.027 -> 0.010 + 0.008 ms.
// One warp per CTA and (group of pairs, part, m), grid (belt groups, cap groups; m): no barrier
// joins warps of unequal work.  Before, a CTA summed an m in shared memory: its warps spent a
// third of their time at the barrier before the epilogue (nside 768), and FP32 atomics in
// shared memory are compare-and-swap loops.
template <int NP>
__global__ void __launch_bounds__(32, NP == 8 ? 17 : 16) k_legana_mx(const MxTables t, int ngroups, const float2 *__restrict__ F,
                                                      float4 *__restrict__ psum)
{
    __shared__ MxAnaShared<NP> S;
    const int m = blockIdx.y, nk = ((t.L - m + 1) >> 1) + 1;
    const long long kb = kbase(t.lmax, m), nks = kbase(t.lmax, t.lmax + 1) + 2;  // nks: entries per part
    // groups nearest the equator (most l above the first kept one) first
    const int g = blockIdx.x;
    if (g < ngroups) mx_analysis<NP, false>(t, m, ngroups - 1 - g, F, &psum[kb].x, S, nk);
    else mx_analysis<NP, true>(t, m, 2 * ngroups - 1 - g, F, &psum[nks + kb].x, S, nk);
}

// Eq. (4) epilogue of the mixed analysis, a CTA per m; clears the sums for the next launch.  Run
// by the last warp at its m inside the kernel above it took 14 % of that kernel (one warp's
// chain of loads per m, nside 768).
__global__ void __launch_bounds__(EPI_THREADS) k_ana_epilogue(const MxTables t, int mode, BlendArgs ba,
                                                      const double2 *__restrict__ low,
                                                      const double2 *__restrict__ a_old, double2 *__restrict__ out,
                                                      double *__restrict__ part, float4 *__restrict__ psum)
{
    __shared__ double red[5][EPI_THREADS];
    const int m = blockIdx.x, nk = ((t.L - m + 1) >> 1) + 1;
    const long long base = mbase(t.lmax, m), kb = kbase(t.lmax, m);
    const long long nks = kbase(t.lmax, t.lmax + 1) + 2;
    float4 *sb = psum + kb, *sc = psum + nks + kb;
    // belt: c mu-sums; cap: even l from E_k, odd l from the fold over E_k and E_{k+1}; the FP64
    // block's l take its values
    const int low_lim = (low && m < t.lc) ? lcm_of(t.lc, m) : 0;
    BlendSums v;
    for (int k = threadIdx.x; 2 * k <= t.lmax - m; k += blockDim.x) {
        const int l = m + 2 * k;
        const long long i = base + 2 * k;
        double2 e = make_double2(0.0, 0.0), o = e;
        if (l < low_lim) {
            if (l <= t.L) e = low[i];
            if (l < t.L) o = low[i + 1];
        } else if (l <= t.L) {
            const float4 b = sb[k], c = sc[k];
            const double4 d = t.kd[kb + k];
            const double ce = t.c64[i];
            e = make_double2(ce * widen(b.x) + d.x * widen(c.x), ce * widen(b.y) + d.x * widen(c.y));
            if (l < t.L) {
                const float4 c2 = sc[k + 1];
                const double r = t.kd[kb + k + 1].z, co = t.c64[i + 1];
                o = make_double2(co * widen(b.z) + (d.y * widen(c.z) + r * widen(c2.z)),
                                 co * widen(b.w) + (d.y * widen(c.w) + r * widen(c2.w)));
            }
        }
        blend_one(l, t.L, i, mode, ba, e, a_old, out, v);
        if (l < t.lmax) blend_one(l + 1, t.L, i + 1, mode, ba, o, a_old, out, v);
    }
    if (mode == LEG_BLEND) blend_sums(v, m, ba, part, red);
    __syncthreads();
    for (int k = threadIdx.x; k < nk; k += blockDim.x) sb[k] = sc[k] = make_float4(0.f, 0.f, 0.f, 0.f);
}

// ---------------------------------------------------------------------------
// launches
// ---------------------------------------------------------------------------
size_t syn_mx_smem(int L) { return (size_t)((L + 1) / 2 + 5) * (sizeof(float4) + sizeof(float2)) + 16; }

template <typename TG>
wf_status launch_syn64(wf_plan p, const double2 *alm, int L, int lcut, cx<TG> *G, int gstride, cudaStream_t s)
{
    const HpTables &t = p->tab;
    const int Lgrid = lcut > 0 ? std::min(L, lcut - 1) : L;
    if (Lgrid < 0) return WF_OK;
    k_legsyn<TG><<<dim3((p->npairs + 31) / 32, Lgrid + 1), 32, 0, s>>>(p->lmax, L, p->npairs, lcut, alm, t.A64, t.c64,
                                                                       t.ls, t.s0_64, t.s1_64, t.xw64, G, gstride);
    WF_COUNT_LAUNCH(p);
    WF_CUDA(cudaGetLastError());
    return WF_OK;
}

// ring pairs from which the FP64 analysis takes two per lane; one / two (us): nside 48 29 / 43, 100
// 68 / 77, 128 128 / 124, 192 356 / 315, 256 665 / 592, 512 4515 / 3619
constexpr int ANA64_MIN_PAIRS = 256;

wf_status launch_ana64(wf_plan p, int L, const double2 *F, LegMode mode, const BlendArgs &ba, const double2 *a_old,
                       double2 *out, cudaStream_t s)
{
    const HpTables &t = p->tab;
    const int np = p->npairs >= ANA64_MIN_PAIRS ? 2 : 1;
    const dim3 grid((p->npairs + 32 * np - 1) / (32 * np), L + 1);
    auto kernel = np == 2 ? k_legana<double, 2> : k_legana<double, 1>;
    kernel<<<grid, 32, 0, s>>>(p->lmax, L, p->npairs, 0, F, t.A64, t.ls, t.s0_64, t.s1_64, t.xw64, t.c64, t.acc64);
    WF_COUNT_LAUNCH(p);
    k_ana64_epilogue<<<L + 1, EPI_THREADS, 0, s>>>(p->lmax, L, (int)mode, ba, a_old, out, p->ws.part_harm, t.acc64);
    WF_COUNT_LAUNCH(p);
    WF_CUDA(cudaGetLastError());
    return WF_OK;
}

// FP64 block of the mixed analysis (adjoint, l < lcm(lcut, m))
wf_status launch_ana64_low(wf_plan p, int L, int lcut, const float2 *F, double2 *out, cudaStream_t s)
{
    const HpTables &t = p->tab;
    const int nm = std::min(L, lcut - 1) + 1;
    if (nm <= 0) return WF_OK;
    WF_CUDA(cudaMemsetAsync(out, 0, (size_t)mbase(p->lmax, nm) * sizeof(double2), s));
    k_legana<float, 1><<<dim3((p->npairs + 31) / 32, nm), 32, 0, s>>>(p->lmax, L, p->npairs, lcut, F, t.A64, t.ls, t.s0_64,
                                                                   t.s1_64, t.xw64, t.c64, out);
    WF_COUNT_LAUNCH(p);
    WF_CUDA(cudaGetLastError());
    return WF_OK;
}

// FP64 block from the double-float table: synthesis into the block's FP32 ring
// coefficients, analysis into the FP64 output that the FP32 analysis epilogue adds
wf_status launch_lowsyn_df(wf_plan p, const double2 *alm, int L, cudaStream_t s)
{
    const HpTables &t = p->tab;
    const int lc = t.lc_mx, nm = std::min(L, lc - 1) + 1;
    if (nm <= 0) return WF_OK;
    const int gx = (p->npairs + LEG_THREADS - 1) / LEG_THREADS;
    const size_t sm = (size_t)(std::min(low_rows(p->lmax, lc, 0), L + 1) + 1) * sizeof(float4);
    k_lowsyn_df<<<dim3(gx, nm), LEG_THREADS, sm, s>>>(p->lmax, L, p->npairs, t.np_pad, lc, t.lowrow, t.lowtab, alm,
                                                       p->ws.Glow, t.glow_cap);
    WF_COUNT_LAUNCH(p);
    WF_CUDA(cudaGetLastError());
    return WF_OK;
}

wf_status launch_lowana_df(wf_plan p, int L, const float2 *F, double2 *out, cudaStream_t s)
{
    const HpTables &t = p->tab;
    const int lc = t.lc_mx, nm = std::min(L, lc - 1) + 1;
    if (nm <= 0) return WF_OK;
    const int rows0 = std::min(low_rows(p->lmax, lc, 0), L + 1);
    const int gx = ((rows0 + 1) / 2 + LOWANA_ROWS - 1) / LOWANA_ROWS;
    const size_t sm = (size_t)t.np_pad * sizeof(float4);
    k_lowana_df<<<dim3(gx, 2, nm), LEG_THREADS, sm, s>>>(p->lmax, L, p->npairs, t.np_pad, lc, t.lowrow, t.lowtab, F,
                                                          out);
    WF_COUNT_LAUNCH(p);
    WF_CUDA(cudaGetLastError());
    return WF_OK;
}

// double-float transforms of a sweep sub-plan (FP64 plan, G and F in FP64)
size_t syn_df_smem(int L) { return (size_t)((L + 2) / 2) * 3 * sizeof(float4); }

wf_status launch_syn_df(wf_plan p, const double2 *alm, int L)
{
    const HpTables &t = p->tab;
    const dim3 grid((p->npairs + LEG_THREADS - 1) / LEG_THREADS, L + 1);
    k_legsyn_df<<<grid, LEG_THREADS, syn_df_smem(L), p->stream>>>(p->lmax, L, p->npairs, alm, t.A64, t.c64, t.ls, t.s0_64,
                                                                  t.s1_64, t.xw64, (double2 *)p->ws.G);
    WF_COUNT_LAUNCH(p);
    WF_CUDA(cudaGetLastError());
    return WF_OK;
}

wf_status launch_ana_df(wf_plan p, int L, LegMode mode, const BlendArgs &ba, const double2 *a_old, double2 *out)
{
    const HpTables &t = p->tab;
    const dim3 grid((p->npairs + 32 * DFP - 1) / (32 * DFP), L + 1);
    k_legana_df<<<grid, 32, 0, p->stream>>>(p->lmax, L, p->npairs, (const double2 *)p->ws.F, t.A64, t.ls, t.s0_64,
                                            t.s1_64, t.xw64, t.c64, t.acc64);
    WF_COUNT_LAUNCH(p);
    k_ana64_epilogue<<<L + 1, EPI_THREADS, 0, p->stream>>>(p->lmax, L, (int)mode, ba, a_old, out, p->ws.part_harm, t.acc64);
    WF_COUNT_LAUNCH(p);
    WF_CUDA(cudaGetLastError());
    return WF_OK;
}

// Device bytes of the block's table for l_c on this plan
long long low_table_bytes(int lmax, int npairs, int lc)
{
    const long long np_pad = (npairs + 31) & ~31;
    long long rows = 0;
    for (int m = 0; m < std::min(lc, lmax + 1); ++m) rows += low_rows(lmax, lc, m);
    return rows * np_pad * (long long)sizeof(float2);
}

}  // namespace

long long hp_low_table_bytes(int lmax, int npairs, int lc) { return low_table_bytes(lmax, npairs, lc); }

// ---------------------------------------------------------------------------
// host: recurrence tables and seeds
// ---------------------------------------------------------------------------
wf_status hp_build_legendre_tables(wf_plan p, const std::vector<double> &xpair, const std::vector<double> &stpair)
{
    const int lmax = p->lmax, np = p->npairs;
    const long long nalm = p->nalm;
    const bool f32 = p->prec != WF_PREC_FP64, tc = tc_prec(p->prec);
    const long long nks = kbase(lmax, lmax + 1) + 2;  // entries of the tables per (m, k)
    std::vector<double> A(nalm), c(nalm), Bm2(tc ? nalm : 0), log2c(lmax + 1), Atop(lmax + 1);
    std::vector<double4> kd(f32 ? nks : 0, make_double4(0.0, 0.0, 0.0, 0.0));
    std::vector<float2> tb(f32 ? nks : 0, make_float2(0.f, 0.f)), tp(f32 ? nks : 0, make_float2(0.f, 0.f));
    std::vector<double> Ax(lmax + 8), cx_(lmax + 8), e(lmax / 2 + 8);
    for (int m = 0; m <= lmax; ++m) {
        const long long b = mbase(lmax, m);
        auto coef = [m](int l) { return std::sqrt((4.0 * l * l - 1.0) / ((double)l * l - (double)m * m)); };
        c[b] = 1.0;
        if (m + 1 <= lmax) c[b + 1] = 1.0;
        for (int l = m + 2; l <= lmax; ++l) c[b + (l - m)] = (coef(l) / coef(l - 1)) * c[b + (l - 2 - m)];
        // scale the l - m odd chain so that c_l / c_{l-1} -> 1 at lmax: the
        // multiplier A_l then tends to 2 x-independently, which the
        // difference form needs
        if (lmax - m >= 2) {
            const double r = c[b + (lmax - m)] / c[b + (lmax - 1 - m)];
            const double f = ((lmax - m) & 1) ? 1.0 / r : r;
            for (int l = m + 1; l <= lmax; l += 2) c[b + (l - m)] *= f;
        }
        A[b] = 0.0;
        if (m + 1 <= lmax) A[b + 1] = std::sqrt(2.0 * m + 3.0) * c[b] / c[b + 1];
        for (int l = m + 2; l <= lmax; ++l) A[b + (l - m)] = coef(l) * c[b + (l - 1 - m)] / c[b + (l - m)];
        if (tc)
            for (int l = m; l <= lmax; ++l) Bm2[b + (l - m)] = A[b + (l - m)] - 2.0;
        if (f32) {
            // A and c a few l past lmax (i = l - m), then the tables of the two-step forms
            const int n = lmax - m + 1, K = n / 2 + 1;  // k = 0 .. K - 1: 2k <= lmax - m + 1
            for (int i = 0; i < n; ++i) {
                Ax[i] = A[b + i];
                cx_[i] = c[b + i];
            }
            for (int i = n; i < n + 5; ++i) {
                const int l = m + i;
                if (i == 1) {
                    cx_[i] = 1.0;
                    Ax[i] = std::sqrt(2.0 * m + 3.0);
                } else {
                    cx_[i] = (coef(l) / coef(l - 1)) * cx_[i - 2];
                    Ax[i] = coef(l) * cx_[i - 1] / cx_[i];
                }
            }
            Atop[m] = Ax[n];
            e[0] = e[1] = 1.0;
            for (int k = 1; k <= K; ++k) e[k + 1] = e[k - 1] * (Ax[2 * k + 2] / Ax[2 * k]);
            // one chain rescaled so that alpha - beta tends to 2 at the top, as A does above
            const int kt = std::max(1, (n - 1) / 2);
            const double r = e[kt] / e[kt - 1];
            for (int k = 1; k <= K + 1; k += 2) e[k] *= (kt & 1) ? 1.0 / r : r;
            const long long kb = kbase(lmax, m);
            for (int k = 0; k < K; ++k) {
                const double A2 = Ax[2 * k + 2], g = e[k + 1] / e[k + 2];
                const double al = Ax[2 * k + 4] * Ax[2 * k + 3] * g, be = (Ax[2 * k + 4] / A2 + 1.0) * g;
                tb[kb + k] = make_float2((float)A2, (float)(Ax[2 * k + 3] * (4.0 / 9.0) / ((double)p->nside * p->nside)));
                tp[kb + k] = make_float2(-(float)al, (float)(al - be - 2.0));
                kd[kb + k] = make_double4(2 * k < n ? cx_[2 * k] * e[k] : 0.0, 2 * k + 1 < n ? cx_[2 * k + 1] * e[k] / A2 : 0.0,
                                          k > 0 && 2 * k - 1 < n ? cx_[2 * k - 1] * e[k] / Ax[2 * k] : 0.0, 1.0 / e[k]);
            }
        }
        // log2 of sqrt((2m+1)/(4 pi) (2m)! / (2^m m!)^2)
        log2c[m] = 0.5 * (std::log(2.0 * m + 1.0) - std::log(4.0 * M_PI) + std::lgamma(2.0 * m + 1.0) -
                          2.0 * std::lgamma(m + 1.0) - 2.0 * m * std::log(2.0)) / std::log(2.0);
    }
    std::vector<double> wpair(np);
    for (int i = 0; i < np; ++i) wpair[i] = 1.0 - xpair[i];
    // 1 - x exactly for the polar-cap rings (1 - z = k^2 / (3 nside^2))
    for (int i = 0; i + 1 < p->nside && i < np; ++i)
        wpair[i] = (double)(i + 1) * (i + 1) / (3.0 * p->nside * p->nside);
    double *dst64 = nullptr, *dlog2c = nullptr;
    wf_status st;
    HpTables &t = p->tab;
    if ((st = plan_alloc(p, (void **)&t.c64, nalm * sizeof(double))) != WF_OK) return st;
    if ((st = plan_alloc(p, (void **)&t.A64, nalm * sizeof(double))) != WF_OK) return st;
    if ((st = plan_alloc(p, (void **)&t.x64, np * sizeof(double))) != WF_OK) return st;
    if ((st = plan_alloc(p, (void **)&dst64, np * sizeof(double))) != WF_OK) return st;
    if ((st = plan_alloc(p, (void **)&t.xw64, np * sizeof(double4))) != WF_OK) return st;
    if (!f32) {
        if ((st = plan_alloc(p, (void **)&t.acc64, nalm * sizeof(double2))) != WF_OK) return st;
        WF_CUDA(cudaMemsetAsync(t.acc64, 0, nalm * sizeof(double2), p->stream));
    }
    std::vector<double4> xw64(np);
    for (int i = 0; i < np; ++i) {
        const double x = xpair[i], X = x * x;
        xw64[i] = make_double4(X, 8.0 * std::fma(x, x, -X), x, i + 1 < np ? 1.0 / x : 0.0);  // the equator's odd values vanish
    }
    if ((st = to_device(p, t.xw64, xw64.data(), np * sizeof(double4))) != WF_OK) return st;
    t.st64 = dst64;
    if ((st = plan_alloc(p, (void **)&dlog2c, (lmax + 1) * sizeof(double))) != WF_OK) return st;
    const long long ns = (long long)(lmax + 1) * np;
    if ((st = plan_alloc(p, (void **)&t.ls, ns * sizeof(int))) != WF_OK) return st;
    if ((st = plan_alloc(p, (void **)&t.s0_64, ns * sizeof(double))) != WF_OK) return st;
    if ((st = plan_alloc(p, (void **)&t.s1_64, ns * sizeof(double))) != WF_OK) return st;
    if ((st = to_device(p, t.A64, A.data(), nalm * sizeof(double))) != WF_OK) return st;
    if ((st = to_device(p, t.c64, c.data(), nalm * sizeof(double))) != WF_OK) return st;
    if ((st = to_device(p, t.x64, xpair.data(), np * sizeof(double))) != WF_OK) return st;
    if ((st = to_device(p, dst64, stpair.data(), np * sizeof(double))) != WF_OK) return st;
    if ((st = to_device(p, dlog2c, log2c.data(), (lmax + 1) * sizeof(double))) != WF_OK) return st;
    {
        const int th = 256;
        const long long nb = (ns + th - 1) / th;
        k_seeds<<<(unsigned)nb, th, 0, p->stream>>>(lmax, np, t.x64, dst64, dlog2c, t.A64, t.c64, t.ls, t.s0_64,
                                                     t.s1_64);
        WF_COUNT_LAUNCH(p);
        WF_CUDA(cudaGetLastError());
    }
    if (f32) {
        if ((st = plan_alloc(p, (void **)&t.x32, np * sizeof(float))) != WF_OK) return st;
        if ((st = plan_alloc(p, (void **)&t.w32, np * sizeof(float))) != WF_OK) return st;
        if ((st = plan_alloc(p, (void **)&t.xw, np * sizeof(float4))) != WF_OK) return st;
        if ((st = plan_alloc(p, (void **)&t.tb, nks * sizeof(float2))) != WF_OK) return st;
        if ((st = plan_alloc(p, (void **)&t.tp, nks * sizeof(float2))) != WF_OK) return st;
        if ((st = plan_alloc(p, (void **)&t.kd, nks * sizeof(double4))) != WF_OK) return st;
        if ((st = plan_alloc(p, (void **)&t.Atop, (lmax + 1) * sizeof(double))) != WF_OK) return st;
        if ((st = plan_alloc(p, (void **)&t.psum, 2 * nks * sizeof(float4))) != WF_OK) return st;
        if ((st = plan_alloc(p, (void **)&t.k0_mx, ns * sizeof(int))) != WF_OK) return st;
        if ((st = plan_alloc(p, (void **)&t.seed_mx, ns * sizeof(float2))) != WF_OK) return st;
        std::vector<float> xf(np), wf(np);
        std::vector<float4> xw(np);
        for (int i = 0; i < np; ++i) {
            xf[i] = (float)xpair[i];
            wf[i] = (float)wpair[i];
            const float ix = i + 1 < np ? (float)(1.0 / xpair[i]) : 0.f;  // the equator's odd values vanish
            if (i < p->nside) {
                const double w2 = wpair[i] * (2.0 - wpair[i]);
                const float w = (float)w2;
                xw[i] = make_float4(w, (float)(-16.0 * (w2 - (double)w)), ix, 0.f);
            } else {
                const float j = (float)(np - 1 - i);
                xw[i] = make_float4(j * j, 0.f, ix, 0.f);
            }
        }
        WF_CUDA(cudaMemsetAsync(t.psum, 0, 2 * nks * sizeof(float4), p->stream));
        if ((st = to_device(p, t.x32, xf.data(), np * sizeof(float))) != WF_OK) return st;
        if ((st = to_device(p, t.w32, wf.data(), np * sizeof(float))) != WF_OK) return st;
        if ((st = to_device(p, t.xw, xw.data(), np * sizeof(float4))) != WF_OK) return st;
        if ((st = to_device(p, t.tb, tb.data(), nks * sizeof(float2))) != WF_OK) return st;
        if ((st = to_device(p, t.tp, tp.data(), nks * sizeof(float2))) != WF_OK) return st;
        if ((st = to_device(p, t.kd, kd.data(), nks * sizeof(double4))) != WF_OK) return st;
        if ((st = to_device(p, t.Atop, Atop.data(), (lmax + 1) * sizeof(double))) != WF_OK) return st;
        if (tc) {  // the tensor-core synthesis keeps the one-step forms
            if ((st = plan_alloc(p, (void **)&t.A32, nalm * sizeof(float))) != WF_OK) return st;
            if ((st = plan_alloc(p, (void **)&t.B32, nalm * sizeof(float))) != WF_OK) return st;
            if ((st = plan_alloc(p, (void **)&t.ls_mx, ns * sizeof(int))) != WF_OK) return st;
            if ((st = plan_alloc(p, (void **)&t.s0_mx, ns * sizeof(float))) != WF_OK) return st;
            if ((st = plan_alloc(p, (void **)&t.s1_mx, ns * sizeof(float))) != WF_OK) return st;
            std::vector<float> Af(nalm), Bf(nalm);
            for (long long i = 0; i < nalm; ++i) {
                Af[i] = (float)A[i];
                Bf[i] = (float)Bm2[i];
            }
            if ((st = to_device(p, t.A32, Af.data(), nalm * sizeof(float))) != WF_OK) return st;
            if ((st = to_device(p, t.B32, Bf.data(), nalm * sizeof(float))) != WF_OK) return st;
        }
        t.lc_mx = -1;
        if ((st = hp_set_low_block(p, 0)) != WF_OK) return st;
    }
    // raise the shared-memory limits of every Legendre kernel this plan can launch to
    // their lmax sizes now, so that no launch (e.g. inside a graph capture) needs to
    if (f32) {
        const void *syn[] = {(const void *)k_legsyn_mx<2>, (const void *)k_legsyn_mx<4>, (const void *)k_legsyn_mx<8>};
        for (const void *f : syn)
            if ((st = raise_smem_limit(f, syn_mx_smem(lmax))) != WF_OK) return st;
        if ((st = raise_smem_limit((const void *)k_lowsyn_df, (size_t)(lmax + 2) * sizeof(float4))) != WF_OK)
            return st;
        if ((st = raise_smem_limit((const void *)k_lowana_df, (size_t)((np + 31) & ~31) * sizeof(float4))) != WF_OK)
            return st;
        if (tc) {
            if ((st = tc_prepare(lmax)) != WF_OK) return st;
            if ((st = plan_alloc(p, (void **)&p->ws.ca32, nalm * sizeof(float2))) != WF_OK) return st;
        }
    } else {
        if ((st = raise_smem_limit((const void *)k_legsyn_df, syn_df_smem(lmax))) != WF_OK) return st;
    }
    WF_CUDA(cudaStreamSynchronize(p->stream));
    return WF_OK;
}

// Select the FP64 block l < lc of the mixed path and build the FP32 seeds
// that restart the recurrence at lc (cached for the current lc).
wf_status hp_set_low_block(wf_plan p, int lc)
{
    HpTables &t = p->tab;
    if (p->prec == WF_PREC_FP64) return WF_OK;
    if (lc < 0) lc = 0;
    if (lc > p->lmax + 1) lc = p->lmax + 1;
    if (lc == t.lc_mx) return WF_OK;
    const long long ns = (long long)(p->lmax + 1) * p->npairs;
    const int th = 256;
    k_restart_seeds<<<(unsigned)((ns + th - 1) / th), th, 0, p->stream>>>(
        p->lmax, p->npairs, lc, p->nside, t.x64, t.A64, t.Atop, t.kd, t.ls, t.s0_64, t.s1_64, t.k0_mx, t.seed_mx,
        t.ls_mx, t.s0_mx, t.s1_mx);
    WF_COUNT_LAUNCH(p);
    WF_CUDA(cudaGetLastError());
    if (lc > 0 && lc > t.glow_cap) {
        wf_status st = plan_alloc(p, (void **)&p->ws.Glow, (size_t)p->npairs * lc * 2 * sizeof(float2));
        if (st != WF_OK) return st;
        t.glow_cap = lc;
    }
    // the block's Legendre table, when it fits the budget (wf_options.mixed_table_bytes)
    t.low_df = 0;
    const long long budget = p->opt.mixed_table_bytes == 0 ? (2LL << 30) : p->opt.mixed_table_bytes;
    const long long bytes = lc > 0 ? low_table_bytes(p->lmax, p->npairs, lc) : 0;
    if (lc > 0 && bytes <= budget) {
        wf_status st;
        const int np_pad = (p->npairs + 31) & ~31, nm = std::min(lc, p->lmax + 1);
        const long long entries = bytes / (long long)sizeof(float2);
        if (entries > t.lowtab_cap) {
            if ((st = plan_alloc(p, (void **)&t.lowtab, (size_t)bytes)) != WF_OK) return st;
            t.lowtab_cap = entries;
        }
        if (!t.lowrow && (st = plan_alloc(p, (void **)&t.lowrow, (size_t)(p->lmax + 2) * sizeof(long long))) != WF_OK)
            return st;
        std::vector<long long> off(nm + 1, 0);
        for (int m = 0; m < nm; ++m) off[m + 1] = off[m] + low_rows(p->lmax, lc, m);
        if ((st = to_device(p, t.lowrow, off.data(), off.size() * sizeof(long long))) != WF_OK) return st;
        k_lowtab_build<<<dim3((np_pad + 255) / 256, nm), 256, 0, p->stream>>>(
            p->lmax, p->npairs, np_pad, lc, t.lowrow, t.A64, t.c64, t.ls, t.s0_64, t.s1_64, t.x64, t.lowtab);
        WF_COUNT_LAUNCH(p);
        WF_CUDA(cudaGetLastError());
        t.np_pad = np_pad;
        t.low_df = 1;
    }
    t.lc_mx = lc;
    return WF_OK;
}

wf_status hp_legendre_synthesis_buf(wf_plan p, const double2 *alm, int L, double2 *G)
{
    if (p->prec != WF_PREC_FP64) return set_error(WF_EUNSUPPORTED, "explicit-buffer transforms need an FP64 plan");
    return launch_syn64<double>(p, alm, L, 0, G, p->lmax + 1, p->stream);
}

wf_status hp_legendre_adjoint_buf(wf_plan p, int L, const double2 *F, double2 *out)
{
    if (p->prec != WF_PREC_FP64) return set_error(WF_EUNSUPPORTED, "explicit-buffer transforms need an FP64 plan");
    WF_CUDA(cudaMemsetAsync(out, 0, p->nalm * sizeof(double2), p->stream));
    BlendArgs none;
    return launch_ana64(p, L, F, LEG_ADJOINT, none, nullptr, out, p->stream);
}

// Mixed precision: the FP64 low-l block (FP64 pipe, few CTAs) runs on the
// plan's auxiliary stream next to the FP32 kernels (FMA pipes); the two write
// disjoint buffers and are joined before their results are combined.
wf_status fork_aux(wf_plan p)
{
    WF_CUDA(cudaEventRecord(p->fork_ev, p->stream));
    WF_CUDA(cudaStreamWaitEvent(p->aux, p->fork_ev, 0));
    return WF_OK;
}

wf_status join_aux(wf_plan p)
{
    WF_CUDA(cudaEventRecord(p->join_ev, p->aux));
    WF_CUDA(cudaStreamWaitEvent(p->stream, p->join_ev, 0));
    return WF_OK;
}

MxTables mx_tables(wf_plan p, int L)
{
    const HpTables &t = p->tab;
    return MxTables{p->lmax, L,    p->npairs, p->nside, t.lc_mx, t.k0_mx, t.seed_mx,
                    t.xw,    t.tb, t.tp,      t.c64,    t.kd};
}

// threads of a CTA that gives one part of the ring pairs (nside of them) to 32 NP pairs per warp
int mx_threads(wf_plan p, int np) { return std::min(LEG_THREADS, 32 * ((p->nside + 32 * np - 1) / (32 * np))); }

// Ring pairs per thread or lane of one launch to band limit L.  A tile set by the user or timed by
// wf_plan_autotune is kept; by default the largest tile that still gives min8 (8 pairs) or min4
// (4 pairs) warps is taken.  The lines lie where the measured times cross (us, tiles 2 / 4 / 8):
// synthesis nside 64 7 / 7 / 9, 128 8.3 / 9.9 / 11.9, 512 50 / 47 / 57, 1024 502 / 462 / 457; analysis
// nside 256 21.8 / 20.6 / 23.1.
constexpr int SYN_MIN_WARPS_8 = 8192, SYN_MIN_WARPS_4 = 4096, ANA_MIN_WARPS = 1824;
int mx_tile(wf_plan p, int L, int tile, bool set, int min8, int min4)
{
    if (set) return tile;
    auto warps = [&](int np) { return 2LL * (L + 1) * ((p->nside + 32 * np - 1) / (32 * np)); };
    return warps(8) >= min8 ? 8 : warps(4) >= min4 ? 4 : 2;
}

template <int NP>
wf_status launch_syn_mx(wf_plan p, const double2 *alm, int L)
{
    const int th = mx_threads(p, NP), gx = (p->nside + NP * th - 1) / (NP * th);
    const size_t sm = syn_mx_smem(L);
    if (wf_status st = raise_smem_limit((const void *)k_legsyn_mx<NP>, sm)) return st;
    k_legsyn_mx<NP><<<dim3(gx, L + 1, 2), th, sm, p->stream>>>(mx_tables(p, L), alm, (float2 *)p->ws.G);
    WF_COUNT_LAUNCH(p);
    WF_CUDA(cudaGetLastError());
    return WF_OK;
}

wf_status hp_legendre_synthesis(wf_plan p, const double2 *alm, int L)
{
    const HpTables &t = p->tab;
    if (p->prec == WF_PREC_FP64)
        return p->df_legendre ? launch_syn_df(p, alm, L)
                              : launch_syn64<double>(p, alm, L, 0, (double2 *)p->ws.G, p->lmax + 1, p->stream);
    wf_status st;
    const bool low = t.lc_mx > 0;
    if (low) {
        if ((st = fork_aux(p)) != WF_OK) return st;
        st = t.low_df ? launch_lowsyn_df(p, alm, L, p->aux)
                      : launch_syn64<float>(p, alm, L, t.lc_mx, p->ws.Glow, t.glow_cap, p->aux);
        if (st != WF_OK) return st;
    }
    if (tc_prec(p->prec)) {
        // in a batch step the group launch (wf_solve_batch) has written G already
        float2 *G = (float2 *)p->ws.G;
        st = p->tc_deferred ? WF_OK : hp_tc_synthesis(p, 1, &alm, &p->ws.ca32, &G, &L, L, p->stream);
    } else {
        switch (mx_tile(p, L, p->tile_syn, p->tile_syn_set, SYN_MIN_WARPS_8, SYN_MIN_WARPS_4)) {
        case 2: st = launch_syn_mx<2>(p, alm, L); break;
        case 8: st = launch_syn_mx<8>(p, alm, L); break;
        default: st = launch_syn_mx<4>(p, alm, L); break;
        }
    }
    if (st != WF_OK) return st;
    if (low) return join_aux(p);
    return WF_OK;
}

namespace {
template <int NP>
wf_status launch_ana_mx_t(wf_plan p, int L, LegMode mode, const BlendArgs &ba, const double2 *low,
                          const double2 *a_old, double2 *out)
{
    const int ng = (p->nside + 32 * NP - 1) / (32 * NP);
    const MxTables t = mx_tables(p, L);
    k_legana_mx<NP><<<dim3(2 * ng, L + 1), 32, 0, p->stream>>>(t, ng, (const float2 *)p->ws.F, p->tab.psum);
    WF_COUNT_LAUNCH(p);
    k_ana_epilogue<<<L + 1, EPI_THREADS, 0, p->stream>>>(t, (int)mode, ba, low, a_old, out, p->ws.part_harm, p->tab.psum);
    WF_COUNT_LAUNCH(p);
    WF_CUDA(cudaGetLastError());
    return WF_OK;
}

wf_status launch_ana_mx(wf_plan p, int L, LegMode mode, const BlendArgs &ba, const double2 *low, const double2 *a_old,
                        double2 *out)
{
    int tile = mx_tile(p, L, p->tile_ana, p->tile_ana_set, ANA_MIN_WARPS, ANA_MIN_WARPS);
    // Two warps that add to zeroed sums give the same bits in either order, three do not: up to nside
    // 256 the default keeps to two groups of a part's ring pairs, and runs repeat exactly (adjoint, tiles
    // 2 / 4: nside 160, lmax 320 51.8 / 54.0 us; 192, 384 55.4 / 56.8; 227, 454 62.4 / 61.4; 256, 256 50.9 / 50.9)
    if (!p->tile_ana_set && tile == 2 && p->nside > 128 && p->nside <= 256) tile = 4;
    switch (tile) {
    case 2: return launch_ana_mx_t<2>(p, L, mode, ba, low, a_old, out);
    case 4: return launch_ana_mx_t<4>(p, L, mode, ba, low, a_old, out);
    default: return launch_ana_mx_t<8>(p, L, mode, ba, low, a_old, out);
    }
}
}  // namespace

// Autotuner of the mixed Legendre tiles: each variant of the synthesis (2, 4
// or 8 ring pairs per thread) and of the analysis (2, 4 or 8 pairs per lane)
// runs on this plan's own buffers at the full band; the fastest is kept.
wf_status hp_autotune(wf_plan p, int reps)
{
    if (p->prec == WF_PREC_FP64) return WF_OK;
    if (reps <= 0) reps = 3;
    const int L = p->lmax;
    WF_CUDA(cudaMemsetAsync(p->ws.a, 0, p->nalm * sizeof(double2), p->stream));
    WF_CUDA(cudaMemsetAsync(p->ws.F, 0, (size_t)p->npairs * (L + 1) * 2 * sizeof(float2), p->stream));
    cudaEvent_t e0, e1;
    WF_CUDA(cudaEventCreate(&e0));
    WF_CUDA(cudaEventCreate(&e1));
    const int saved_syn = p->tile_syn, saved_ana = p->tile_ana;
    const bool set_syn = p->tile_syn_set, set_ana = p->tile_ana_set;
    p->tile_syn_set = p->tile_ana_set = true;
    const int np[3] = {2, 4, 8};
    float best_syn = 1e30f, best_ana = 1e30f;
    int pick_syn = saved_syn, pick_ana = saved_ana;
    wf_status st = WF_OK;
    BlendArgs none;
    for (int v = 0; v < 3 && st == WF_OK; ++v) {
        p->tile_syn = np[v];
        p->tile_ana = np[v];
        float ms[2] = {0.f, 0.f};
        for (int which = 0; which < 2 && st == WF_OK; ++which) {
            for (int r = -1; r < reps && st == WF_OK; ++r) {  // r = -1: untimed warm-up
                if (r == 0) cudaEventRecord(e0, p->stream);
                if (which == 0)
                    st = np[v] == 2 ? launch_syn_mx<2>(p, p->ws.a, L)
                                    : np[v] == 8 ? launch_syn_mx<8>(p, p->ws.a, L) : launch_syn_mx<4>(p, p->ws.a, L);
                else
                    st = launch_ana_mx(p, L, LEG_ADJOINT, none, nullptr, nullptr, p->ws.b);
            }
            cudaEventRecord(e1, p->stream);
            cudaEventSynchronize(e1);
            cudaEventElapsedTime(&ms[which], e0, e1);
        }
        if (st != WF_OK) break;
        if (ms[0] < best_syn) { best_syn = ms[0]; pick_syn = np[v]; }
        if (ms[1] < best_ana) { best_ana = ms[1]; pick_ana = np[v]; }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    p->tile_syn = st == WF_OK ? pick_syn : saved_syn;
    p->tile_ana = st == WF_OK ? pick_ana : saved_ana;
    if (st != WF_OK) {
        p->tile_syn_set = set_syn;
        p->tile_ana_set = set_ana;
    }
    return st;
}

wf_status hp_legendre_analysis(wf_plan p, int L, LegMode mode, const BlendArgs &ba_in, const double2 *a_old,
                               double2 *out)
{
    const HpTables &t = p->tab;
    BlendArgs ba = ba_in;
    if (mode == LEG_BLEND && ba.epi_ready) {
        ba.epi = p->ws.epi;  // the ring pass of this iteration has filled it
    } else if (mode == LEG_BLEND) {
        k_epi_table<<<(p->lmax + 256) / 256, 256, 0, p->stream>>>(
            EpiArgs{p->lmax, ba.S, p->omega, ba.lam_tauh, ba.tauh, p->ws.epi});
        WF_COUNT_LAUNCH(p);
        WF_CUDA(cudaGetLastError());
        ba.epi = p->ws.epi;
    }
    if (p->prec == WF_PREC_FP64)
        return p->df_legendre ? launch_ana_df(p, L, mode, ba, a_old, out)
                              : launch_ana64(p, L, (const double2 *)p->ws.F, mode, ba, a_old, out, p->stream);
    const int lc = t.lc_mx;
    if (lc <= 0) return launch_ana_mx(p, L, mode, ba, nullptr, a_old, out);
    // sequential: the FP32 epilogue of m < lc reads the block's result
    wf_status st = t.low_df ? launch_lowana_df(p, L, (const float2 *)p->ws.F, p->ws.b_low, p->stream)
                            : launch_ana64_low(p, L, lc, (const float2 *)p->ws.F, p->ws.b_low, p->stream);
    if (st != WF_OK) return st;
    return launch_ana_mx(p, L, mode, ba, p->ws.b_low, a_old, out);
}

}  // namespace wf
