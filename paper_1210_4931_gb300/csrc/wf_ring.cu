// Ring part of the HEALPix basis change (Sect. 2.1 / Sect. 3) and the
// pixel-space blend of Eq. (3), fused into the synthesis side.
//
// Each HEALPix ring r has n_r equally spaced pixels at longitudes
// phi_j = (2j + q) pi / n_r.  Synthesis on a ring is
//     f_j = sum_{m=-L..L} G_m e^{i m phi_j}      (G_{-m} = conj G_m)
//         = sum_{k<n} H_k e^{2 pi i k j / n},   H_k = sum_{m = k mod n} G_m e^{i pi m q / n},
// an inverse DFT of the folded coefficients H; analysis is the forward DFT
// F_m = e^{-i pi m q / n} DFT(f)[m mod n].  The north and south rings of a
// pair have the same n and q, so both are packed into one complex DFT
// (z = f_N + i f_S).
//
// Every ring length is n = 4k.  A DFT of n splits into four DFTs of length k
// and one radix-4 step with the twiddles w_n^{rq} (decimation in time for the
// synthesis, in frequency for the analysis), and the radix-4 step of both
// directions touches the pixels q, q + k, q + 2k, q + 3k of one thread: in the
// messenger step a thread combines its four pixels, blends them (Eq. 3) and
// splits them again in registers.  The four length-k DFTs run
//   k <= 8              as direct sums;
//   k = 2^b >= 16       as FFTs of length N = k;
//   otherwise           by Bluestein's chirp convolution
//                       X_p = c_p sum_j (x_j c_j) conj(c_{p-j}), c_j = e^{-i pi j^2 / k},
//                       circular of length N = 2^b >= 2k - 1: FFT, product with the
//                       tabulated filter spectrum, inverse FFT.
//
// Pixel blend (Eq. 3 solved for t with nu = N^-1, r = nu d):
//     t = s + lambda tau (r - nu s) / (1 + (lambda - 1) tau nu)
// and the pixel term of chi^2 (Eq. 6, x-independent part dropped):
//     sum (nu s^2 - 2 r s) / (1 + (lambda - 1) tau nu).
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <map>

#include "wf_internal.cuh"

namespace wf {

namespace {

int ilog2(long long v)
{
    int l = 0;
    while ((1LL << l) < v) ++l;
    return l;
}

bool is_pow2(long long v) { return v > 0 && (v & (v - 1)) == 0; }

// host radix-2 FFT (FP64), forward e^{-2 pi i jk / n}; used once per ring
// length to tabulate the Bluestein filters
void host_fft(std::vector<double2> &x)
{
    const size_t n = x.size();
    const int lg = ilog2((long long)n);
    for (size_t i = 0; i < n; ++i) {
        size_t j = 0;
        for (int b = 0; b < lg; ++b)
            if (i & (1ull << b)) j |= 1ull << (lg - 1 - b);
        if (i < j) std::swap(x[i], x[j]);
    }
    for (size_t half = 1; half < n; half <<= 1) {
        for (size_t pos = 0; pos < half; ++pos) {
            const double ang = -M_PI * (double)pos / (double)half;
            const double2 w = make_double2(std::cos(ang), std::sin(ang));
            for (size_t i0 = pos; i0 < n; i0 += 2 * half) {
                const size_t i1 = i0 + half;
                const double2 u = x[i0], v = cmul(x[i1], w);
                x[i0] = cadd(u, v);
                x[i1] = csub(u, v);
            }
        }
    }
}

// ---------------------------------------------------------------------------
// register DFTs (forward, e^{-2 pi i nk / R}; the synthesis conjugates around
// them), natural order in and out
// ---------------------------------------------------------------------------
template <typename T> __device__ __forceinline__ cx<T> mul_mi(cx<T> a) { return mk<T>(a.y, -a.x); }  // -i a

template <typename T> __device__ __forceinline__ void dft4(cx<T> &a0, cx<T> &a1, cx<T> &a2, cx<T> &a3)
{
    const cx<T> s02 = cadd(a0, a2), d02 = csub(a0, a2), s13 = cadd(a1, a3), d13 = mul_mi<T>(csub(a1, a3));
    a0 = cadd(s02, s13);
    a1 = cadd(d02, d13);
    a2 = csub(s02, s13);
    a3 = csub(d02, d13);
}

// the same with a2 = a3 = 0 on entry
template <typename T> __device__ __forceinline__ void dft4_half(cx<T> &a0, cx<T> &a1, cx<T> &a2, cx<T> &a3)
{
    const cx<T> x = a0, y = a1, z = mul_mi<T>(a1);
    a0 = cadd(x, y);
    a1 = cadd(x, z);
    a2 = csub(x, y);
    a3 = csub(x, z);
}

template <typename T, int R> __device__ __forceinline__ void dft_small(cx<T> *v)
{
    if constexpr (R == 2) {
        const cx<T> a = v[0];
        v[0] = cadd(a, v[1]);
        v[1] = csub(a, v[1]);
    } else if constexpr (R == 4) {
        dft4<T>(v[0], v[1], v[2], v[3]);
    } else if constexpr (R == 8) {
        const T h = (T)0.70710678118654752440;
        cx<T> e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
        dft4<T>(e[0], e[1], e[2], e[3]);
        dft4<T>(o[0], o[1], o[2], o[3]);
        o[1] = mk<T>(h * (o[1].x + o[1].y), h * (o[1].y - o[1].x));
        o[2] = mul_mi<T>(o[2]);
        o[3] = mk<T>(h * (o[3].y - o[3].x), -h * (o[3].x + o[3].y));
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[k] = cadd(e[k], o[k]);
            v[k + 4] = csub(e[k], o[k]);
        }
    }
}

// 16 = 4 x 4; HALF: v[8..15] are zero on entry (and need not be set)
template <typename T, bool HALF> __device__ __forceinline__ void dft16(cx<T> (&v)[16])
{
    const T c1 = (T)0.92387953251128675613, s1 = (T)0.38268343236508977173, h = (T)0.70710678118654752440;
#pragma unroll
    for (int n = 0; n < 4; ++n) {
        if (HALF) dft4_half<T>(v[n], v[4 + n], v[8 + n], v[12 + n]);
        else dft4<T>(v[n], v[4 + n], v[8 + n], v[12 + n]);
    }
    // v[4 k + n] *= w16^{k n}
    auto w1 = [&](cx<T> a, T c, T s) { return mk<T>(a.x * c + a.y * s, a.y * c - a.x * s); };  // a e^{-i angle}
    v[5] = w1(v[5], c1, s1);
    v[6] = mk<T>(h * (v[6].x + v[6].y), h * (v[6].y - v[6].x));
    v[7] = w1(v[7], s1, c1);
    v[9] = mk<T>(h * (v[9].x + v[9].y), h * (v[9].y - v[9].x));
    v[10] = mul_mi<T>(v[10]);
    v[11] = mk<T>(h * (v[11].y - v[11].x), -h * (v[11].x + v[11].y));
    v[13] = w1(v[13], s1, c1);
    v[14] = mk<T>(h * (v[14].y - v[14].x), -h * (v[14].x + v[14].y));
    v[15] = w1(v[15], -c1, -s1);
#pragma unroll
    for (int k = 0; k < 4; ++k) dft4<T>(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
    // slot 4 k1 + k2 holds output k1 + 4 k2: transpose (register renaming)
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = a + 1; b < 4; ++b) {
            const cx<T> x = v[4 * a + b];
            v[4 * a + b] = v[4 * b + a];
            v[4 * b + a] = x;
        }
}

// v[k] *= w_N^{t k} (conjugated for INV), N = 2^B, t < N/16, from the table of every
// N: tw[N - 32 + k N/16 + t].  FP32 reads k = 1, 4, 8 and forms the other powers (three
// products deep at most); FP64, whose arithmetic is the scarce part, reads all of them.
template <typename T, int B, bool INV>
__device__ __forceinline__ void tw16(cx<T> (&v)[16], int t, const cx<T> *__restrict__ tw)
{
    constexpr int st = 1 << (B - 4);
    const cx<T> *p = tw + ((1 << B) - 32) + t;
    auto ld = [&](int k) {
        cx<T> w = __ldg(p + k * st);
        if (INV) w.y = -w.y;
        return w;
    };
    if constexpr (sizeof(T) == 4) {
        const cx<T> a = ld(1), q = ld(4), o = ld(8);
        const cx<T> b = cmul(a, a), c = cmul(b, a), e = cmul(o, q);
        v[1] = cmul(v[1], a);
        v[2] = cmul(v[2], b);
        v[3] = cmul(v[3], c);
        v[4] = cmul(v[4], q);
        v[5] = cmul(v[5], cmul(q, a));
        v[6] = cmul(v[6], cmul(q, b));
        v[7] = cmul(v[7], cmul(q, c));
        v[8] = cmul(v[8], o);
        v[9] = cmul(v[9], cmul(o, a));
        v[10] = cmul(v[10], cmul(o, b));
        v[11] = cmul(v[11], cmul(o, c));
        v[12] = cmul(v[12], e);
        v[13] = cmul(v[13], cmul(e, a));
        v[14] = cmul(v[14], cmul(e, b));
        v[15] = cmul(v[15], cmul(e, c));
    } else {
#pragma unroll
        for (int k = 1; k < 16; ++k) v[k] = cmul(v[k], ld(k));
    }
}

// shared buffers are padded by one entry per 16: the strides of the exchanges
// below (16, R, 16 R entries) would otherwise fall on a few banks
__host__ __device__ __forceinline__ int pidx(int i) { return i + (i >> 4); }
inline size_t padded_len(size_t n) { return n + n / 16 + 1; }

// ---------------------------------------------------------------------------
// One DFT of length N = 2^B by a team of N/16 threads, 16 values each, in
// registers.  Thread t enters with x[e N/16 + t] in v[e].
//   B <= 8:  radix 16, exchange, radix R = N/16
//   B >= 9:  radix 16, exchange, radix 16, exchange, radix R = N/256
// The last exchange (the only one for B <= 8) stays inside groups of R <= 16
// consecutive threads: a warp barrier.  The first needs the team's barrier
// (a warp barrier again for B = 9, whose team is one warp).  The forward
// transform leaves X in the registers in the order fft_index gives; the
// inverse starts from that order and runs the same steps backwards, so a
// convolution needs no reordering and its shared-memory traffic is four
// exchanges.  In the backward run every thread writes the addresses it read
// last, so no barrier guards the buffer between steps.
// ---------------------------------------------------------------------------
template <int B> struct Team {
    static constexpr int N = 1 << B, NT = N / 16;           // values, threads
    static constexpr int R = B <= 8 ? N / 16 : N / 256;     // last radix (B = 4: none)
};

// frequency held in register e of thread t after the forward transform of length 2^B
__host__ __device__ inline int fft_index(int B, int t, int e)
{
    if (B == 4) return e;
    if (B <= 8) {
        const int R = 1 << (B - 4), u = e / R, k2 = e % R;
        return t * (16 / R) + u + 16 * k2;
    }
    const int R = 1 << (B - 8), u = e / R, k3 = e % R, k1 = t / R, t2 = t % R;
    return k1 + 16 * (t2 * (16 / R) + u) + 256 * k3;
}

template <int B> __device__ __forceinline__ void team_sync(int slot, unsigned mask)
{
    if constexpr (B <= 9) __syncwarp(mask);
    else asm volatile("bar.sync %0, %1;" ::"r"(1 + slot), "r"(Team<B>::NT) : "memory");
}

// The addresses split into a part of the thread and a compile-time offset: pidx(a + b) =
// pidx(a) + pidx(b) wherever b is a multiple of a power of two above a mod 16.
template <typename T, int B, bool HALF>
__device__ __forceinline__ void fft_forward(cx<T> (&v)[16], cx<T> *ex, int t, int slot, unsigned mask,
                                            const cx<T> *__restrict__ tw)
{
    constexpr int NT = Team<B>::NT, R = Team<B>::R;
    dft16<T, HALF>(v);
    if constexpr (B > 4) {
        tw16<T, B, false>(v, t, tw);
        cx<T> *e1 = ex + pidx(t);
#pragma unroll
        for (int k = 0; k < 16; ++k) e1[pidx(k * NT)] = v[k];
        team_sync<B>(slot, mask);
        if constexpr (B > 8) {
            cx<T> *e2 = ex + pidx((t / R) * NT + t % R);
#pragma unroll
            for (int k = 0; k < 16; ++k) v[k] = e2[pidx(k * R)];
            dft16<T, false>(v);
            tw16<T, B - 4, false>(v, t % R, tw);
#pragma unroll
            for (int k = 0; k < 16; ++k) e2[pidx(k * R)] = v[k];
            __syncwarp(mask);
        }
        const cx<T> *e3 = ex + 17 * t;  // pidx(16 t)
#pragma unroll
        for (int e = 0; e < 16; ++e) v[e] = e3[e];
        if constexpr (R == 16) {
            dft16<T, false>(v);
        } else {
#pragma unroll
            for (int u = 0; u < 16; u += R) dft_small<T, R>(v + u);
        }
    }
}

// inverse (unnormalised) of fft_forward on the conjugate: takes conj X, returns conj x
template <typename T, int B>
__device__ __forceinline__ void fft_backward(cx<T> (&v)[16], cx<T> *ex, int t, int slot, unsigned mask,
                                             const cx<T> *__restrict__ tw)
{
    constexpr int NT = Team<B>::NT, R = Team<B>::R;
    if constexpr (B > 4) {
        if constexpr (R == 16) {
            dft16<T, false>(v);
        } else {
#pragma unroll
            for (int u = 0; u < 16; u += R) dft_small<T, R>(v + u);
        }
        cx<T> *e3 = ex + 17 * t;
#pragma unroll
        for (int e = 0; e < 16; ++e) e3[e] = v[e];
        if constexpr (B > 8) {
            __syncwarp(mask);
            cx<T> *e2 = ex + pidx((t / R) * NT + t % R);
#pragma unroll
            for (int k = 0; k < 16; ++k) v[k] = e2[pidx(k * R)];
            tw16<T, B - 4, false>(v, t % R, tw);
            dft16<T, false>(v);
#pragma unroll
            for (int k = 0; k < 16; ++k) e2[pidx(k * R)] = v[k];
        }
        team_sync<B>(slot, mask);
        const cx<T> *e1 = ex + pidx(t);
#pragma unroll
        for (int k = 0; k < 16; ++k) v[k] = e1[pidx(k * NT)];
        tw16<T, B, false>(v, t, tw);
    }
    dft16<T, false>(v);
}

// threads of a ring CTA, one ring pair each: a team of 256 holds the longest Bluestein FFT
// (N = 4096) with 16 values per thread; shorter ones run up to four of the pair's sub-DFTs
// side by side
constexpr int RING_CTA = 256;

// position of value j of a ring (or of frequency j) in the padded buffer: the four
// length-k sequences j mod 4 one after another
__device__ __forceinline__ int zpos(int j, int k) { return pidx((j & 3) * k + (j >> 2)); }

template <typename P> __device__ __forceinline__ const P *opaque(const P *p)
{
    asm volatile("" : "+l"(p));
    return p;
}
__device__ __forceinline__ int opaque(int t)
{
    asm volatile("" : "+r"(t));
    return t;
}

// The four length-k DFTs (forward; FLIP conjugates in and out, i.e. the inverse) of the
// sequences at zb[pidx(r k + j)], in place.
template <typename T, int B, bool BLUE>
__device__ __noinline__ void sub_dfts(cx<T> *zb, cx<T> *exch, int k, bool flip, const cx<T> *V0,
                                      const cx<T> *chirp0, const cx<T> *tw0)
{
    constexpr int N = Team<B>::N, NT = Team<B>::NT, R = Team<B>::R;
    constexpr int SLOTS = NT * 4 <= RING_CTA ? 4 : RING_CTA / NT;
    const int slot = threadIdx.x / NT, t0 = threadIdx.x % NT;
    if (slot >= SLOTS) return;  // whole warps, or the lanes that `mask` leaves out
    const unsigned mask = SLOTS * NT >= 32 ? 0xffffffffu : (1u << (SLOTS * NT)) - 1u;
    cx<T> *ex = exch + slot * (N + N / 16);
    const T sg = flip ? (T)-1 : (T)1;
#pragma unroll 1
    for (int r = slot; r < 4; r += SLOTS) {
        // opaque: addresses and table values are formed again in every round (tables from L1);
        // held in registers across the rounds and the FFTs they spill
        const int t = opaque(t0);
        const cx<T> *__restrict__ tw = opaque(tw0);
        cx<T> v[16];
        if constexpr (BLUE) {
            const cx<T> *__restrict__ V = opaque(V0), *__restrict__ chirp = opaque(chirp0);
            // value j = e NT + t of sequence r
            cx<T> *z = zb + pidx(r * k + t);
            auto at = [&](int e) -> cx<T> & { return NT >= 16 ? z[pidx(e * NT)] : zb[pidx(r * k + e * NT + t)]; };
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int j = e * NT + t;
                v[e] = mk<T>(0, 0);
                if (j < k) {
                    cx<T> u = at(e);
                    u.y *= sg;
                    v[e] = cmul(u, __ldg(chirp + j));
                }
            }
            fft_forward<T, B, true>(v, ex, t, slot, mask, tw);
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                v[e] = cmul(v[e], __ldg(V + e * NT + t));
                v[e].y = -v[e].y;
            }
            fft_backward<T, B>(v, ex, t, slot, mask, opaque(tw0));
            const cx<T> *__restrict__ chirp2 = opaque(chirp0);
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int j = e * NT + t;
                if (j < k) {
                    cx<T> y = cmul(cconj(v[e]), __ldg(chirp2 + j));
                    y.y *= sg;
                    at(e) = y;
                }
            }
        } else {
            cx<T> *zr = zb + pidx(r * N), *z = zr + pidx(t);
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                v[e] = z[pidx(e * NT)];
                v[e].y *= sg;
            }
            if (r >= SLOTS) team_sync<B>(slot, mask);  // the exchange buffer's last readers are done
            fft_forward<T, B, false>(v, ex, t, slot, mask, tw);
            // outputs land where other threads of the team may still read inputs (B = 4: its own)
            team_sync<B>(slot, mask);
            // pidx(fft_index(B, t, e)) as a part of the thread and a constant
            cx<T> *o = zr + (B == 4 ? 0 : B <= 8 ? t * (16 / R) : t / R + 17 * (t % R) * (16 / R));
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                v[e].y *= sg;
                o[B == 4 ? e : B <= 8 ? e / R + 17 * (e % R) : 17 * (e / R + 16 * (e % R))] = v[e];
            }
        }
    }
}

// The same for k <= 8 by direct sums, one value per thread of the first warp; root: e^{i pi t / 4k}.
// What bounds a grid of such rings alone (nside <= 8) is the chain of one pair: as a Bluestein FFT
// of length 16 a DFT is one thread's, some 600 FP64 operations in a row.  Synthesis / adjoint in FP64
// (whole calls) at nside 2 35.9 / 46.5 -> 22.1 / 30.8 us, at nside 8 39.9 / 50.7 -> 27.1 / 37.0 us.
template <typename T>
__device__ __noinline__ void short_dfts(cx<T> *zb, int k, bool flip, const cx<T> *__restrict__ root)
{
    const int t = threadIdx.x, r = t / k, p = t - r * k;
    if (t >= 32) return;
    cx<T> s = mk<T>(0, 0);
    if (r < 4) {
        cx<T> w[RING_SHORT_K];
        int i = 0;  // j p mod k
#pragma unroll
        for (int j = 0; j < RING_SHORT_K; ++j) {  // every load in flight before the sum
            w[j] = root[8 * i];
            i += p;
            if (i >= k) i -= k;
        }
#pragma unroll
        for (int j = 0; j < RING_SHORT_K; ++j) {
            if (j == k) break;
            if (!flip) w[j].y = -w[j].y;
            s = cadd(s, cmul(zb[pidx(r * k + j)], w[j]));
        }
    }
    __syncwarp();
    if (r < 4) zb[pidx(t)] = s;
}

template <typename T>
__device__ __forceinline__ void ring_sub_dfts(const RingTab &R, cx<T> *zb, cx<T> *ex, bool flip,
                                              const cx<T> *__restrict__ V, const cx<T> *__restrict__ chirp,
                                              const cx<T> *__restrict__ tw, const cx<T> *__restrict__ root)
{
    const cx<T> *v = V + R.vOff, *c = chirp + R.cOff;
    const int k = R.n >> 2;
    if (R.kind == RING_SHORT) {
        short_dfts<T>(zb, k, flip, root);
    } else if (R.kind == RING_POW2) {
        switch (R.logF) {
        case 4: sub_dfts<T, 4, false>(zb, ex, k, flip, v, c, tw); break;
        case 5: sub_dfts<T, 5, false>(zb, ex, k, flip, v, c, tw); break;
        case 6: sub_dfts<T, 6, false>(zb, ex, k, flip, v, c, tw); break;
        case 7: sub_dfts<T, 7, false>(zb, ex, k, flip, v, c, tw); break;
        case 8: sub_dfts<T, 8, false>(zb, ex, k, flip, v, c, tw); break;
        case 9: sub_dfts<T, 9, false>(zb, ex, k, flip, v, c, tw); break;
        case 10: sub_dfts<T, 10, false>(zb, ex, k, flip, v, c, tw); break;
        default: sub_dfts<T, 11, false>(zb, ex, k, flip, v, c, tw); break;
        }
    } else {
        switch (R.logF) {
        case 5: sub_dfts<T, 5, true>(zb, ex, k, flip, v, c, tw); break;
        case 6: sub_dfts<T, 6, true>(zb, ex, k, flip, v, c, tw); break;
        case 7: sub_dfts<T, 7, true>(zb, ex, k, flip, v, c, tw); break;
        case 8: sub_dfts<T, 8, true>(zb, ex, k, flip, v, c, tw); break;
        case 9: sub_dfts<T, 9, true>(zb, ex, k, flip, v, c, tw); break;
        case 10: sub_dfts<T, 10, true>(zb, ex, k, flip, v, c, tw); break;
        case 11: sub_dfts<T, 11, true>(zb, ex, k, flip, v, c, tw); break;
        default: sub_dfts<T, 12, true>(zb, ex, k, flip, v, c, tw); break;
        }
    }
    __syncthreads();
}

__device__ __forceinline__ double block_sum(double v, double *red)
{
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
    return s;
}

template <typename T> struct RingArgs {
    int lmax, L;
    const RingTab *rings;
    const int *order;      // ring pairs by decreasing cost: CTA i takes pair order[i]
    const cx<T> *roots, *V, *chirp, *tw;
    int zlen;              // padded length of the ring buffer; the exchange buffer follows it
    const cx<T> *G;        // synthesis input
    const float2 *Glow;    // mixed path: FP64-block coefficients for m < lc, rounded to FP32 (or null)
    int lc, glow_stride;
    int mode;              // RingSynMode, or RS_ANA
    const T *r, *nu;       // blend
    T lam, tau;
    T *tmap;               // synthesis: output map; analysis: null
    double *omap;          // RS_MAP output
    const T *amap;         // RS_ANA input
    double *part;          // per ring pair: chi^2 pixel term
    cx<T> *F;              // analysis output
    int npairs;
    EpiArgs epi;           // messenger step: CTAs past the pairs fill the blend table of the analysis
};

constexpr int RS_ANA = 16;  // analysis only (beside RingSynMode)

// north and south coefficient of one m (adjacent in memory): one 16-byte load in FP32
__device__ __forceinline__ void load_ns(const float2 *g, float2 &n, float2 &s)
{
    const float4 v = *reinterpret_cast<const float4 *>(g);
    n = make_float2(v.x, v.y);
    s = make_float2(v.z, v.w);
}
__device__ __forceinline__ void load_ns(const double2 *g, double2 &n, double2 &s)
{
    n = g[0];
    s = g[1];
}
__device__ __forceinline__ void store_ns(float2 *g, float2 n, float2 s)
{
    *reinterpret_cast<float4 *>(g) = make_float4(n.x, n.y, s.x, s.y);
}
__device__ __forceinline__ void store_ns(double2 *g, double2 n, double2 s)
{
    g[0] = n;
    g[1] = s;
}

// Fold H_k = sum_{m = k mod n} G_m e^{i pi m q / n} + conj terms of -m, for the packed
// north/south pair.  e^{i pi m / n} at m = k + a n is (-1)^a e^{i pi k / n}: the aliases of a
// bin are summed with alternating signs and take the phase once.  Rings longer than L have
// at most one alias of each sign, independent bins with several loads in flight; shorter
// rings sum each bin over S lanes of a warp (S up to 32 for the polar rings, whose bins
// collect ~2L/n aliases), combined by shuffles in a fixed order.
template <typename T>
__device__ __forceinline__ void fold_ring(const RingArgs<T> &A, const RingTab &R, const cx<T> *__restrict__ g,
                                          const float2 *__restrict__ gl, bool south, cx<T> *zb)
{
    const int n = R.n, q = R.q, L = A.L, k4 = n >> 2, lc = gl ? A.lc : 0;
    const cx<T> *root = A.roots + R.rootOff;
    auto coef = [&](int m, cx<T> &a, cx<T> &b) {
        load_ns(g + 2 * m, a, b);
        if (m < lc) {
            const float2 x = gl[2 * m], y = gl[2 * m + 1];
            a.x += (T)x.x;
            a.y += (T)x.y;
            b.x += (T)y.x;
            b.y += (T)y.y;
        }
    };
    if (n > L) {
#pragma unroll 4
        for (int k = threadIdx.x; k < n; k += RING_CTA) {
            cx<T> hn = mk<T>(0, 0), hs = mk<T>(0, 0), a, b;
            if (k <= L) {
                coef(k, a, b);
                const cx<T> ph = root[q ? k : 0];
                hn = cmul(a, ph);
                hs = cmul(b, ph);
            }
            const int mneg = n - k;
            if (k > 0 && mneg <= L) {
                coef(mneg, a, b);
                const cx<T> ph = root[q ? mneg : 0];
                hn = cadd(hn, cconj(cmul(a, ph)));
                hs = cadd(hs, cconj(cmul(b, ph)));
            }
            if (!south) hs = mk<T>(0, 0);
            zb[zpos(k, k4)] = mk<T>(hn.x - hs.y, hn.y + hs.x);
        }
        return;
    }
    int S = 1;
    while (S < 32 && 2 * S * n <= RING_CTA) S *= 2;
    const int sub = threadIdx.x & (S - 1), nb = RING_CTA / S;
    for (int base = 0; base < n; base += nb) {
        const int k = base + threadIdx.x / S;
        cx<T> pn = mk<T>(0, 0), ps = pn, mn = pn, ms = pn, a, b;
        if (k < n) {
            const int m0 = k == 0 ? n : n - k;
            // alternating signs over the alias number (q = 1; the belt's q = 0 rings are longer than L
            // or take no sign)
#pragma unroll 2
            for (int i = sub, m = k + sub * n; m <= L; i += S, m += S * n) {
                coef(m, a, b);
                const T s = (q && (i & 1)) ? (T)-1 : (T)1;
                pn.x = fma(s, a.x, pn.x);
                pn.y = fma(s, a.y, pn.y);
                ps.x = fma(s, b.x, ps.x);
                ps.y = fma(s, b.y, ps.y);
            }
#pragma unroll 2
            for (int i = sub, m = m0 + sub * n; m <= L; i += S, m += S * n) {
                coef(m, a, b);
                const T s = (q && (i & 1)) ? (T)-1 : (T)1;
                mn.x = fma(s, a.x, mn.x);
                mn.y = fma(s, a.y, mn.y);
                ms.x = fma(s, b.x, ms.x);
                ms.y = fma(s, b.y, ms.y);
            }
            const cx<T> ph = root[q ? k : 0], pm = root[q ? m0 : 0];
            pn = cadd(cmul(pn, ph), cconj(cmul(mn, pm)));
            ps = cadd(cmul(ps, ph), cconj(cmul(ms, pm)));
        }
        for (int o = S >> 1; o >= 1; o >>= 1) {
            pn.x += __shfl_xor_sync(0xffffffffu, pn.x, o);
            pn.y += __shfl_xor_sync(0xffffffffu, pn.y, o);
            ps.x += __shfl_xor_sync(0xffffffffu, ps.x, o);
            ps.y += __shfl_xor_sync(0xffffffffu, ps.y, o);
        }
        if (k < n && sub == 0) {
            if (!south) ps = mk<T>(0, 0);
            zb[zpos(k, k4)] = mk<T>(pn.x - ps.y, pn.y + ps.x);
        }
    }
}

// Unfold a forward ring DFT of the packed pair (z = f_N + i f_S) to
// F_m = e^{-i pi m q / n} DFT(f)[m mod n] for both rings, m <= L.
template <typename T>
__device__ __forceinline__ void unfold_ring(const RingArgs<T> &A, const RingTab &R, const cx<T> *zb, bool south,
                                            cx<T> *__restrict__ f)
{
    const int n = R.n, k4 = n >> 2, L = A.L;
    const cx<T> *root = A.roots + R.rootOff;
#pragma unroll 4
    for (int m = threadIdx.x; m <= L; m += RING_CTA) {
        const unsigned al = __umulhi((unsigned)m, R.inv);  // m / n
        const int k = m - (int)al * n;
        const int nk = k ? n - k : 0;
        const cx<T> zk = zb[zpos(k, k4)], znk = zb[zpos(nk, k4)];
        cx<T> ph = mk<T>(1, 0);
        if (R.q) {
            ph = root[k];
            const T s = (al & 1) ? (T)-1 : (T)1;
            ph = mk<T>(s * ph.x, -s * ph.y);
        }
        const cx<T> tn = mk<T>((T)0.5 * (zk.x + znk.x), (T)0.5 * (zk.y - znk.y));
        const cx<T> ts = mk<T>((T)0.5 * (zk.y + znk.y), (T)-0.5 * (zk.x - znk.x));
        store_ns(f + 2 * m, cmul(ph, tn), south ? cmul(ph, ts) : mk<T>(0, 0));
    }
}

// One ring pair per CTA: fold, four inverse sub-DFTs, radix-4 step with the pixels (blend, or a
// map written or read), four forward sub-DFTs, unfold.
//
// What bounds it: the latency of one pair's chain of steps, covered by the SM's other CTAs.  An
// earlier version gave a pair a 1024-thread CTA and in-place radix-8 passes in shared memory,
// each between two CTA barriers (~60 barriers per Bluestein pair, the first stall).  Here a
// pair takes 256 threads and keeps its values in registers between two exchanges per FFT.
// Mean over the ring passes of one solve (cooling and full-band steps, output map), FP32: nside
// 2048 1.28 -> 0.53 ms, nside 512 0.153 -> 0.057 ms, nside 128 0.042 -> 0.019 ms (cold caches);
// FP64: nside 512 0.93 -> 0.55 ms and nside 100 0.21 -> 0.073 ms, bound by the FP64 pipe.
//
// MINB CTAs per SM set the register budget: FP32 at 128 registers (2) or 80 with some 210 bytes
// spilled per thread in the Bluestein FFTs of 2048 and 4096 (3).  Three are faster where shared
// memory holds three and there are pairs for them (a map pass at nside 1024 0.131 -> 0.112 ms, a
// step at nside 512 0.066 -> 0.057 ms), two where it does not (nside 2048: 0.525 against 0.570 ms
// averaged over a solve) or where one wave holds every pair (nside 128: 18.5 against 20.6 us).
// FP64: two at 128 registers against one at 255: nside 100 0.126 -> 0.073 ms, nside 512
// 0.60 -> 0.55 ms.
template <typename T, int MINB>
__global__ void __launch_bounds__(RING_CTA, MINB) k_ring(const RingArgs<T> A)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double red[RING_CTA / 32];
    if ((int)blockIdx.x >= A.npairs) {  // (a launch of its own costs 3.5 us an iteration)
        epi_entry(A.epi, (blockIdx.x - A.npairs) * RING_CTA + threadIdx.x);
        return;
    }
    cx<T> *zb = reinterpret_cast<cx<T> *>(smem_raw), *ex = zb + A.zlen;
    const int pair = A.order[blockIdx.x], mode = A.mode;
    const RingTab R = A.rings[pair];
    const int n = R.n, k = n >> 2;
    const bool south = R.offS >= 0, syn = mode != RS_ANA, blend = mode == RS_BLEND || mode == RS_BLEND_ANA;
    const bool ana = mode == RS_ANA || mode == RS_BLEND_ANA;
    const cx<T> *root = A.roots + R.rootOff;
    const size_t row = (size_t)pair * (A.lmax + 1) * 2;
    if (syn) {
        fold_ring<T>(A, R, A.G + row, A.Glow ? A.Glow + (size_t)pair * A.glow_stride * 2 : nullptr, south, zb);
        __syncthreads();
        ring_sub_dfts<T>(R, zb, ex, true, A.V, A.chirp, A.tw, root);
    }
    const T lt = A.lam * A.tau, lm1t = (A.lam - (T)1) * A.tau;
    T chi = 0;
    auto blend1 = [&](T s, T rv, T nv) {
        const T id = (T)1 / ((T)1 + lm1t * nv);  // one division for both (FP64 divides are a dozen operations)
        chi += (nv * s * s - (T)2 * rv * s) * id;
        return s + lt * (rv - nv * s) * id;
    };
#pragma unroll 2
    for (int p = threadIdx.x; p < k; p += RING_CTA) {
        const int z0 = pidx(p), z1 = pidx(k + p), z2 = pidx(2 * k + p), z3 = pidx(3 * k + p);
        cx<T> w1 = root[2 * p], w2, w3;
        if constexpr (sizeof(T) == 4) {
            w2 = cmul(w1, w1);
            w3 = cmul(w2, w1);
        } else {
            w2 = root[4 * p];
            w3 = root[6 * p];
        }
        // x[s]: pixel p + s k of the north (re) and south (im) ring
        cx<T> x[4];
        const long long iN = R.offN + p, iS = R.offS + p;
        if (syn) {
            // the four sub-DFTs conjugated: x_s = conj sum_r (-i)^{rs} conj(w^{rp} X_r)
            x[0] = cconj(zb[z0]);
            x[1] = cconj(cmul(zb[z1], w1));
            x[2] = cconj(cmul(zb[z2], w2));
            x[3] = cconj(cmul(zb[z3], w3));
            dft4<T>(x[0], x[1], x[2], x[3]);
#pragma unroll
            for (int s = 0; s < 4; ++s) x[s].y = -x[s].y;
            if (mode == RS_MAP) {
#pragma unroll
                for (int s = 0; s < 4; ++s) {
                    A.omap[iN + s * k] = (double)x[s].x;
                    if (south) A.omap[iS + s * k] = (double)x[s].y;
                }
            } else if (blend) {
                T rN[4], nN[4], rS[4], nS[4];
#pragma unroll
                for (int s = 0; s < 4; ++s) {
                    rN[s] = A.r[iN + s * k];
                    nN[s] = A.nu[iN + s * k];
                    rS[s] = south ? A.r[iS + s * k] : (T)0;
                    nS[s] = south ? A.nu[iS + s * k] : (T)0;
                }
#pragma unroll
                for (int s = 0; s < 4; ++s) {
                    x[s].x = blend1(x[s].x, rN[s], nN[s]);
                    x[s].y = south ? blend1(x[s].y, rS[s], nS[s]) : (T)0;
                }
            }
            if (mode == RS_SYN || mode == RS_BLEND) {
#pragma unroll
                for (int s = 0; s < 4; ++s) {
                    A.tmap[iN + s * k] = x[s].x;
                    if (south) A.tmap[iS + s * k] = x[s].y;
                }
            }
        } else {
#pragma unroll
            for (int s = 0; s < 4; ++s) x[s] = mk<T>(A.amap[iN + s * k], south ? A.amap[iS + s * k] : (T)0);
        }
        if (ana) {
            dft4<T>(x[0], x[1], x[2], x[3]);
            zb[z0] = x[0];
            zb[z1] = cmul(x[1], cconj(w1));
            zb[z2] = cmul(x[2], cconj(w2));
            zb[z3] = cmul(x[3], cconj(w3));
        }
    }
    if (blend) {  // per-pair partial: the reduction order does not depend on the schedule
        const double s = block_sum((double)chi, red);
        if (threadIdx.x == 0) A.part[pair] = s;
    }
    if (ana) {
        __syncthreads();
        ring_sub_dfts<T>(R, zb, ex, false, A.V, A.chirp, A.tw, root);
        unfold_ring<T>(A, R, zb, south, A.F + row);
    }
}

template <typename T> struct RingLaunch {
    static RingArgs<T> args(wf_plan p, int L, int mode)
    {
        const HpTables &t = p->tab;
        RingArgs<T> a{};
        a.lmax = p->lmax;
        a.L = L;
        a.rings = t.rings;
        a.order = t.order;
        a.roots = (const cx<T> *)t.roots;
        a.V = (const cx<T> *)t.V;
        a.chirp = (const cx<T> *)t.chirp;
        a.tw = (const cx<T> *)t.tw;
        a.zlen = (int)padded_len(t.nmax);
        a.npairs = p->npairs;
        a.mode = mode;
        return a;
    }
    static wf_status launch(wf_plan p, const RingArgs<T> &a)
    {
        const size_t sm = smem_bytes(p->tab);
        auto kernel = k_ring<T, 2>;
        if constexpr (sizeof(T) == 4)
            if (p->tab.ring_ctas == 3) kernel = k_ring<T, 3>;
        const int extra = a.epi.epi ? (a.epi.lmax + RING_CTA) / RING_CTA : 0;
        kernel<<<p->npairs + extra, RING_CTA, sm, p->stream>>>(a);
        WF_COUNT_LAUNCH(p);
        WF_CUDA(cudaGetLastError());
        return WF_OK;
    }
    static wf_status syn(wf_plan p, int L, RingSynMode mode, double lam, double tau, double *omap)
    {
        return syn_buf(p, L, mode, lam, tau, p->ws.G, p->ws.t, omap);
    }
    static wf_status syn_buf(wf_plan p, int L, RingSynMode mode, double lam, double tau, const void *G, void *tmap,
                             double *omap)
    {
        const HpTables &t = p->tab;
        if (p->prec != WF_PREC_FP64 && t.lc_mx > 0)
            return syn_buf_low(p, L, mode, lam, tau, G, p->ws.Glow, t.lc_mx, t.glow_cap, tmap, omap);
        return syn_buf_low(p, L, mode, lam, tau, G, nullptr, 0, 0, tmap, omap);
    }
    // with the FP64 block's coefficients (m < lc, [pair][m][hemisphere] with
    // glow_stride columns per pair) added to G, or none (glow null)
    static wf_status syn_buf_low(wf_plan p, int L, RingSynMode mode, double lam, double tau, const void *G,
                                 const float2 *glow, int lc, int glow_stride, void *tmap, double *omap,
                                 void *F = nullptr, const EpiArgs *epi = nullptr)
    {
        RingArgs<T> a = args(p, L, (int)mode);
        if (epi) a.epi = *epi;
        if (glow && lc > 0) {
            a.Glow = glow;
            a.lc = lc;
            a.glow_stride = glow_stride;
        }
        a.G = (const cx<T> *)G;
        a.r = (const T *)p->ws.r;
        a.nu = (const T *)p->ws.nu;
        a.lam = (T)lam;
        a.tau = (T)tau;
        a.tmap = (T *)tmap;
        a.omap = omap;
        a.part = p->ws.part_pix;
        a.F = (cx<T> *)F;
        return launch(p, a);
    }
    // messenger step on the rings: fold, inverse DFT, Eq. 3, forward DFT, unfold into F
    static wf_status syn_ana(wf_plan p, int L, double lam, double tau, const EpiArgs &epi)
    {
        const HpTables &t = p->tab;
        if (p->prec != WF_PREC_FP64 && t.lc_mx > 0)
            return syn_buf_low(p, L, RS_BLEND_ANA, lam, tau, p->ws.G, p->ws.Glow, t.lc_mx, t.glow_cap, nullptr,
                               nullptr, p->ws.F, &epi);
        return syn_buf_low(p, L, RS_BLEND_ANA, lam, tau, p->ws.G, nullptr, 0, 0, nullptr, nullptr, p->ws.F, &epi);
    }
    static wf_status ana(wf_plan p, int L, const void *map) { return ana_buf(p, L, map, p->ws.F); }
    static wf_status ana_buf(wf_plan p, int L, const void *map, void *F)
    {
        RingArgs<T> a = args(p, L, RS_ANA);
        a.amap = (const T *)map;
        a.F = (cx<T> *)F;
        return launch(p, a);
    }
    static size_t smem_bytes(const HpTables &t) { return (padded_len(t.nmax) + padded_len(t.exmax)) * sizeof(cx<T>); }
    // The dynamic shared-memory limit is raised once per kernel and size, before
    // any launch that needs it, and never lowered: plans of several sizes may
    // launch concurrently from different host threads.
    static wf_status prepare(wf_plan p)
    {
        const size_t sm = smem_bytes(p->tab);
        if (wf_status st = raise_smem_limit((const void *)k_ring<T, 2>, sm)) return st;
        int b = 0;
        WF_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_ring<T, 2>, RING_CTA, sm));
        if (b < 1) return set_error(WF_EUNSUPPORTED, "ring kernel does not fit on an SM (smem %zu bytes)", sm);
        p->tab.ring_ctas = 2;
        if constexpr (sizeof(T) == 4) {
            if (p->npairs > 2 * p->nsm) {
                int b3 = 0;
                if (wf_status st = raise_smem_limit((const void *)k_ring<T, 3>, sm)) return st;
                WF_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b3, k_ring<T, 3>, RING_CTA, sm));
                if (b3 >= 3) p->tab.ring_ctas = 3;
            }
        }
        return WF_OK;
    }
};

template <typename T>
wf_status upload_cx(wf_plan p, void **dst, const std::vector<double2> &src)
{
    wf_status st = plan_alloc(p, dst, src.size() * sizeof(cx<T>) + 16);
    if (st != WF_OK) return st;
    std::vector<cx<T>> tmp(src.size());
    for (size_t i = 0; i < src.size(); ++i) tmp[i] = mk<T>((T)src[i].x, (T)src[i].y);
    if ((st = to_device(p, *dst, tmp.data(), tmp.size() * sizeof(cx<T>))) != WF_OK) return st;
    return WF_OK;
}

}  // namespace

// how the DFTs of a ring of n = 4k pixels are done, and log2 of their FFT length (short rings: 0)
RingKind ring_kind(int n, int *logF)
{
    const int k = n / 4;
    const RingKind kind = k <= RING_SHORT_K ? RING_SHORT : is_pow2(k) ? RING_POW2 : RING_BLUESTEIN;
    *logF = kind == RING_SHORT ? 0 : ilog2(kind == RING_POW2 ? k : 2LL * k - 1);
    return kind;
}

wf_status hp_build_ring_tables(wf_plan p)
{
    const int nside = p->nside, np = p->npairs;
    const int R = 4 * nside - 1;
    if (nside > RING_MAX_K) return set_error(WF_EUNSUPPORTED, "rings longer than %d pixels (nside > %d)", 4 * RING_MAX_K, RING_MAX_K);
    // ring offsets (RING order)
    std::vector<long long> off(R + 1, 0);
    std::vector<int> nr(R), qr(R);
    for (int i = 1; i <= R; ++i) {
        const int k = (i <= 2 * nside) ? i : 4 * nside - i;
        if (k < nside) {
            nr[i - 1] = 4 * k;
            qr[i - 1] = 1;
        } else {
            nr[i - 1] = 4 * nside;
            qr[i - 1] = ((i + nside) & 1) ? 0 : 1;
        }
        off[i] = off[i - 1] + nr[i - 1];
    }
    std::vector<RingTab> rt(np);
    std::map<int, long long> rootOff, vOff, cOff;
    std::vector<double2> roots, Vtab, chirp;
    int exmax = 0, logmax = 0;
    for (int pr = 0; pr < np; ++pr) {
        RingTab &t = rt[pr];
        const int i0 = pr;  // north ring, 0-based
        t.n = nr[i0];
        t.q = qr[i0];
        t.offN = off[i0];
        t.offS = (pr < np - 1) ? off[R - 1 - pr] : -1;
        const int n = t.n, k = n / 4;
        t.inv = (unsigned)((0x100000000ull + n - 1) / n);
        if (!rootOff.count(n)) {
            rootOff[n] = (long long)roots.size();
            for (int q = 0; q < 2 * n; ++q) {
                const double a = M_PI * (double)q / (double)n;
                roots.push_back(make_double2(std::cos(a), std::sin(a)));
            }
        }
        t.rootOff = rootOff[n];
        t.vOff = 0;
        t.cOff = 0;
        t.kind = ring_kind(n, &t.logF);
        if (t.kind == RING_SHORT) continue;
        logmax = std::max(logmax, t.logF);
        const int N = 1 << t.logF, nt = N / 16;
        exmax = std::max(exmax, N * std::min(4, RING_CTA / nt));
        if (t.kind == RING_BLUESTEIN) {
            if (!vOff.count(k)) {
                vOff[k] = (long long)Vtab.size();
                std::vector<double2> v(N, make_double2(0.0, 0.0));
                for (long long j = 0; j < k; ++j) {
                    const long long e = (j * j) % (2LL * k);
                    const double a = M_PI * (double)e / (double)k;  // conj(c_j) = e^{+i pi j^2 / k}
                    v[j] = make_double2(std::cos(a), std::sin(a));
                    if (j > 0) v[N - j] = v[j];
                }
                host_fft(v);
                // in the order the forward transform leaves the frequencies in, 1/N folded in
                for (int e = 0; e < 16; ++e)
                    for (int th = 0; th < nt; ++th) Vtab.push_back(cscale(v[fft_index(t.logF, th, e)], 1.0 / (double)N));
                cOff[k] = (long long)chirp.size();
                for (long long j = 0; j < k; ++j) {  // c_j = e^{-i pi j^2 / k}, j^2 reduced mod 2k exactly
                    const double a = -M_PI * (double)((j * j) % (2LL * k)) / (double)k;
                    chirp.push_back(make_double2(std::cos(a), std::sin(a)));
                }
            }
            t.vOff = vOff[k];
            t.cOff = cOff[k];
        }
    }
    // twiddles of every FFT length N = 32 .. 2^logmax: tw[N - 32 + k N/16 + t] = e^{-2 pi i t k / N}
    std::vector<double2> tw(std::max(1, ring_tw_len(logmax)));
    for (int N = 32; N <= 1 << logmax; N *= 2)
        for (int kk = 0; kk < 16; ++kk)
            for (int t = 0; t < N / 16; ++t) {
                const double a = -2.0 * M_PI * (double)(t * kk) / (double)N;
                tw[N - 32 + kk * (N / 16) + t] = make_double2(std::cos(a), std::sin(a));
            }
    if (Vtab.empty()) Vtab.push_back(make_double2(0, 0));
    if (chirp.empty()) chirp.push_back(make_double2(0, 0));
    p->tab.nmax = 4 * nside;
    p->tab.exmax = exmax;
    wf_status st;
    if ((st = plan_alloc(p, (void **)&p->tab.rings, rt.size() * sizeof(RingTab))) != WF_OK) return st;
    if ((st = to_device(p, p->tab.rings, rt.data(), rt.size() * sizeof(RingTab))) != WF_OK) return st;
    const bool f32 = p->prec != WF_PREC_FP64;
    if (f32) {
        if ((st = upload_cx<float>(p, &p->tab.roots, roots)) != WF_OK) return st;
        if ((st = upload_cx<float>(p, &p->tab.V, Vtab)) != WF_OK) return st;
        if ((st = upload_cx<float>(p, &p->tab.chirp, chirp)) != WF_OK) return st;
        if ((st = upload_cx<float>(p, &p->tab.tw, tw)) != WF_OK) return st;
        if ((st = RingLaunch<float>::prepare(p)) != WF_OK) return st;
    } else {
        if ((st = upload_cx<double>(p, &p->tab.roots, roots)) != WF_OK) return st;
        if ((st = upload_cx<double>(p, &p->tab.V, Vtab)) != WF_OK) return st;
        if ((st = upload_cx<double>(p, &p->tab.chirp, chirp)) != WF_OK) return st;
        if ((st = upload_cx<double>(p, &p->tab.tw, tw)) != WF_OK) return st;
        if ((st = RingLaunch<double>::prepare(p)) != WF_OK) return st;
    }
    // pairs by decreasing cost (two FFTs of N per Bluestein sub-DFT): the grid hands them out in
    // this order, so the launch ends on its cheapest pairs
    std::vector<int> order(np);
    std::vector<double> cost(np);
    for (int i = 0; i < np; ++i) {
        order[i] = i;
        const RingTab &t = rt[i];
        const double F = 4.0 * (double)(1LL << t.logF) * (t.logF + 2);
        cost[i] = (t.kind == RING_BLUESTEIN ? 2.0 : 1.0) * F + 8.0 * t.n + 4.0 * p->lmax;
    }
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return cost[x] > cost[y]; });
    if ((st = plan_alloc(p, (void **)&p->tab.order, np * sizeof(int))) != WF_OK) return st;
    return to_device(p, p->tab.order, order.data(), np * sizeof(int));
}

wf_status hp_ring_synthesis(wf_plan p, int L, RingSynMode mode, double lam, double tau, double *out_map)
{
    return p->prec == WF_PREC_FP64 ? RingLaunch<double>::syn(p, L, mode, lam, tau, out_map)
                                   : RingLaunch<float>::syn(p, L, mode, lam, tau, out_map);
}

wf_status hp_ring_synthesis_analysis(wf_plan p, int L, double lam, double tau, const EpiArgs &epi)
{
    return p->prec == WF_PREC_FP64 ? RingLaunch<double>::syn_ana(p, L, lam, tau, epi)
                                   : RingLaunch<float>::syn_ana(p, L, lam, tau, epi);
}

wf_status hp_ring_synthesis_buf(wf_plan p, int L, RingSynMode mode, double lam, double tau, const void *G,
                                void *tmap, double *out_map)
{
    return p->prec == WF_PREC_FP64 ? RingLaunch<double>::syn_buf(p, L, mode, lam, tau, G, tmap, out_map)
                                   : RingLaunch<float>::syn_buf(p, L, mode, lam, tau, G, tmap, out_map);
}

wf_status hp_ring_synthesis_buf_low(wf_plan p, int L, RingSynMode mode, double lam, double tau, const void *G,
                                    const float2 *glow, int lc, int glow_stride, void *tmap, double *out_map)
{
    if (p->prec == WF_PREC_FP64) return set_error(WF_EINVAL, "FP64 plans have no FP64 block");
    return RingLaunch<float>::syn_buf_low(p, L, mode, lam, tau, G, glow, lc, glow_stride, tmap, out_map);
}

wf_status hp_ring_analysis_buf(wf_plan p, int L, const void *map_T, void *F)
{
    return p->prec == WF_PREC_FP64 ? RingLaunch<double>::ana_buf(p, L, map_T, F)
                                   : RingLaunch<float>::ana_buf(p, L, map_T, F);
}

wf_status hp_ring_analysis(wf_plan p, int L, const void *map_T)
{
    return p->prec == WF_PREC_FP64 ? RingLaunch<double>::ana(p, L, map_T) : RingLaunch<float>::ana(p, L, map_T);
}

}  // namespace wf
