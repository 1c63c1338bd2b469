// Flat-sky messenger-field Wiener filter on a periodic n x n grid with the
// unitary 2-D DFT (the "e.g. Fourier space" basis of Sect. 2.1).
//
// The whole solve -- every iteration of Eqs. (3)-(4), the chi^2 of Eq. (6),
// the residual and the cooling schedule -- runs in ONE cooperative launch of
// n/2 + 1 CTAs of n threads.  CTA c owns spectrum column kx = c and (c < n/2)
// the pixel rows 2c, 2c + 1; thread t keeps one mode (a, and the factors of
// Eq. 4) and two pixels (r, nu, the factors of Eq. 3) in registers for the whole
// solve.  One iteration:
//   1. inverse FFT (ky) of the column, written to global memory (L2)
//   2. grid barrier; every CTA sums all CTAs' partials of the previous iteration in
//      the same order and takes the same schedule decision; inverse FFT of its
//      two rows (packed, below), the pixel blend of Eq. (3), forward FFT
//   3. grid barrier; forward FFT (ky) of the column, the harmonic blend of Eq. (4)
//      with its chi^2 and lambda = 1 residual sums.
// Two real rows go through one complex FFT: the inverse DFT of Xa + i Xb (both
// Hermitian) is xa + i xb, and the forward DFT Z of ta + i tb gives
// Ta = (Z_k + conj Z_-k) / 2 and Tb = (Z_k - conj Z_-k) / 2i.
//
// What bounds it: FP64 runs at 1/64 of the FP32 rate (two lanes per clock and SM), so an
// iteration wants many SMs: one FFT per SM, one value per thread, 32 FP64 operations per
// thread and FFT.  The
// rest is two grid barriers and their exchanges through L2.  A cluster of 16 CTAs (the
// largest) with four to five FFTs each in one warp took 42.5 us per iteration of the
// 128 x 128 grid, 18 to 21 us of it FP64 issue, three cluster barriers;
// this kernel takes 14.2 us (4.25 ms for 300 iterations against 12.6), and 11.3 against 18.5 us on
// the 32 x 32 grid, where both are bound by the barriers.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <vector>

#include "wf_internal.cuh"

namespace wf {

constexpr int FLAT_MAXN = 128;
constexpr int FLAT_NP = 2;  // partial sums per CTA: chi^2, residual^2

struct FlatStatus {
    int iters, converged, levels, stop_reason;  // 0 schedule/replay end, 1 converged, 2 maxiter, 3 diverged, 4 barrier gave up
    double final_resid, chi2_final, bnorm;
};

struct FlatPlan {
    int n = 0, nh = 0;
    double *r = nullptr, *nu = nullptr;  // device pixel maps
    double2 *xch = nullptr;              // FlatScratch of the launch
    double *levels = nullptr;            // device lambda levels
    double *tr_lam = nullptr, *tr_chi2 = nullptr, *tr_res = nullptr;
    int tr_cap = 0;
    FlatStatus *status = nullptr;
    double *replay = nullptr;
    int replay_cap = 0;
};

namespace {

// exchange buffers (column layout, [kx][y]), two generations of partial sums, barrier counter
inline size_t flat_scratch_bytes(int n)
{
    const size_t nh = n / 2 + 1;
    return 2 * nh * n * sizeof(double2) + 2 * nh * FLAT_NP * sizeof(double) + 256;
}

struct FlatArgs {
    int n, nh;
    const double *r, *nu, *S;
    const double *g1;      // fluct: unit draws in pixel space (or null)
    const double2 *g2;     // fluct: unit harmonic draws (or null)
    const double *levels;
    int nlevels;
    const double *replay;  // lambda per iteration (or null)
    int nreplay;
    double tau, sigma, eta, tol;
    int level_cap, maxiter;
    double *s_out;
    double2 *alm_out;
    double *tr_lam, *tr_chi2, *tr_res;
    int tr_cap;
    FlatStatus *status;
    double2 *x1, *x2;      // columns after step 1, row spectra after step 2
    double *part;
    unsigned *bar;         // zero at launch
};

void flat_set_scratch(FlatArgs &A, void *base, int n)
{
    const size_t nh = n / 2 + 1;
    A.x1 = (double2 *)base;
    A.x2 = A.x1 + nh * n;
    A.part = (double *)(A.x2 + nh * n);
    A.bar = (unsigned *)(A.part + 2 * nh * FLAT_NP);
}

__device__ __forceinline__ double flip(double v, bool neg)
{
    return __hiloint2double(__double2hiint(v) ^ (neg ? 0x80000000 : 0), __double2loint(v));
}

// FFT of length n = 2^logn over the CTA's first n threads, one value per thread, natural order in
// and out (Stockham, decimation in frequency: radix 4, a last radix 2 where logn is odd; thread t
// computes output t of every pass, six additions and one twiddle product).  sign -1:
// e^{-2 pi i jk/n}, +1: conjugated.  buf: 2 n entries, used alternately, so one barrier a pass.
__device__ double2 cta_fft(double2 v, int n, int sign, double2 *buf, const double2 *tw /* e^{-2 pi i j / n} */)
{
    const int t = threadIdx.x;
    int s = 1, nc = n;  // stride, remaining length
    double2 *cur = buf, *nxt = buf + n;
    while (nc > 1) {
        if (t < n) cur[t] = v;
        __syncthreads();
        if (t < n) {
            const int q = t & (s - 1), u = t / s;
            if (nc == 2) {
                const double2 x0 = cur[q], x1 = cur[q + s];
                v = make_double2(x0.x + flip(x1.x, u & 1), x0.y + flip(x1.y, u & 1));
            } else {
                const int m = nc >> 2, r = u & 3, p = u >> 2, i0 = q + s * p, st = s * m;
                const double2 x0 = cur[i0], x1 = cur[i0 + st], x2 = cur[i0 + 2 * st], x3 = cur[i0 + 3 * st];
                const bool odd = r & 1;
                const double ax = x0.x + flip(x2.x, odd), ay = x0.y + flip(x2.y, odd);
                const double bx = x1.x + flip(x3.x, odd), by = x1.y + flip(x3.y, odd);
                // b (sign i)^r: r = 2 negates; r odd swaps, one part negated
                const bool pos = sign > 0;
                const double rx = odd ? flip(by, (r == 1) == pos) : flip(bx, r == 2);
                const double ry = odd ? flip(bx, (r == 3) == pos) : flip(by, r == 2);
                v = make_double2(ax + rx, ay + ry);
                if (m > 1) {
                    double2 w = tw[p * r * s];
                    w.y = flip(w.y, pos);
                    v = cmul(v, w);
                }
            }
        }
        const int R = nc == 2 ? 2 : 4;
        s *= R;
        nc /= R;
        double2 *x = cur;
        cur = nxt;
        nxt = x;
    }
    __syncthreads();  // the buffers are free
    return v;
}

// sum over a warp, in every lane (same order always)
__device__ __forceinline__ double warp_sum(double v)
{
    for (int o = 16; o >= 1; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

constexpr int FLAT_MAX_POLLS = 1 << 22;  // seconds; the launch is cooperative, so a barrier takes microseconds

// all CTAs have arrived (and their global writes are visible) when it returns true; false, in every
// thread of the CTA, when the wait gave up
__device__ __forceinline__ bool grid_barrier(unsigned *bar, unsigned target, int *ok)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        // (release and acquire carry the CTA's other threads' accesses through the CTA barriers)
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
        unsigned v = 0;
        int polls = 0;
        do {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
        } while ((int)(v - target) < 0 && ++polls < FLAT_MAX_POLLS);  // (the count may wrap)
        *ok = (int)(v - target) >= 0;
    }
    __syncthreads();
    return *ok != 0;
}

__global__ void __launch_bounds__(FLAT_MAXN) k_flat_solve(const FlatArgs A)
{
    __shared__ double2 buf[2 * FLAT_MAXN], tw[FLAT_MAXN];
    __shared__ double red[FLAT_MAXN / 32][FLAT_NP];
    __shared__ int ok;
    const int n = A.n, nh = A.nh, c = blockIdx.x, t = threadIdx.x;
    const bool mode = t < n, row = mode && c < n / 2;
    const int ya = 2 * c, yb = 2 * c + 1;
    const double inv_tau = 1.0 / A.tau, dn = (double)n, wk = (c == 0 || 2 * c == n) ? 1.0 : 2.0;
    const double wkn = wk * dn * dn;  // weight of a mode's squares, for a over n
    unsigned arrivals = 0;
    for (int i = t; i < n; i += blockDim.x) {
        double sn, cs;
        sincospi(-2.0 * i / n, &sn, &cs);
        tw[i] = make_double2(cs, sn);
    }
    // this thread's mode (ky = t, kx = c); a is kept over n, so that neither FFT needs its 1/n.  The
    // n^2 of the squares stays out of 1 / S, which may be next to the largest FP64 number
    const double S = mode ? A.S[(size_t)t * nh + c] : 0.0;
    const double si = S > 0.0 ? 1.0 / S : 0.0;                         // chi^2
    const double kr = S > 0.0 ? si + inv_tau : 0.0;                    // residual
    double2 a = make_double2(0.0, 0.0);
    double f = 0.0;                                                    // S / (S + lam tau) / (2 n^2)
    // its two pixels (rows ya, yb; x = t)
    double ra = 0.0, rb = 0.0, na = 0.0, nb = 0.0, ia = 1.0, ib = 1.0;  // r, nu, 1 / (1 + (lam - 1) tau nu)
    double la = 0.0, lb = 0.0;                                          // lam tau ia, lam tau ib
    if (row) {
        ra = A.r[(size_t)ya * n + t];
        rb = A.r[(size_t)yb * n + t];
        na = A.nu[(size_t)ya * n + t];
        nb = A.nu[(size_t)yb * n + t];
    }
    __syncthreads();

    auto barrier = [&]() {
        arrivals += gridDim.x;
        return grid_barrier(A.bar, arrivals, &ok);
    };
    // step 1: the column's inverse FFT of v into x1
    auto columns_out = [&](double2 v) {
        v = cta_fft(v, n, +1, buf, tw);
        if (mode) __stcg(A.x1 + (size_t)c * n + t, v);
    };
    // row spectra from x1: this thread's entry of the packed inverse FFT
    auto rows_load = [&]() {
        double2 z = make_double2(0.0, 0.0);
        if (row) {
            const bool up = t >= nh;
            const double2 *x = A.x1 + (size_t)(up ? n - t : t) * n + ya;
            const double2 va = __ldcg(x), vb = __ldcg(x + 1);
            z = make_double2(va.x - flip(vb.y, up), flip(va.y, up) + vb.x);
        }
        return z;
    };
    auto rows_in = [&](double2 z) { return c < n / 2 ? cta_fft(z, n, +1, buf, tw) : z; };
    // rows to x2: twice the forward FFTs of the pixel values ta, tb
    auto rows_out = [&](double ta, double tb) {
        if (c >= n / 2) return;
        const double2 z = cta_fft(make_double2(ta, tb), n, -1, buf, tw);
        if (mode) buf[t] = z;
        __syncthreads();
        if (t < nh) {
            const double2 y = buf[(n - t) & (n - 1)];  // conj Z_-k = (y.x, -y.y)
            double2 *x = A.x2 + (size_t)t * n + ya;
            __stcg(x, make_double2(z.x + y.x, z.y - y.y));
            __stcg(x + 1, make_double2(z.y + y.y, y.x - z.x));
        }
        __syncthreads();
    };
    // column from x2: 2 n times this thread's mode of the pixel values
    auto columns_in = [&]() {
        const double2 v = mode ? __ldcg(A.x2 + (size_t)c * n + t) : make_double2(0.0, 0.0);
        return cta_fft(v, n, -1, buf, tw);
    };
    // partial sums: written before a barrier, read after it; generations alternate.  Every warp
    // adds all CTAs' partials itself.
    auto put_part = [&](int gen, double p0, double p1) {
        p0 = warp_sum(p0);
        p1 = warp_sum(p1);
        if ((t & 31) == 0) {
            red[t >> 5][0] = p0;
            red[t >> 5][1] = p1;
        }
        __syncthreads();
        if (t < FLAT_NP) {
            double q = red[0][t];
            for (int i = 1; i < (int)(blockDim.x >> 5); ++i) q += red[i][t];
            __stcg(A.part + ((size_t)(gen & 1) * nh + c) * FLAT_NP + t, q);
        }
    };
    auto load_part = [&](int gen) {
        double2 q = make_double2(0.0, 0.0);
        const double2 *x = reinterpret_cast<const double2 *>(A.part) + (size_t)(gen & 1) * nh;
        for (int i = t & 31; i < nh; i += 32) {
            const double2 v = __ldcg(x + i);
            q.x += v.x;
            q.y += v.y;
        }
        return q;
    };
    auto gave_up = [&]() {
        if (t == 0) A.status->stop_reason = 4;
    };

    double2 tot;
    // ---- fluctuation source: r = nu^1/2 g1 + F^-1 (S^-1/2 g2) ----
    if (A.g1) {
        double2 v = make_double2(0.0, 0.0);
        if (mode && S > 0.0) v = cscale(A.g2[(size_t)t * nh + c], rsqrt(S) / dn);
        columns_out(v);
        if (!barrier()) return gave_up();
        const double2 s = rows_in(rows_load());
        if (row) {
            ra = sqrt(na) * A.g1[(size_t)ya * n + t] + s.x;
            rb = sqrt(nb) * A.g1[(size_t)yb * n + t] + s.y;
        }
    }
    // ---- prologue: |b| = |F r| ----
    rows_out(ra, rb);
    if (!barrier()) return gave_up();
    {
        const double2 v = cscale(columns_in(), 0.5 / dn);
        const double b2 = S > 0.0 ? wk * (v.x * v.x + v.y * v.y) : 0.0;
        put_part(1, 0.0, b2);
    }

    // ---- iterations ----
    // (the sums of iteration k - 1 are read behind the first barrier of iteration k, which step 1
    // of iteration k does not wait for; k = 0 reads |b|)
    int k = 0, lev = 0, level_iters = 0, have_prev = 0, converged = 0, stop_reason = 0;
    double prev = 0.0, last_res = NAN, best = INFINITY, bnorm = 0.0, lam = NAN, cur_lam = NAN;
    for (;; ++k) {
        columns_out(a);
        if (!barrier()) return gave_up();
        tot = load_part(k + 1);
        const double2 z = rows_load();  // in flight while the schedule is decided
        tot.x = warp_sum(tot.x);
        tot.y = warp_sum(tot.y);
        if (k == 0) {
            bnorm = sqrt(tot.y);
        } else {  // absorb iteration k - 1, which ran at lam
            const double chi2 = tot.x;
            const bool full = lam == 1.0;
            const double resid = full ? sqrt(tot.y) / bnorm : NAN;
            if (c == 0 && t == 0 && k - 1 < A.tr_cap) {
                A.tr_lam[k - 1] = lam;
                A.tr_chi2[k - 1] = chi2;
                A.tr_res[k - 1] = resid;
            }
            if (full) {
                last_res = resid;
                if (!isfinite(resid) || (k > 50 && resid > 1e3 * best)) {
                    stop_reason = 3;
                    break;
                }
                best = fmin(best, resid);
            }
            if (!A.replay) {
                bool advanced = false;
                if (full) {
                    if (resid < A.tol) {
                        converged = 1;
                        stop_reason = 1;
                        break;
                    }
                } else {
                    ++level_iters;
                    const bool plateau = have_prev && fabs(chi2 - prev) < A.eta * A.sigma;
                    if (plateau || level_iters >= A.level_cap) {
                        lev = min(lev + 1, A.nlevels - 1);
                        level_iters = 0;
                        have_prev = 0;
                        advanced = true;
                    }
                }
                if (!advanced) {
                    prev = chi2;
                    have_prev = 1;
                }
            }
        }
        if (A.replay) {
            if (k >= A.nreplay) break;
            lam = A.replay[k];
        } else {
            if (k >= A.maxiter) {
                stop_reason = 2;
                break;
            }
            lam = A.levels[lev];
        }
        const double lt = lam * A.tau;
        if (!(lam == cur_lam)) {  // FP64 divisions once per cooling level, not once per iteration
            const double lm1t = (lam - 1.0) * A.tau;
            ia = 1.0 / (1.0 + lm1t * na);
            ib = 1.0 / (1.0 + lm1t * nb);
            la = lt * ia;
            lb = lt * ib;
            f = S > 0.0 ? S / (S + lt) / (2.0 * dn * dn) : 0.0;
            cur_lam = lam;
        }
        const double2 s = rows_in(z);
        // Eq. 3 and its chi^2 term (nu s^2 - 2 r s) id = -s (e + r) id with e = r - nu s
        const double ea = ra - na * s.x, eb = rb - nb * s.y;
        rows_out(s.x + la * ea, s.y + lb * eb);
        // sums that need no exchange before the second barrier, while its first arrivals wait
        double ch = S > 0.0 ? wkn * ((a.x * a.x + a.y * a.y) * si) : 0.0, rs = 0.0;
        ch -= s.x * ((ea + ra) * ia) + s.y * ((eb + rb) * ib);
        if (!barrier()) return gave_up();
        const double2 th = columns_in();
        if (S > 0.0) {
            const double2 an = cscale(th, f);
            if (lam == 1.0) {
                const double dx = kr * (a.x - an.x), dy = kr * (a.y - an.y);
                rs = wkn * (dx * dx + dy * dy);
            }
            a = an;
        }
        put_part(k, ch, rs);
    }
    if (A.replay && isfinite(last_res) && last_res < A.tol) converged = 1;
    // ---- output: s = F^-1 a (its columns are in x1), chi^2(s, 1) ----
    const double2 s = rows_in(rows_load());
    double pc = wkn * ((a.x * a.x + a.y * a.y) * si);
    if (row) {
        A.s_out[(size_t)ya * n + t] = s.x;
        A.s_out[(size_t)yb * n + t] = s.y;
        const double ea = ra - na * s.x, eb = rb - nb * s.y;
        if (na > 0.0) pc += ea * ea / na;  // nu (d - s)^2
        if (nb > 0.0) pc += eb * eb / nb;
    }
    if (mode && A.alm_out) A.alm_out[(size_t)t * nh + c] = cscale(a, dn);
    put_part(k, pc, 0.0);
    if (!barrier()) return gave_up();
    if (c != 0) return;
    tot = load_part(k);
    tot.x = warp_sum(tot.x);
    if (t == 0) {
        A.status->iters = k;
        A.status->converged = converged;
        A.status->levels = lev + 1;
        A.status->stop_reason = stop_reason;
        A.status->final_resid = last_res;
        A.status->chi2_final = tot.x;
        A.status->bnorm = bnorm;
    }
}

// nu = N^-1 (0 where masked), r = nu d; per CTA the minimum of N and the count over observed
// pixels and whether an input is invalid, combined on the host (one CTA's FP64 divisions took
// 80 us at n = 128)
__global__ void __launch_bounds__(256) k_flat_setup(int npix, const double *__restrict__ d,
                                                    const double *__restrict__ nv, const uint8_t *__restrict__ mask,
                                                    double *__restrict__ r, double *__restrict__ nu,
                                                    double *__restrict__ out /* per CTA [min, count, flag] */)
{
    __shared__ double smin[8], scnt[8], sfl[8];
    double mn = INFINITY, cnt = 0, fl = 0;
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i < npix) {
        const bool obs = mask ? mask[i] != 0 : true;
        double rv = 0.0, nuv = 0.0;
        if (obs) {
            const double N = nv[i], dv = d ? d[i] : 0.0;
            if (!(N > 0.0) || !isfinite(N) || !isfinite(dv)) fl = 1;
            else {
                nuv = 1.0 / N;
                rv = dv / N;
                mn = N;
                cnt = 1;
            }
        }
        r[i] = rv;
        nu[i] = nuv;
    }
    for (int o = 16; o >= 1; o >>= 1) {
        mn = fmin(mn, __shfl_xor_sync(0xffffffffu, mn, o));
        cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
        fl = fmax(fl, __shfl_xor_sync(0xffffffffu, fl, o));
    }
    if ((threadIdx.x & 31) == 0) {
        smin[threadIdx.x >> 5] = mn;
        scnt[threadIdx.x >> 5] = cnt;
        sfl[threadIdx.x >> 5] = fl;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = INFINITY, b = 0, f = 0;
        for (int w = 0; w < 8; ++w) {
            a = fmin(a, smin[w]);
            b += scnt[w];
            f = fmax(f, sfl[w]);
        }
        out[3 * blockIdx.x] = a;
        out[3 * blockIdx.x + 1] = b;
        out[3 * blockIdx.x + 2] = f;
    }
}

constexpr int FLAT_SETUP_CTAS = FLAT_MAXN * FLAT_MAXN / 256;

// launches the setup; h: host, 3 * FLAT_SETUP_CTAS entries, valid after the stream synchronises (tmp: device)
wf_status flat_setup(int n, const double *d, const double *noise_var, const uint8_t *mask, double *r, double *nu,
                     double *tmp, double *h, cudaStream_t stream)
{
    const int npix = n * n, g = (npix + 255) / 256;
    k_flat_setup<<<g, 256, 0, stream>>>(npix, d, noise_var, mask, r, nu, tmp);
    WF_CUDA(cudaGetLastError());
    WF_CUDA(cudaMemcpyAsync(h, tmp, (size_t)3 * g * sizeof(double), cudaMemcpyDeviceToHost, stream));
    return WF_OK;
}

// [min, count, flag] of the whole map into h[0..2]
void flat_setup_combine(int n, double *h)
{
    for (int i = 1; i < (n * n + 255) / 256; ++i) {
        h[0] = std::fmin(h[0], h[3 * i]);
        h[1] += h[3 * i + 1];
        h[2] = std::fmax(h[2], h[3 * i + 2]);
    }
}

// one solve: a cooperative launch of n/2 + 1 CTAs (the barriers need them co-resident)
wf_status flat_launch(const FlatArgs &A, cudaStream_t stream)
{
    WF_CUDA(cudaMemsetAsync(A.bar, 0, sizeof(unsigned), stream));
    WF_CUDA(cudaMemsetAsync(A.status, 0, sizeof(FlatStatus), stream));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(A.nh);
    cfg.blockDim = dim3(std::max(32, A.n));
    cfg.stream = stream;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeCooperative;
    at.val.cooperative = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    WF_CUDA(cudaLaunchKernelEx(&cfg, k_flat_solve, A));
    return WF_OK;
}

wf_status flat_result(const FlatStatus &fs)
{
    if (fs.stop_reason == 4) return set_error(WF_ETIMEOUT, "a bounded wait at a grid barrier gave up");
    if (fs.stop_reason == 3) return set_error(WF_EDIVERGE, "residual grew (%.3e)", fs.final_resid);
    if (fs.stop_reason == 2) return set_error(WF_ENOCONV, "iteration cap reached (residual %.3e)", fs.final_resid);
    return WF_OK;
}

}  // namespace

wf_status flat_create(wf_plan p)
{
    const int n = p->g.nx;
    if (p->g.ny != n) return set_error(WF_EUNSUPPORTED, "flat grid must be square");
    if (n < 16 || n > FLAT_MAXN || (n & (n - 1))) return set_error(WF_EUNSUPPORTED, "flat n must be a power of two in [16, 128]");
    FlatPlan *f = new (std::nothrow) FlatPlan();
    if (!f) return set_error(WF_ENOMEM, "host allocation");
    p->flat = f;
    f->n = n;
    f->nh = n / 2 + 1;
    p->npix = (long long)n * n;
    p->nalm = (long long)n * f->nh;
    p->omega = 1.0;
    wf_status st;
    if ((st = plan_alloc(p, (void **)&f->r, p->npix * 8)) != WF_OK) return st;
    if ((st = plan_alloc(p, (void **)&f->nu, p->npix * 8)) != WF_OK) return st;
    if ((st = plan_alloc(p, (void **)&f->levels, 64 * 8)) != WF_OK) return st;
    if ((st = plan_alloc(p, (void **)&f->status, sizeof(FlatStatus))) != WF_OK) return st;
    if ((st = plan_alloc(p, (void **)&f->xch, flat_scratch_bytes(n))) != WF_OK) return st;
    return WF_OK;
}

void flat_destroy(wf_plan p)
{
    delete p->flat;
    p->flat = nullptr;
}

static wf_status ensure_trace(wf_plan p, int cap)
{
    FlatPlan *f = p->flat;
    if (f->tr_cap >= cap) return WF_OK;
    wf_status st;
    if ((st = plan_alloc(p, (void **)&f->tr_lam, (size_t)cap * 8)) != WF_OK) return st;
    if ((st = plan_alloc(p, (void **)&f->tr_chi2, (size_t)cap * 8)) != WF_OK) return st;
    if ((st = plan_alloc(p, (void **)&f->tr_res, (size_t)cap * 8)) != WF_OK) return st;
    f->tr_cap = cap;
    return WF_OK;
}

wf_status flat_solve(wf_plan p, const double *d, const double *noise_var, const uint8_t *mask, const double *S,
                     double tol, bool fluct, const double *g1, const double *g2, double *s_out, double *alm_out,
                     wf_info *info)
{
    FlatPlan *f = p->flat;
    const wf_options o = [&] {
        wf_options q = p->opt;
        if (q.maxiter <= 0) q.maxiter = 20000;
        if (q.level_cap <= 0) q.level_cap = 200;
        if (!(q.eta > 0)) q.eta = 1e-2;
        if (!(q.lambda_max > 0)) q.lambda_max = 100.0;
        return q;
    }();
    const int n = f->n, nh = f->nh;
    Prof pr(p, info, p->opt.profile != 0);
    double h[3 * FLAT_SETUP_CTAS];
    if (wf_status ls = flat_setup(n, fluct ? nullptr : d, noise_var, mask, f->r, f->nu, (double *)f->xch, h, p->stream))
        return ls;
    WF_COUNT_LAUNCH(p);
    WF_CUDA(cudaStreamSynchronize(p->stream));
    flat_setup_combine(n, h);
    if (h[2] != 0.0) return set_error(WF_EINVAL, "noise variance must be finite and > 0 (and d finite) on observed pixels");
    if (h[1] == 0.0) return set_error(WF_EINVAL, "every pixel is masked");
    const double tau = h[0];
    const long long ndof = (long long)h[1];

    // lambda levels: k_iter = 1, 2, 4, ...; lambda = clip(max S on |k| = k_iter / tau, 1, lambda_max)
    std::vector<double> Sh((size_t)n * nh);
    wf_status st = to_host(p, Sh.data(), S, Sh.size() * 8);
    if (st != WF_OK) return st;
    for (size_t i = 0; i < Sh.size(); ++i)
        if (!(Sh[i] >= 0.0 && std::isfinite(Sh[i])))
            return set_error(WF_EINVAL, "the prior S must be finite and >= 0 (mode %zu: %g)", i, Sh[i]);
    std::vector<double> lev{o.lambda_max};
    int kmax = 0;
    std::vector<int> kr(Sh.size());
    for (int ky = 0; ky < n; ++ky)
        for (int kx = 0; kx < nh; ++kx) {
            const int sy = ky < (n + 1) / 2 ? ky : ky - n;
            const int r = (int)std::lrint(std::sqrt((double)sy * sy + (double)kx * kx));
            kr[(size_t)ky * nh + kx] = r;
            kmax = std::max(kmax, r);
        }
    for (int kit = 2; lev.back() != 1.0; kit *= 2) {
        double lam = 1.0;
        if (kit <= kmax) {
            double smax = -1.0;
            for (size_t i = 0; i < Sh.size(); ++i)
                if (kr[i] == kit) smax = std::max(smax, Sh[i]);
            if (smax >= 0.0) lam = std::min(o.lambda_max, std::max(1.0, smax / tau));
        }
        if (lam != lev.back()) lev.push_back(lam);
        if ((int)lev.size() >= 60) { lev.push_back(1.0); break; }
    }
    WF_CUDA(cudaMemcpyAsync(f->levels, lev.data(), lev.size() * 8, cudaMemcpyHostToDevice, p->stream));
    const bool replay = !p->replay_lambda.empty();
    const int nrep = (int)p->replay_lambda.size();
    if (replay && nrep > f->replay_cap) {
        wf_status st = plan_alloc(p, (void **)&f->replay, (size_t)nrep * 8);
        if (st != WF_OK) return st;
        f->replay_cap = nrep;
    }
    if (replay)
        WF_CUDA(cudaMemcpyAsync(f->replay, p->replay_lambda.data(), nrep * 8, cudaMemcpyHostToDevice, p->stream));
    const int cap = replay ? nrep : o.maxiter;
    st = ensure_trace(p, std::max(cap, 1));
    if (st != WF_OK) return st;

    FlatArgs A{};
    A.n = n;
    A.nh = nh;
    flat_set_scratch(A, f->xch, n);
    A.r = f->r;
    A.nu = f->nu;
    A.S = S;
    A.g1 = fluct ? g1 : nullptr;
    A.g2 = fluct ? (const double2 *)g2 : nullptr;
    A.levels = f->levels;
    A.nlevels = (int)lev.size();
    A.replay = replay ? f->replay : nullptr;
    A.nreplay = nrep;
    A.tau = tau;
    A.sigma = std::sqrt(2.0 * (double)ndof);
    A.eta = o.eta;
    A.tol = tol;
    A.level_cap = o.level_cap;
    A.maxiter = o.maxiter;
    A.s_out = s_out;
    A.alm_out = (double2 *)alm_out;
    A.tr_lam = f->tr_lam;
    A.tr_chi2 = f->tr_chi2;
    A.tr_res = f->tr_res;
    A.tr_cap = f->tr_cap;
    A.status = f->status;
    pr.begin(WF_K_FLAT);
    if (wf_status ls = flat_launch(A, p->stream)) return ls;
    WF_COUNT_LAUNCH(p);
    pr.end();
    FlatStatus fs;
    WF_CUDA(cudaMemcpyAsync(&fs, f->status, sizeof fs, cudaMemcpyDeviceToHost, p->stream));
    WF_CUDA(cudaStreamSynchronize(p->stream));
    pr.collect();
    pr.finish();
    if (info) {
        info->iters = fs.iters;
        info->converged = fs.converged;
        info->final_residual = fs.final_resid;
        info->chi2_over_ndof = fluct ? NAN : fs.chi2_final / (double)ndof;
        info->n_dof = ndof;
        info->tau = tau;
        info->n_levels = fs.levels;
        info->refine_sweeps = 0;
        const int nt = std::min(fs.iters, info->trace_cap);
        if (nt > 0) {
            std::vector<double> tl(nt), tc(nt), trs(nt);
            if ((st = to_host(p, tl.data(), f->tr_lam, nt * 8)) != WF_OK) return st;
            if ((st = to_host(p, tc.data(), f->tr_chi2, nt * 8)) != WF_OK) return st;
            if ((st = to_host(p, trs.data(), f->tr_res, nt * 8)) != WF_OK) return st;
            for (int i = 0; i < nt; ++i) {
                if (info->lambda_trace) info->lambda_trace[i] = tl[i];
                if (info->L_trace) info->L_trace[i] = -1;
                if (info->chi2_trace) info->chi2_trace[i] = tc[i];
                if (info->resid_trace) info->resid_trace[i] = trs[i];
            }
        }
    }
    return flat_result(fs);
}

wf_status flat_alm2map(wf_plan p, const double *alm, double *map)
{
    return set_error(WF_EUNSUPPORTED, "flat-grid basis change is internal to the fused solve");
}

wf_status flat_map2alm(wf_plan p, const double *map, double *alm)
{
    return set_error(WF_EUNSUPPORTED, "flat-grid basis change is internal to the fused solve");
}

// ---------------------------------------------------------------------------
// Flat-grid solve that allocates nothing (wf_flat_solve_noalloc).
//
// For callers that cannot allocate device memory at solve time -- code that
// runs inside another framework's memory pool (a cudaMalloc there would go
// around the pool's accounting), or on a context where allocation is locked
// down -- this entry point runs the same two kernels as wf_solve on the flat grid
// (k_flat_setup, k_flat_solve), with the solver's scratch (the source and
// inverse-noise maps, the lambda levels, the status block and the per-
// iteration traces) in one file-scope device array instead of plan memory.
// Limits: n <= 128 (a power of two >= 16) and at most 20000 iterations;
// the array is 0.97 MiB and stays resident on every device that loads the
// library.  In host code the array's symbol is not a device address: every
// call looks up its address on the current device with cudaGetSymbolAddress,
// so no address outlives the context it belongs to (a cudaDeviceReset between
// calls is safe).  All calls share the one array: calls that overlap on the
// GPU race; everything a call reads is written by that call first.  The prior
// S must be finite and >= 0 (the largest S per radius is taken as an integer
// maximum over the bit patterns, an order that holds for S >= 0 only).
// ---------------------------------------------------------------------------
namespace {
constexpr int NOALLOC_MAXN = 128;
constexpr int NOALLOC_MAXITER = 20000;
constexpr int NOALLOC_LEVELS = 64;
constexpr size_t NA_PIX = (size_t)NOALLOC_MAXN * NOALLOC_MAXN;
constexpr size_t NA_R = 0;
constexpr size_t NA_NU = NA_R + NA_PIX * sizeof(double);
constexpr size_t NA_LEV = NA_NU + NA_PIX * sizeof(double);
constexpr size_t NA_RAD = NA_LEV + NOALLOC_LEVELS * sizeof(double);
constexpr size_t NA_STATUS = NA_RAD + 32 * sizeof(double);
constexpr size_t NA_TRACE = NA_STATUS + 256;
constexpr size_t NA_XCH = NA_TRACE + 3 * (size_t)NOALLOC_MAXITER * sizeof(double);
constexpr size_t NA_BYTES = NA_XCH + 2 * (NOALLOC_MAXN / 2 + 1) * (size_t)NOALLOC_MAXN * sizeof(double2) +
                            2 * (NOALLOC_MAXN / 2 + 1) * (size_t)FLAT_NP * sizeof(double) + 256;

// max S over the half-plane modes whose rounded |k| equals 2^j, j = 1..15
// (-1 where no mode has that radius): the priors the flat schedule needs.
// out[16] counts the modes whose S is not finite and >= 0 (rejected by the
// caller: the maximum below compares bit patterns, valid for S >= 0 only).
__global__ void k_flat_radial_max(int n, const double *__restrict__ S, double *__restrict__ out)
{
    __shared__ unsigned long long best[16];
    __shared__ unsigned int bad;
    if (threadIdx.x < 16) best[threadIdx.x] = 0ull;
    if (threadIdx.x == 0) bad = 0u;
    __syncthreads();
    const int nh = n / 2 + 1;
    for (int i = threadIdx.x; i < n * nh; i += blockDim.x) {
        if (!(S[i] >= 0.0 && isfinite(S[i]))) {
            atomicAdd(&bad, 1u);
            continue;
        }
        const int ky = i / nh, kx = i % nh;
        const int sy = ky < (n + 1) / 2 ? ky : ky - n;
        const long r = lrint(sqrt((double)sy * sy + (double)kx * kx));
        if (r >= 2 && (r & (r - 1)) == 0) {
            int j = 0;
            while ((1L << j) < r) ++j;
            if (j < 16) atomicMax(&best[j], (unsigned long long)__double_as_longlong(S[i]) | 0ull);
        }
    }
    __syncthreads();
    if (threadIdx.x < 16) {
        const unsigned long long b = best[threadIdx.x];
        out[threadIdx.x] = b ? __longlong_as_double((long long)b) : -1.0;
    }
    if (threadIdx.x == 0) out[16] = (double)bad;
}
}  // namespace

static __device__ __align__(256) unsigned char g_flat_noalloc_scratch[NA_BYTES];

namespace {
wf_status noalloc_base(unsigned char **out)
{
    void *p = nullptr;
    WF_CUDA(cudaGetSymbolAddress(&p, g_flat_noalloc_scratch));
    *out = (unsigned char *)p;
    return WF_OK;
}
}  // namespace

}  // namespace wf

extern "C" wf_status wf_flat_solve_noalloc(int n, const double *d, const double *noise_var, const uint8_t *mask,
                                           const double *S, double tol, const wf_options *opt, void *cuda_stream,
                                           double *s_wf, double *alm_out, wf_info *info)
{
    using namespace wf;
    if (!d || !noise_var || !S || !s_wf) return set_error(WF_EINVAL, "null argument");
    if (n < 16 || n > NOALLOC_MAXN || (n & (n - 1)))
        return set_error(WF_EINVAL, "wf_flat_solve_noalloc: n must be a power of two in [16, %d] (got %d)",
                         NOALLOC_MAXN, n);
    if (!(tol > 0)) return set_error(WF_EINVAL, "tol must be > 0");
    wf_options o = opt ? *opt : wf_options{};
    if (o.maxiter <= 0) o.maxiter = NOALLOC_MAXITER;
    if (o.maxiter > NOALLOC_MAXITER)
        return set_error(WF_EINVAL, "wf_flat_solve_noalloc: maxiter %d exceeds the %d iterations its scratch holds",
                         o.maxiter, NOALLOC_MAXITER);
    if (o.level_cap <= 0) o.level_cap = 200;
    if (!(o.eta > 0)) o.eta = 1e-2;
    if (!(o.lambda_max > 0)) o.lambda_max = 100.0;
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    unsigned char *base = nullptr;
    wf_status st = noalloc_base(&base);
    if (st != WF_OK) return st;
    double *r = (double *)(base + NA_R), *nu = (double *)(base + NA_NU), *lev_d = (double *)(base + NA_LEV);
    double *rad = (double *)(base + NA_RAD);
    FlatStatus *status = (FlatStatus *)(base + NA_STATUS);
    double *tr = (double *)(base + NA_TRACE);
    const int nh = n / 2 + 1;

    double h[3 * FLAT_SETUP_CTAS], smax[17];
    if (wf_status ls = flat_setup(n, d, noise_var, mask, r, nu, (double *)(base + NA_XCH), h, stream)) return ls;
    k_flat_radial_max<<<1, 256, 0, stream>>>(n, S, rad);
    WF_CUDA(cudaGetLastError());
    WF_CUDA(cudaMemcpyAsync(smax, rad, sizeof smax, cudaMemcpyDeviceToHost, stream));
    WF_CUDA(cudaStreamSynchronize(stream));
    flat_setup_combine(n, h);
    if (h[2] != 0.0) return set_error(WF_EINVAL, "noise variance must be finite and > 0 (and d finite) on observed pixels");
    if (h[1] == 0.0) return set_error(WF_EINVAL, "every pixel is masked");
    if (smax[16] != 0.0)
        return set_error(WF_EINVAL, "the prior S must be finite and >= 0 (%.0f modes are not)", smax[16]);
    const double tau = h[0];
    const long long ndof = (long long)h[1];

    // lambda levels of the flat schedule: k_iter = 1, 2, 4, ..., first level at lambda_max
    double lev[NOALLOC_LEVELS];
    int nlev = 0;
    lev[nlev++] = o.lambda_max;
    for (int j = 1; lev[nlev - 1] != 1.0 && nlev < NOALLOC_LEVELS - 1; ++j) {
        double lam = 1.0;
        if (j < 16 && smax[j] >= 0.0) lam = std::min(o.lambda_max, std::max(1.0, smax[j] / tau));
        if (j >= 16) lam = 1.0;
        if (lam != lev[nlev - 1]) lev[nlev++] = lam;
    }
    if (lev[nlev - 1] != 1.0) lev[nlev++] = 1.0;
    WF_CUDA(cudaMemcpyAsync(lev_d, lev, nlev * sizeof(double), cudaMemcpyHostToDevice, stream));

    FlatArgs A{};
    A.n = n;
    A.nh = nh;
    flat_set_scratch(A, base + NA_XCH, n);
    A.r = r;
    A.nu = nu;
    A.S = S;
    A.levels = lev_d;
    A.nlevels = nlev;
    A.tau = tau;
    A.sigma = std::sqrt(2.0 * (double)ndof);
    A.eta = o.eta;
    A.tol = tol;
    A.level_cap = o.level_cap;
    A.maxiter = o.maxiter;
    A.s_out = s_wf;
    A.alm_out = (double2 *)alm_out;
    A.tr_lam = tr;
    A.tr_chi2 = tr + NOALLOC_MAXITER;
    A.tr_res = tr + 2 * NOALLOC_MAXITER;
    A.tr_cap = NOALLOC_MAXITER;
    A.status = status;
    if (wf_status ls = flat_launch(A, stream)) return ls;
    FlatStatus fs;
    WF_CUDA(cudaMemcpyAsync(&fs, status, sizeof fs, cudaMemcpyDeviceToHost, stream));
    WF_CUDA(cudaStreamSynchronize(stream));
    if (info) {
        info->iters = fs.iters;
        info->converged = fs.converged;
        info->final_residual = fs.final_resid;
        info->chi2_over_ndof = fs.chi2_final / (double)ndof;
        info->n_dof = ndof;
        info->tau = tau;
        info->n_levels = fs.levels;
        info->refine_sweeps = 0;
        info->mixed_lc = 0;
        info->launches = 3;
        const int nt = std::min(fs.iters, info->trace_cap);
        if (nt > 0) {
            // ordered on the caller's stream like every other copy of this call
            if (info->lambda_trace)
                WF_CUDA(cudaMemcpyAsync(info->lambda_trace, A.tr_lam, nt * 8, cudaMemcpyDeviceToHost, stream));
            if (info->chi2_trace)
                WF_CUDA(cudaMemcpyAsync(info->chi2_trace, A.tr_chi2, nt * 8, cudaMemcpyDeviceToHost, stream));
            if (info->resid_trace)
                WF_CUDA(cudaMemcpyAsync(info->resid_trace, A.tr_res, nt * 8, cudaMemcpyDeviceToHost, stream));
            WF_CUDA(cudaStreamSynchronize(stream));
            if (info->L_trace)
                for (int i = 0; i < nt; ++i) info->L_trace[i] = -1;
        }
    }
    return flat_result(fs);
}
