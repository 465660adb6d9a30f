// Harmonic synthesis of a band-limited HEALPix map on the GPU: the unlensed
// input of the remap (Sec. 3.2 draws it from C_l and synthesises it; Table 2
// counts that transform in the total time).  Spin s = 0, 1, 2:
//
//   spin 0:  T(theta, phi) = sum_{l,m} a_lm sY_lm,
//   spin s:  P = -sum_{l,m} (E + iB)_lm sY_lm  (P = Q + iU for s = 2; for s = 1
//            with E_lm = sqrt(l(l+1)) phi_lm it is the gradient d_theta + i d_phi),
//
// with sY_lm(theta, phi) = (-1)^s N_l e^{i m phi} d^l_{m,-s}(theta),
// N_l = sqrt((2l+1)/(4 pi)) (Appendix A), and real E, B fields
// (a_{l,-m} = (-1)^m a_lm^*).  Per ring the sum over l gives coefficients
//
//   spin 0:  F_m = sum_l a_lm N_l d^l_{m,0}                       (m >= 0),
//   spin s:  P_m  = -(-1)^s sum_l (E + iB)_lm N_l d^l_{m,-s},
//            P_-m = -sum_l (E^* + iB^*)_lm N_l d^l_{m,s}            (m >= 1),
//
// and the ring values are the Fourier sums sum_m F_m e^{i m phi_j}, done by
// folding m modulo the ring length n and an inverse DFT of length n.  The
// 2 Nside + 1 equatorial rings (n = 4 Nside) share one batched cuFFT plan.
// The polar rings (n = 4i, i < Nside) use Bluestein's algorithm: with
// w_t = exp(i pi t^2 / n), x_j = sum_k H_k e^{2 pi i jk/n} = w_j (a * b)_j for
// a_k = H_k w_k and b_t = conj(w_t), a linear convolution done with FFTs of
// a power-of-two length M >= 2n - 1; the transforms of b are tabulated per
// ring size at plan time, and the rings of equal M share one batched plan, so
// a plan holds at most 14 cuFFT plans whatever Nside.
//
// The l-sums use the Wigner-d three-term recurrence in l at fixed (m, m'):
//   d^{l+1} = (A_l x - B_l) d^l - C_l d^{l-1},  A_l = (2l+1) l (l+1) / D_l,
//   B_l = (2l+1) m m' / D_l,  C_l = (l+1) sqrt((l^2-m^2)(l^2-m'^2)) / D_l,
//   D_l = l sqrt(((l+1)^2-m^2)((l+1)^2-m'^2)),  x = cos(theta),
// started at l0 = max(m, |m'|) from the closed form
//   d^l_{l,b} = (-1)^{l-b} sqrt((2l)! / ((l+b)!(l-b)!)) c^{l+b} s^{l-b},
//   d^l_{-l,b} = sqrt((2l)! / ((l+b)!(l-b)!)) c^{l-b} s^{l+b}   (c, s = cos, sin theta/2)
// with d^l_{m,m'} = d^l_{-m',-m} when |m'| > m.  The start is formed in
// base-2 logarithms and carried as v 2^E (E an integer, raised in steps of 256
// while |v| > 2^256), so columns whose start underflows (large m near the
// poles) still reach their oscillatory range.  One thread runs the columns of
// one (ring, m) pair for the northern ring and, through
//   d^l_{m,m'}(pi - theta) = (-1)^{l+m} d^l_{m,-m'}(theta),
// for its southern mirror as well.
#include <cuda_runtime.h>
#include <cufft.h>

#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <vector>

#include "common.cuh"
#include "flints.h"

namespace {

constexpr double PI_D = 3.14159265358979323846;

struct SynthRing {
    double x;          // cos(theta)
    double lc, ls;     // log2 cos(theta/2), log2 sin(theta/2)
    double phi0;       // azimuth of the first pixel / pi
    long long first;   // RING index of the first pixel
    long long off;     // equatorial ring: offset of its FFT input; polar ring: offset of its Bluestein slot
    long long fboff;   // polar ring: offset of the transformed chirp for its size
    int n;             // pixels in the ring
    int M;             // polar ring: Bluestein length (0: equatorial ring)
};

// w_t = exp(i pi t^2 / n), with t^2 reduced modulo 2n (exact in integers)
__device__ __forceinline__ double2 chirp(long long t, int n) {
    const long long q = (t * t) % (2LL * n);
    double sp, cp;
    sincospi((double)q / (double)n, &sp, &cp);
    return make_double2(cp, sp);
}

thread_local char g_msg[512] = "no error";

int sfail(int code, const char *fmt, ...) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_msg, sizeof g_msg, fmt, ap);
    va_end(ap);
    return code;
}

constexpr int CHUNK = 256;  // l values staged per pass in shared memory (FP64 kernel)
constexpr unsigned FULL_WARP = 0xffffffffu;

// Start of a column: d^l0_{m,m'} = (sign) sqrt((2l)! / ((l+b)!(l-b)!)) c^pc s^ps.
__device__ __forceinline__ void start_powers(int m, int mp, int &pc, int &ps, bool &neg) {
    if (m >= abs(mp)) {  // first index +l = m, second b = m'
        pc = m + mp;
        ps = m - mp;
        neg = ((m - mp) & 1) != 0;
    } else if (mp < 0) {  // d_{m,m'} = d_{-m',-m}: first index -m' = +l, b = -m
        pc = -mp - m;
        ps = -mp + m;
        neg = ((m - mp) & 1) != 0;
    } else {  // first index -m' = -l, b = -m
        pc = mp + m;
        ps = mp - m;
        neg = false;
    }
}

// log2 of sqrt((2l)! / ((l+b)!(l-b)!)) at l = max(m, s), b = min(m, s)
__device__ __forceinline__ double start_factor(int m, int s) {
    const int l = m > s ? m : s, b = m > s ? s : m;
    const double lf = 0.5 * (lgamma(2.0 * l + 1.0) - lgamma((double)(l + b) + 1.0) - lgamma((double)(l - b) + 1.0));
    return lf * 1.4426950408889634;
}

// One recurrence column carried as v 2^E.
struct Col {
    double v, prev, mult;
    int e;
    __device__ __forceinline__ void init(double lg, bool neg) {
        const double fl = floor(lg);
        e = (int)fl;
        v = exp2(lg - fl);
        if (neg) v = -v;
        prev = 0.0;
        mult = e < -1074 ? 0.0 : ldexp(1.0, e);
    }
    __device__ __forceinline__ void step(double a, double b, double c, double x) {
        const double nv = fma(fma(a, x, -b), v, -c * prev);
        prev = v;
        v = nv;
        if (fabs(v) > 1.157920892373162e77) {  // 2^256
            v *= 8.636168555094445e-78;
            prev *= 8.636168555094445e-78;
            e += 256;
            mult = e < -1074 ? 0.0 : ldexp(1.0, e);
        }
    }
    __device__ __forceinline__ double value() const { return v * mult; }
};

// F layout: spin 0: [ring][m], m = 0..lmax;  spin s: [ring][lmax + m], m = -lmax..lmax.
// Rings are 1..4N-1, stored at index ring-1.  Threads: x = northern ring (1..2N), y = m.
template <int S>
__global__ void __launch_bounds__(128) legendre_kernel(int lmax, int nside, const SynthRing *__restrict__ rings,
                                                       const double2 *__restrict__ alm, const double2 *__restrict__ blm,
                                                       double2 *__restrict__ F) {
    __shared__ double sA[CHUNK], sB[CHUNK], sC[CHUNK];
    __shared__ double2 sWp[CHUNK], sWm[CHUNK];
    const int m = blockIdx.y;
    const int ring = blockIdx.x * blockDim.x + threadIdx.x + 1;  // northern ring incl. the equator
    const int nnorth = 2 * nside;
    const bool active = ring <= nnorth;
    const int NM = S == 0 ? lmax + 1 : 2 * lmax + 1;
    const int l0 = m > S ? m : S;
    const double inv4pi = 1.0 / (4.0 * PI_D);
    SynthRing rg{};
    if (active) rg = rings[ring - 1];
    // columns: A = d_{m,-s}, B = d_{m,+s} (spin 0: A only)
    Col ca{}, cb{};
    if (active && l0 <= lmax) {
        const double lg = start_factor(m, S);
        int pc, ps;
        bool neg;
        start_powers(m, -S, pc, ps, neg);
        ca.init(lg + pc * rg.lc + ps * rg.ls, neg);
        if (S > 0) {
            start_powers(m, S, pc, ps, neg);
            cb.init(lg + pc * rg.lc + ps * rg.ls, neg);
        }
    }
    // accumulators by parity of l + m (e: even, o: odd); the parity is uniform
    // across the block (same l and m), so the branches below do not diverge
    double2 pAe{}, pAo{}, pBe{}, pBo{}, mAe{}, mAo{}, mBe{}, mBo{};
    for (int c0 = l0; c0 <= lmax; c0 += CHUNK) {
        const int c1 = min(c0 + CHUNK, lmax + 1);
        __syncthreads();
        for (int l = c0 + threadIdx.x; l < c1; l += blockDim.x) {
            const int k = l - c0;
            const double ld = (double)l, lp = ld + 1.0;
            const double md = (double)m, sd = (double)S;
            const double den = ld * sqrt((lp * lp - md * md) * (lp * lp - sd * sd));
            if (l == 0 || !(den > 0.0)) {  // l = m = s = 0: d^1 = x d^0
                sA[k] = 1.0;
                sB[k] = 0.0;
                sC[k] = 0.0;
            } else {
                sA[k] = (2.0 * ld + 1.0) * ld * lp / den;
                sB[k] = (2.0 * ld + 1.0) * md * sd / den;  // for m' = +s; m' = -s takes -sB
                sC[k] = lp * sqrt((ld * ld - md * md) * (ld * ld - sd * sd)) / den;
            }
            const double nl = sqrt((2.0 * ld + 1.0) * inv4pi);
            const double2 a = alm[(size_t)l * (lmax + 1) + m];
            if (S == 0) {
                sWp[k] = make_double2(a.x * nl, a.y * nl);
            } else {
                const double2 b = blm ? blm[(size_t)l * (lmax + 1) + m] : make_double2(0.0, 0.0);
                // (E + iB) N and (E^* + iB^*) N
                sWp[k] = make_double2((a.x - b.y) * nl, (a.y + b.x) * nl);
                sWm[k] = make_double2((a.x + b.y) * nl, (b.x - a.y) * nl);
            }
        }
        __syncthreads();
        if (active) {
            for (int l = c0; l < c1; ++l) {
                const int k = l - c0;
                const bool odd = ((l + m) & 1) != 0;
                const double da = ca.value();
                const double2 wp = sWp[k];
                double2 &pa = odd ? pAo : pAe;
                pa.x = fma(wp.x, da, pa.x);
                pa.y = fma(wp.y, da, pa.y);
                if (S > 0) {
                    const double db = cb.value();
                    const double2 wm = sWm[k];
                    double2 &pb = odd ? pBo : pBe;
                    double2 &ma = odd ? mAo : mAe;
                    double2 &mb = odd ? mBo : mBe;
                    pb.x = fma(wp.x, db, pb.x);
                    pb.y = fma(wp.y, db, pb.y);
                    ma.x = fma(wm.x, da, ma.x);
                    ma.y = fma(wm.y, da, ma.y);
                    mb.x = fma(wm.x, db, mb.x);
                    mb.y = fma(wm.y, db, mb.y);
                }
                if (l < lmax) {
                    ca.step(sA[k], -sB[k], sC[k], rg.x);
                    if (S > 0) cb.step(sA[k], sB[k], sC[k], rg.x);
                }
            }
        }
    }
    if (!active) return;
    const int south = 4 * nside - ring;  // mirror ring (== ring at the equator)
    double2 *Fn = F + (size_t)(ring - 1) * NM;
    double2 *Fs = F + (size_t)(south - 1) * NM;
    if (S == 0) {
        Fn[m] = make_double2(pAe.x + pAo.x, pAe.y + pAo.y);
        if (south != ring) Fs[m] = make_double2(pAe.x - pAo.x, pAe.y - pAo.y);
        return;
    }
    // P_m = -(-1)^s sum wp d_{m,-s}; south: d_{m,-s}(pi - t) = (-1)^{l+m} d_{m,s}(t)
    const double sg = (S & 1) ? 1.0 : -1.0;  // -(-1)^s
    Fn[lmax + m] = make_double2(sg * (pAe.x + pAo.x), sg * (pAe.y + pAo.y));
    if (south != ring) Fs[lmax + m] = make_double2(sg * (pBe.x - pBo.x), sg * (pBe.y - pBo.y));
    if (m > 0) {  // P_-m = -sum wm d_{m,s}; south: d_{m,s}(pi - t) = (-1)^{l+m} d_{m,-s}(t)
        Fn[lmax - m] = make_double2(-(mBe.x + mBo.x), -(mBe.y + mBo.y));
        if (south != ring) Fs[lmax - m] = make_double2(-(mAe.x - mAo.x), -(mAe.y - mAo.y));
    }
}

// --------------------------------------------------- the l-sums in fixed point
// The mixed precision of the synthesis.
// Per (ring, m) column the recurrence is run on g_l = d^l / alpha_l with
// alpha_{l+1} = C_l alpha_{l-1} and alpha = 1 at the two largest l, which leaves
//   g_{l+1} = (a_l x -+ b_l) g_l - g_{l-1},   a_l = A_l alpha_l / alpha_{l+1}, b_l likewise:
// alpha falls with l (C_l < 1), so |g| <= |d| <= 1, and one product per column and step is
// gone.  Everything is an integer: x in units of 2^-62, a of 2^-54, b, t = a x -+ b and g of
// 2^-59, the weights alpha_l N_l (E + iB) of a unit chosen per m (synth_weight_kernel) so that
// a sum's high word cannot overflow; its cross word is folded every 16 steps.  Three stretches of l per warp: while every lane's columns are below 2^-64 the
// recurrence alone; then columns v 2^E with sums; and once every lane oscillates (|t| < 2:
// no growth left, E = 0) the plain loop, which most steps take.  Coefficients depend on
// (l, m) alone and are tabulated per plan, weights once per call (every block of 128 rings
// formed both anew, in FP64).
// What bounds it: issue.  A plain step at spin 2 is 37 IMAD.WIDE (two issue cycles each)
// and some 50 other instructions; the double-float form took 273.  Words carry an offset of
// 2^31, so splitting one into signed halves is one XOR.  Measured (GB300, Q/U at
// Nside 1024, lmax 2048, whole synthesis): 40.7 -> 27.0 ms, error against 64 bits 7.6e-13 ->
// 1.7e-13 of the map.
constexpr int GS = 59, AS = 54;

// The signed halves of v when V = v + 2^31.  (The pairs here are never negated, so they keep
// every bit: a lowest bit always set would shift every coefficient the same way, and near the
// poles, where the recurrence answers a constant push with its square, that showed.)
constexpr long long OFF = 1ll << 31;
__device__ __forceinline__ flints::fx halves(long long V) {
    return {(int)(V >> 32), (int)((uint32_t)V ^ 0x80000000u)};
}
struct alignas(16) SynthStep {
    flints::fx a;  // units of 2^-AS
    long long b;   // units of 2^-GS
};

// Row m of the (l, m) tables: l = m .. lmax, contiguous.
__host__ __device__ __forceinline__ long long tri_row(int lmax, int m) {
    return (long long)m * (lmax + 1) - (long long)m * (m - 1) / 2 - m;
}

// What depends on l alone: with q_l = sqrt((l^2 - m^2)(l^2 - s^2)) / l, q_l = g sqrt(l^2 - m^2).
struct alignas(16) SynthOrder {
    double g, ig, igl;  // sqrt(1 - s^2 / l^2) and its reciprocal, a pair of doubles (0 for l <= s)
    double n, b;        // N_l = sqrt((2l + 1) / 4 pi), s / (l (l + 1))
    double pad;
};
// what 1 / sqrt(x) adds to r, its value in FP64
__device__ __forceinline__ double rsqrt_rest(double x, double r) {
    const double p = x * r, pl = fma(x, r, -p);
    return 0.5 * r * (fma(-p, r, 1.0) - pl * r);
}
__global__ void synth_order_kernel(int lmax, int s, SynthOrder *__restrict__ ord, double *__restrict__ start) {
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l > lmax) return;
    const double ld = l, sd = s;
    SynthOrder o{0.0, 0.0, 0.0, sqrt((2.0 * ld + 1.0) / (4.0 * PI_D)), s > 0 && l > 0 ? sd / (ld * (ld + 1.0)) : 0.0, 0.0};
    if (l > s) {
        const double x = (ld - sd) * (ld + sd), r = rsqrt(x);
        o.g = sqrt(x) / ld;
        o.ig = ld * r;
        o.igl = fma(ld, r, -o.ig) + ld * rsqrt_rest(x, r);
    }
    ord[l] = o;
    start[l] = start_factor(l, s);  // m = l
}

// C_l = q_l / q_{l+1}, so alpha_l alpha_{l-1} q_l is the same for all l, and
// alpha_l = alpha_{l+2} q_{l+2} / q_{l+1}: two chains of products downwards in l.  One block per
// m; a thread multiplies along its stretch of both chains, and by what lies above it.  The coefficients are a_l = (2l + 1) / q_{l+1} alpha_l / alpha_{l+1}
// and b_l = a_l m s / (l (l + 1)), with the quotient of the alphas as they are stored; a_l is
// formed as a pair of doubles, because its error moves the recurrence's phase (FP64 alone
// leaves two to four units of 2^-54).
// What bounds it: the FP64 pipe, one reciprocal square root and one division per (l, m).
// Measured (GB300, lmax 4096, spin 2): 0.77 ms; with a chain per thread, a division a step and
// the roots in FP64 divisions 5.1 ms, of which the host's FFT planning hid none: the plan's
// set-up took 16.2 ms, 11.4 now, an FP64 plan's 11.0.
constexpr int COEF_THREADS = 256;
__global__ void __launch_bounds__(COEF_THREADS) synth_coef_kernel(int lmax, int s, const SynthOrder *__restrict__ ord,
                                                                  SynthStep *steps, double *na, double *start) {
    __shared__ double prod[2][COEF_THREADS];
    const int m = blockIdx.x, l0 = m > s ? m : s, tid = threadIdx.x;
    SynthStep *st = steps + tri_row(lmax, m);
    double *n = na + tri_row(lmax, m);
    // 1 / sqrt(l^2 - m^2), kept in the steps' places until these are formed
    auto root = [&](int l) { return __longlong_as_double(st[l].b); };
    for (int l = l0 + tid; l <= lmax; l += COEF_THREADS) {
        const int x = (l - m) * (l + m);
        st[l].b = __double_as_longlong(x > 0 ? rsqrt((double)x) : 0.0);
    }
    __syncthreads();
    auto ratio = [&](int l) {  // q_{l+2} / q_{l+1}
        const double above = (double)((l + 2 - m) * (l + 2 + m)) * root(l + 2) * ord[l + 2].g;
        return above * (root(l + 1) * ord[l + 1].ig);
    };
    const int pairs = (lmax - l0 + 2) / 2, per = (pairs + COEF_THREADS - 1) / COEF_THREADS;
    const int p0 = tid * per < pairs ? tid * per : pairs, p1 = p0 + per < pairs ? p0 + per : pairs;
    double c0 = 1.0, c1 = 1.0;  // alpha = 1 at lmax and lmax - 1
    for (int p = p0; p < p1; ++p) {
        const int l = lmax - 2 * p;
        if (p > 0) c0 *= ratio(l);
        n[l] = c0;
        if (l > l0) {
            if (p > 0) c1 *= ratio(l - 1);
            n[l - 1] = c1;
        }
    }
    prod[0][tid] = c0;
    prod[1][tid] = c1;
    __syncthreads();
    if (tid < 2) {  // in order: the last alpha of a stretch is then exactly what the next one is multiplied by
        double v = 1.0;
        for (int t = 0; t < COEF_THREADS; ++t) {
            const double c = prod[tid][t];
            prod[tid][t] = v;
            v *= c;
        }
    }
    __syncthreads();
    c0 = prod[0][tid];
    c1 = prod[1][tid];
    for (int p = p0; p < p1; ++p) {
        const int l = lmax - 2 * p;
        n[l] *= c0;
        if (l > l0) n[l - 1] *= c1;
    }
    __syncthreads();
    for (int base = l0; base <= lmax; base += COEF_THREADS) {  // upwards: what lies above l is read before its block overwrites it
        const int l = base + tid;
        const double cur = l <= lmax ? n[l] : 1.0, up = l < lmax ? n[l + 1] : 1.0, r = l < lmax ? root(l + 1) : 0.0;
        if (l == l0) start[m] -= log2(cur);
        __syncthreads();
        if (l > lmax) continue;
        n[l] = ord[l].n * cur;
        double a = 0.0, al = 0.0;  // (lmax: no step)
        if (l < lmax) {
            const double k = 2.0 * l + 1.0, iu = 1.0 / up, v = cur * iu, vl = fma(-v, up, cur) * iu;
            const double ig = ord[l + 1].ig, t = k * r, tl = fma(k, r, -t) + k * rsqrt_rest((double)((l + 1 - m) * (l + 1 + m)), r);
            const double u = t * ig, ul = fma(t, ig, -u) + tl * ig + t * ord[l + 1].igl;
            a = u * v;
            al = fma(u, v, -a) + ul * v + u * vl;
        }
        const double b = a * ((double)m * ord[l].b);
        st[l] = SynthStep{halves(flints::fx_of(a, AS) + flints::fx_of(al, AS) + OFF), (long long)flints::fx_of(b, GS)};
    }
}

// One block per m: weights W_l = alpha_l N_l (E + iB) and, spin s, alpha_l N_l (E^* + iB^*) in
// units of 2^-ws, ws the largest with sum_l |W_l| < 2^66 units (a sum's high word, whose terms
// are at most 2^(GS - 32) times a weight's, stays below 2^61) and |W_l| < 2^59 (eight terms of
// its cross word stay below 2^62).  The low words' products that the sums drop are then 2^-51
// of the sum of the weights' sizes at most; ws = WE_BAD where that sum is not finite.
constexpr int WE_BAD = 1 << 20;
template <int S>
__global__ void synth_weight_kernel(int lmax, const double *__restrict__ na, const double2 *__restrict__ alm,
                                    const double2 *__restrict__ blm, flints::fxc *__restrict__ W, int *__restrict__ we) {
    __shared__ double part[256], peak[256];
    const int m = blockIdx.x, l0 = m > S ? m : S, tid = threadIdx.x;
    const double *n = na + tri_row(lmax, m);
    auto weights = [&](int l, double2 &p, double2 &q) {
        const double nl = n[l];
        const double2 a = alm[(size_t)l * (lmax + 1) + m];
        const double2 b = (S > 0 && blm) ? blm[(size_t)l * (lmax + 1) + m] : make_double2(0.0, 0.0);
        p = make_double2((a.x - b.y) * nl, (a.y + b.x) * nl);
        q = make_double2((a.x + b.y) * nl, (b.x - a.y) * nl);
    };
    double sum = 0.0, big = 0.0;
    for (int l = l0 + tid; l <= lmax; l += blockDim.x) {
        double2 p, q;
        weights(l, p, q);
        double t = fabs(p.x) + fabs(p.y);
        if (S > 0) t += fabs(q.x) + fabs(q.y);
        sum += t;
        big = fmax(big, t);
    }
    part[tid] = sum;
    peak[tid] = big;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (tid < o) {
            part[tid] += part[tid + o];
            peak[tid] = fmax(peak[tid], peak[tid + o]);
        }
        __syncthreads();
    }
    const bool bad = !(part[0] <= 1.7e308);
    // a value below 2^expo (one more than its own exponent for the sum, whose rounding may carry)
    auto expo = [](double v) {
        const int ex = (int)(((unsigned long long)__double_as_longlong(v) >> 52) & 0x7ff);
        return ex == 0 ? -960 : ex - 1022;
    };
    const int e0 = 66 - (expo(part[0]) + 1), e1 = 59 - expo(peak[0]), ws = e0 < e1 ? e0 : e1;
    if (tid == 0) we[m] = bad ? WE_BAD : ws;
    flints::fxc *w = W + (S > 0 ? 2 : 1) * tri_row(lmax, m);
    auto put = [&](flints::fxc &dst, double2 v) {
        dst = flints::fxc{halves((bad ? 0 : flints::fx_of(v.x, ws)) + OFF), halves((bad ? 0 : flints::fx_of(v.y, ws)) + OFF)};
    };
    for (int l = l0 + tid; l <= lmax; l += blockDim.x) {
        double2 p, q;
        weights(l, p, q);
        if constexpr (S == 0) {  // two real weights per l
            put(w[l], p);
        } else {
            put(w[2 * l], p);
            put(w[2 * l + 1], q);
        }
    }
}

// x y / 2^DOWN + offs, rounded; the low words' product enters by its top halves
template <int DOWN>
__device__ __forceinline__ long long mul_off(flints::fx x, flints::fx y, uint64_t offs) {
    flints::fxacc a{0, (offs << (DOWN - 32)) + ((uint64_t)1 << (DOWN - 33))};
    flints::fx_mac(a, x, y);
    flints::mad_wide(a.cr, x.lo >> 16, y.lo >> 16);
    return flints::fx_down<DOWN>(a);
}

// One column v 2^(E - GS); prev on the same scale.
struct ColFx {
    long long v, prev;
    int e;
    __device__ __forceinline__ void init(double lg, bool neg) {
        const double fl = floor(lg);
        e = (int)fl - 1;
        v = (long long)(exp2(lg - fl) * 1152921504606846976.0);  // 2^60 to 2^61
        if (neg) v = -v;
        prev = 0;
    }
    // to the next l with t = T 2^-AS, |T| < 2^(AS + k): v is kept below 2^(62 - k), lim its high word's bound
    __device__ __forceinline__ void step(long long T, int lim) {
        if (e < 0) {
            const int th = (int)(T >> 32);
            int k = 0;
            if ((th < 0 ? ~th : th) < (2 << (AS - 32)) && e > -24) {
                k = -e;  // the column oscillates: the common scale holds what it needs
            } else {
                int h = (int)(v >> 32);
                h = h < 0 ? ~h : h;
                if (h >= lim) {
                    k = __clz((unsigned)lim) - __clz((unsigned)h) + 5;
                    k = k < -e ? k : -e;
                }
            }
            v >>= k;
            prev >>= k;
            e += k;
        }
        const long long nv = (long long)((uint64_t)mul_off<AS>(halves(T + OFF), halves(v + OFF), 0) - (uint64_t)prev);
        prev = v;
        v = nv;
    }
    __device__ __forceinline__ flints::fx value() const { return halves((v >> (e > -63 ? -e : 63)) + OFF); }
};

template <int S>
__global__ void __launch_bounds__(128) legendre_fx_kernel(int lmax, int nside, const SynthRing *__restrict__ rings,
                                                          const SynthStep *__restrict__ steps,
                                                          const flints::fxc *__restrict__ W, const int *__restrict__ we,
                                                          const double *__restrict__ start, double2 *__restrict__ F) {
    using flints::fx;
    using flints::fxacc;
    using flints::fxc;
    constexpr int NS = S == 0 ? 1 : 4;  // sums: pA (spin 0: the only one), pB, mA, mB
    const int m = blockIdx.y;
    const int ring = blockIdx.x * blockDim.x + threadIdx.x + 1;  // northern ring incl. the equator
    const int nnorth = 2 * nside;
    const bool active = ring <= nnorth;
    const int NM = S == 0 ? lmax + 1 : 2 * lmax + 1;
    int l = m > S ? m : S;
    SynthRing rg{};
    if (active) rg = rings[ring - 1];
    const fx x = halves(flints::fx_of(rg.x, 62) + OFF);
    ColFx ca{0, 0, -(1 << 20)}, cb{0, 0, -(1 << 20)};
    if (active && l <= lmax) {  // columns A = d_{m,-s}, B = d_{m,s}
        const double lg = __ldg(start + m);
        int pc, ps;
        bool neg;
        start_powers(m, -S, pc, ps, neg);
        ca.init(lg + pc * rg.lc + ps * rg.ls, neg);
        if (S > 0) {
            start_powers(m, S, pc, ps, neg);
            cb.init(lg + pc * rg.lc + ps * rg.ls, neg);
        }
    }
    // Columns that stay evanescent: left of its turning point l sin(theta) = M = m - s a column is
    // at most exp(-M (acosh(1/r) - sqrt(1 - r^2))), r = (l + 1/2) sin(theta) / M (WKB; the
    // factor it leaves out is below 1).  Below 2^-93 at lmax nothing of it reaches a sum's last bit.
    const float M = (float)(m - S), r = ((float)lmax + 0.5f) * sqrtf(fmaxf(0.0f, (float)((1.0 - rg.x) * (1.0 + rg.x)))) / fmaxf(M, 1.0f);
    bool never = !active;
    if (active && r < 1.0f) {
        const float c = sqrtf(1.0f - r * r);
        never = M * (logf((1.0f + c) / fmaxf(r, 1e-30f)) - c) > 64.5f;  // 93 ln 2
    }
    if (__all_sync(FULL_WARP, never)) l = lmax + 1;
    const SynthStep *st = steps + tri_row(lmax, m);
    const fxc *w = W + (S > 0 ? 2 : 1) * tri_row(lmax, m);
    auto ld_step = [&](int i) {
        const float4 q = __ldg(reinterpret_cast<const float4 *>(st + i));
        SynthStep r;
        r.a = fx{(int)__float_as_uint(q.x), (int)__float_as_uint(q.y)};
        r.b = (long long)(((uint64_t)__float_as_uint(q.w) << 32) | __float_as_uint(q.z));
        return r;
    };
    auto ld_w = [&](int i) {
        const float4 q = __ldg(reinterpret_cast<const float4 *>(w + i));
        return fxc{fx{(int)__float_as_uint(q.x), (int)__float_as_uint(q.y)},
                   fx{(int)__float_as_uint(q.z), (int)__float_as_uint(q.w)}};
    };
    auto top_of = [](const SynthStep &c) {  // above a + |b|, units of 2^(32 - AS)
        const int bh = (int)(c.b >> (32 + GS - AS));
        return c.a.hi + (bh < 0 ? ~bh : bh) + 2;
    };
    auto advance = [&](const SynthStep &c) {
        const long long b = c.b >> (GS - AS);
        const int lim = 1 << (30 - (32 - __clz((unsigned)top_of(c)) - (AS - 32)));
        const long long ax = mul_off<62>(c.a, x, 0);
        ca.step(ax + b, lim);
        if (S > 0) cb.step(ax - b, lim);
    };
    // no lane's columns above 2^-64: the recurrence alone
    while (l < lmax) {
        if (__any_sync(FULL_WARP, ca.e > -64 || (S > 0 && cb.e > -64))) break;
        const int stop = l + 8 < lmax ? l + 8 : lmax;
        for (; l < stop; ++l) advance(ld_step(l));
    }
    // sums by parity of l + l1, l1 the first summed l (re, im)
    const int l1 = l;
    fxacc acc[2][NS][2];
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int i = 0; i < NS; ++i) acc[h][i][0] = acc[h][i][1] = fxacc{0, 0};
    auto fold = [&]() {  // the cross words' upper halves into the high words
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int i = 0; i < NS; ++i)
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    acc[h][i][c].hh += (uint64_t)((int64_t)acc[h][i][c].cr >> 32);
                    acc[h][i][c].cr &= 0xffffffffull;
                }
    };
    auto add = [&](fxacc(&s)[NS][2], const fxc &p, const fxc &q, const fx &da, const fx &db) {
        flints::fx_mac(s[0][0], p.re, da);
        flints::fx_mac(s[0][1], p.im, da);
        if constexpr (S > 0) {
            flints::fx_mac(s[1][0], p.re, db);
            flints::fx_mac(s[1][1], p.im, db);
            flints::fx_mac(s[2][0], q.re, da);
            flints::fx_mac(s[2][1], q.im, da);
            flints::fx_mac(s[3][0], q.re, db);
            flints::fx_mac(s[3][1], q.im, db);
        }
    };
    constexpr int WN = S > 0 ? 2 : 1;  // weight pairs per l
    while (l <= lmax) {
        const bool plain = !active || (ca.e == 0 && (S == 0 || cb.e == 0));
        if (l < lmax && top_of(ld_step(l)) < (7 << (AS - 32)) && __all_sync(FULL_WARP, plain)) break;
#pragma unroll 1
        for (int j = 0; j < 4 && l <= lmax; ++j) {
            add(acc[0], ld_w(WN * l), ld_w(WN * l + WN - 1), ca.value(), cb.value());
            if (l < lmax) advance(ld_step(l));
            if (++l > lmax) break;
            add(acc[1], ld_w(WN * l), ld_w(WN * l + WN - 1), ca.value(), cb.value());
            if (l < lmax) advance(ld_step(l));
            ++l;
        }
        fold();
    }
    // every column on the common scale and |t| < 7 from here on (a and |b| fall with l)
    long long va = ca.v + OFF, pa = ca.prev + OFF, vb = cb.v + OFF, pb = cb.prev + OFF;
    auto plain_step = [&](fxacc(&s)[NS][2], int at) {
        const fxc p = ld_w(WN * at), q = ld_w(WN * at + WN - 1);
        const SynthStep c = ld_step(at < lmax ? at : lmax);
        const fx da = halves(va), db = halves(vb);
        add(s, p, q, da, db);
        const long long ax = mul_off<62 + AS - GS>(c.a, x, OFF);  // units of 2^-GS
        const long long na = (long long)((uint64_t)mul_off<GS>(halves(ax + c.b), da, 2 * OFF) - (uint64_t)pa);
        pa = va;
        va = na;
        if constexpr (S > 0) {
            const long long nb = (long long)((uint64_t)mul_off<GS>(halves(ax - c.b), db, 2 * OFF) - (uint64_t)pb);
            pb = vb;
            vb = nb;
        }
    };
    while (l + 1 <= lmax) {
#pragma unroll 1
        for (int j = 0; j < 8 && l + 1 <= lmax; ++j, l += 2) {
            plain_step(acc[0], l);
            plain_step(acc[1], l + 1);
        }
        fold();
    }
    if (l <= lmax) plain_step(acc[0], l);
    fold();
    if (!active) return;
    const int ws = __ldg(we + m);
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
    auto val = [&](const fxacc &s) {  // units of 2^-(ws + GS), hh of 2^64 and cr of 2^32 of them
        return ws == WE_BAD ? nan : flints::fx_scale2((double)(int64_t)s.hh, 64 - ws - GS) +
                                        flints::fx_scale2((double)(int64_t)s.cr, 32 - ws - GS);
    };
    const bool odd = ((l1 + m) & 1) != 0;  // acc[0] holds the terms of odd l + m
    auto sum = [&](int i, double sg_o, double sg) {
        const double r0 = val(acc[0][i][0]), r1 = val(acc[1][i][0]), i0 = val(acc[0][i][1]), i1 = val(acc[1][i][1]);
        return odd ? make_double2(sg * (r1 + sg_o * r0), sg * (i1 + sg_o * i0))
                   : make_double2(sg * (r0 + sg_o * r1), sg * (i0 + sg_o * i1));
    };
    const int south = 4 * nside - ring;  // mirror ring (== ring at the equator)
    double2 *Fn = F + (size_t)(ring - 1) * NM;
    double2 *Fs = F + (size_t)(south - 1) * NM;
    if constexpr (S == 0) {
        Fn[m] = sum(0, 1.0, 1.0);
        if (south != ring) Fs[m] = sum(0, -1.0, 1.0);
    } else {
        // P_m = -(-1)^s sum wp d_{m,-s}; south: d_{m,-s}(pi - t) = (-1)^{l+m} d_{m,s}(t)
        const double sg = (S & 1) ? 1.0 : -1.0;  // -(-1)^s
        Fn[lmax + m] = sum(0, 1.0, sg);
        if (south != ring) Fs[lmax + m] = sum(1, -1.0, sg);
        if (m > 0) {  // P_-m = -sum wm d_{m,s}; south: d_{m,s}(pi - t) = (-1)^{l+m} d_{m,-s}(t)
            Fn[lmax - m] = sum(3, 1.0, -1.0);
            if (south != ring) Fs[lmax - m] = sum(2, -1.0, -1.0);
        }
    }
}

// Fold the coefficients of one ring modulo its length n, with the phase of the
// first pixel: H_k = sum_{m = k mod n} F_m e^{i m phi0}.  Spin 0 (real field,
// F_-m = F_m^*): k = 0..n/2 for a complex-to-real FFT; spin s: k = 0..n-1.
// Polar rings (rg.M > 0) write a_k = H_k w_k, k < n, zero-padded to M, into
// their Bluestein slot in A; equatorial rings write H into H.
template <int S>
__global__ void fold_kernel(int lmax, const SynthRing *__restrict__ rings, const double2 *__restrict__ F,
                            double2 *__restrict__ H, double2 *__restrict__ A) {
    const int r = blockIdx.x;  // ring index - 1
    const SynthRing rg = rings[r];
    const int n = rg.n;
    const int NM = S == 0 ? lmax + 1 : 2 * lmax + 1;
    const double2 *Fr = F + (size_t)r * NM;
    const bool polar = rg.M > 0;
    double2 *Hr = polar ? A + rg.off : H + rg.off;
    if (polar)
        for (int k = n + threadIdx.x; k < rg.M; k += blockDim.x) Hr[k] = make_double2(0.0, 0.0);
    const int nk = (S == 0 && !polar) ? n / 2 + 1 : n;
    for (int k = threadIdx.x; k < nk; k += blockDim.x) {
        double hr = 0.0, hi = 0.0;
        // m = k + j n: e^{i m phi0} = e^{i k phi0} (-1)^j where phi0 is half a pixel, and 1 where it is 0
        const bool half = rg.phi0 > 0.0;
        if (S == 0) {
            double sg = 1.0;
            for (int m = k; m <= lmax; m += n) {  // m >= 0
                const double2 f = Fr[m];
                hr = fma(sg, f.x, hr);
                hi = fma(sg, f.y, hi);
                if (half) sg = -sg;
            }
            sg = half ? -1.0 : 1.0;  // -m = k - (j + 1) n
            for (int m = (k == 0 ? n : n - k); m <= lmax; m += n) {  // m >= 1, -m = k mod n: conj
                const double2 f = Fr[m];
                hr = fma(sg, f.x, hr);
                hi = fma(-sg, f.y, hi);
                if (half) sg = -sg;
            }
        } else {
            const int j0 = (k + lmax) / n;  // first m = k - j0 n >= -lmax
            double sg = (half && (j0 & 1)) ? -1.0 : 1.0;
            for (int m = k - j0 * n; m <= lmax; m += n) {
                const double2 f = Fr[lmax + m];
                hr = fma(sg, f.x, hr);
                hi = fma(sg, f.y, hi);
                if (half) sg = -sg;
            }
        }
        // one phase per k: polar rings e^{i k phi0} w_k = exp(i pi k (k + 1) / n), reduced in integers
        double sp = 0.0, cp = 1.0;
        if (polar) sincospi((double)(((long long)k * (k + 1)) % (2LL * n)) / (double)n, &sp, &cp);
        else if (half) sincospi((double)k / (double)n, &sp, &cp);
        Hr[k] = make_double2(hr * cp - hi * sp, hr * sp + hi * cp);
    }
}

// Bluestein middle step: the transformed slot times the transformed chirp, / M.
__global__ void chirp_mul_kernel(const SynthRing *__restrict__ rings, const int *__restrict__ polar,
                                 const double2 *__restrict__ FB, double2 *__restrict__ A) {
    const SynthRing rg = rings[polar[blockIdx.x]];
    const double inv = 1.0 / (double)rg.M;
    double2 *a = A + rg.off;
    const double2 *b = FB + rg.fboff;
    for (int k = threadIdx.x; k < rg.M; k += blockDim.x) {
        const double2 x = a[k], y = b[k];
        a[k] = make_double2((x.x * y.x - x.y * y.y) * inv, (x.x * y.y + x.y * y.x) * inv);
    }
}

// Bluestein last step: x_j = w_j c_j, written to the ring's pixels.
template <int S>
__global__ void chirp_out_kernel(const SynthRing *__restrict__ rings, const int *__restrict__ polar,
                                 const double2 *__restrict__ A, double *__restrict__ map) {
    const SynthRing rg = rings[polar[blockIdx.x]];
    const double2 *a = A + rg.off;
    for (int j = threadIdx.x; j < rg.n; j += blockDim.x) {
        const double2 w = chirp(j, rg.n), c = a[j];
        const double xr = w.x * c.x - w.y * c.y, xi = w.x * c.y + w.y * c.x;
        if (S == 0) {
            map[rg.first + j] = xr;
        } else {
            reinterpret_cast<double2 *>(map)[rg.first + j] = make_double2(xr, xi);
        }
    }
}

// Chirp b_t = conj(w_t) for |t| < n in a length-M cyclic buffer (one block per ring size).
__global__ void chirp_fill_kernel(const int *__restrict__ sizes_n, const int *__restrict__ sizes_M,
                                  const long long *__restrict__ sizes_off, double2 *__restrict__ FB) {
    const int n = sizes_n[blockIdx.x], M = sizes_M[blockIdx.x];
    double2 *b = FB + sizes_off[blockIdx.x];
    for (int t = threadIdx.x; t < M; t += blockDim.x) {
        double2 v = make_double2(0.0, 0.0);
        if (t < n) {
            const double2 w = chirp(t, n);
            v = make_double2(w.x, -w.y);
        } else if (t > M - n) {
            const double2 w = chirp(M - t, n);
            v = make_double2(w.x, -w.y);
        }
        b[t] = v;
    }
}

}  // namespace

struct flints_synth_s {
    int device;
    int64_t nside;
    int lmax, spin, precision;
    SynthRing *d_rings;
    int *d_polar;      // indices of the polar rings
    double2 *d_F, *d_H, *d_A, *d_FB;
    SynthStep *d_steps;    // recurrence coefficients per (m, l); these and the next three lie behind F
    double *d_na;          // alpha_l N_l per (m, l)
    double *d_start;       // log2 of the columns' start factor per m
    int *d_we;             // exponents of the weights per m, of the call in hand
    // the weights themselves, per (m, l), lie in d_H: the l-sums have read them before the fold
    // writes there
    flints::fxc *weights() const { return reinterpret_cast<flints::fxc *>(d_H); }
    void *d_work;
    std::vector<SynthRing> rings;
    int npolar;
    cufftHandle belt;                 // equatorial rings, batched
    std::vector<cufftHandle> groups;  // polar rings: one C2C plan per Bluestein length M
    std::vector<long long> group_off; // first slot of each group in A
    bool belt_made;
};

static void synth_release(flints_synth_s *s) {
    if (s->belt_made) cufftDestroy(s->belt);
    for (cufftHandle h : s->groups) cufftDestroy(h);
    cudaFree(s->d_rings);
    cudaFree(s->d_polar);
    cudaFree(s->d_F);
    cudaFree(s->d_H);
    cudaFree(s->d_A);
    cudaFree(s->d_FB);
    cudaFree(s->d_work);
}

static int synth_bail(flints_synth_s *s, int code, const char *what, cudaError_t e = cudaSuccess) {
    synth_release(s);
    delete s;
    if (e != cudaSuccess) return sfail(code, "flints_synth_plan: %s: %s", what, cudaGetErrorString(e));
    return sfail(code, "flints_synth_plan: %s", what);
}

// weights, l-sums and the fold of one synthesis
template <int S>
static void launch_sums(flints_synth_s *s, const double2 *alm, const double2 *blm, cudaStream_t st) {
    const int N = (int)s->nside, lmax = s->lmax, nr = 4 * N - 1;
    const dim3 grid((2 * N + 127) / 128, lmax + 1);
    if (s->precision == FLINTS_MIXED) {
        synth_weight_kernel<S><<<lmax + 1, 256, 0, st>>>(lmax, s->d_na, alm, blm, s->weights(), s->d_we);
        legendre_fx_kernel<S><<<grid, 128, 0, st>>>(lmax, N, s->d_rings, s->d_steps, s->weights(), s->d_we, s->d_start, s->d_F);
    } else {
        legendre_kernel<S><<<grid, 128, 0, st>>>(lmax, N, s->d_rings, alm, blm, s->d_F);
    }
    fold_kernel<S><<<nr, 256, 0, st>>>(lmax, s->d_rings, s->d_F, s->d_H, s->d_A);
}

extern "C" {

const char *flints_synth_last_error(void) { return g_msg; }

int flints_synth_plan(flints_synth_t *out, int64_t nside, int lmax, int spin, int precision, void *stream) {
    if (!out) return sfail(FLINTS_EINVAL, "flints_synth_plan: out is NULL");
    *out = nullptr;
    if (nside < 1 || nside > 8192) return sfail(FLINTS_EINVAL, "flints_synth_plan: nside outside [1, 8192]");
    if (spin != 0 && spin != 1 && spin != 2) return sfail(FLINTS_EINVAL, "flints_synth_plan: spin must be 0, 1 or 2");
    if (lmax < spin || lmax > 16384) return sfail(FLINTS_EINVAL, "flints_synth_plan: lmax outside [spin, 16384]");
    if (precision != FLINTS_FP64 && precision != FLINTS_MIXED)
        return sfail(FLINTS_EINVAL, "flints_synth_plan: precision must be FLINTS_FP64 or FLINTS_MIXED");
    const int64_t N = nside;
    const int nr = (int)(4 * N - 1);
    flints_synth_s *s = new flints_synth_s();
    cudaGetDevice(&s->device);
    s->nside = nside;
    s->lmax = lmax;
    s->spin = spin;
    s->precision = precision;
    s->d_rings = nullptr;
    s->d_polar = nullptr;
    s->d_F = s->d_H = s->d_A = s->d_FB = nullptr;
    s->d_steps = nullptr;
    s->d_na = s->d_start = nullptr;
    s->d_we = nullptr;
    s->d_work = nullptr;
    s->belt_made = false;
    // ring geometry (host, FP64)
    s->rings.resize(nr);
    for (int i = 1; i <= nr; ++i) {
        SynthRing rg{};
        double z, f;
        int nq;
        long long first;
        if (i < N) {
            nq = i;
            z = 1.0 - (double)i * i / (3.0 * N * N);
            first = 2LL * i * (i - 1);
            f = 0.5;
        } else if (i <= 3 * N) {
            nq = (int)N;
            z = (4.0 * N - 2.0 * i) / (3.0 * N);
            first = 2LL * N * (N - 1) + 4LL * N * (i - N);
            f = ((i + N) & 1) ? 0.0 : 0.5;
        } else {
            const int ip = (int)(4 * N - i);
            nq = ip;
            z = -(1.0 - (double)ip * ip / (3.0 * N * N));
            first = 12LL * N * N - 2LL * ip * (ip + 1);
            f = 0.5;
        }
        const double th = acos(z);
        rg.x = z;
        rg.lc = log2(cos(0.5 * th));
        rg.ls = log2(sin(0.5 * th));
        rg.phi0 = f / (2.0 * nq);
        rg.first = first;
        rg.n = 4 * nq;
        s->rings[i - 1] = rg;
    }
    // equatorial FFT inputs, contiguous in ring order
    const long long nkb = spin == 0 ? 2 * N + 1 : 4 * N;  // per equatorial ring
    for (int i = (int)N; i <= 3 * N; ++i) s->rings[i - 1].off = (long long)(i - N) * nkb;
    const long long hsize = (2 * N + 1) * nkb;
    // polar rings: Bluestein length M = next power of two >= 2n - 1, slots grouped by M
    std::vector<int> polar, sz_n, sz_M;
    std::vector<long long> sz_off;
    std::vector<int> group_M;
    std::vector<int> group_batch;
    long long aoff = 0, fboff = 0;
    for (int i = 1; i < N; ++i) {
        const int n = 4 * i;
        int M = 1;
        while (M < 2 * n - 1) M <<= 1;
        if (group_M.empty() || group_M.back() != M) {
            group_M.push_back(M);
            group_batch.push_back(0);
            s->group_off.push_back(aoff);
        }
        sz_n.push_back(n);
        sz_M.push_back(M);
        sz_off.push_back(fboff);
        for (int r : {i, (int)(4 * N - i)}) {
            SynthRing &rg = s->rings[r - 1];
            rg.M = M;
            rg.off = aoff;
            rg.fboff = fboff;
            aoff += M;
            polar.push_back(r - 1);
            group_batch.back() += 1;
        }
        fboff += M;
    }
    s->npolar = (int)polar.size();
    const size_t NM = spin == 0 ? (size_t)lmax + 1 : 2 * (size_t)lmax + 1;
    const size_t npair = (size_t)(lmax + 1) * (lmax + 2) / 2;
    // tables of a mixed plan, behind F: steps, alpha_l N_l, starts, exponents
    const size_t tbytes = precision == FLINTS_MIXED
                              ? (sizeof(SynthStep) + sizeof(double)) * npair + (sizeof(double) + sizeof(int)) * (lmax + 1)
                              : 0;
    // the belt's FFT inputs and, before them in a call, the weights (mixed)
    const size_t wbytes = precision == FLINTS_MIXED ? sizeof(flints::fxc) * npair * (spin == 0 ? 1 : 2) : 0;
    const size_t hbytes = sizeof(double2) * (size_t)hsize > wbytes ? sizeof(double2) * (size_t)hsize : wbytes;
    cudaError_t e;
    if ((e = cudaMalloc(&s->d_rings, sizeof(SynthRing) * nr)) != cudaSuccess ||
        (e = cudaMalloc(&s->d_F, sizeof(double2) * NM * nr + tbytes)) != cudaSuccess ||
        (e = cudaMalloc(&s->d_H, hbytes)) != cudaSuccess)
        return synth_bail(s, e == cudaErrorMemoryAllocation ? FLINTS_ENOMEM : FLINTS_ECUDA, "allocation", e);
    if (precision == FLINTS_MIXED) {
        s->d_steps = reinterpret_cast<SynthStep *>(s->d_F + NM * nr);
        s->d_na = reinterpret_cast<double *>(s->d_steps + npair);
        s->d_start = s->d_na + npair;
        s->d_we = reinterpret_cast<int *>(s->d_start + lmax + 1);
    }
    if (s->npolar > 0 &&
        ((e = cudaMalloc(&s->d_polar, sizeof(int) * polar.size())) != cudaSuccess ||
         (e = cudaMalloc(&s->d_A, sizeof(double2) * (size_t)aoff)) != cudaSuccess ||
         (e = cudaMalloc(&s->d_FB, sizeof(double2) * (size_t)fboff)) != cudaSuccess))
        return synth_bail(s, e == cudaErrorMemoryAllocation ? FLINTS_ENOMEM : FLINTS_ECUDA, "allocation", e);
    cudaStream_t st = (cudaStream_t)stream;
    if ((e = cudaMemcpyAsync(s->d_rings, s->rings.data(), sizeof(SynthRing) * nr, cudaMemcpyHostToDevice, st)) !=
        cudaSuccess)
        return synth_bail(s, FLINTS_ECUDA, "copy", e);
    if (s->npolar > 0 && (e = cudaMemcpyAsync(s->d_polar, polar.data(), sizeof(int) * polar.size(),
                                              cudaMemcpyHostToDevice, st)) != cudaSuccess)
        return synth_bail(s, FLINTS_ECUDA, "copy", e);
    if (precision == FLINTS_MIXED) {
        // (the orders' table lies in d_F, which no call has written yet)
        SynthOrder *ord = reinterpret_cast<SynthOrder *>(s->d_F);
        static_assert(sizeof(SynthOrder) <= 3 * sizeof(double2), "F holds at least 3 (lmax + 1) complex numbers");
        synth_order_kernel<<<(lmax + 256) / 256, 256, 0, st>>>(lmax, spin, ord, s->d_start);
        synth_coef_kernel<<<lmax + 1, COEF_THREADS, 0, st>>>(lmax, spin, ord, s->d_steps, s->d_na, s->d_start);
        if ((e = cudaGetLastError()) != cudaSuccess) return synth_bail(s, FLINTS_ECUDA, "coefficients", e);
    }
    // cuFFT plans sharing one work area
    size_t work_max = 0;
    auto make = [&](cufftHandle &h, int n, long long idist, long long odist, cufftType type, int batch) -> bool {
        if (cufftCreate(&h) != CUFFT_SUCCESS) return false;
        cufftSetAutoAllocation(h, 0);
        int nn[1] = {n}, inembed[1] = {(int)idist}, onembed[1] = {(int)odist};
        size_t ws = 0;
        if (cufftMakePlanMany(h, 1, nn, inembed, 1, (int)idist, onembed, 1, (int)odist, type, batch, &ws) !=
            CUFFT_SUCCESS) {
            cufftDestroy(h);
            return false;
        }
        if (ws > work_max) work_max = ws;
        return true;
    };
    if (!make(s->belt, (int)(4 * N), nkb, 4 * N, spin == 0 ? CUFFT_Z2D : CUFFT_Z2Z, (int)(2 * N + 1)))
        return synth_bail(s, FLINTS_ECUDA, "cuFFT plan creation failed");
    s->belt_made = true;
    for (size_t g = 0; g < group_M.size(); ++g) {
        cufftHandle h;
        if (!make(h, group_M[g], group_M[g], group_M[g], CUFFT_Z2Z, group_batch[g]))
            return synth_bail(s, FLINTS_ECUDA, "cuFFT plan creation failed");
        s->groups.push_back(h);
    }
    if (work_max && (e = cudaMalloc(&s->d_work, work_max)) != cudaSuccess)
        return synth_bail(s, FLINTS_ENOMEM, "FFT work area", e);
    cufftSetWorkArea(s->belt, s->d_work);
    for (cufftHandle h : s->groups) cufftSetWorkArea(h, s->d_work);
    // transformed chirps, one per polar ring size
    if (s->npolar > 0) {
        int *d_n = nullptr, *d_M = nullptr;
        long long *d_off = nullptr;
        const size_t ns = sz_n.size();
        if ((e = cudaMalloc(&d_n, sizeof(int) * ns)) != cudaSuccess ||
            (e = cudaMalloc(&d_M, sizeof(int) * ns)) != cudaSuccess ||
            (e = cudaMalloc(&d_off, sizeof(long long) * ns)) != cudaSuccess) {
            cudaFree(d_n);
            cudaFree(d_M);
            return synth_bail(s, FLINTS_ENOMEM, "chirp tables", e);
        }
        cudaMemcpyAsync(d_n, sz_n.data(), sizeof(int) * ns, cudaMemcpyHostToDevice, st);
        cudaMemcpyAsync(d_M, sz_M.data(), sizeof(int) * ns, cudaMemcpyHostToDevice, st);
        cudaMemcpyAsync(d_off, sz_off.data(), sizeof(long long) * ns, cudaMemcpyHostToDevice, st);
        chirp_fill_kernel<<<(unsigned)ns, 256, 0, st>>>(d_n, d_M, d_off, s->d_FB);
        e = cudaGetLastError();
        // forward transforms of the chirps, group by group (one per ring size in a group)
        for (size_t g = 0; e == cudaSuccess && g < group_M.size(); ++g) {
            size_t k0 = 0;
            while (k0 < ns && sz_M[k0] != group_M[g]) ++k0;
            size_t k1 = k0;
            while (k1 < ns && sz_M[k1] == group_M[g]) ++k1;
            cufftHandle h;
            if (!make(h, group_M[g], group_M[g], group_M[g], CUFFT_Z2Z, (int)(k1 - k0))) {
                e = cudaErrorUnknown;
                break;
            }
            void *tmp = nullptr;
            size_t ws = 0;
            cufftGetSize(h, &ws);
            if (ws && cudaMalloc(&tmp, ws) != cudaSuccess) {
                cufftDestroy(h);
                e = cudaErrorMemoryAllocation;
                break;
            }
            cufftSetWorkArea(h, tmp);
            cufftSetStream(h, st);
            cufftDoubleComplex *p = reinterpret_cast<cufftDoubleComplex *>(s->d_FB + sz_off[k0]);
            if (cufftExecZ2Z(h, p, p, CUFFT_FORWARD) != CUFFT_SUCCESS) e = cudaErrorUnknown;
            cudaStreamSynchronize(st);
            cufftDestroy(h);
            cudaFree(tmp);
        }
        cudaStreamSynchronize(st);
        cudaFree(d_n);
        cudaFree(d_M);
        cudaFree(d_off);
        if (e != cudaSuccess) return synth_bail(s, FLINTS_ECUDA, "chirp transforms", e);
    }
    if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return synth_bail(s, FLINTS_ECUDA, "set-up", e);
    *out = s;
    return FLINTS_OK;
}

int flints_synthesize(flints_synth_t s, const double *alm, const double *blm, double *map, void *stream) {
    if (!s) return sfail(FLINTS_EINVAL, "flints_synthesize: plan is NULL");
    if (!alm || !map) return sfail(FLINTS_EINVAL, "flints_synthesize: alm and map must not be NULL");
    if (((uintptr_t)alm | (uintptr_t)map | (uintptr_t)blm) & 15u)
        return sfail(FLINTS_EINVAL, "flints_synthesize: alm, blm and map must be 16-byte aligned");
    int cur = -1;
    cudaGetDevice(&cur);
    if (cur != s->device) return sfail(FLINTS_EINVAL, "flints_synthesize: plan made on another device");
    cudaStream_t st = (cudaStream_t)stream;
    const int N = (int)s->nside;
    const double2 *a = reinterpret_cast<const double2 *>(alm);
    const double2 *b = s->spin == 0 ? nullptr : reinterpret_cast<const double2 *>(blm);
    switch (s->spin) {
        case 0: launch_sums<0>(s, a, b, st); break;
        case 1: launch_sums<1>(s, a, b, st); break;
        default: launch_sums<2>(s, a, b, st); break;
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return sfail(FLINTS_ECUDA, "flints_synthesize: kernel launch: %s", cudaGetErrorString(e));
    // equatorial rings: one batched inverse transform straight into the map
    if (cufftSetStream(s->belt, st) != CUFFT_SUCCESS) return sfail(FLINTS_ECUDA, "flints_synthesize: cufftSetStream");
    {
        const SynthRing &r0 = s->rings[N - 1];
        cufftDoubleComplex *in = reinterpret_cast<cufftDoubleComplex *>(s->d_H);
        cufftResult fr = s->spin == 0
                             ? cufftExecZ2D(s->belt, in, reinterpret_cast<cufftDoubleReal *>(map + r0.first))
                             : cufftExecZ2Z(s->belt, in, reinterpret_cast<cufftDoubleComplex *>(map) + r0.first,
                                            CUFFT_INVERSE);
        if (fr != CUFFT_SUCCESS) return sfail(FLINTS_ECUDA, "flints_synthesize: cuFFT execution failed (%d)", (int)fr);
    }
    if (s->npolar == 0) return FLINTS_OK;
    // polar rings: Bluestein convolution
    for (size_t g = 0; g < s->groups.size(); ++g) {
        cufftSetStream(s->groups[g], st);
        cufftDoubleComplex *p = reinterpret_cast<cufftDoubleComplex *>(s->d_A + s->group_off[g]);
        if (cufftExecZ2Z(s->groups[g], p, p, CUFFT_FORWARD) != CUFFT_SUCCESS)
            return sfail(FLINTS_ECUDA, "flints_synthesize: cuFFT execution failed");
    }
    chirp_mul_kernel<<<s->npolar, 256, 0, st>>>(s->d_rings, s->d_polar, s->d_FB, s->d_A);
    for (size_t g = 0; g < s->groups.size(); ++g) {
        cufftDoubleComplex *p = reinterpret_cast<cufftDoubleComplex *>(s->d_A + s->group_off[g]);
        if (cufftExecZ2Z(s->groups[g], p, p, CUFFT_INVERSE) != CUFFT_SUCCESS)
            return sfail(FLINTS_ECUDA, "flints_synthesize: cuFFT execution failed");
    }
    if (s->spin == 0)
        chirp_out_kernel<0><<<s->npolar, 256, 0, st>>>(s->d_rings, s->d_polar, s->d_A, map);
    else
        chirp_out_kernel<1><<<s->npolar, 256, 0, st>>>(s->d_rings, s->d_polar, s->d_A, map);
    e = cudaGetLastError();
    if (e != cudaSuccess) return sfail(FLINTS_ECUDA, "flints_synthesize: kernel launch: %s", cudaGetErrorString(e));
    return FLINTS_OK;
}

void flints_synth_free(flints_synth_t s) {
    if (!s) return;
    int cur = 0;
    cudaGetDevice(&cur);
    if (cur != s->device) cudaSetDevice(s->device);
    synth_release(s);
    if (cur != s->device) cudaSetDevice(cur);
    delete s;
}

}  // extern "C"
