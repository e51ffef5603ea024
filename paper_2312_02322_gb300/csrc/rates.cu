// Post-processing of cross sections (Sec. III): the symmetrised cross sections of Eq. 20 and
// the Maxwell-Boltzmann rate coefficients of both directions of every transition.
//
// Readings (the paper defers the integration to its ref. [44]):
//   R1  U, the energy at which Eq. 19 compares both directions, is the mean of the incoming and
//       outgoing translational energies;
//   R2  k_{a->b}(T) = (8/(pi mu))^(1/2) (kT)^(-3/2) exp(-(E_b - E_a)/(2kT)) / g_a
//                      * int_{u0}^inf sigma~_ab(U) U exp(-U/kT) dU,
//       so that g_a k_{a->b} = g_b k_{b->a} exp(-(E_b - E_a)/kT) holds exactly;
//   R3  natural cubic spline of sigma~ in U through the computed energies, negative values
//       taken as zero;
//   R4  u0 = |E_b - E_a| / 2; below U_1 a linear ramp from zero at u0, or the spline cut at u0
//       when u0 >= U_1;
//   R5  above U_K the power law sigma~_K (U/U_K)^p, p the log-log slope of the last two points
//       clipped to [-1, 0], integrated in closed form with the upper incomplete gamma function.
//
// One thread per unordered pair of levels and chunk of temperatures.  The spline's second derivatives
// are a fixed linear map of the knot values (set up on the host from the energy grid).  Two forms of
// the integral:
//   closed form  when no piece of the spline at or above u0 can be negative (its Bernstein coefficients
//       are >= 0, so the cubic is): the integral over every whole piece is linear in the knot values with
//       weights that depend on the temperature alone (host tables, rate_tables); the piece that u0
//       cuts (or the ramp) is a quartic times exp(-(U - u0)/kT), i.e. five lower incomplete gamma functions
//       of integer order; the tail's Gamma(2 + p, x), x = U_K/kT, is a Chebyshev series in p per temperature
//       for x >= 0.1 and evaluated for the pair below (kRateChebX).
//       About 170 FP64 instructions per pair and temperature instead of about 4400: the kernel is bound
//       by the FP64 pipe, so the instruction count is its time.
//   quadrature  (k_rates_quad) for every other pair (a value below zero is taken as zero, R3), a u0 at or above U_K, and
//       temperatures or energies outside [1e-12, 1e6] hartree: 16-point Gauss-Legendre panels no
//       wider than 4 kT (the exponential at the nodes as a panel factor times node factors shared by the
//       panels of a piece); the walk stops at the first panel whose remainder bound
//       (4 max|y| kT (U + kT) exp(-(U - u0)/kT) at its lower edge U) is below 1e-17 of the integral so
//       far; the tail is then dropped too.
// The integrand carries exp(-(U - u0)/kT) so that neither exponential factor of R2 overflows.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "internal.h"

namespace mqct {

namespace {

constexpr int kRateMaxK = MQCT_RATE_MAX_ENERGIES;
constexpr int kRateMaxT = MQCT_RATE_MAX_TEMPS;
constexpr int kGl = 16;
constexpr int kRateThreads = 128;          // a block's tile of pairs: 16 levels a x 8 levels b
constexpr int kRateTa = 16, kRateTb = 8;
constexpr size_t kRatePass = (size_t)1 << 26;  // pairs of levels of one pass (all up to 11 585 levels): 512 MB of list
constexpr int kRateCheb = 16;              // Chebyshev coefficients of the tail per temperature
// The series expands x^-(1+p) Gamma(2+p, x) e^x, which varies over a factor 1/x in p as x = U_K/kT falls: sixteen
// terms hold the integral to 2e-14 at x = 0.1, 2e-12 at 0.03, 1e-10 at 0.01 and lose every digit by 1e-7.  A
// temperature with x below this bound evaluates the incomplete gamma function for each pair.
constexpr double kRateChebX = 0.1;

struct RateArgs {
    double u[kRateMaxK];
    double Q[kRateMaxK][kRateMaxK];  // second derivatives of the natural spline: M = Q y
    double gx[kGl], gw[kGl];         // Gauss-Legendre nodes and weights on [-1, 1]
    double kT[kRateMaxT];
    double ikT[kRateMaxT];           // 1 / kT
    double pref[kRateMaxT];          // (8 / (pi mu))^(1/2) kT^(-3/2)
    double ln_uK;                    // ln(U_K / U_{K-1})
    int K, L, n_T;
    int t_chunk;                     // temperatures of one block
    int closed;                      // the closed form is allowed (ranges of kT and U)
    // per temperature: [K][K] weights of the whole pieces at and above knot j, [K] exp(-(U_K - U_j)/kT),
    // the tail's Chebyshev coefficients
    const double *tab;
};

// the pairs whose rates k_rates leaves to k_rates_quad, listed from the front (whole warps of them, which stay
// together: their panel counts are alike) and from the back (the others); the next item of k_rates_quad
struct RateQueue {
    unsigned long long front, back, next, pad;
};

// tiles before row j of tiles (eight levels b): row i has those a-tiles (16 levels) with a <= 8 i + 7, i / 2 + 1 of them
__host__ __device__ constexpr long long rate_tiles(long long j) { return (j / 2) * (j / 2 + 1) + (j % 2) * (j / 2 + 1); }

// doubles of A.tab per temperature
__host__ __device__ constexpr int rate_tab_stride(int K) { return K * K + K + kRateCheb; }

// Gamma(s, x) e^x for 1 <= s <= 2, x > 0.  Below x = s + 1 the power series of the lower
// function gamma(s, x) = x^s e^-x sum_n x^n / (s (s+1) ... (s+n)) (Abramowitz & Stegun 6.5.29)
// is subtracted from Gamma(s); above, Legendre's continued fraction (A&S 6.5.31) is evaluated
// by the modified Lentz algorithm.
__device__ double upper_gamma_scaled(double s, double x)
{
    if (s == 1.0) return 1.0;
    if (s == 2.0) return 1.0 + x;
    if (x < s + 1.0) {
        double term = 1.0 / s, sum = term;
        for (int n = 1; n < 200; ++n) {
            term *= x / (s + n);
            sum += term;
            if (fabs(term) < 1e-17 * sum) break;
        }
        return tgamma(s) * exp(x) - pow(x, s) * sum;
    }
    const double tiny = 1e-300;
    double b = x + 1.0 - s, c = 1.0 / tiny, d = 1.0 / b, f = d;
    for (int i = 1; i < 300; ++i) {
        const double an = -i * (i - s);
        b += 2.0;
        d = an * d + b;
        if (fabs(d) < tiny) d = tiny;
        c = b + an / c;
        if (fabs(c) < tiny) c = tiny;
        d = 1.0 / d;
        const double del = d * c;
        f *= del;
        if (fabs(del - 1.0) < 1e-16) break;
    }
    return pow(x, s) * f;
}

// the closed form's tail factor x^-(1+p) Gamma(2+p, x) e^x for one pair
__device__ __noinline__ double rate_tail(double p, double x) { return pow(x, -(1.0 + p)) * upper_gamma_scaled(2.0 + p, x); }

// int sigma~ U exp(-(U - u0)/kT) dU by quadrature, piece by piece in increasing U (y, M: the knot values
// and second derivatives of this thread's pair, `st` doubles apart)
__device__ __noinline__ double rate_quadrature(const RateArgs &A, const double *y, const double *M, int st, double ymax,
                                               double u0, double th, double ith)
{
    const int K = A.K;
    double acc = 0.0;
    bool done = false;
    auto piece = [&](double lo, double hi, int kind, int k) {
        // remainder above lo bounded by 4 max|y| kT (lo + kT) exp(-(lo - u0)/kT)
        if (done || hi <= lo) return;
        if (4.0 * ymax * th * (lo + th) * exp(-(lo - u0) * ith) <= 1e-17 * acc) { done = true; return; }
        const int np = (int)fmin(256.0, fmax(1.0, ceil((hi - lo) * 0.25 * ith)));
        const double hp = (hi - lo) / np;
        const double h = kind ? A.u[k + 1] - A.u[k] : 0.0;
        // reciprocals once per piece (an FP64 division costs ~10 FMA slots on this GPU's FP64 pipe)
        const double ih = kind ? 1.0 / h : 0.0, iramp = kind ? 0.0 : y[0] / (A.u[0] - u0);
        const double y0 = y[k * st], y1 = kind ? y[(k + 1) * st] : 0.0, M0 = M[k * st], M1 = kind ? M[(k + 1) * st] : 0.0;
        const double h26 = h * h * (1.0 / 6.0);
        // exp(-(U - u0)/kT) = exp(-(c - u0)/kT) exp(-(hp/2) x_j / kT): the node factors are the same
        // for every panel of the piece
        double ef[kGl];
#pragma unroll
        for (int j = 0; j < kGl; ++j) ef[j] = exp(-0.5 * hp * A.gx[j] * ith);
        // the same remainder bound at each panel's lower edge c - hp/2, from the panel factor:
        // exp(-(c - hp/2 - u0)/kT) = exp(-(c - u0)/kT) exp(hp/(2kT))
        const double bnd = 4.0 * ymax * th * exp(0.5 * hp * ith);
        for (int p = 0; p < np; ++p) {
            const double c = lo + hp * (p + 0.5);
            const double ec = exp(-(c - u0) * ith);
            if (p > 0 && bnd * (c - 0.5 * hp + th) * ec <= 1e-17 * acc) { done = true; return; }
            double s = 0.0;
#pragma unroll
            for (int j = 0; j < kGl; ++j) {
                const double U = fma(0.5 * hp, A.gx[j], c);
                double v;
                if (kind == 0) {
                    v = (U - u0) * iramp;
                } else {
                    const double tt = (U - A.u[k]) * ih, sr = 1.0 - tt;
                    v = sr * y0 + tt * y1 + h26 * ((sr * sr * sr - sr) * M0 + (tt * tt * tt - tt) * M1);
                    v = fmax(v, 0.0);
                }
                s = fma(A.gw[j], v * U * (ec * ef[j]), s);
            }
            acc = fma(0.5 * hp, s, acc);
        }
    };
    if (u0 < A.u[0]) piece(u0, A.u[0], 0, 0);
    for (int k = 0; k + 1 < K; ++k) piece(fmax(A.u[k], u0), A.u[k + 1], 1, k);
    {
        // tail: y_K U_K^-p int_a^inf U^(1+p) exp(-(U - u0)/kT) dU
        //     = y_K U_K^-p kT^s [Gamma(s, a/kT) e^(a/kT)] exp(-(a - u0)/kT),  s = 2 + p
        const double a = fmax(A.u[K - 1], u0), yK = y[(K - 1) * st], yJ = y[(K - 2) * st];
        double p = 0.0;
        if (yK > 0.0 && yJ > 0.0) p = fmin(0.0, fmax(-1.0, log(yK / yJ) / A.ln_uK));
        if (yK != 0.0 && !done) {
            const double s = 2.0 + p, x = a * ith;
            acc += yK * pow(A.u[K - 1], -p) * pow(th, s) * upper_gamma_scaled(s, x) * exp(-(a - u0) * ith);
        }
    }
    return acc;
}

// Lower incomplete gamma functions gamma(1..5, z) from ez = exp(-z).  z >= 2: upward recurrence
// gamma(m + 1) = m gamma(m) - z^m e^-z (loses less than one digit there); below, the power series of
// gamma(5, z) (Abramowitz & Stegun 6.5.29; 21 terms reach 1e-18 at z = 2) and the downward recurrence, all
// of whose terms are positive.
__device__ __forceinline__ void lower_gammas(double z, double ez, double G[5])
{
    const double z2 = z * z;
    if (z >= 2.0) {
        G[0] = 1.0 - ez;
        G[1] = fma(-z, ez, G[0]);
        G[2] = fma(2.0, G[1], -z2 * ez);
        G[3] = fma(3.0, G[2], -z2 * z * ez);
        G[4] = fma(4.0, G[3], -z2 * z2 * ez);
    } else {
        // sum_n z^n / (5 6 ... (5 + n)) = (1/5)(1 + z/6 (1 + z/7 (...)))
        double s = 1.0;
#pragma unroll
        for (int n = 25; n >= 6; --n) s = fma(s, z * (1.0 / n), 1.0);
        const double z4e = z2 * z2 * ez;
        G[4] = 0.2 * s * z * z4e;
        G[3] = 0.25 * (G[4] + z4e);
        G[2] = (1.0 / 3.0) * (G[3] + z2 * z * ez);
        G[1] = 0.5 * (G[2] + z2 * ez);
        G[0] = fma(z, ez, G[1]);
    }
}

// both rates of a pair from its integral (x0 = u0/kT): exp(-dE/(2kT)) exp(-u0/kT) is exp(-|dE|/kT) for an
// excitation, 1 for a quenching
__device__ __forceinline__ void rate_store(const RateArgs &A, double *rate, int t, double acc, double dE, double x0,
                                           double ga, double gb, int ia, int ib)
{
    const double c = A.pref[t] * acc, ex = exp(-2.0 * x0);
    rate[(size_t)ia * A.L + ib] = c * (dE >= 0.0 ? ex : 1.0) * (1.0 / ga);
    rate[(size_t)ib * A.L + ia] = c * (dE >= 0.0 ? 1.0 : ex) * (1.0 / gb);
}

// One thread per unordered pair (a <= b): the symmetrised cross sections of Eq. 20 (sym, or NULL) and, where the
// closed form holds, both rates; the other pairs join the list that k_rates_quad integrates, so that no thread waits
// for a quadrature.  A block takes a tile of 16 x 8 pairs, so that the transposed reads sigma[k][a][b] of its warps
// share 32-byte sectors; only tiles with pairs a <= b have a block (rate_tiles), since the empty blocks of a
// rectangular grid leave the others unevenly spread over the SMs.  Bound by the FP64 pipe: a call with 1032 levels x
// 10 energies x 5 temperatures, all in closed form, takes 1.20 ms (the kernel 0.94); with the quadrature of every
// pair 27 ms.
__global__ void __launch_bounds__(kRateThreads, 3) k_rates(const __grid_constant__ RateArgs A, const double *sigma,
                                                         const double *g, const double *E, double *sym, double *rate,
                                                         long long first, RateQueue *queue, int2 *list, size_t list_n)
{
    extern __shared__ double rsm[];
    const int K = A.K, L = A.L;
    // tile first + blockIdx.x: row j of tiles is the last one with rate_tiles(j) at or below it
    const long long tile = first + blockIdx.x;
    long long j8 = (long long)sqrtf(4.f * (float)tile);
    while (rate_tiles(j8) > tile) --j8;
    while (rate_tiles(j8 + 1) <= tile) ++j8;
    const int ia = (int)(tile - rate_tiles(j8)) * kRateTa + threadIdx.x % kRateTa, ib = (int)j8 * kRateTb + threadIdx.x / kRateTa;
    if (ia >= L || ib >= L || ia > ib) return;
    constexpr int st = kRateThreads;
    double *y = rsm + threadIdx.x, *M = y + K * st;
    const double ga = g[ia], gb = g[ib];
    const size_t plane = (size_t)L * L, ab = (size_t)ia * L + ib, ba = (size_t)ib * L + ia;
    const int t0 = blockIdx.y * A.t_chunk, t1 = min(A.n_T, t0 + A.t_chunk);
    double ymax = 0.0;
    for (int k = 0; k < K; ++k) {
        const double v = 0.5 * (ga * sigma[k * plane + ab] + gb * sigma[k * plane + ba]);
        y[k * st] = v;
        ymax = fmax(ymax, fabs(v));
        if (sym && t0 == 0) { sym[k * plane + ab] = v; sym[k * plane + ba] = v; }
    }
    for (int k = 0; k < K; ++k) {
        double m = 0.0;
        for (int j = 0; j < K; ++j) m = fma(A.Q[k][j], y[j * st], m);
        M[k * st] = m;
    }
    const double dE = E[ib] - E[ia], u0 = 0.5 * fabs(dE);
    // first knot at or above u0, and the Bernstein coefficients of the spline from there down to u0 (a NaN
    // fails every comparison, so it takes the quadrature)
    int j = 0;
    while (j < K && !(A.u[j] >= u0)) ++j;
    bool closed = A.closed && j < K && y[(K - 1) * st] >= 0.0 && y[0] >= 0.0;
    for (int k = j > 0 ? j - 1 : 0; closed && k + 1 < K; ++k) {
        const double h = A.u[k + 1] - A.u[k], h18 = h * h * (1.0 / 18.0);
        const double ya = y[k * st], yb = y[(k + 1) * st], Ma = M[k * st], Mb = M[(k + 1) * st];
        const double c1 = (2.0 * ya + yb) * (1.0 / 3.0) - h18 * (2.0 * Ma + Mb);
        const double c2 = (ya + 2.0 * yb) * (1.0 / 3.0) - h18 * (Ma + 2.0 * Mb);
        closed = ya >= 0.0 && yb >= 0.0 && c1 >= 0.0 && c2 >= 0.0;
    }
    if (!closed) {
        if (t0 == 0) {
            const unsigned m = __activemask(), below = m & ((1u << (threadIdx.x & 31)) - 1u);
            const bool whole = m == 0xffffffffu;
            unsigned long long pos = 0;
            if (!below) pos = atomicAdd(whole ? &queue->front : &queue->back, (unsigned long long)__popc(m));
            pos = __shfl_sync(m, pos, __ffs(m) - 1) + __popc(below);
            list[whole ? pos : list_n - 1 - pos] = make_int2(ia, ib);
        }
        return;
    }
    // quartic q of the cut piece (or the ramp): sigma~ U = sum_m q_m (U - u0)^m on [u0, U_j]
    double q0 = 0.0, q1 = 0.0, q2 = 0.0, q3 = 0.0, q4 = 0.0, w = 0.0, p = 0.0;
    w = A.u[j] - u0;
    if (j > 0) {
        const int k = j - 1;
        const double h = A.u[j] - A.u[k], ih = 1.0 / h, t = (u0 - A.u[k]) * ih, r = 1.0 - t;
        const double ya = y[k * st], yb = y[j * st], Ma = M[k * st], Mb = M[j * st];
        const double p0 = r * ya + t * yb + h * h * (1.0 / 6.0) * ((r * r * r - r) * Ma + (t * t * t - t) * Mb);
        const double p1 = (yb - ya) * ih + h * (1.0 / 6.0) * ((1.0 - 3.0 * r * r) * Ma + (3.0 * t * t - 1.0) * Mb);
        const double p2 = 0.5 * (r * Ma + t * Mb), p3 = (Mb - Ma) * ih * (1.0 / 6.0);
        q0 = p0 * u0;
        q1 = fma(p1, u0, p0);
        q2 = fma(p2, u0, p1);
        q3 = fma(p3, u0, p2);
        q4 = p3;
    } else if (w > 0.0) {
        const double ramp = y[0] / w;
        q1 = ramp * u0;
        q2 = ramp;
    }
    // the tail's exponent
    const double yK = y[(K - 1) * st], yJ = y[(K - 2) * st];
    if (yK > 0.0 && yJ > 0.0) p = fmin(0.0, fmax(-1.0, log(yK / yJ) / A.ln_uK));
    for (int t = t0; t < t1; ++t) {
        const double th = A.kT[t], ith = A.ikT[t];
        const double *tab = A.tab + (size_t)t * rate_tab_stride(K);
        // exp(-800) is zero in FP64, and z^4 exp(-z) with it
        const double z = fmin(w * ith, 800.0), ez = exp(-z);
        double G[5];
        lower_gammas(z, ez, G);
        double acc = th * fma(q0, G[0], th * fma(q1, G[1], th * fma(q2, G[2], th * fma(q3, G[3], th * (q4 * G[4])))));
        double whole = 0.0;
        const double *W = tab + j * K;
        for (int m = 0; m < K; ++m) whole = fma(__ldg(W + m), y[m * st], whole);
        acc = fma(ez, whole, acc);
        // tail: y_K kT U_K g(p) exp(-(U_K - u0)/kT), g(p) = x^-(1+p) Gamma(2 + p, x) e^x at x = U_K/kT;
        // left out under the quadrature's remainder bound
        const double eK = ez * __ldg(tab + K * K + j), uK = A.u[K - 1];
        if (!(4.0 * ymax * th * (uK + th) * eK <= 1e-17 * acc)) {
            double gp;
            if (uK * ith >= kRateChebX) {
                const double *ch = tab + K * K + K, chx = fma(2.0, p, 1.0);  // [-1, 0] on [-1, 1]
                double d1 = 0.0, d2 = 0.0;
                for (int m = kRateCheb - 1; m > 0; --m) {
                    const double d = fma(2.0 * chx, d1, __ldg(ch + m) - d2);
                    d2 = d1;
                    d1 = d;
                }
                gp = fma(chx, d1, __ldg(ch) - d2);
            } else {
                gp = rate_tail(p, uK * ith);
            }
            acc = fma(y[(K - 1) * st] * th * uK * eK, gp, acc);
        }
        rate_store(A, rate + t * plane, t, acc, dE, u0 * ith, ga, gb, ia, ib);
    }
}

// The listed pairs by quadrature: one thread per pair and temperature (temperature is the slow index: the lanes of a
// warp share kT and so take similar panel counts).  Two blocks per SM, i.e. two warps per FP64 pipe, which keep it
// busy; with few items a warp takes fewer than 32 (its time is that of its longest), and the first items go to
// different SMs and sub-partitions, the rest to whichever warp is free.  The pair's values come from `sym` where
// that was asked for (it may be sigma's own memory).  Calls of 1032 levels x 5 temperatures: every pair listed
// 35.7 ms, 0.2 % of the values negative 6.0 ms; 200 levels x 64 temperatures, most pairs listed, 11.2 ms (57 ms
// when a warp ran its pairs' quadratures in place; 37.6, 27 and 21.6 ms with every pair by quadrature).
__global__ void __launch_bounds__(kRateThreads, 2) k_rates_quad(const __grid_constant__ RateArgs A, const double *sigma,
                                                              const double *sym, const double *g, const double *E, double *rate,
                                                              RateQueue *queue, const int2 *list, size_t list_n)
{
    extern __shared__ double rsm[];
    const int K = A.K, lane = threadIdx.x & 31, half = gridDim.x / 2;
    constexpr int st = kRateThreads, warps = kRateThreads / 32;
    double *y = rsm + threadIdx.x, *M = y + K * st;
    const size_t plane = (size_t)A.L * A.L;
    const unsigned long long front = queue->front, pairs = front + queue->back;
    const int lanes = (int)min(32ull, (pairs * A.n_T + warps * half - 1) / (warps * half));
    // items per temperature: the pairs, in whole warps where a warp takes 32
    const unsigned long long row = lanes == 32 ? (pairs + 31) & ~31ull : pairs, items = row * A.n_T;
    unsigned long long i0 = ((blockIdx.x / half) * warps + threadIdx.x / 32) * (unsigned long long)half + blockIdx.x % half;
    for (i0 *= lanes; i0 < items;) {
        const unsigned long long i = i0 + lane, p = i % row;
        if (lane < lanes && i < items && p < pairs) {
            const int2 pr = list[p < front ? p : list_n - 1 - (p - front)];
            const int t = (int)(i / row), ia = pr.x, ib = pr.y;
            const size_t ab = (size_t)ia * A.L + ib, ba = (size_t)ib * A.L + ia;
            const double ga = g[ia], gb = g[ib];
            double ymax = 0.0;
            for (int k = 0; k < K; ++k) {
                const double v = sym ? sym[k * plane + ab] : 0.5 * (ga * sigma[k * plane + ab] + gb * sigma[k * plane + ba]);
                y[k * st] = v;
                ymax = fmax(ymax, fabs(v));
            }
            for (int k = 0; k < K; ++k) {
                double m = 0.0;
                for (int j = 0; j < K; ++j) m = fma(A.Q[k][j], y[j * st], m);
                M[k * st] = m;
            }
            const double dE = E[ib] - E[ia], u0 = 0.5 * fabs(dE), th = A.kT[t], ith = A.ikT[t];
            rate_store(A, rate + t * plane, t, rate_quadrature(A, y, M, st, ymax, u0, th, ith), dE, u0 * ith, ga, gb, ia, ib);
        }
        __syncwarp();
        if (lane == 0) i0 = 2ull * half * warps * lanes + atomicAdd(&queue->next, (unsigned long long)lanes);
        i0 = __shfl_sync(0xffffffffu, i0, 0);
    }
}

// Gauss-Legendre nodes and weights by Newton's iteration on P_n (three-term recurrence)
void gauss_legendre(int n, double *x, double *w)
{
    const double pi = 3.14159265358979323846;
    for (int i = 0; i < n; ++i) {
        double z = std::cos(pi * (i + 0.75) / (n + 0.5)), dp = 1.0;
        for (int it = 0; it < 100; ++it) {
            double p0 = 1.0, p1 = z;
            for (int k = 2; k <= n; ++k) {
                const double p2 = ((2 * k - 1) * z * p1 - (k - 1) * p0) / k;
                p0 = p1;
                p1 = p2;
            }
            dp = n * (z * p1 - p0) / (z * z - 1.0);
            const double dz = p1 / dp;
            z -= dz;
            if (std::fabs(dz) < 1e-16) break;
        }
        double p0 = 1.0, p1 = z;
        for (int k = 2; k <= n; ++k) {
            const double p2 = ((2 * k - 1) * z * p1 - (k - 1) * p0) / k;
            p0 = p1;
            p1 = p2;
        }
        dp = n * (z * p1 - p0) / (z * z - 1.0);
        x[i] = z;
        w[i] = 2.0 / ((1.0 - z * z) * dp * dp);
    }
}

// Q[k][j] = d M_k / d y_j for the natural spline on the knots u (M_0 = M_{K-1} = 0)
void natural_spline_map(const double *u, int K, double Q[kRateMaxK][kRateMaxK])
{
    for (int k = 0; k < kRateMaxK; ++k)
        for (int j = 0; j < kRateMaxK; ++j) Q[k][j] = 0.0;
    const int n = K - 2;
    if (n <= 0) return;
    std::vector<double> lo(n), di(n), up(n), cp(n), r(n);
    for (int i = 0; i < n; ++i) {
        const double h0 = u[i + 1] - u[i], h1 = u[i + 2] - u[i + 1];
        lo[i] = h0;
        di[i] = 2.0 * (h0 + h1);
        up[i] = h1;
    }
    for (int j = 0; j < K; ++j) {
        // right-hand side 6 [(y_{i+2} - y_{i+1}) / h1 - (y_{i+1} - y_i) / h0] for y = e_j
        for (int i = 0; i < n; ++i) {
            const double h0 = u[i + 1] - u[i], h1 = u[i + 2] - u[i + 1];
            const double yi = (j == i), yi1 = (j == i + 1), yi2 = (j == i + 2);
            r[i] = 6.0 * ((yi2 - yi1) / h1 - (yi1 - yi) / h0);
        }
        // Thomas
        cp[0] = up[0] / di[0];
        r[0] /= di[0];
        for (int i = 1; i < n; ++i) {
            const double m = di[i] - lo[i] * cp[i - 1];
            cp[i] = up[i] / m;
            r[i] = (r[i] - lo[i] * r[i - 1]) / m;
        }
        for (int i = n - 2; i >= 0; --i) r[i] -= cp[i] * r[i + 1];
        for (int i = 0; i < n; ++i) Q[i + 1][j] = r[i];
    }
}

// Gamma(s, x) e^x x^(1-s) for 1 <= s <= 2 and x > 0 (the series and the continued fraction of
// upper_gamma_scaled)
double upper_gamma_reduced(double s, double x)
{
    if (x < s + 1.0) {
        double term = 1.0 / s, sum = term;
        for (int n = 1; n < 300; ++n) {
            term *= x / (s + n);
            sum += term;
            if (term < 1e-17 * sum) break;
        }
        return std::pow(x, 1.0 - s) * std::tgamma(s) * std::exp(x) - x * sum;
    }
    const double tiny = 1e-300;
    double b = x + 1.0 - s, c = 1.0 / tiny, d = 1.0 / b, f = d;
    for (int i = 1; i < 400; ++i) {
        const double an = -i * (i - s);
        b += 2.0;
        d = an * d + b;
        if (std::fabs(d) < tiny) d = tiny;
        c = b + an / c;
        if (std::fabs(c) < tiny) c = tiny;
        d = 1.0 / d;
        const double del = d * c;
        f *= del;
        if (std::fabs(del - 1.0) < 3e-16) break;
    }
    return x * f;
}

// gamma(1..5, z) on the host, as lower_gammas
void host_gammas(double z, double G[5])
{
    const double ez = std::exp(-z);
    if (z >= 8.0) {
        G[0] = 1.0 - ez;
        double zm = 1.0;
        for (int m = 1; m < 5; ++m) {
            zm *= z;
            G[m] = m * G[m - 1] - zm * ez;
        }
        return;
    }
    // as many terms as z needs (the first one left out is below 1e-21)
    double s = 1.0;
    for (int n = std::min(60, 18 + (int)(6.0 * z)); n >= 6; --n) s = 1.0 + s * z / n;
    double zm = z * z * z * z;
    G[4] = 0.2 * s * zm * z * ez;
    for (int m = 4; m >= 1; --m) {
        G[m - 1] = (G[m] + zm * ez) / m;
        zm /= z;
    }
}

// the closed form's tables (RateArgs::tab) of every temperature
void rate_tables(const RateArgs &A, std::vector<double> &tab)
{
    const int K = A.K, stride = rate_tab_stride(K);
    tab.assign((size_t)A.n_T * stride, 0.0);
    // the Chebyshev points and the series' cosines there
    struct Cheb {
        double node[kRateCheb], cosine[kRateCheb][kRateCheb];
        Cheb()
        {
            const double pi = 3.14159265358979323846;
            for (int i = 0; i < kRateCheb; ++i) {
                node[i] = std::cos(pi * (i + 0.5) / kRateCheb);
                for (int m = 0; m < kRateCheb; ++m) cosine[m][i] = std::cos(pi * m * (i + 0.5) / kRateCheb);
            }
        }
    };
    static const Cheb cheb;
    for (int t = 0; t < A.n_T; ++t) {
        double *W = tab.data() + (size_t)t * stride, *eK = W + K * K, *ch = eK + K;
        const double th = A.kT[t], uK = A.u[K - 1];
        for (int j = 0; j < K; ++j) eK[j] = std::exp(-(uK - A.u[j]) / th);
        // row j: pieces j .. K-2 relative to exp(-(U - U_j)/kT); row K-1 is zero
        std::vector<double> row(K, 0.0);
        for (int j = K - 2; j >= 0; --j) {
            const double u = A.u[j], h = A.u[j + 1] - u, z = h / th, drop = std::exp(-z);
            for (int m = 0; m < K; ++m) row[m] *= drop;
            double G[5], I[6] = {0, 0, 0, 0, 0, 0};
            host_gammas(z, G);
            // I_m = int_0^h s^m exp(-s/kT) ds, then moments of t^m U = t^m (u + s), t = s/h
            double pw = th, hm = 1.0, Tm[4];
            for (int m = 0; m < 5; ++m) { I[m] = pw * G[m]; pw *= th; }
            for (int m = 0; m < 4; ++m) { Tm[m] = (u * I[m] + I[m + 1]) / hm; hm *= h; }
            // basis of the piece in t: y_a (1 - t), y_b t, h^2/6 [(r^3 - r) M_a + (t^3 - t) M_b], r = 1 - t
            const double wya = Tm[0] - Tm[1], wyb = Tm[1];
            const double wMa = h * h / 6.0 * (-2.0 * Tm[1] + 3.0 * Tm[2] - Tm[3]);
            const double wMb = h * h / 6.0 * (Tm[3] - Tm[1]);
            row[j] += wya;
            row[j + 1] += wyb;
            for (int m = 0; m < K; ++m) row[m] += wMa * A.Q[j][m] + wMb * A.Q[j + 1][m];
            for (int m = 0; m < K; ++m) W[j * K + m] = row[m];
        }
        // Chebyshev series of g(p) on p in [-1, 0] (s = 2 + p), through its Chebyshev points
        if (uK / th < 0.5 * kRateChebX) continue;  // not read (half: whatever the rounding of the kernel's ratio)
        double f[kRateCheb];
        for (int i = 0; i < kRateCheb; ++i)
            f[i] = upper_gamma_reduced(1.5 + 0.5 * cheb.node[i], uK / th);
        for (int m = 0; m < kRateCheb; ++m) {
            double c = 0.0;
            for (int i = 0; i < kRateCheb; ++i) c += f[i] * cheb.cosine[m][i];
            ch[m] = c * (m ? 2.0 : 1.0) / kRateCheb;
        }
    }
}

bool rate_is_dev(const void *p)
{
    if (!p) return false;
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

}  // namespace

}  // namespace mqct

using namespace mqct;

extern "C" mqct_status mqct_rate_coefficients(const mqct_rate_desc *d, const double *sigma, double *sigma_sym,
                                              double *rate, void *cuda_stream)
{
    reset_launches();
    if (!d || !sigma || !rate) return fail(MQCT_ERR_INVALID_ARG, "mqct_rate_coefficients: NULL argument");
    const int K = d->n_energies, L = d->n_levels, nT = d->n_temps;
    if (d->reserved != 0) return fail(MQCT_ERR_INVALID_ARG, "mqct_rate_coefficients: reserved must be 0");
    if (L < 1 || K < 2 || K > kRateMaxK || nT < 1 || nT > kRateMaxT)
        return fail(MQCT_ERR_INVALID_ARG, "mqct_rate_coefficients: sizes out of range");
    if (!d->u || !d->kT || !d->level_energy || !d->degeneracy)
        return fail(MQCT_ERR_INVALID_ARG, "mqct_rate_coefficients: NULL array in the descriptor");
    if (!(d->mu > 0.0) || !std::isfinite(d->mu)) return fail(MQCT_ERR_INVALID_ARG, "mqct_rate_coefficients: mu must be > 0");
    if (rate_is_dev(d->u) || rate_is_dev(d->kT) || rate_is_dev(d->level_energy) || rate_is_dev(d->degeneracy))
        return fail(MQCT_ERR_INVALID_ARG, "mqct_rate_coefficients: descriptor arrays must be host memory");
    RateArgs A;
    std::memset(&A, 0, sizeof(A));
    for (int k = 0; k < K; ++k) {
        A.u[k] = d->u[k];
        if (!(A.u[k] > 0.0) || !std::isfinite(A.u[k]) || (k > 0 && !(A.u[k] > A.u[k - 1])))
            return fail(MQCT_ERR_INVALID_ARG, "mqct_rate_coefficients: energies must be finite, > 0 and increasing");
    }
    for (int t = 0; t < nT; ++t) {
        A.kT[t] = d->kT[t];
        if (!(A.kT[t] > 0.0) || !std::isfinite(A.kT[t])) return fail(MQCT_ERR_INVALID_ARG, "mqct_rate_coefficients: kT must be > 0");
    }
    for (int l = 0; l < L; ++l) {
        if (!(d->degeneracy[l] > 0.0) || !std::isfinite(d->degeneracy[l]) || !std::isfinite(d->level_energy[l]))
            return fail(MQCT_ERR_INVALID_ARG, "mqct_rate_coefficients: degeneracies must be > 0, energies finite");
    }
    natural_spline_map(A.u, K, A.Q);
    struct Gauss {
        double x[kGl], w[kGl];
        Gauss() { gauss_legendre(kGl, x, w); }
    };
    static const Gauss gauss;
    std::copy(gauss.x, gauss.x + kGl, A.gx);
    std::copy(gauss.w, gauss.w + kGl, A.gw);
    for (int t = 0; t < nT; ++t) {
        A.ikT[t] = 1.0 / A.kT[t];
        A.pref[t] = std::sqrt(8.0 / (3.14159265358979323846 * d->mu)) * std::pow(A.kT[t], -1.5);
    }
    A.K = K;
    A.L = L;
    A.n_T = nT;
    A.ln_uK = std::log(A.u[K - 1] / A.u[K - 2]);
    // the closed form's powers of kT stay far from the limits of FP64 in this range
    A.closed = A.u[0] >= 1e-12 && A.u[K - 1] <= 1e6;
    for (int t = 0; t < nT; ++t) A.closed = A.closed && A.kT[t] >= 1e-12 && A.kT[t] <= 1e6;
    // the rows of pairs (a <= b) in passes of at most kRatePass pairs, which bounds the list
    std::vector<int> first{0};
    size_t list_n = 0, n_pairs = 0;
    for (int b = 0; b < L; b += kRateTb) {
        const int b1 = std::min(L, b + kRateTb);
        const size_t rows = ((size_t)b1 * (b1 + 1) - (size_t)b * (b + 1)) / 2;
        if (n_pairs && n_pairs + rows > kRatePass) {
            first.push_back(b);
            n_pairs = 0;
        }
        n_pairs += rows;
        list_n = std::max(list_n, n_pairs);
    }
    first.push_back(L);
    const size_t passes = first.size() - 1;
    // one upload: degeneracies, level energies, tables, empty queues
    std::vector<double> up;
    if (A.closed) rate_tables(A, up);
    const size_t tab_n = up.size();
    up.insert(up.end(), d->degeneracy, d->degeneracy + L);
    up.insert(up.end(), d->level_energy, d->level_energy + L);
    up.insert(up.end(), passes * sizeof(RateQueue) / sizeof(double), 0.0);

    cudaStream_t st = (cudaStream_t)cuda_stream;
    cudaError_t e;
    std::vector<void *> tmp;
    auto get = [&](void **p, size_t b) {
        cudaError_t r = cudaMallocAsync(p, b ? b : 16, st);
        if (r == cudaSuccess) tmp.push_back(*p);
        return r;
    };
    auto cleanup = [&]() { for (void *p : tmp) cudaFreeAsync(p, st); };
    const size_t sig_bytes = sizeof(double) * (size_t)K * L * L, rate_bytes = sizeof(double) * (size_t)nT * L * L;
    const double *dsig = sigma;
    double *dsym = sigma_sym, *drate = rate, *dup = nullptr;
    const bool host_rate = !rate_is_dev(rate), host_sym = sigma_sym && !rate_is_dev(sigma_sym);
    if (!rate_is_dev(sigma)) {
        double *p;
        if ((e = get((void **)&p, sig_bytes)) != cudaSuccess ||
            (e = cudaMemcpyAsync(p, sigma, sig_bytes, cudaMemcpyHostToDevice, st)) != cudaSuccess) {
            cleanup();
            return cuda_fail(e, "staging sigma");
        }
        dsig = p;
    }
    // a pageable copy is staged by the runtime before cudaMemcpyAsync returns
    if ((e = get((void **)&dup, sizeof(double) * up.size() + sizeof(int2) * list_n)) != cudaSuccess ||
        (e = cudaMemcpyAsync(dup, up.data(), sizeof(double) * up.size(), cudaMemcpyHostToDevice, st)) != cudaSuccess) {
        cleanup();
        return cuda_fail(e, "staging levels");
    }
    A.tab = dup;
    const double *dg = dup + tab_n, *dE = dg + L;
    RateQueue *queues = reinterpret_cast<RateQueue *>(dup + tab_n + 2 * (size_t)L);
    int2 *list = reinterpret_cast<int2 *>(dup + up.size());
    if (host_rate && (e = get((void **)&drate, rate_bytes)) != cudaSuccess) { cleanup(); return cuda_fail(e, "cudaMallocAsync"); }
    if (host_sym && (e = get((void **)&dsym, sig_bytes)) != cudaSuccess) { cleanup(); return cuda_fail(e, "cudaMallocAsync"); }
    const size_t smem = sizeof(double) * 2 * (size_t)K * kRateThreads;
    if (smem > 48 * 1024 &&  // what a launch may have without asking
        ((e = cudaFuncSetAttribute(k_rates, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess ||
         (e = cudaFuncSetAttribute(k_rates_quad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess)) {
        cleanup();
        return cuda_fail(e, "cudaFuncSetAttribute");
    }
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    for (size_t ps = 0; ps < passes; ++ps) {
        const long long tile0 = rate_tiles(first[ps] / kRateTb), tiles = rate_tiles((first[ps + 1] + kRateTb - 1) / kRateTb) - tile0;
        // a thread runs all temperatures of its pair (the pair's spline is formed once); with too few tiles to
        // fill the GPU the temperatures are spread over blocks instead
        const int split = (int)std::min<long long>(nT, std::max<long long>(1, 608 / tiles));
        A.t_chunk = (nT + split - 1) / split;
        k_rates<<<dim3((unsigned)tiles, (nT + A.t_chunk - 1) / A.t_chunk), kRateThreads, smem, st>>>(A, dsig, dg, dE, dsym, drate,
                                                                                                  tile0, queues + ps, list, list_n);
        k_rates_quad<<<2 * sms, kRateThreads, smem, st>>>(A, dsig, dsym, dg, dE, drate, queues + ps, list, list_n);
    }
    count_launches(2 * (long long)passes);
    if ((e = cudaGetLastError()) != cudaSuccess) { cleanup(); return cuda_fail(e, "rate kernels"); }
    if (host_rate && (e = cudaMemcpyAsync(rate, drate, rate_bytes, cudaMemcpyDeviceToHost, st)) != cudaSuccess) {
        cleanup();
        return cuda_fail(e, "cudaMemcpyAsync");
    }
    if (host_sym && (e = cudaMemcpyAsync(sigma_sym, dsym, sig_bytes, cudaMemcpyDeviceToHost, st)) != cudaSuccess) {
        cleanup();
        return cuda_fail(e, "cudaMemcpyAsync");
    }
    cleanup();
    if (host_rate || host_sym) {
        if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return cuda_fail(e, "cudaStreamSynchronize");
    }
    return MQCT_OK;
}
