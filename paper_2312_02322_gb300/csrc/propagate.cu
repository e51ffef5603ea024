// Persistent RK4 trajectory kernels and mqct_propagate.
//
// One CTA integrates one trajectory at a time, claiming trajectories from a device
// work queue (longest estimated first) until the queue is empty; the whole RK4 loop of a
// trajectory runs on the device with its amplitudes resident in shared memory.  The warps have
// three roles; per RK4 stage (Eqs. 4-10):
//   element warps  16 rows at a time, two lanes per row (real and imaginary part): the coupling
//       w = M(R) c, u = M'(R) c of the phase-rotated stage amplitudes c = exp(-i E t_s) a_s over the
//       32-row sliced-ELL slices
//         PLAIN:      M_nm(R) from the spline table of Sec. III, M = sum_p T_p x^p,
//                     computed as w = sum_p x^p (T_p c), u = sum_p p x^(p-1) (T_p c);
//         FACTORISED: w = sum_l v_l(R) (G^l c), u = sum_l v_l'(R) (G^l c)  (Eq. 12);
//       then, in the same pass, da/dt = conj(p) (-i w + (dPhi/dt / 2) (J+ - J-) c) (Eq. 5; p the phase
//       factor, the ladder partners share it), the RK4 accumulation and the next stage's c into the
//       other of two buffers, with the sums of force, torque Re(c^dag (J+ - J-) w) = -Re(((J+ - J-) c)^dag w)
//       (Eq. 10) and, at stage 0, diagnostics;
//   classical warp the stage update of R, P_R, Phi, P_Phi (Eqs. 7-9), half a stage behind: while the
//       element warps contract stage s it sums the force and torque of stage s-1, publishes dPhi/dt
//       of stage s (an mbarrier the element warps wait on before their update) and looks ahead to
//       the spline quantities of stage s+1, whose R depends on P_R of stage s only;
//   phase warp     the phase factors of the stage times ahead; phase arguments E_n t are FP64 and
//       evaluated per level (states of a level share E_n).
// One barrier per stage.  Bound by the FP64 pipe (one warp instruction per 64 cycles and sub-partition):
// the passes are ordered for the fewest FP64 instructions, and no chain of them runs while the
// element warps wait.  Measured against a kernel that wrote w to shared memory for a second pass (two
// barriers and one thread's FP64 chain per stage): N = 49, 32 trajectories 34 -> 12 us per step; N = 441 PLAIN, 256
// trajectories 471 -> 297 ms (FP64 pipe 75 -> 89 % busy, 14 % fewer FP64 instructions, 15 % fewer padded
// entries); N = 210 FACTORISED, 304 trajectories 424 -> 244 ms.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cub/device/device_radix_sort.cuh>
#include <cub/device/device_select.cuh>
#include <type_traits>
#include <vector>

#include "internal.h"
#include "mqct_probe.h"
#include "tc_ptx.cuh"
#include "traj_common.cuh"

namespace mqct {

constexpr int kPropElem = 14;              // element warps at most
constexpr long long kPropWait = 1ll << 17;  // polls of at most ~1 us

struct Ctl {
    double q[4], qs[4], lacc[4], q0[4];  // classical state, stage input, accumulator; start of an adaptive step
    double ir, i2m, phid, t1, dinv;      // current stage: 1/R, 1/(mu R^2), dPhi/dt, P_Phi^2/(mu R^3), dx/dR
    double r_n, ir_n, i2m_n, dinv_n;     // looked ahead (dx/dR of the spline variable: 1, or 1/R on the log grid)
    double i2m0, vid0;                   // of stage 0, for the diagnostics
    // per stage parity: dPhi/dt / 2; offset in the interval, 2 x and 3 x^2; identity terms' v and v'; v_l, v_l'
    double hp[2], x[2], x2[2], x3[2], vid[2], dvid[2];
    double v[2][kMaxTerms], dv[2][kMaxTerms];
    double imu, h, hh, h6, t0, r_end;    // 1/mu; length of the step, its half and sixth; start time
    double line_b, line_v, line_t0;      // prescribed straight line (MQCT_PRESCRIBED_TRAJ)
    double e0, j0, ndev, edev, jdev;
    double err, tcur;
    double red[kPropElem][6];            // sums of one stage per element warp
    int kint[2];
    int below_n, status, steps, done, max_steps, item;
    int timeout;                         // a bounded wait ran out: the trajectory's results are void
    __align__(8) uint64_t published;     // mbarrier: classical and phase warp are done with what a stage needs
};

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// spline of the expansion terms at R (factorised path and initial mean field)
__device__ __forceinline__ void term_at(const DevSys &S, int l, int k, double x, double &v, double &dv)
{
    dbl4 c = S.vcoef[(size_t)l * S.n_int + k];
    v = c.x + x * (c.y + x * (c.z + x * c.w));
    dv = c.y + x * (2.0 * c.z + 3.0 * x * c.w);
}

// prescribed straight line at time t
__device__ __forceinline__ double line_r(const Ctl &c, double t)
{
    const double s = c.line_v * (t - c.line_t0);
    return sqrt(c.line_b * c.line_b + s * s);
}

// ---- classical warp (every function is called by all 32 lanes; lane 0 writes) ----------------

// spline quantities at R into the slot of parity `par`, and the looked-ahead 1/R etc.
__device__ void cls_look(const DevSys &S, Ctl &c, int lane, double R, int par)
{
    int k;
    double x;
    bool below;
    locate_interval(S, R, k, x, below);
    const double dinv = S.grid_log ? 1.0 / R : 1.0;
    const bool fact = S.path == MQCT_PATH_FACTORISED;
    if (lane == 0) {
        c.kint[par] = k;
        c.x[par] = x;
        c.x2[par] = 2.0 * x;
        c.x3[par] = 3.0 * x * x;
        c.below_n = R < S.r_min;
        c.r_n = R;
        c.dinv_n = dinv;
    }
    if (fact)
        for (int l = lane; l < S.L; l += 32) {
            double v, dv;
            term_at(S, l, k, x, v, dv);
            c.v[par][l] = v;
            c.dv[par][l] = dv * dinv;
        }
    __syncwarp();
    if (fact || (S.flags & MQCT_DECOUPLED_TRAJ)) {
        // the identity terms' sum (also the isotropic potential that drives the decoupled motion)
        double vid = 0.0, dvid = 0.0;
        for (unsigned long long m = S.id_mask; m; m &= m - 1) {
            const int l = __ffsll((long long)m) - 1;
            double v, dv;
            if (fact) { v = c.v[par][l]; dv = c.dv[par][l]; }
            else { term_at(S, l, k, x, v, dv); dv *= dinv; }
            vid += v;
            dvid += dv;
        }
        if (lane == 0) { c.vid[par] = vid; c.dvid[par] = dvid; }
    }
    const double ir = 1.0 / R, i2m = c.imu * ir * ir;
    if (lane == 0) { c.ir_n = ir; c.i2m_n = i2m; }
    __syncwarp();
}

// the looked-ahead stage becomes the current one
__device__ void cls_enter(const DevSys &S, Ctl &c, int lane)
{
    const double ir = c.ir_n, i2m = c.i2m_n, pp = c.qs[3];
    const double phid = (S.flags & MQCT_PRESCRIBED_TRAJ) ? c.line_b * c.line_v * (ir * ir) : pp * i2m;
    const double t1 = pp * phid * ir;
    __syncwarp();
    if (lane == 0) {
        c.ir = ir; c.i2m = i2m; c.dinv = c.dinv_n; c.phid = phid; c.t1 = t1;
        if (c.below_n) c.status |= MQCT_TRAJ_TABLE_RANGE;
    }
    __syncwarp();
}

// looks ahead from stage s of the step (t_next: time of its end on the prescribed line)
__device__ void cls_ahead(const DevSys &S, Ctl &c, int lane, int s, double t_next)
{
    double R;
    if (S.flags & MQCT_PRESCRIBED_TRAJ) {
        R = line_r(c, s == 3 ? t_next : (s == 2 ? c.t0 + c.h : c.t0 + 0.5 * c.h));
    } else {
        double lacc = c.lacc[0];
        stage_component(s, c.imu, c.qs[1], 0.0, c.hh, c.h, c.h6, c.q[0], R, lacc);
    }
    __syncwarp();
    cls_look(S, c, lane, R, (s + 1) & 1);
}

// the classical update of stage sp from its sums; afterwards the stage quantities are those of the
// next stage
__device__ void cls_advance(const DevSys &S, Ctl &c, int lane, int sp, int nelem)
{
    const unsigned full = 0xffffffffu;
    // lanes 0-7 sum the force, 8-15 the torque (16-31 copies)
    const int w = lane & 7;
    double v = w < nelem ? c.red[w][(lane >> 3) & 1] : 0.0;
    if (nelem > 8) v += w + 8 < nelem ? c.red[w + 8][(lane >> 3) & 1] : 0.0;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(full, v, o);
    double F = -__shfl_sync(full, v, 0), T = -__shfl_sync(full, v, 8);
    if (S.path == MQCT_PATH_PLAIN && S.grid_log) F *= c.dinv;
    if (S.flags & MQCT_DECOUPLED_TRAJ) { F = -c.dvid[sp & 1]; T = 0.0; }  // isotropic potential alone, no torque
    const bool presc = S.flags & MQCT_PRESCRIBED_TRAJ;                    // the motion is prescribed
    const int sc = lane & 3;
    const double q = c.q[sc], pr = c.qs[1];
    const double X = presc ? 0.0 : (sc == 0 ? pr : (sc == 1 ? F : (sc == 2 ? c.phid : T)));
    const double alpha = sc == 0 ? c.imu : 1.0, beta = sc == 1 && !presc ? c.t1 : 0.0;
    double qs = c.qs[sc], lacc = c.lacc[sc];
    stage_component(sp, alpha, X, beta, c.hh, c.h, c.h6, q, qs, lacc);
    if (presc && sc == 0) qs = c.r_n;
    const bool bad = __any_sync(full, !finite64(qs)) && sp == 3;
    if (lane == 0 && sp == 0) { c.i2m0 = c.i2m; c.vid0 = c.vid[0]; }
    if (lane < 4) {
        c.qs[sc] = qs;
        c.lacc[sc] = lacc;
        if (sp == 3) c.q[sc] = qs;
    }
    if (lane == 0 && bad) { c.status |= MQCT_TRAJ_NONFINITE; c.done = 1; }
    __syncwarp();
    if (!bad) cls_enter(S, c, lane);
}

// total energy, P_Phi + <J_y> and norm of the state at the start of a step (or of the final state) from
// its stage-0 sums: running maxima of their deviations; `first` sets the reference values
__device__ void cls_bookkeeping(const DevSys &S, Ctl &c, int lane, int nelem, bool first)
{
    const unsigned full = 0xffffffffu;
    // lanes 8 k .. 8 k + 7 sum quantity k of (V, <J_y>, |a|^2, E|a|^2)
    const int w = lane & 7;
    double v = w < nelem ? c.red[w][2 + (lane >> 3)] : 0.0;
    if (nelem > 8) v += w + 8 < nelem ? c.red[w + 8][2 + (lane >> 3)] : 0.0;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(full, v, o);
    const double V = __shfl_sync(full, v, 0), JY = __shfl_sync(full, v, 8);
    const double NR = __shfl_sync(full, v, 16), ER = __shfl_sync(full, v, 24);
    const double PR = c.q[1], PP = c.q[3];
    const bool dec = S.flags & MQCT_DECOUPLED_TRAJ;
    const double et = 0.5 * (c.imu * PR * PR + PP * PP * c.i2m0) + (dec ? c.vid0 : ER + V);
    const double jt = dec ? PP : PP + 0.5 * JY;
    if (lane == 0) {
        if (first) { c.e0 = et; c.j0 = jt; }
        c.ndev = fmax(c.ndev, fabs(NR - 1.0));
        c.edev = fmax(c.edev, fabs(et - c.e0));
        c.jdev = fmax(c.jdev, fabs(jt - c.j0));
    }
    __syncwarp();
}

// ---- phase warp: factors exp(-i E_l t) of every level -----------------------------------------
__device__ void phase_factors(const DevSys &S, int lane, double t, double2 *PH)
{
    for (int l = lane; l < S.n_levels; l += 32) {
        double sn, cs;
        sincos(S.lev_energy[l] * t, &sn, &cs);
        PH[l] = make_double2(cs, -sn);
    }
}

// ---- element warps -----------------------------------------------------------------------------

// one component (real or imaginary part) of w = M c and u = M' c for the lane's row; u without dx/dR
// on the PLAIN path (cls_advance applies it to the force)
__device__ __forceinline__ void coupling_row(const DevSys &S, const Ctl &c, int par, const double *__restrict__ Cc,
                                             int sl, int rl, double c0, double &w, double &u)
{
    if (S.path == MQCT_PATH_PLAIN) {
        const int off = S.sl_off[sl], width = (S.sl_off[sl + 1] - off) / kSlice;
        const size_t base = (size_t)c.kint[par] * S.nnz_pad + off + rl;
        const double2 *t01 = S.T01 + base, *t23 = S.T23 + base;
        const int *cl = S.cols + off + rl;
        double u0 = 0.0, u1 = 0.0, u2 = 0.0, u3 = 0.0;
#pragma unroll 3
        for (int k = 0; k < width; ++k) {
            const double2 a = __ldg(t01 + k * kSlice), b = __ldg(t23 + k * kSlice);
            const double z = Cc[2 * __ldg(cl + k * kSlice)];
            u0 = fma(a.x, z, u0);
            u1 = fma(a.y, z, u1);
            u2 = fma(b.x, z, u2);
            u3 = fma(b.y, z, u3);
        }
        const double x = c.x[par];
        w = fma(x, fma(x, fma(x, u3, u2), u1), u0);
        u = fma(c.x3[par], u3, fma(c.x2[par], u2, u1));
    } else {
        w = c.vid[par] * c0;
        u = c.dvid[par] * c0;
        for (int f = 0; f < S.n_f; ++f) {
            const int *so = S.f_sl_off + (size_t)f * (S.n_slices + 1);
            const int off = __ldg(so + sl), width = (__ldg(so + sl + 1) - off) / kSlice;
            const int *cl = S.f_cols + off + rl;
            const double *gv = S.f_val + off + rl;
            double y = 0.0;
#pragma unroll 4
            for (int k = 0; k < width; ++k) y = fma(__ldg(gv + k * kSlice), Cc[2 * __ldg(cl + k * kSlice)], y);
            const int l = __ldg(S.f_term + f);
            w = fma(c.v[par][l], y, w);
            u = fma(c.dv[par][l], y, u);
        }
    }
}

// one stage of every row: S0 is stage 0 (diagnostics; with c.done the sums only, no update)
template <bool S0>
__device__ __forceinline__ void elem_stage(const DevSys &S, Ctl &c, int s, int nelem, unsigned phase, double *A, double *ACC,
                                           double *C0, double *C1, const double2 *PHa, const double2 *PHb)
{
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int cp = lane & 1, par = s & 1, n = S.n, n_half = (n + 15) >> 4;
    const double *Cc = (par ? C1 : C0) + cp;
    double *Cn = (par ? C0 : C1) + cp;
    const double2 *PHc = (S0 || s == 3) ? PHa : PHb, *PHn = (S0 || s == 1) ? PHb : PHa;
    const double hb = (!S0 && s == 3) ? c.h6 : (s == 2 ? c.h : c.hh);
    double f = 0.0, t = 0.0, ve = 0.0, jy = 0.0, nr = 0.0, er = 0.0;
    // every lane of the warp waits for the views of this stage, and the warp converges again afterwards (bounded;
    // after one wait ran out the trajectory's others return at once)
    auto wait = [&]() {
        if (!*(volatile int *)&c.timeout && !tc_mbar_wait(&c.published, phase & 1u, kPropWait)) c.timeout = 1;
        __syncwarp();
    };
    // the last (shortest) row groups go to the warps that share an FP64 pipe with the classical and the phase
    // warp when nelem is a multiple of 4
    const int hs0 = nelem > 1 ? (warp + nelem - 2) % nelem : 0;
    if (hs0 >= n_half) wait();
    for (int hs = hs0; hs < n_half; hs += nelem) {
        const int r = 16 * hs + (lane >> 1);
        const bool on = r < n;
        const int rr = on ? r : 0;
        const double c0 = on ? Cc[2 * rr] : 0.0;
        double w, u;
        coupling_row(S, c, par, Cc, hs >> 1, 16 * (hs & 1) + (lane >> 1), c0, w, u);
        const double dc = on ? S.adn[rr] * Cc[2 * S.dn[rr]] - S.aup[rr] * Cc[2 * S.up[rr]] : 0.0;
        if (hs == hs0) wait();
        f = fma(c0, u, f);
        t = fma(dc, w, t);
        const double a0 = A[2 * rr + cp];
        if (S0) {
            const double dc_o = __shfl_xor_sync(full, dc, 1);
            const double a1 = on ? a0 : 0.0, pp = a1 * a1;
            ve = fma(c0, w, ve);
            jy = fma(c0, cp ? -dc_o : dc_o, jy);  // Im(c^dag D c): the phases of a level's states cancel
            nr += pp;
            er = fma(S.lev_energy[S.lev[rr]], pp, er);
            if (c.done) continue;
        }
        const int lev = S.lev[rr];
        const double2 p = PHc[lev];
        const double w_o = __shfl_xor_sync(full, w, 1);
        const double z = fma(c.hp[par], dc, cp ? -w_o : w_o);
        const double z_o = __shfl_xor_sync(full, z, 1);
        const double k = fma(cp ? -p.y : p.y, z_o, p.x * z);
        double acc = k;
        if (!S0) acc = fma(s == 3 ? 1.0 : 2.0, k, ACC[2 * rr + cp]);
        const double y = fma(hb, (!S0 && s == 3) ? acc : k, a0);
        const double y_o = __shfl_xor_sync(full, y, 1);
        // the next stage's time differs from this one's at stages 0 and 2 only
        const double2 q = (S0 || s == 2) ? PHn[lev] : p;
        const double cn = fma(cp ? q.y : -q.y, y_o, q.x * y);
        if (on) {
            if (!S0 && s == 3) A[2 * rr + cp] = y;
            else ACC[2 * rr + cp] = acc;
            Cn[2 * rr] = cn;
        }
    }
    __syncwarp();
    // sums over the warp, two (stage 0: six) quantities with one exchange per halving of what a lane carries
    {
        const bool hi = lane & 16;
        double v = (hi ? t : f) + __shfl_xor_sync(full, hi ? f : t, 16);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(full, v, o);
        if ((lane & 15) == 0) c.red[warp][lane >> 4] = v;
    }
    if (S0) {
        const bool h4 = lane & 16, h3 = lane & 8;
        const double a = (h4 ? nr : ve) + __shfl_xor_sync(full, h4 ? ve : nr, 16);
        const double b = (h4 ? er : jy) + __shfl_xor_sync(full, h4 ? jy : er, 16);
        double v = (h3 ? b : a) + __shfl_xor_sync(full, h3 ? a : b, 8);
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(full, v, o);
        if ((lane & 7) == 0) c.red[warp][2 + (lane >> 3)] = v;  // (V, <J_y>, |a|^2, E|a|^2)
    }
    __syncwarp();
}

// T threads at most, MINB CTAs per SM at least (register budget): <320, 2> up to eight element warps, else <512, 1>
template <int T, int MINB>
__global__ void __launch_bounds__(T, MINB) k_propagate_fp64(PropArgs a)
{
    extern __shared__ double2 smem[];
    __shared__ Ctl c;
    __shared__ DevSys S;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nelem = (blockDim.x >> 5) - 2, nte = 32 * nelem;
    const bool elem = warp < nelem, classical = warp == nelem;  // the last warp is the phase warp
    const int NN = a.smem_n;
    double2 *A = smem, *ACC = A + NN, *C0 = ACC + NN, *C1 = C0 + NN;
    double2 *PHa = C1 + NN, *PHb = PHa + a.smem_lev;
    double2 *A0 = PHb + a.smem_lev, *A1 = A0 + NN;  // adaptive steps only (a.adapt)
    double *Ad = reinterpret_cast<double *>(A), *ACCd = reinterpret_cast<double *>(ACC);
    double *C0d = reinterpret_cast<double *>(C0), *C1d = reinterpret_cast<double *>(C1);
    unsigned phase = 0;  // stages published so far (parity of the mbarrier)
    if (tid == 0) tc_mbar_init(&c.published, 2);

    for (;;) {
        if (tid == 0) c.item = atomicAdd(a.queue, 1);
        __syncthreads();
        const int item = c.item;
        if (item >= a.n) break;
        const int t = a.order ? a.order[item] : item;
        const mqct_traj tr = a.trajs[t];
        // trajectories that live in device memory were not seen by the host: validate here
        bool ok = tr.system_idx >= 0 && tr.system_idx < a.n_systems && tr.dt > 0.0 && tr.e_coll > 0.0 &&
                  tr.b >= 0.0 && tr.r0 > 0.0 && tr.b < tr.r0 && isfinite(tr.r_end) && tr.max_steps >= 0;
        if (ok) ok = tr.init_state >= 0 && tr.init_state < a.sys[tr.system_idx].n;
        if (!ok) {
            if (a.diag && tid == 0) {
                mqct_diag d = {0, MQCT_TRAJ_INVALID, 0.0, 0.0, 0.0, 0.0};
                a.diag[t] = d;
            }
            __syncthreads();
            continue;
        }
        if (tid == 0) {
            S = a.sys[tr.system_idx];
            c.timeout = a.fail_every > 0 && (item + 1) % a.fail_every == 0;
            if (a.t_start) a.t_start[t] = mqct_clock_ns();
        }
        __syncthreads();
        const int n = S.n;
        const int s0 = S.inv[tr.init_state];
        const bool adaptive = S.adapt_tol > 0.0, presc = S.flags & MQCT_PRESCRIBED_TRAJ;
        const double dt = tr.dt;
        // ---- initial state
        if (elem) {
            for (int r = tid; r < n; r += nte) {
                double2 v = make_double2(r == s0 ? 1.0 : 0.0, 0.0);
                A[r] = v; C0[r] = v;  // phase at t = 0 is 1
            }
        } else if (classical) {
            int k;
            double x;
            bool below;
            locate_interval(S, tr.r0, k, x, below);
            const bool dec = S.flags & MQCT_DECOUPLED_TRAJ;
            double m00 = 0.0;
            for (int l = lane; l < S.L; l += 32) {
                double v, dv;
                term_at(S, l, k, x, v, dv);
                // decoupled motion starts in the isotropic potential, not the state's mean field
                m00 += dec ? (((S.id_mask >> l) & 1ull) ? v : 0.0) : v * S.diag_g[(size_t)l * n + s0];
            }
            m00 = warp_sum(m00);
            double q4[4];
            initial_state(S, tr, m00, q4);
            if (lane == 0) {
                c.imu = 1.0 / S.mu;
                c.h = dt; c.hh = 0.5 * dt; c.h6 = dt / 6.0; c.t0 = 0.0; c.r_end = tr.r_end; c.max_steps = tr.max_steps;
                if (presc) {
                    // the straight line R(t) = sqrt(b^2 + v^2 (t - t_0)^2), time-symmetric about t_0
                    c.line_b = tr.b;
                    c.line_v = sqrt(2.0 * tr.e_coll / S.mu);
                    c.line_t0 = 0.5 * tr.max_steps * tr.dt;
                    q4[0] = line_r(c, 0.0);
                    q4[1] = q4[2] = q4[3] = 0.0;
                }
                for (int i = 0; i < 4; ++i) { c.q[i] = c.qs[i] = q4[i]; c.lacc[i] = 0.0; }
                c.status = tr.max_steps <= 0 ? MQCT_TRAJ_MAX_STEPS : 0;
                c.steps = 0;
                c.done = tr.max_steps <= 0;
                c.ndev = c.edev = c.jdev = 0.0;
                c.tcur = 0.0;
            }
            __syncwarp();
            cls_look(S, c, lane, c.q[0], 0);
            cls_enter(S, c, lane);
        } else {
            for (int l = lane; l < S.n_levels; l += 32) PHa[l] = make_double2(1.0, 0.0);
            phase_factors(S, lane, 0.5 * dt, PHb);  // fixed steps: the first half time
        }
        __syncthreads();

        // one stage: the element warps' pass beside the classical and the phase warp's work.  `adv`: the
        // stage before is to be advanced (not the first stage of a trajectory or of an adaptive trial)
        auto stage = [&](int s, bool adv, bool first_step, double t_next) {
            if (elem) {
                if (s == 0) elem_stage<true>(S, c, s, nelem, phase, Ad, ACCd, C0d, C1d, PHa, PHb);
                else elem_stage<false>(S, c, s, nelem, phase, Ad, ACCd, C0d, C1d, PHa, PHb);
            } else if (classical) {
                if (adv) {
                    cls_advance(S, c, lane, (s + 3) & 3, nelem);
                    if (s == 0 && lane == 0) {  // end of a fixed step
                        c.steps += 1;
                        c.tcur = c.steps * dt;
                        c.t0 = c.tcur;
                        if (!(c.status & MQCT_TRAJ_NONFINITE)) {
                            if (!presc && c.q[0] >= c.r_end && c.q[1] > 0.0) c.done = 1;
                            else if (c.steps >= c.max_steps) {
                                c.status |= presc ? 0 : MQCT_TRAJ_MAX_STEPS;
                                c.done = 1;
                            }
                        }
                    }
                }
                if (lane == 0) c.hp[s & 1] = 0.5 * c.phid;
                __syncwarp();
                if (lane == 0) tc_mbar_arrive(&c.published);
                if (s > 0 || !c.done) {
                    cls_ahead(S, c, lane, s, t_next);
                    if (s == 1) cls_bookkeeping(S, c, lane, nelem, first_step);
                }
            } else {
                // phases: t + h once stage 0 has read those of t; the half time ahead of the step that reads
                // it (adaptive steps: during its stage 0, their length is known no earlier)
                if (s == 0 && adaptive) {
                    phase_factors(S, lane, c.t0 + 0.5 * c.h, PHb);
                    __syncwarp();
                }
                if (lane == 0) tc_mbar_arrive(&c.published);
                if (s == 1) phase_factors(S, lane, c.t0 + c.h, PHa);
                if (s == 3 && !adaptive) phase_factors(S, lane, (c.steps + 1) * dt + 0.5 * dt, PHb);
            }
            ++phase;
            __syncwarp();
            __syncthreads();
        };

        if (adaptive) {
            // step doubling (the adaptive step of Sec. III in the reading of the header): one step of
            // h against two of h/2 from the same state; the two-half result is kept when
            // max_n |a_n(halves) - a_n(one step)| <= tol or h = dt, else h halves and the step is
            // retried; h doubles (up to hmax) after a step whose error was <= tol / 64
            const double hmax = dt * S.adapt_hmax;
            double h = hmax, tcur = 0.0;
            // one RK4 step of length hs from the state at ts, with the classical state of its end
            auto trial = [&](double ts, double hs, bool first) {
                if (tid == 0) { c.h = hs; c.hh = 0.5 * hs; c.h6 = hs / 6.0; c.t0 = ts; }
                __syncthreads();
                for (int s = 0; s < 4; ++s) stage(s, s > 0, first, ts + hs);
                if (classical) cls_advance(S, c, lane, 3, nelem);
                __syncthreads();
            };
            // back to the start of the step: amplitudes A0 at time tcur (C0 = exp(-iEt) A0 with fresh
            // phase factors), classical state q0, stage quantities
            auto restore = [&]() {
                if (!elem && !classical) phase_factors(S, lane, tcur, PHa);
                if (classical) {
                    if (lane == 0) {
                        for (int i = 0; i < 4; ++i) c.q[i] = c.qs[i] = c.q0[i];
                        c.status &= ~MQCT_TRAJ_NONFINITE;
                        c.done = 0;
                    }
                    __syncwarp();
                    cls_look(S, c, lane, c.q[0], 0);
                    cls_enter(S, c, lane);
                }
                __syncthreads();
                if (elem)
                    for (int r = tid; r < n; r += nte) {
                        const double2 a0 = A0[r], p = PHa[S.lev[r]];
                        A[r] = a0;
                        C0[r] = make_double2(p.x * a0.x - p.y * a0.y, p.x * a0.y + p.y * a0.x);
                    }
                __syncthreads();
            };
            while (!c.done) {
                if (elem)
                    for (int r = tid; r < n; r += nte) A0[r] = A[r];
                if (tid == 0)
                    for (int i = 0; i < 4; ++i) c.q0[i] = c.q[i];
                __syncthreads();
                trial(tcur, h, c.steps == 0);
                if (elem)
                    for (int r = tid; r < n; r += nte) A1[r] = A[r];
                __syncthreads();
                restore();
                trial(tcur, 0.5 * h, false);
                if (!(c.status & MQCT_TRAJ_NONFINITE)) trial(tcur + 0.5 * h, 0.5 * h, false);
                // error: max over the states of |a(halves) - a(one step)| (independent of the order)
                double err = 0.0;
                if (elem)
                    for (int r = tid; r < n; r += nte) {
                        const double2 x = A[r], y = A1[r];
                        err = fmax(err, hypot(x.x - y.x, x.y - y.y));
                    }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) err = fmax(err, __shfl_xor_sync(0xffffffffu, err, o));
                __syncthreads();
                if (elem && lane == 0) c.red[warp][0] = err;
                __syncthreads();
                if (tid == 0) {
                    double e2 = 0.0;
                    for (int w2 = 0; w2 < nelem; ++w2) e2 = fmax(e2, c.red[w2][0]);
                    c.err = e2;
                }
                __syncthreads();
                if (!(c.status & MQCT_TRAJ_NONFINITE) && !(c.err <= S.adapt_tol) && h > dt) {
                    restore();
                    h *= 0.5;
                    continue;
                }
                if (tid == 0) {
                    c.steps += 1;
                    if (!(c.status & MQCT_TRAJ_NONFINITE)) {
                        if (c.q[0] >= c.r_end && c.q[1] > 0.0) c.done = 1;
                        else if (c.steps >= c.max_steps) { c.status |= MQCT_TRAJ_MAX_STEPS; c.done = 1; }
                    }
                    c.tcur = tcur + h;
                }
                __syncthreads();
                tcur = c.tcur;
                if (64.0 * c.err <= S.adapt_tol && h < hmax) h *= 2.0;
            }
            stage(0, false, false, 0.0);  // the sums of the final state
        } else {
            bool adv = false;
            for (;;) {
                stage(0, adv, false, 0.0);  // with c.done: the sums of the final state
                if (c.done) break;
                const double t_next = (c.steps + 1) * dt;
                const bool first = c.steps == 0;
#pragma unroll 1
                for (int s = 1; s < 4; ++s) stage(s, true, first, t_next);
                adv = true;
            }
        }
        // ---- diagnostics of the final state
        const bool out = c.timeout;
        if (classical) {
            if (!(c.status & MQCT_TRAJ_NONFINITE)) {
                if (lane == 0) { c.i2m0 = c.i2m; c.vid0 = c.vid[0]; }
                __syncwarp();
                cls_bookkeeping(S, c, lane, nelem, c.steps == 0);
            }
            if (lane == 0) {
                if (a.diag) {
                    mqct_diag d;
                    d.steps = c.steps; d.status = c.status | (out ? MQCT_TRAJ_TIMEOUT : 0);
                    d.norm_dev = c.ndev; d.energy_dev = c.edev; d.angmom_dev = c.jdev;
                    d.t_final = c.tcur;
                    a.diag[t] = d;
                }
                if (a.t_done) a.t_done[t] = mqct_clock_ns();
            }
        }
        // ---- outputs in the caller's state order (NaN after a timeout)
        if (elem && out)
            for (int r = tid; r < n; r += nte) {
                const double nan = __longlong_as_double(0x7ff8000000000000ll);
                A[r] = make_double2(nan, nan);
            }
        if (elem) {
            if (a.pop)
                for (int r = tid; r < n; r += nte) {
                    const double2 y = A[r];
                    a.pop[(size_t)t * a.nmax + S.perm[r]] = y.x * y.x + y.y * y.y;
                }
            if (a.amp)
                for (int r = tid; r < n; r += nte) {
                    const double2 y = A[r];
                    a.amp[((size_t)t * a.nmax + S.perm[r]) * 2] = y.x;
                    a.amp[((size_t)t * a.nmax + S.perm[r]) * 2 + 1] = y.y;
                }
        }
        __syncthreads();
    }
}

constexpr size_t kPropBasisBytes = 229216;  // of an SM's 232448 bytes per CTA

// Element warps of a CTA: a warp takes 16 rows at a time, and there are as many as the rows feed, at most 14
// (a 16-warp CTA, one per SM): N = 441, 256 trajectories 297 ms against 369 ms with eight warps and two CTAs
// per SM, whose last trajectories leave half the GPU idle; 64 trajectories 208 against 224 ms.  Four trajectories
// per SM are the exception (600 take 615 ms against 602 with eight warps): 2 % that no bound on the count
// separates from the 20 % of a batch with a tail.  A basis of at most eight row groups with more than two trajectories per SM
// takes half as many warps as groups, two row groups a warp (N = 49, 600 trajectories 504 against 580 ms; N = 100,
// 400 trajectories 628 against 690 ms): its stage is a chain of barriers that other CTAs fill.
cudaError_t launch_propagate(PropArgs pa, int maxlev, bool adapt, cudaStream_t st)
{
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int n_half = (pa.nmax + 15) / 16;
    const int want = n_half <= 8 && pa.n > 2 * sms ? (n_half + 1) / 2 : kPropElem;
    const int threads = 32 * (std::max(1, std::min(want, n_half)) + 2);
    pa.smem_n = pa.nmax;
    pa.smem_lev = maxlev;
    pa.adapt = adapt ? 1 : 0;
    const size_t smem = sizeof(double2) * ((adapt ? 6 : 4) * (size_t)pa.nmax + 2 * (size_t)maxlev);
    // the bases taken are those whose six vectors (with adaptive steps eight) would fit: this layout needs four
    // (six), but the call keeps refusing what it refused (N above 2380 or so)
    if (sizeof(double2) * ((adapt ? 8 : 6) * (size_t)pa.nmax + 2 * (size_t)maxlev) > kPropBasisBytes) return cudaErrorInvalidValue;
    auto go = [&](auto kern) -> cudaError_t {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem);
        if (e != cudaSuccess) return e;
        if (per_sm < 1) return cudaErrorInvalidConfiguration;
        kern<<<std::min(pa.n, sms * per_sm), threads, smem, st>>>(pa);
        count_launches(1);
        return cudaGetLastError();
    };
    return threads > 320 ? go(k_propagate_fp64<512, 1>) : go(k_propagate_fp64<320, 2>);
}

// work-order keys: estimated cost of a trajectory (steps ~ 2 r0 / v, work per step ~ nnz)
__global__ void k_order_keys(const DevSys *sys, int n_systems, const mqct_traj *trajs, int n, float *keys, int *idx)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const mqct_traj tr = trajs[i];
    idx[i] = i;
    if (tr.system_idx < 0 || tr.system_idx >= n_systems) { keys[i] = 0.0f; return; }
    const DevSys &S = sys[tr.system_idx];
    double v = sqrt(2.0 * fmax(tr.e_coll, 1e-30) / S.mu);
    double steps = fmin(2.0 * tr.r0 / (v * tr.dt), (double)tr.max_steps);
    double work = S.path == MQCT_PATH_PLAIN ? (double)S.nnz_pad : (double)S.n * (S.n_f + 1);
    keys[i] = (float)(-(steps * (work + 64.0 * S.n)));  // ascending sort = longest first
}

}  // namespace mqct

using namespace mqct;

namespace {

bool is_device_ptr(const void *p)
{
    if (!p) return false;
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

struct StreamAllocs {
    cudaStream_t st;
    std::vector<void *> ptrs;
    explicit StreamAllocs(cudaStream_t s) : st(s) {}
    cudaError_t get(void **p, size_t bytes)
    {
        cudaError_t e = cudaMallocAsync(p, bytes ? bytes : 16, st);
        if (e == cudaSuccess) ptrs.push_back(*p);
        return e;
    }
    ~StreamAllocs()
    {
        for (void *p : ptrs) cudaFreeAsync(p, st);
    }
};

}  // namespace

namespace {

// trajectory index i of the work order belongs to system s
struct IsSystem {
    const mqct_traj *tr;
    int s;
    __device__ bool operator()(const int &i) const { return tr[i].system_idx == s; }
};

// estimated work of each system: sum of its trajectories' (negated) order keys
__global__ void k_system_work(const mqct_traj *trajs, const int *order, const float *keys, int n, int n_systems,
                              double *work)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int s = trajs[order[i]].system_idx;
    if (s >= 0 && s < n_systems) atomicAdd(work + s, -(double)keys[i]);
}

}  // namespace

extern "C" mqct_status mqct_propagate(const mqct_system *systems, int32_t n_systems, const mqct_traj *trajs, int32_t n,
                                      double *final_pop, double *final_amp, mqct_diag *diag, void *cuda_stream)
{
    return mqct_propagate_ex(systems, n_systems, trajs, n, final_pop, final_amp, diag, nullptr, cuda_stream);
}

// mqct_propagate_ex; fail_every as in mqct_probe_propagate_timeout
static mqct_status propagate_impl(const mqct_system *systems, int32_t n_systems, const mqct_traj *trajs, int32_t n,
                                  double *final_pop, double *final_amp, mqct_diag *diag,
                                  const mqct_propagate_opts *opts, int fail_every, void *cuda_stream)
{
    reset_launches();
    const mqct_propagate_opts no_opts{};
    const mqct_propagate_opts &op = opts ? *opts : no_opts;
    auto shape_of = [&](int i) { return op.batch_shape ? op.batch_shape[i] : 0; };
    auto slots_of = [&](int i) { return op.tc_slots ? op.tc_slots[i] : 0; };
    for (int i = 0; i < std::max(0, (int)n_systems); ++i) {
        if (shape_of(i) < 0 || shape_of(i) > 7) return fail(MQCT_ERR_INVALID_ARG, "mqct_propagate: batch_shape outside [0, 7]");
        if (slots_of(i) < 0 || slots_of(i) > 8192) return fail(MQCT_ERR_INVALID_ARG, "mqct_propagate: tc_slots outside [0, 8192]");
    }
    if (!systems || n_systems < 1) return fail(MQCT_ERR_INVALID_ARG, "mqct_propagate: no systems");
    if (n < 0) return fail(MQCT_ERR_INVALID_ARG, "mqct_propagate: n < 0");
    if (n > 0 && !trajs) return fail(MQCT_ERR_INVALID_ARG, "mqct_propagate: trajs is NULL");
    cudaStream_t st = (cudaStream_t)cuda_stream;
    int nmax = 0, maxlev = 0;
    int path = -1, prec = -1;
    for (int i = 0; i < n_systems; ++i) {
        if (!systems[i]) return fail(MQCT_ERR_INVALID_ARG, "mqct_propagate: NULL system");
        const DevSys &h = systems[i]->s.h;
        nmax = std::max(nmax, h.n);
        maxlev = std::max(maxlev, h.n_levels);
        if (path < 0) { path = h.path; prec = h.precision; }
        if (h.path != path || h.precision != prec)
            return fail(MQCT_ERR_INVALID_ARG, "mqct_propagate: systems differ in path or precision");
    }
    // FP32 factorised systems run the persistent batched kernel; FP32 PLAIN systems (large bases
    // with the FP32 spline table) and BF16X3 systems the stage-synchronous path
    const bool stage_sync = prec == MQCT_BF16X3 || (prec == MQCT_FP32 && path == MQCT_PATH_PLAIN);
    if (prec == MQCT_FP32 && !stage_sync)
        for (int i = 0; i < n_systems; ++i) {
            const DevSys &h = systems[i]->s.h;
            if (batched_width(h) == 0) return fail(MQCT_ERR_UNSUPPORTED, "mqct_propagate: basis too large for the batched kernel");
            if (shape_of(i) > 0 && !batched_shape_fits(h, shape_of(i) - 1))
                return fail(MQCT_ERR_UNSUPPORTED, "mqct_propagate: batch_shape does not fit a system's basis");
        }
    if (n == 0) return MQCT_OK;

    const bool trajs_dev = is_device_ptr(trajs);
    // host trajectories are validated on the host
    if (!trajs_dev) {
        for (int i = 0; i < n; ++i) {
            const mqct_traj &t = trajs[i];
            if (t.system_idx < 0 || t.system_idx >= n_systems) return fail(MQCT_ERR_INVALID_ARG, "trajectory system_idx out of range");
            const DevSys &h = systems[t.system_idx]->s.h;
            if (t.init_state < 0 || t.init_state >= h.n) return fail(MQCT_ERR_INVALID_ARG, "trajectory init_state out of range");
            if (!(t.dt > 0) || !(t.e_coll > 0) || !(t.b >= 0) || !(t.r0 > 0) || t.max_steps < 0 || !std::isfinite(t.r_end))
                return fail(MQCT_ERR_INVALID_ARG, "trajectory with invalid e_coll, b, r0, r_end, dt or max_steps");
            double q = 2.0 * h.mu * t.e_coll - 2.0 * h.mu * t.e_coll * (t.b * t.b) / (t.r0 * t.r0);
            if (!(q > 0)) return fail(MQCT_ERR_INVALID_ARG, "trajectory starts inside its centrifugal barrier (b >= r0)");
        }
    }
    StreamAllocs sa(st);
    cudaError_t e;
    // device view of the system array
    DevSys *dsys = nullptr;
    {
        std::vector<DevSys> hv(n_systems);
        for (int i = 0; i < n_systems; ++i) hv[i] = systems[i]->s.h;
        if ((e = sa.get((void **)&dsys, sizeof(DevSys) * n_systems)) != cudaSuccess) return cuda_fail(e, "cudaMallocAsync");
        // pageable source: the copy is staged before cudaMemcpyAsync returns
        if ((e = cudaMemcpyAsync(dsys, hv.data(), sizeof(DevSys) * n_systems, cudaMemcpyHostToDevice, st)) != cudaSuccess)
            return cuda_fail(e, "cudaMemcpyAsync");
    }
    const mqct_traj *dtr = trajs;
    if (!trajs_dev) {
        mqct_traj *p = nullptr;
        if ((e = sa.get((void **)&p, sizeof(mqct_traj) * n)) != cudaSuccess) return cuda_fail(e, "cudaMallocAsync");
        if ((e = cudaMemcpyAsync(p, trajs, sizeof(mqct_traj) * n, cudaMemcpyHostToDevice, st)) != cudaSuccess)
            return cuda_fail(e, "cudaMemcpyAsync");
        dtr = p;
    }
    // outputs: device pointers are written directly, host ones through staging buffers
    const bool pop_dev = is_device_ptr(final_pop), amp_dev = is_device_ptr(final_amp), diag_dev = is_device_ptr(diag);
    const bool any_host = (final_pop && !pop_dev) || (final_amp && !amp_dev) || (diag && !diag_dev);
    double *dpop = final_pop, *damp = final_amp;
    mqct_diag *ddiag = nullptr;
    if (final_pop && !pop_dev && (e = sa.get((void **)&dpop, sizeof(double) * (size_t)n * nmax)) != cudaSuccess)
        return cuda_fail(e, "cudaMallocAsync");
    if (final_amp && !amp_dev && (e = sa.get((void **)&damp, sizeof(double) * 2 * (size_t)n * nmax)) != cudaSuccess)
        return cuda_fail(e, "cudaMallocAsync");
    if (diag && diag_dev) ddiag = diag;
    else if ((diag || any_host) && (e = sa.get((void **)&ddiag, sizeof(mqct_diag) * (size_t)n)) != cudaSuccess)
        return cuda_fail(e, "cudaMallocAsync");
    long long *dts = reinterpret_cast<long long *>(op.t_start_ns), *dtd = reinterpret_cast<long long *>(op.t_done_ns);
    const bool ts_host = op.t_start_ns && !is_device_ptr(op.t_start_ns), td_host = op.t_done_ns && !is_device_ptr(op.t_done_ns);
    if (ts_host && (e = sa.get((void **)&dts, sizeof(long long) * (size_t)n)) != cudaSuccess) return cuda_fail(e, "cudaMallocAsync");
    if (td_host && (e = sa.get((void **)&dtd, sizeof(long long) * (size_t)n)) != cudaSuccess) return cuda_fail(e, "cudaMallocAsync");
    // work order: longest estimated trajectory first
    float *keys = nullptr, *keys2 = nullptr;
    int *idx = nullptr, *order = nullptr, *queue = nullptr;
    if ((e = sa.get((void **)&keys, sizeof(float) * n)) != cudaSuccess || (e = sa.get((void **)&keys2, sizeof(float) * n)) != cudaSuccess ||
        (e = sa.get((void **)&idx, sizeof(int) * n)) != cudaSuccess || (e = sa.get((void **)&order, sizeof(int) * n)) != cudaSuccess ||
        (e = sa.get((void **)&queue, sizeof(int))) != cudaSuccess)
        return cuda_fail(e, "cudaMallocAsync");
    k_order_keys<<<(n + 255) / 256, 256, 0, st>>>(dsys, n_systems, dtr, n, keys, idx);
    count_launches(1);
    size_t tmp_bytes = 0;
    cub::DeviceRadixSort::SortPairs(nullptr, tmp_bytes, keys, keys2, idx, order, n, 0, 32, st);
    void *tmp = nullptr;
    if ((e = sa.get(&tmp, tmp_bytes)) != cudaSuccess) return cuda_fail(e, "cudaMallocAsync");
    if ((e = cub::DeviceRadixSort::SortPairs(tmp, tmp_bytes, keys, keys2, idx, order, n, 0, 32, st)) != cudaSuccess)
        return cuda_fail(e, "cub::DeviceRadixSort");
    if ((e = cudaMemsetAsync(queue, 0, sizeof(int), st)) != cudaSuccess) return cuda_fail(e, "cudaMemsetAsync");

    if (prec != MQCT_FP64) {
        // uneven batch of several systems: the work order split per system (stable, so each list
        // stays longest first) and the estimated work of each system, all on the device
        int *lists = order, *counts = nullptr, *queues = queue;
        double *work = nullptr;
        if (n_systems > 1) {
            if ((e = sa.get((void **)&lists, sizeof(int) * (size_t)n * n_systems)) != cudaSuccess ||
                (e = sa.get((void **)&counts, sizeof(int) * n_systems)) != cudaSuccess ||
                (e = sa.get((void **)&queues, sizeof(int) * n_systems)) != cudaSuccess ||
                (e = sa.get((void **)&work, sizeof(double) * n_systems)) != cudaSuccess)
                return cuda_fail(e, "cudaMallocAsync");
            cudaMemsetAsync(queues, 0, sizeof(int) * n_systems, st);
            cudaMemsetAsync(work, 0, sizeof(double) * n_systems, st);
            k_system_work<<<(n + 255) / 256, 256, 0, st>>>(dtr, order, keys2, n, n_systems, work);
            count_launches(1);
            size_t sel_bytes = 0;
            cub::DeviceSelect::If(nullptr, sel_bytes, order, lists, counts, n, IsSystem{dtr, 0}, st);
            void *sel_tmp = nullptr;
            if ((e = sa.get(&sel_tmp, sel_bytes)) != cudaSuccess) return cuda_fail(e, "cudaMallocAsync");
            for (int i = 0; i < n_systems; ++i)
                if ((e = cub::DeviceSelect::If(sel_tmp, sel_bytes, order, lists + (size_t)i * n, counts + i, n,
                                               IsSystem{dtr, i}, st)) != cudaSuccess)
                    return cuda_fail(e, "cub::DeviceSelect");
        }
        if (!stage_sync) {
            // one persistent launch over every system of the call (at most kBatchMaxSystems per
            // launch): CTAs bind to systems on the device
            BatchMultiArgs ma{};
            ma.trajs = dtr; ma.pop = dpop; ma.amp = damp; ma.diag = ddiag; ma.nmax = nmax;
            ma.t_start = dts; ma.t_done = dtd; ma.n = n; ma.fail_every = fail_every;
            int shape = 0;
            for (int i = 0; i < n_systems && !shape; ++i) shape = shape_of(i);
            for (int g0 = 0; g0 < n_systems; g0 += kBatchMaxSystems) {
                const int ng = std::min(kBatchMaxSystems, n_systems - g0);
                ma.sys = dsys + g0; ma.lists = lists + (size_t)g0 * n; ma.counts = counts ? counts + g0 : nullptr;
                ma.queues = queues + g0; ma.work = work ? work + g0 : nullptr; ma.n_systems = ng; ma.sys_base = g0;
                std::vector<const DevSys *> hs;
                for (int i = 0; i < ng; ++i) hs.push_back(&systems[g0 + i]->s.h);
                if ((e = run_batched(ma, hs, shape, st)) != cudaSuccess) return cuda_fail(e, "batched launch");
            }
        } else {
            BatchArgs ba{};
            ba.trajs = dtr; ba.pop = dpop; ba.amp = damp; ba.diag = ddiag; ba.nmax = nmax;
            ba.t_start = dts; ba.t_done = dtd;
            if (n_systems == 1) {
                ba.sys = systems[0]->s.d; ba.order = order; ba.n = n; ba.queue = queue; ba.sys_idx = 0;
                ba.tc_slots = slots_of(0);
                const mqct_status ts = run_tc_batched(ba, systems[0]->s.h, st);
                if (ts != MQCT_OK) return ts;
            } else {
                // the stage-synchronous path fills the GPU with one system at a time
                std::vector<int> hc(n_systems);
                if ((e = cudaMemcpyAsync(hc.data(), counts, sizeof(int) * n_systems, cudaMemcpyDeviceToHost, st)) != cudaSuccess ||
                    (e = cudaStreamSynchronize(st)) != cudaSuccess)
                    return cuda_fail(e, "work partition");
                for (int i = 0; i < n_systems; ++i) {
                    if (hc[i] == 0) continue;
                    BatchArgs bi = ba;
                    bi.sys = systems[i]->s.d; bi.order = lists + (size_t)i * n; bi.n = hc[i]; bi.queue = queues + i;
                    bi.sys_idx = i; bi.tc_slots = slots_of(i);
                    const mqct_status ts = run_tc_batched(bi, systems[i]->s.h, st);
                    if (ts != MQCT_OK) return ts;
                }
            }
        }
    } else {
    bool adapt = false;
    for (int i = 0; i < n_systems; ++i) adapt |= systems[i]->s.h.adapt_tol > 0.0;
    PropArgs pa{};
    pa.sys = dsys; pa.trajs = dtr; pa.order = order; pa.n = n; pa.n_systems = n_systems; pa.queue = queue;
    pa.pop = dpop; pa.amp = damp; pa.diag = ddiag; pa.nmax = nmax;
    pa.t_start = dts; pa.t_done = dtd; pa.fail_every = fail_every;
    if ((e = launch_propagate(pa, maxlev, adapt, st)) != cudaSuccess) {
        if (e == cudaErrorInvalidConfiguration) return fail(MQCT_ERR_UNSUPPORTED, "mqct_propagate: kernel does not fit on an SM");
        return cuda_fail(e, "k_propagate_fp64 launch (basis too large for shared memory?)");
    }
    }

    if (ts_host && (e = cudaMemcpyAsync(op.t_start_ns, dts, sizeof(long long) * (size_t)n, cudaMemcpyDeviceToHost, st)) != cudaSuccess)
        return cuda_fail(e, "cudaMemcpyAsync");
    if (td_host && (e = cudaMemcpyAsync(op.t_done_ns, dtd, sizeof(long long) * (size_t)n, cudaMemcpyDeviceToHost, st)) != cudaSuccess)
        return cuda_fail(e, "cudaMemcpyAsync");
    if (!any_host) {
        if ((ts_host || td_host) && (e = cudaStreamSynchronize(st)) != cudaSuccess) return cuda_fail(e, "cudaStreamSynchronize");
        return MQCT_OK;
    }
    if (final_pop && !pop_dev &&
        (e = cudaMemcpyAsync(final_pop, dpop, sizeof(double) * (size_t)n * nmax, cudaMemcpyDeviceToHost, st)) != cudaSuccess)
        return cuda_fail(e, "cudaMemcpyAsync");
    if (final_amp && !amp_dev &&
        (e = cudaMemcpyAsync(final_amp, damp, sizeof(double) * 2 * (size_t)n * nmax, cudaMemcpyDeviceToHost, st)) != cudaSuccess)
        return cuda_fail(e, "cudaMemcpyAsync");
    std::vector<mqct_diag> hd(n);
    mqct_diag *dst = (diag && !diag_dev) ? diag : hd.data();
    if ((e = cudaMemcpyAsync(dst, ddiag, sizeof(mqct_diag) * (size_t)n, cudaMemcpyDeviceToHost, st)) != cudaSuccess)
        return cuda_fail(e, "cudaMemcpyAsync");
    if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return cuda_fail(e, "cudaStreamSynchronize");
    int all = 0;
    for (int i = 0; i < n; ++i) all |= dst[i].status;
    if (all & MQCT_TRAJ_TIMEOUT) return fail(MQCT_ERR_TIMEOUT, "mqct_propagate: a bounded device wait ran out");
    if (all) return fail(MQCT_ERR_TRAJ, "at least one trajectory ended with a non-zero status");
    return MQCT_OK;
}

extern "C" mqct_status mqct_propagate_ex(const mqct_system *systems, int32_t n_systems, const mqct_traj *trajs,
                                         int32_t n, double *final_pop, double *final_amp, mqct_diag *diag,
                                         const mqct_propagate_opts *opts, void *cuda_stream)
{
    return propagate_impl(systems, n_systems, trajs, n, final_pop, final_amp, diag, opts, 0, cuda_stream);
}

extern "C" mqct_status mqct_probe_propagate_timeout(const mqct_system *systems, int32_t n_systems, const mqct_traj *trajs,
                                                    int32_t n, double *final_pop, double *final_amp, mqct_diag *diag,
                                                    const mqct_propagate_opts *opts, int32_t fail_every, void *cuda_stream)
{
    if (fail_every < 0) return fail(MQCT_ERR_INVALID_ARG, "mqct_probe_propagate_timeout: fail_every < 0");
    return propagate_impl(systems, n_systems, trajs, n, final_pop, final_amp, diag, opts, fail_every, cuda_stream);
}
