// Batched mixed-precision trajectory kernel (factorised path, FP32 amplitudes).
//
// One CTA integrates B trajectories ("slots") at once; finished slots are refilled from the
// device work queue, so trajectories of uneven length share a CTA.  Their phase-rotated stage
// amplitudes form the N x B block C (FP32, shared memory, real and imaginary planes [row][slot], two
// buffers by stage parity).  The warps have two roles:
//
//   element warps  own units (row r, 4 slots) with their amplitudes (up to two units per thread) and RK4
//     accumulators in registers; per RK4 stage
//     contraction (Eq. 12): for every pair of stored terms, Y_l = G^l C over the row's non-zeros (one
//         column and two values per entry, so a neighbour that both terms couple to is read once), folded
//         with the FP32 spline values: w = M(R_b) c_b and u = M'(R_b) c_b;
//     update: Coriolis stencil Dc = (J+ - J-) c, stage derivative da/dt = -i exp(iEt) w +
//         (dPhi/dt / 2) exp(iEt) Dc (Eq. 5), RK4 accumulation and the next stage's input into the other
//         C buffer; the partial sums of the force -Re(c^dag u) (Eq. 9), the torque
//         Re(c^dag D w) = -Re((Dc)^dag w) (Eq. 10) and, at stage 0, Re(c^dag w), |a|^2, E|a|^2, <J_y>; the step
//         update a + (dt/6) acc is compensated (two-sum), its rounding error carried into the next
//         step's accumulator;
//   slot warps     hold the FP64 classical state of the slots in registers, one lane per
//     (component, slot): lane 8 c + j carries component c of (R, P_R, Phi, P_Phi) of slot j, so
//     one FP64 instruction advances all four components of eight trajectories.
//
// One barrier per stage.  The slot warps are half a stage behind: while the element warps contract
// stage s (whose spline values were looked ahead, since R of stage s depends only on P_R of stage
// s-1), they sum the force and torque of stage s-1, advance the classical state and publish dPhi/dt
// and the slots' states of stage s (an mbarrier that the element warps wait on between contraction and
// update, by then long complete); then they look ahead to the spline values of stage s+1 and do the
// bookkeeping of norm, total energy and P_Phi + <J_y>, the outputs and the refill of a finished slot.
// Every chain of dependent FP64 instructions so runs beside the contraction.
//
// What bounds it: shared-memory reads of the neighbours' amplitudes (8 bytes per non-zero and slot) and
// instruction issue.  Amplitude arithmetic is on packed pairs of slots (fma.rn.f32x2), which the planar
// layout makes possible without moves; a unit's four slots are one 128-bit access per plane,
// and consecutive rows of a warp are contiguous, so the accesses are free of bank conflicts but for the
// borders of the m-blocks.  Measured (equal lengths, against two barriers per stage with scalar
// arithmetic, interleaved complex C and one entry per term and column): N = 441, 1216 trajectories 42.8 -> 72 M
// traj-steps/s, 2102 warp instructions per trajectory-stage (3974 before), issue slots 51 % busy,
// shared-memory data path 78 % (two CTAs of four slots per SM); N = 1600, 1216 trajectories 8.6 -> 16.3 M (its tables
// come from L2).
//
// Uneven batches (trajectories of several systems, i.e. basis sizes, in one call) run in this one
// persistent launch: a CTA binds to a system (its share of the grid at the start is proportional
// to the systems' estimated work), takes trajectories from that system's work list (longest
// first) with as many slots as the system's basis allows in the CTA's shared memory, and when the
// list is exhausted and its slots have drained it binds to the system with the most estimated
// work left.
//
// On this GPU an FP64 instruction holds its sub-partition's FP64 pipe for tens of cycles
// whatever the number of active lanes, so the kernel keeps FP64 off the per-element work:
// the phase arguments are 64-bit fixed-point turn counts (traj_common.cuh), the partial sums
// are FP32 within a warp and compensated FP32 (two-sum) across warps, converted to FP64 once per
// trajectory and stage.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>
#include <vector>

#include "internal.h"
#include "tc_ptx.cuh"
#include "traj_common.cuh"

namespace mqct {


enum { SLOT_IDLE = 0, SLOT_ACTIVE = 1, SLOT_FINAL = 2, SLOT_WAIT = 3 };

// slot warps for B slots (eight slots per warp, four component lanes per slot)
__host__ __device__ constexpr int batch_slot_warps(int B) { return B > 8 ? B / 8 : 1; }

// ---- packed arithmetic on two slots (each half rounded as the scalar instruction)
__device__ __forceinline__ float2 mul2(float2 a, float2 b)
{
    float2 d;
    asm("mul.rn.f32x2 %0, %1, %2;"
        : "=l"(reinterpret_cast<unsigned long long &>(d))
        : "l"(reinterpret_cast<const unsigned long long &>(a)), "l"(reinterpret_cast<const unsigned long long &>(b)));
    return d;
}
__device__ __forceinline__ float2 add2(float2 a, float2 b)
{
    float2 d;
    asm("add.rn.f32x2 %0, %1, %2;"
        : "=l"(reinterpret_cast<unsigned long long &>(d))
        : "l"(reinterpret_cast<const unsigned long long &>(a)), "l"(reinterpret_cast<const unsigned long long &>(b)));
    return d;
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return make_float2(__fsub_rn(a.x, b.x), __fsub_rn(a.y, b.y)); }
__device__ __forceinline__ float2 dup2(float x) { return make_float2(x, x); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }

// one plane (real or imaginary parts) of a unit's four slots, as two packed pairs
struct Q4 {
    float2 p[2];
};
__device__ __forceinline__ Q4 neg4(const Q4 &a)
{
    Q4 r;
    r.p[0] = neg2(a.p[0]);
    r.p[1] = neg2(a.p[1]);
    return r;
}
__device__ __forceinline__ Q4 ldq(const float *p)
{
    const float4 v = *reinterpret_cast<const float4 *>(p);
    Q4 r;
    r.p[0] = make_float2(v.x, v.y);
    r.p[1] = make_float2(v.z, v.w);
    return r;
}
__device__ __forceinline__ void stq(float *p, const Q4 &r)
{
    *reinterpret_cast<float4 *>(p) = make_float4(r.p[0].x, r.p[0].y, r.p[1].x, r.p[1].y);
}
__device__ __forceinline__ float qget(const Q4 &r, int j) { return (j & 1) ? r.p[j >> 1].y : r.p[j >> 1].x; }
__device__ __forceinline__ void qset(Q4 &r, int j, float v)
{
    if (j & 1) r.p[j >> 1].y = v;
    else r.p[j >> 1].x = v;
}

// Sums over the lanes of a warp that share lane % G4 of eight values per lane (G4 in {1, 2, 4}): each
// exchange halves the values a lane carries, so 15 shuffles or fewer take the place of 8 x 5.  On
// return v[0] of the lane is the sum of the value whose index has bits (2, 1, 0) = lane bits (4, 3, 2).
__device__ __forceinline__ float reduce8(float (&v)[8], int lane, int G4)
{
    const unsigned full = 0xffffffffu;
    const bool h4 = lane & 16, h3 = lane & 8, h2 = lane & 4;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float keep = h4 ? v[i + 4] : v[i], send = h4 ? v[i] : v[i + 4];
        v[i] = keep + __shfl_xor_sync(full, send, 16);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const float keep = h3 ? v[i + 2] : v[i], send = h3 ? v[i] : v[i + 2];
        v[i] = keep + __shfl_xor_sync(full, send, 8);
    }
    const float keep = h2 ? v[1] : v[0], send = h2 ? v[0] : v[1];
    float x = keep + __shfl_xor_sync(full, send, 4);
    if (G4 < 4) x += __shfl_xor_sync(full, x, 2);
    if (G4 < 2) x += __shfl_xor_sync(full, x, 1);
    return x;
}

// per-slot values the element warps read during one stage: vid, dvid are looked ahead (written during
// the stage before), the others published during the stage (double-buffered by stage parity)
template <int B>
struct SlotView {
    __align__(16) float hp[B];    // dPhi/dt / 2 (FP32 view)
    __align__(16) float dtf[B], hdtf[B], h6f[B], ih6f[B];  // dt, dt/2, dt/6, 6/dt (FP32 views)
    __align__(16) float vid[B];   // sum of the identity terms' v_l (FP32 spline)
    __align__(16) float dvid[B];  // and of their v_l'
    __align__(16) int state[B];
    __align__(16) int steps[B];
    int traj[B], s0[B];
};

// per-slot values of the slot warps that are not needed at every stage (shared memory keeps
// them out of the registers)
struct SlotCold {
    double e0, j0, ndev, edev, jdev;  // initial E_tot and P_Phi + <J_y>, running deviations
    double last_dt, r_end, i2m0;      // dt of the phase increments; stop radius; (1/mu)/R^2 at stage 0
    int status, max_steps, traj, s0;
    float dtf, ih6f;
};

// shared state of one CTA besides the big per-element arrays
template <int B>
struct BatchShared {
    DevSys S;
    SlotView<B> view[2];
    SlotCold cold[B];
    int live[B > 8 ? B / 8 : 1];  // per slot warp: some slot of it is not idle (set at stage 0)
    int cur;                      // system the CTA is bound to (-1: no work left)
    // a bounded wait of an element warp ran out (since the CTA bound to this system): what the slots hold is void,
    // the CTA claims nothing more and binds anew once they have ended
    int timeout;
    __align__(8) uint64_t published;  // mbarrier: the slot warps have published a stage's views
};

constexpr long long kBatchWait = 1ll << 17;  // polls of at most ~1 us

// dynamic shared memory of a CTA bound to a system with B slots: inc [NL][B] (u64), C [2][re, im][n][B], with more than
// two units per thread the amplitudes [re, im][n][B], PHa, PHb [re, im][NL][B], vv, dvv [2][2 groups][B], red [NE][6][B], elev [NL] (float)
template <int BMAX, int T, int kUpt>
size_t batched_smem(const DevSys &h, int B)
{
    constexpr int NE = T / 32 - batch_slot_warps(BMAX);
    const size_t nl = h.n_levels, n = h.n, nv = 2 * h.n_grp;
    return 8 * nl * B + 4 * ((kUpt <= 2 ? 4 : 6) * n * B + 4 * nl * B + 4 * nv * B + nl + (size_t)NE * 6 * B) + 16;
}

template <int T>
constexpr int batched_min_blocks() { return T >= 512 ? 1 : (T >= 256 ? 2 : 4); }

// the system a CTA binds to next: at the start, the CTA's share of the grid by estimated work;
// afterwards the system with the most estimated work left (-1: none)
__device__ int pick_system(const BatchMultiArgs &a, bool first)
{
    const int ns = a.n_systems;
    auto count_of = [&](int s) { return a.counts ? a.counts[s] : a.n; };
    if (first && ns > 1 && a.work) {
        double tot = 0.0;
        for (int s = 0; s < ns; ++s) tot += a.work[s];
        const double target = (blockIdx.x + 0.5) / gridDim.x * tot;
        double acc = 0.0;
        for (int s = 0; s < ns; ++s) {
            acc += a.work[s];
            if (acc >= target && count_of(s) > 0) return s;
        }
    }
    int best = -1;
    double best_score = -1.0;
    for (int s = 0; s < ns; ++s) {
        const int c = count_of(s);
        const int q = *((volatile const int *)(a.queues + s));
        const int rem = c - (q < c ? q : c);
        if (rem <= 0) continue;
        const double score = rem * (a.work ? a.work[s] / c : 1.0);
        if (score > best_score) {
            best_score = score;
            best = s;
        }
    }
    return best;
}

// the results of a trajectory that a timeout made void (row offset o): NaN; by four lanes, this one the c-th
__device__ __noinline__ void batched_void(double *pop, double *amp, size_t o, int n, int c)
{
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
    for (int r = c; r < n; r += 4) {
        if (pop) pop[o + r] = nan;
        if (amp) amp[2 * (o + r)] = amp[2 * (o + r) + 1] = nan;
    }
}

// everything a CTA does while bound to system `cur`: with BC > 0 its slot count is the compile-time
// constant BC, with BC = 0 the system's entry of a.slots; `phase` counts the stages published
template <int BC, int BMAX, int T, int kUpt>
__device__ __forceinline__ void batched_system(const BatchMultiArgs &a, BatchShared<BMAX> &sh, int cur,
                                               unsigned char *smraw, unsigned &phase)
{
    static_assert(BC % 4 == 0 && BC <= BMAX, "slots per CTA");
    constexpr int NS = batch_slot_warps(BMAX);  // slot warps (the last NS warps)
    constexpr int NW = T / 32, NE = NW - NS;    // element warps
    constexpr int TE = NE * 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool slot_warp = warp >= NE;
    const unsigned full = 0xffffffffu;
    const DevSys &S = sh.S;
    const int B = BC > 0 ? BC : a.slots[cur];    // slots (4, 8, 16 or 32)
    const int G4 = B / 4;                        // four-slot groups per row
    const int lg4 = G4 == 1 ? 0 : (G4 == 2 ? 1 : (G4 == 4 ? 2 : 3));
    const int n = S.n, NL = S.n_levels, L = S.L, ng = S.n_grp, NV = 2 * ng;
    const int np = n * B;  // floats of one plane of C
    const int *order = a.lists + (size_t)cur * a.n;
    int *queue = a.queues + cur;
    const int count = a.counts ? a.counts[cur] : a.n;
    float *C = reinterpret_cast<float *>(smraw);           // [2][re, im][np]
    [[maybe_unused]] float *Asm = C + 4 * np;              // [re, im][np] when the amplitudes are not in registers
    float *PHa = C + (kUpt <= 2 ? 4 : 6) * np, *PHb = PHa + 2 * NL * B;  // [re, im][NL][B]
    float *vv = PHb + 2 * NL * B, *dvv = vv + 2 * NV * B;  // [2][NV][B]
    float *red = dvv + 2 * NV * B;                         // [NE][6][B]
    unsigned long long *inc = reinterpret_cast<unsigned long long *>(red + NE * 6 * B);  // [NL][B]
    float *elev = reinterpret_cast<float *>(inc + NL * B);
    for (int l = tid; l < NL; l += T) elev[l] = (float)S.lev_energy[l];
    // spline-weight rows of groups of one term stay zero in their second half
    for (int i = tid; i < 4 * NV * B; i += T) vv[i] = 0.f;
    __syncthreads();

    // The two roles run separate code with the same barriers (one per stage), so that the
    // registers of one role are not kept alive in the other.
    if (slot_warp) {
    const int sc = lane >> 3, sj = lane & 7;
    const int sb = 8 * (warp - NE) + sj;
    const unsigned m4 = 0x01010101u << sj;  // the four component lanes of this slot
    // slot-warp registers (lane 8 c + j: component c of (R, P_R, Phi, P_Phi) of slot 8 (warp - NE) + j)
    double q = 0.0, qs = 0.0, lacc = 0.0;
    double imu = 1.0 / S.mu, dtd = 1.0, hdt = 0.5, h6 = 1.0 / 6.0;
    double ir = 0.0, i2m = 0.0, phid = 0.0, t1 = 0.0;  // 1/R, (1/mu)/R^2, dPhi/dt, P_Phi^2/(mu R^3)
    double ir_n = 0.1, i2m_n = 0.0;                   // look-ahead
    int steps = 0, state = SLOT_IDLE;
    bool below_n = false;
    float2 bk = make_float2(0.f, 0.f);  // stage-0 sum of lane c: V, <J_y>, |a|^2, E|a|^2

    // Every lane of a slot warp runs the same instructions (lanes of slots >= B compute on copies
    // and store nothing), so that the shuffles between the four component lanes of a slot are
    // warp-uniform.
    const bool slot_lane = sb < B;
    const int sbc = sb < B ? sb : B - 1;   // a valid index for reads of the lanes past B
    SlotCold &cs = sh.cold[sbc];
    if (slot_lane && sc == 0) {
        cs.last_dt = -1.0;
        cs.status = 0;
    }
    __syncwarp();

    auto comp = [&](double v, int c2) { return __shfl_sync(full, v, 8 * c2 + sj); };

    // publish this slot's view for stage `stage`
    auto publish = [&](int stage) {
        if (slot_lane && sc == 0) {
            SlotView<BMAX> &vw = sh.view[stage & 1];
            vw.state[sb] = state;
            vw.traj[sb] = cs.traj;
            vw.s0[sb] = cs.s0;
            vw.steps[sb] = steps;
            vw.dtf[sb] = cs.dtf;
            vw.hdtf[sb] = 0.5f * cs.dtf;
            vw.h6f[sb] = cs.dtf * (1.0f / 6.0f);
            vw.ih6f[sb] = cs.ih6f;
            vw.hp[sb] = (float)phid * 0.5f;
        }
    };

    // claim the next valid trajectory for this slot (its four lanes together, shuffles over m4);
    // on return the slot is WAIT (column to be initialised at the next stage 3) or IDLE
    auto claim = [&]() {
        for (;;) {
            int item = count;
            if (sc == 0 && !sh.timeout) item = atomicAdd(queue, 1);
            item = __shfl_sync(m4, item, sj);
            if (item >= count) {
                state = SLOT_IDLE;
                return;
            }
            if (a.fail_every && sc == 0 && (item + 1) % a.fail_every == 0) sh.timeout = 1;
            const int t = order ? order[item] : item;
            const mqct_traj tr = a.trajs[t];
            if (!traj_valid(tr, S, a.sys_base + cur)) {
                if (a.diag && sc == 0) {
                    mqct_diag d = {0, MQCT_TRAJ_INVALID, 0.0, 0.0, 0.0, 0.0};
                    a.diag[t] = d;
                }
                __syncwarp(m4);
                continue;
            }
            if (a.t_start && sc == 0) a.t_start[t] = mqct_clock_ns();
            const int s0 = S.inv[tr.init_state];
            int k0;
            double x0;
            bool bl;
            locate_interval(S, tr.r0, k0, x0, bl);
            // initial mean field M_ss(r0): the four lanes split the terms
            double m = 0.0;
            for (int l = sc; l < L; l += 4) m += spline_fp64(S, l, k0, x0) * S.diag_g[(size_t)l * n + s0];
            m += __shfl_xor_sync(m4, m, 8);
            m += __shfl_xor_sync(m4, m, 16);
            double q4[4];
            initial_state(S, tr, m, q4);
            q = q4[sc];
            qs = q;
            lacc = 0.0;
            dtd = tr.dt;
            hdt = 0.5 * tr.dt;
            h6 = tr.dt / 6.0;
            steps = 0;
            state = SLOT_WAIT;
            const bool new_dt = tr.dt != cs.last_dt;
            __syncwarp(m4);
            if (sc == 0) {
                cs.traj = t;
                cs.s0 = s0;
                cs.dtf = (float)tr.dt;
                cs.ih6f = 6.0f / (float)tr.dt;
                cs.r_end = tr.r_end;
                cs.max_steps = tr.max_steps;
                cs.status = 0;
                cs.ndev = cs.edev = cs.jdev = 0.0;
                cs.last_dt = tr.dt;
            }
            // fixed-point phase increments of every level for this dt (kept while dt repeats)
            if (new_dt)
                for (int l = sc; l < NL; l += 4) inc[l * B + sb] = phase_increment(S.lev_energy[l], tr.dt);
            __syncwarp(m4);
            return;
        }
    };

    // look-ahead for stage s+1 (s = -1: a slot that starts at the next stage 0): R, its interval and
    // the spline values of every term, written to vv / dvv [(s+1) & 1]; then 1/R
    auto look_ahead = [&](int s) {
        const int par = (s + 1) & 1;
        const bool act = slot_lane && state == SLOT_ACTIVE;
        const bool start = slot_lane && state == SLOT_WAIT && (s == 3 || s == -1);
        const double q0 = comp(q, 0), pr = comp(qs, 1), la0 = comp(lacc, 0);
        double qs0 = 0.0, lacc0 = la0;
        stage_component(s < 0 ? 0 : s, imu, pr, 0.0, hdt, dtd, h6, q0, qs0, lacc0);
        double Rn = act ? qs0 : (start ? q0 : 10.0);  // any finite R for slots not running
        int k;
        double x;
        locate_interval(S, Rn, k, x, below_n);
        const float xf = (float)x;
        float v0 = 0.f, d0 = 0.f;
        for (int l = sc; l < L; l += 4) {
            float v = 0.f, dv = 0.f;
            if (act || start) {
                const float4 c = __ldg(S.vcoef_f + (size_t)l * S.n_int + k);
                v = fmaf(xf, fmaf(xf, fmaf(xf, c.w, c.z), c.y), c.x);
                dv = fmaf(xf, fmaf(3.0f * xf, c.w, 2.0f * c.z), c.y);
            }
            const int row = __ldg(S.grp_row + l);
            if (slot_lane && row >= 0) {
                vv[(par * NV + row) * B + sb] = v;
                dvv[(par * NV + row) * B + sb] = dv;
            }
            if ((S.id_mask >> l) & 1ull) { v0 += v; d0 += dv; }
        }
        v0 += __shfl_xor_sync(full, v0, 8);
        v0 += __shfl_xor_sync(full, v0, 16);
        d0 += __shfl_xor_sync(full, d0, 8);
        d0 += __shfl_xor_sync(full, d0, 16);
        if (slot_lane && sc == 0) {
            sh.view[par].vid[sb] = v0;
            sh.view[par].dvid[sb] = d0;
        }
        ir_n = 1.0 / Rn;
        i2m_n = imu * ir_n * ir_n;
    };

    // compensated FP32 sum of quantity qq of this lane's slot over the element warps w0, w0 + dw, ...
    auto wsum = [&](int qq, int w0, int dw) {
        float hi = 0.f, lo = 0.f;
#pragma unroll 4
        for (int w2 = w0; w2 < NE; w2 += dw) {
            float e2;
            two_sum(hi, red[(w2 * 6 + qq) * B + sbc], hi, e2);
            lo += e2;
        }
        return make_float2(hi, lo);
    };

    // total energy, P_Phi + <J_y> and norm of the state at the start of a step (or of the final
    // state) from its stage-0 sums: running maxima of their deviations, for the slots where
    // `apply` holds
    auto bookkeeping = [&](bool apply) {
        const double val = (double)bk.x + (double)bk.y;
        const double V = comp(val, 0), JY = comp(val, 1), NR = comp(val, 2), ER = comp(val, 3);
        const double PR = comp(q, 1), PP = comp(q, 3);
        const double et = 0.5 * (imu * PR * PR + PP * PP * cs.i2m0) + ER + V;
        const double jt = PP + 0.5 * JY;
        const double e0 = steps == 0 ? et : cs.e0, j0 = steps == 0 ? jt : cs.j0;
        const double nd = fmax(cs.ndev, fabs(NR - 1.0));
        const double ed = fmax(cs.edev, fabs(et - e0));
        const double jd = fmax(cs.jdev, fabs(jt - j0));
        __syncwarp();
        if (apply && sc == 0) {
            cs.e0 = e0; cs.j0 = j0;
            cs.ndev = nd; cs.edev = ed; cs.jdev = jd;
        }
        __syncwarp();
    };

    // the classical stage update from the sums of stage sp, the stop rule (sp = 3) and the start of
    // waiting slots; afterwards state, dPhi/dt and 1/R are those of the next stage
    auto advance = [&](int sp) {
        // lanes c = 0, 1 sum the force, c = 2, 3 the torque, over half of the element warps each
        float2 pv = wsum(sc >> 1, sc & 1, 2);
        {
            const float ohi = __shfl_xor_sync(full, pv.x, 8), olo = __shfl_xor_sync(full, pv.y, 8);
            float hi, e2;
            two_sum(pv.x, ohi, hi, e2);
            pv = make_float2(hi, pv.y + olo + e2);
        }
        const double X2 = (double)pv.x + (double)pv.y;
        const double pr = comp(qs, 1);
        if (sp == 0 && slot_lane && sc == 0) cs.i2m0 = i2m;
        const bool act = slot_lane && state == SLOT_ACTIVE;
        const bool start = slot_lane && state == SLOT_WAIT && sp == 3;
        {
            // derivative l_c: (P_R / mu, F + P_Phi^2/(mu R^3), dPhi/dt, torque) (Eqs. 7-10)
            const double X = sc == 0 ? pr : (sc == 2 ? phid : X2);
            const double alpha = sc == 0 ? imu : 1.0, beta = sc == 1 ? t1 : 0.0;
            double qs2 = qs, lacc2 = lacc;
            stage_component(sp, alpha, X, beta, hdt, dtd, h6, q, qs2, lacc2);
            if (act) { qs = qs2; lacc = lacc2; }
        }
        int add_status = 0;
        if (sp == 3) {
            const unsigned bad = __ballot_sync(full, act && !finite64(qs));
            const double R = comp(qs, 0), PR = comp(qs, 1);
            if (act) {
                q = qs;
                steps += 1;
                if ((bad >> sj) & 0x01010101u) {
                    add_status |= MQCT_TRAJ_NONFINITE;
                    state = SLOT_FINAL;
                } else if (ge_pos(R, cs.r_end) && __double_as_longlong(PR) > 0) {
                    state = SLOT_FINAL;
                } else if (steps >= cs.max_steps) {
                    add_status |= MQCT_TRAJ_MAX_STEPS;
                    state = SLOT_FINAL;
                }
            }
        }
        const double pp3 = comp(qs, 3);
        if ((act && !(add_status & MQCT_TRAJ_NONFINITE)) || start) {
            if (below_n) add_status |= MQCT_TRAJ_TABLE_RANGE;
            ir = ir_n;
            i2m = i2m_n;
            phid = pp3 * i2m_n;
        }
        if (start) {
            const int ms = cs.max_steps;
            state = ms > 0 ? SLOT_ACTIVE : SLOT_FINAL;
            if (ms <= 0) add_status |= MQCT_TRAJ_MAX_STEPS;
        }
        __syncwarp();
        if (slot_lane && sc == 0 && add_status) cs.status |= add_status;
    };

    // ---------------------------------------------------------------- start
    {
        if (slot_lane) claim();
        __syncwarp();
        look_ahead(-1);
        if (slot_lane && state == SLOT_WAIT) {
            const int ms = cs.max_steps;
            state = ms > 0 ? SLOT_ACTIVE : SLOT_FINAL;
            __syncwarp(m4);
            if (sc == 0) cs.status |= (ms <= 0 ? MQCT_TRAJ_MAX_STEPS : 0) | (below_n ? MQCT_TRAJ_TABLE_RANGE : 0);
            ir = ir_n;
            i2m = i2m_n;
        }
        const double pp3 = comp(q, 3);
        if (slot_lane && state != SLOT_IDLE) phid = pp3 * i2m;
        publish(0);
    }
    __syncthreads();
    __syncthreads();  // the element warps have set up the columns
    bool run = true, first = true;
    while (run) {
        for (int s = 0; s < 4; ++s) {
            // ---- while the element warps contract stage s: the classical stage from the sums of the
            // stage before, and this stage's views
            if (!first) {
                advance((s + 3) & 3);
                publish(s);
            }
            first = false;
            if (s == 0) {
                const unsigned live = __ballot_sync(full, slot_lane && state != SLOT_IDLE);
                if (lane == 0) sh.live[warp - NE] = live != 0;
                if (NS > 1) {
                    asm volatile("bar.sync 1, %0;" ::"r"(NS * 32) : "memory");
                    run = false;
#pragma unroll
                    for (int i = 0; i < NS; ++i) run |= sh.live[i] != 0;
                } else {
                    run = live != 0;
                }
            }
            __syncwarp();
            if (lane == 0) tc_mbar_arrive(&sh.published);
            if (!run) {  // the element warps read `live` after the barrier
                __syncthreads();
                break;
            }
            // ---- bookkeeping of stage 0 (a finished slot at stage 1, before its refill; running slots
            // at stage 2), the diagnostics and refill of a finished slot, then the look-ahead
            if (s == 1) {
                bk = wsum(2 + sc, 0, 1);
                const bool fin_any = __any_sync(full, slot_lane && state == SLOT_FINAL);
                if (fin_any) {
                    bookkeeping(slot_lane && state == SLOT_FINAL);
                    if (slot_lane && state == SLOT_FINAL) {
                        const int out = __shfl_sync(m4, sh.timeout, sj);
                        if (out) batched_void(a.pop, a.amp, (size_t)cs.traj * a.nmax, n, sc);
                        if (sc == 0) {
                            if (a.diag) {
                                mqct_diag d;
                                d.steps = steps; d.status = cs.status | (out ? MQCT_TRAJ_TIMEOUT : 0);
                                d.norm_dev = cs.ndev; d.energy_dev = cs.edev; d.angmom_dev = cs.jdev;
                                d.t_final = steps * dtd;
                                a.diag[cs.traj] = d;
                            }
                            if (a.t_done) a.t_done[cs.traj] = mqct_clock_ns();
                        }
                        __syncwarp(m4);
                        claim();  // WAIT or IDLE: phases and column at stage 3
                    }
                    __syncwarp();
                }
            }
            look_ahead(s);
            const double pp3 = comp(qs, 3);
            if (slot_lane && state == SLOT_ACTIVE) t1 = pp3 * phid * ir;  // P_Phi^2 / (mu R^3)
            if (s == 2) bookkeeping(slot_lane && state == SLOT_ACTIVE);
            __syncthreads();
        }
    }
    } else {
    const int g = tid & (G4 - 1);
    // amplitudes and RK4 accumulators of the units' four slots in registers; with more than two units per
    // thread the amplitudes in shared memory (own values only)
    constexpr bool kRegA = kUpt <= 2;
    Q4 Rx[kRegA ? kUpt : 1] = {}, Ry[kRegA ? kUpt : 1] = {}, Kx[kUpt], Ky[kUpt];
    auto get_a = [&](int k, int o, Q4 &x, Q4 &y) {
        if constexpr (kRegA) { x = Rx[k]; y = Ry[k]; }
        else { x = ldq(Asm + o); y = ldq(Asm + np + o); }
    };
    auto set_a = [&](int k, int o, const Q4 &x, const Q4 &y) {
        if constexpr (kRegA) { Rx[k] = x; Ry[k] = y; }
        else { stq(Asm + o, x); stq(Asm + np + o, y); }
    };
    __syncthreads();
    // columns of the slots that start at the first stage 0: e_s0, accumulators 0, phase of t = dt/2
    bool any = false;
#pragma unroll
    for (int j = 0; j < 4; ++j) any |= sh.view[0].state[4 * g + j] != SLOT_IDLE;
#pragma unroll
    for (int k = 0; k < kUpt; ++k) {
        const int r = (tid + k * TE) >> lg4;
        Q4 x, y;
        Kx[k].p[0] = Kx[k].p[1] = Ky[k].p[0] = Ky[k].p[1] = y.p[0] = y.p[1] = make_float2(0.f, 0.f);
#pragma unroll
        for (int j = 0; j < 4; ++j)
            qset(x, j, sh.view[0].state[4 * g + j] != SLOT_IDLE && r == sh.view[0].s0[4 * g + j] ? 1.0f : 0.0f);
        if (r < n) {
            set_a(k, r * B + 4 * g, x, y);
            stq(C + r * B + 4 * g, x);
            stq(C + np + r * B + 4 * g, y);
        }
    }
    for (int i = tid; i < NL * B; i += TE) {
        const float2 p = sh.view[0].state[i % B] != SLOT_IDLE ? phase_factor(inc[i], 1u) : make_float2(1.f, 0.f);
        PHb[i] = p.x;
        PHb[NL * B + i] = p.y;
        PHa[i] = 1.f;  // t = 0
        PHa[NL * B + i] = 0.f;
    }
    __syncthreads();

    // one RK4 stage of this warp's units
    auto stage = [&](auto s0c, int s) {
        constexpr bool S0 = decltype(s0c)::value;
        const int par = s & 1;
        const SlotView<BMAX> &vw = sh.view[par];
        const float *Cc = C + par * 2 * np + 4 * g;
        float *Cn = C + (par ^ 1) * 2 * np + 4 * g;
        const float *PHc = ((S0 || s == 3) ? PHa : PHb) + 4 * g, *PHn = ((S0 || s == 1) ? PHb : PHa) + 4 * g;
        const float *vvs = vv + par * NV * B + 4 * g, *dvvs = dvv + par * NV * B + 4 * g;
        bool act = any, regular = false;
        // the views of this stage, which the slot warps publish during the contraction: every lane of the
        // warp waits, and the warp converges again afterwards
        auto wait = [&]() {
            // (bounded; after one wait ran out the others return at once: the stages go on with whatever the views
            // hold, whose indices are in range at any time, and the results are void)
            if (!*(volatile int *)&sh.timeout && !tc_mbar_wait(&sh.published, phase & 1u, kBatchWait)) sh.timeout = 1;
            __syncwarp();
            const int4 st4 = *reinterpret_cast<const int4 *>(vw.state + 4 * g);
            regular = st4.x == SLOT_ACTIVE && st4.y == SLOT_ACTIVE && st4.z == SLOT_ACTIVE && st4.w == SLOT_ACTIVE;
            if (S0) {
                const int4 sp = *reinterpret_cast<const int4 *>(vw.steps + 4 * g);
                regular = regular && sp.x > 0 && sp.y > 0 && sp.z > 0 && sp.w > 0;
            }
            act = st4.x != SLOT_IDLE || st4.y != SLOT_IDLE || st4.z != SLOT_IDLE || st4.w != SLOT_IDLE;
        };
        float2 f2[2], t2[2], v2[2], j2[2], m2[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) f2[i] = t2[i] = v2[i] = j2[i] = m2[i] = make_float2(0.f, 0.f);
#pragma unroll
        for (int k = 0; k < kUpt; ++k) {
            const int r = (tid + k * TE) >> lg4;
            const bool on = r < n && any;
            const int ro = r * B;
            // ---- contraction
            Q4 wx, wy, ux, uy;
#pragma unroll
            for (int i = 0; i < 2; ++i) wx.p[i] = wy.p[i] = ux.p[i] = uy.p[i] = make_float2(0.f, 0.f);
            if (on) {
            const int sl = r >> 5;
            const int o0 = __ldg(S.g_off + sl) + (r & 31);
            const float2 *pv = S.g_val + o0;
            const unsigned short *pc = S.g_col + o0;
            const int *pw = S.g_width + sl * ng;
            for (int gi = 0; gi < ng; ++gi) {
                const int wd = __ldg(pw + gi), width = wd & 0xffff;
                Q4 ax, ay, bx, by;
#pragma unroll
                for (int i = 0; i < 2; ++i) ax.p[i] = ay.p[i] = bx.p[i] = by.p[i] = make_float2(0.f, 0.f);
                const float *vr = vvs + 2 * gi * B, *dr = dvvs + 2 * gi * B;
                // two entries at a time: their table and amplitude reads are in flight together
                auto entries = [&](auto two) {
                    auto one = [&](float2 gv, const Q4 &zx, const Q4 &zy) {
                        const float2 ga = dup2(gv.x), gb = dup2(gv.y);
#pragma unroll
                        for (int i = 0; i < 2; ++i) {
                            ax.p[i] = fma2(ga, zx.p[i], ax.p[i]); ay.p[i] = fma2(ga, zy.p[i], ay.p[i]);
                            if constexpr (decltype(two)::value) {
                                bx.p[i] = fma2(gb, zx.p[i], bx.p[i]); by.p[i] = fma2(gb, zy.p[i], by.p[i]);
                            }
                        }
                    };
                    int e = width;
                    for (; e >= 2; e -= 2) {
                        const float2 g0 = __ldg(pv), g1 = __ldg(pv + kSlice);
                        const float *z0 = Cc + __ldg(pc) * B, *z1 = Cc + __ldg(pc + kSlice) * B;
                        const Q4 x0 = ldq(z0), y0 = ldq(z0 + np), x1 = ldq(z1), y1 = ldq(z1 + np);
                        pv += 2 * kSlice;
                        pc += 2 * kSlice;
                        one(g0, x0, y0);
                        one(g1, x1, y1);
                    }
                    if (e) {
                        const float2 g0 = __ldg(pv);
                        const float *z0 = Cc + __ldg(pc) * B;
                        const Q4 x0 = ldq(z0), y0 = ldq(z0 + np);
                        pv += kSlice;
                        pc += kSlice;
                        one(g0, x0, y0);
                    }
                };
                if (wd >> 16) {
                    entries(std::true_type{});
                    const Q4 v = ldq(vr + B), d = ldq(dr + B);
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        wx.p[i] = fma2(v.p[i], bx.p[i], wx.p[i]); wy.p[i] = fma2(v.p[i], by.p[i], wy.p[i]);
                        ux.p[i] = fma2(d.p[i], bx.p[i], ux.p[i]); uy.p[i] = fma2(d.p[i], by.p[i], uy.p[i]);
                    }
                } else {
                    entries(std::false_type{});
                }
                const Q4 v = ldq(vr), d = ldq(dr);
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    wx.p[i] = fma2(v.p[i], ax.p[i], wx.p[i]); wy.p[i] = fma2(v.p[i], ay.p[i], wy.p[i]);
                    ux.p[i] = fma2(d.p[i], ax.p[i], ux.p[i]); uy.p[i] = fma2(d.p[i], ay.p[i], uy.p[i]);
                }
            }
            }
            if (k == 0) wait();
            // ---- update
            if (!on) continue;
            // identity terms
            const Q4 cx = ldq(Cc + ro), cy = ldq(Cc + np + ro);
            {
                const Q4 vi = ldq(vw.vid + 4 * g), dvi = ldq(vw.dvid + 4 * g);
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    wx.p[i] = fma2(vi.p[i], cx.p[i], wx.p[i]); wy.p[i] = fma2(vi.p[i], cy.p[i], wy.p[i]);
                    ux.p[i] = fma2(dvi.p[i], cx.p[i], ux.p[i]); uy.p[i] = fma2(dvi.p[i], cy.p[i], uy.p[i]);
                }
            }
            const int4 ri = __ldg(S.row_info + r);
            const float *cu = Cc + (ri.x & 0xffff) * B, *cd = Cc + (int)((unsigned)ri.x >> 16) * B;
            const int lo = ri.y * B;
            Q4 px = ldq(PHc + lo), py = ldq(PHc + NL * B + lo);
            const float2 nau = dup2(-__int_as_float(ri.z)), ad = dup2(__int_as_float(ri.w));
            Q4 dcx, dcy;
            {
                const Q4 ux_ = ldq(cu), uy_ = ldq(cu + np), dx_ = ldq(cd), dy_ = ldq(cd + np);
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    dcx.p[i] = fma2(ad, dx_.p[i], mul2(nau, ux_.p[i]));
                    dcy.p[i] = fma2(ad, dy_.p[i], mul2(nau, uy_.p[i]));
                }
            }
            if (S0 && !regular) {
                // the first stage of a trajectory is at t = 0, where every phase factor is 1
                const int4 sp = *reinterpret_cast<const int4 *>(vw.steps + 4 * g);
                const int spj[4] = {sp.x, sp.y, sp.z, sp.w};
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (spj[j] == 0) { qset(px, j, 1.f); qset(py, j, 0.f); }
            }
            // the next stage's time differs from this one's at stages 0 and 2 only
            const Q4 npy = neg4(py);
            Q4 qx = px, qy = py, nqy = npy;
            if (S0 || s == 2) { qx = ldq(PHn + lo); qy = ldq(PHn + NL * B + lo); nqy = neg4(qy); }
            const Q4 hp = ldq(vw.hp + 4 * g), nhp = neg4(hp);
            // dt/6, dt or dt/2
            const Q4 hs = ldq((!S0 && s == 3 ? vw.h6f : (s == 2 ? vw.dtf : vw.hdtf)) + 4 * g), nhs = neg4(hs);
            Q4 ih6;
            if (!S0 && s == 3) ih6 = ldq(vw.ih6f + 4 * g);
            Q4 nx, ny, Ax, Ay;  // the next stage's input; the amplitudes at the start of the step
            get_a(k, ro + 4 * g, Ax, Ay);
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                f2[i] = fma2(cx.p[i], ux.p[i], f2[i]); f2[i] = fma2(cy.p[i], uy.p[i], f2[i]);
                t2[i] = fma2(dcx.p[i], wx.p[i], t2[i]); t2[i] = fma2(dcy.p[i], wy.p[i], t2[i]);
                // k = conj(p) (-i w + (dPhi/dt / 2) Dc), the imaginary part carried negated (ny = -Im), so
                // that no operand needs a sign change (packed instructions have none)
                const float2 zx = fma2(hp.p[i], dcx.p[i], wy.p[i]), zy = fma2(nhp.p[i], dcy.p[i], wx.p[i]);
                const float2 kx = fma2(npy.p[i], zy, mul2(px.p[i], zx));
                const float2 ky = fma2(px.p[i], zy, mul2(py.p[i], zx));
                const float2 ax = Ax.p[i], ay = Ay.p[i];
                if (S0) {
                    v2[i] = fma2(cx.p[i], wx.p[i], v2[i]); v2[i] = fma2(cy.p[i], wy.p[i], v2[i]);
                    // <J_y>: Im(a^dag D a) = Im(c^dag D c), the phases of a level's states cancel
                    j2[i] = fma2(cx.p[i], dcy.p[i], j2[i]); m2[i] = fma2(cy.p[i], dcx.p[i], m2[i]);
                    // the accumulator enters the step holding the rounding error of the last update
                    Kx[k].p[i] = add2(kx, Kx[k].p[i]);
                    Ky[k].p[i] = add2(ky, Ky[k].p[i]);
                } else {
                    const float2 wg = dup2(s == 3 ? 1.0f : 2.0f);
                    Kx[k].p[i] = fma2(wg, kx, Kx[k].p[i]);
                    Ky[k].p[i] = fma2(wg, ky, Ky[k].p[i]);
                }
                float2 yx, yy;
                if (!S0 && s == 3) {
                    // compensated a + (dt/6) acc (two-sum): far from the collision the
                    // interaction-picture amplitudes change by increments a plain FP32 add
                    // would round away; the error is carried to the next accumulator
                    auto step2 = [&](float2 a0, float2 &acc, float2 h, float2 ih) {
                        const float2 b0 = mul2(h, acc);
                        const float2 sum = add2(a0, b0);
                        const float2 bb = sub2(sum, a0);
                        const float2 er = add2(sub2(a0, sub2(sum, bb)), sub2(b0, bb));
                        acc = mul2(er, ih);
                        return sum;
                    };
                    yx = step2(ax, Kx[k].p[i], hs.p[i], ih6.p[i]);
                    yy = step2(ay, Ky[k].p[i], nhs.p[i], neg2(ih6.p[i]));
                    Ax.p[i] = yx;
                    Ay.p[i] = yy;
                } else {
                    yx = fma2(hs.p[i], kx, ax);
                    yy = fma2(nhs.p[i], ky, ay);
                }
                nx.p[i] = fma2(nqy.p[i], yy, mul2(qx.p[i], yx));
                ny.p[i] = fma2(qx.p[i], yy, mul2(qy.p[i], yx));
            }
            if (!regular) {
                // slots that are not running: their arithmetic above is discarded
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int stj = vw.state[4 * g + j];
                    if (S0 && stj == SLOT_FINAL) {
                        const float fx = qget(Ax, j), fy = qget(Ay, j);
                        const size_t oo = (size_t)vw.traj[4 * g + j] * a.nmax + __ldg(S.perm + r);
                        if (a.pop) a.pop[oo] = (double)fmaf(fx, fx, fy * fy);
                        if (a.amp) { a.amp[2 * oo] = fx; a.amp[2 * oo + 1] = fy; }
                    }
                    if (stj == SLOT_WAIT && !S0 && s == 3) {
                        const float v = r == vw.s0[4 * g + j] ? 1.0f : 0.0f;
                        qset(Ax, j, v); qset(Ay, j, 0.f);
                        qset(Kx[k], j, 0.f); qset(Ky[k], j, 0.f);
                        qset(nx, j, v); qset(ny, j, 0.f);
                    }
                }
            }
            if (!S0 && s == 3) set_a(k, ro + 4 * g, Ax, Ay);
            stq(Cn + ro, nx);
            stq(Cn + np + ro, ny);
        }
        __syncwarp();
        ++phase;
        // phase factors of the stages ahead: t + dt once stage 0 has read those of t, the next step's half
        // time once stage 2 has read this one's (t = 0 of a starting slot needs none)
        if (!S0 && s != 2) {
            float *dst = s == 1 ? PHa : PHb;
            for (int i = tid; i < NL * B; i += TE) {
                const int bb = i % B, stb = vw.state[bb];
                if (stb == SLOT_ACTIVE || (stb == SLOT_WAIT && s == 3)) {
                    const unsigned nh = stb == SLOT_WAIT ? 1u : 2u * (unsigned)vw.steps[bb] + (s == 1 ? 2u : 3u);
                    const float2 p = phase_factor(inc[i], nh);
                    dst[i] = p.x;
                    dst[NL * B + i] = p.y;
                }
            }
        }
        __syncwarp();
        // per-slot sums over the warp (lanes of one group), FP32; six quantities at stage 0, two
        // (force, torque) at the others
        float *rw = red + warp * 6 * B;
        // quantities q0 and q0 + 1 from their packed pairs
        auto warp_sums = [&](int q0, const float2 (&s0)[2], const float2 (&s1)[2]) {
            float part[8] = {s0[0].x, s0[0].y, s0[1].x, s0[1].y, s1[0].x, s1[0].y, s1[1].x, s1[1].y};
            if (G4 <= 4) {
                const float x = reduce8(part, lane, G4);
                const int idx = ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);
                if ((lane & 3) == g) rw[(q0 + (idx >> 2)) * B + 4 * g + (idx & 3)] = x;
            } else {
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    part[i] += __shfl_xor_sync(full, part[i], 8);
                    part[i] += __shfl_xor_sync(full, part[i], 16);
                    if (lane < 8) rw[(q0 + (i >> 2)) * B + 4 * g + (i & 3)] = part[i];
                }
            }
        };
#pragma unroll
        for (int i = 0; i < 2; ++i) { f2[i] = neg2(f2[i]); t2[i] = neg2(t2[i]); }
        warp_sums(0, f2, t2);
        if constexpr (S0) {
#pragma unroll
            for (int i = 0; i < 2; ++i) j2[i] = sub2(j2[i], m2[i]);
            warp_sums(2, v2, j2);
            // |a|^2 and E|a|^2 (their own pass: fewer sums live at once)
            float2 n2[2], e2[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) n2[i] = e2[i] = make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < kUpt; ++k) {
                const int r = (tid + k * TE) >> lg4;
                if (r >= n || !any) continue;
                Q4 Ax, Ay;
                get_a(k, r * B + 4 * g, Ax, Ay);
                const float2 el = dup2(elev[__ldg(S.row_info + r).y]);
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const float2 pp = fma2(Ax.p[i], Ax.p[i], mul2(Ay.p[i], Ay.p[i]));
                    n2[i] = add2(n2[i], pp);
                    e2[i] = fma2(el, pp, e2[i]);
                }
            }
            __syncwarp();
            warp_sums(4, n2, e2);
        }
        any = act;
        __syncwarp();
    };
    for (;;) {
        stage(std::true_type{}, 0);
        __syncthreads();
        // (read behind the barrier: whether or not a wait ran out, both roles leave at the same stage)
        bool run = false;
#pragma unroll
        for (int i = 0; i < NS; ++i) run |= sh.live[i] != 0;
        if (!run) break;
#pragma unroll 1
        for (int s = 1; s < 4; ++s) {
            stage(std::false_type{}, s);
            __syncthreads();
        }
    }
    }
}

// EXACT: every system of the launch runs BMAX slots per CTA (compile-time slot count); otherwise
// each system runs the slot count of a.slots
template <int BMAX, int T, int kUpt, bool EXACT>  // kUpt: (row, 4-column) units per element thread at most
__global__ void __launch_bounds__(T, batched_min_blocks<T>()) k_batched_f32(BatchMultiArgs a)
{
    static_assert(BMAX % 4 == 0 && BMAX <= 32, "batch width");
    static_assert(T / 32 - batch_slot_warps(BMAX) >= 1, "no element warps");
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ BatchShared<BMAX> sh;
    bool first = true;
    unsigned phase = 0;  // stages published so far (parity of the mbarrier)
    if (threadIdx.x == 0) tc_mbar_init(&sh.published, batch_slot_warps(BMAX));
    for (;;) {
        // bind to a system
        if (threadIdx.x == 0) {
            const int s = pick_system(a, first);
            sh.cur = s;
            sh.timeout = 0;
            if (s >= 0) sh.S = a.sys[s];
        }
        __syncthreads();
        first = false;
        const int cur = sh.cur;
        if (cur < 0) break;
        batched_system<EXACT ? BMAX : 0, BMAX, T, kUpt>(a, sh, cur, smraw, phase);
        __syncthreads();  // both roles are done with this system before the CTA binds to the next
    }
}

// the largest slot count (4, 8, 16 or 32, at most BMAX) with which a system fits a CTA of the shape; 0 if
// none.  The first bound (`cap` bytes for three amplitude arrays, two values per term and slot and eight
// partial sums) says which bases a shape takes, whatever the layout, so that a shape that a caller keeps
// stays valid; the layout above it is at most 16 L B bytes larger, which fits for every such basis with
// four slots.
template <int BMAX, int T, int kUpt>
int batched_slots(const DevSys &h, size_t cap)
{
    constexpr int NE = T / 32 - batch_slot_warps(BMAX);
    constexpr size_t kMaxBytes = 232448;  // shared memory of a CTA
    static_assert(kUpt * NE * 32 <= kBatchMaxRows, "the group tables are built for at most kBatchMaxRows rows");
    const size_t n = h.n, nl = h.n_levels, L = h.L;
    for (int b = BMAX; b >= 4; b >>= 1) {
        const size_t bound = 24 * (n + nl) * b + 16 * L * b + 4 * nl + 32 * (size_t)NE * b + 16 + 400 + 200 * BMAX;
        if (n * (b / 4) <= (size_t)kUpt * NE * 32 && bound <= cap &&
            batched_smem<BMAX, T, kUpt>(h, b) + sizeof(BatchShared<BMAX>) <= kMaxBytes)
            return b;
    }
    return 0;
}

template <int BMAX, int T, int kUpt>
cudaError_t launch_batched(BatchMultiArgs a, const std::vector<const DevSys *> &hs, size_t cap, int sms,
                           cudaStream_t st)
{
    size_t smem = 0;
    int minb = BMAX;
    for (size_t i = 0; i < hs.size(); ++i) {
        const int b = batched_slots<BMAX, T, kUpt>(*hs[i], cap);
        if (b == 0) return cudaErrorInvalidConfiguration;
        a.slots[i] = b;
        minb = std::min(minb, b);
        smem = std::max(smem, batched_smem<BMAX, T, kUpt>(*hs[i], b));
    }
    const bool exact = minb == BMAX;
    const void *kern = exact ? (const void *)k_batched_f32<BMAX, T, kUpt, true>
                             : (const void *)k_batched_f32<BMAX, T, kUpt, false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, T, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    const int grid = std::max(1, std::min(sms * per_sm, (a.n + minb - 1) / minb));
    if (exact) k_batched_f32<BMAX, T, kUpt, true><<<grid, T, smem, st>>>(a);
    else k_batched_f32<BMAX, T, kUpt, false><<<grid, T, smem, st>>>(a);
    count_launches(1);
    return cudaGetLastError();
}

// Shapes (slots per CTA at most, threads), kBatchShapes; a CTA of 256 threads leaves room for two
// per SM (half the shared memory each).
static size_t shape_cap(int i) { return (i == 2 || i == 6) ? 110 * 1024 : 220 * 1024; }

// slot count of shape index i for the system (0: does not fit) and the shared memory it takes
template <int BMAX, int T, int kUpt>
static int shape_slots_of(const DevSys &h, size_t cap, size_t *smem)
{
    const int b = batched_slots<BMAX, T, kUpt>(h, cap);
    if (smem) *smem = b ? batched_smem<BMAX, T, kUpt>(h, b) + sizeof(BatchShared<BMAX>) : 0;
    return b;
}

static int shape_slots(const DevSys &h, int i, size_t *smem = nullptr)
{
    const size_t cap = shape_cap(i);
    switch (i) {
        case 0: return shape_slots_of<32, 512, 4>(h, cap, smem);
        case 1: return shape_slots_of<16, 512, 4>(h, cap, smem);
        case 2: return shape_slots_of<8, 256, 4>(h, cap, smem);
        case 3: return shape_slots_of<8, 512, 2>(h, cap, smem);
        case 4: return shape_slots_of<4, 512, 4>(h, cap, smem);
        case 5: return shape_slots_of<16, 256, 4>(h, cap, smem);
        case 6: return shape_slots_of<4, 256, 2>(h, cap, smem);
        default: return 0;
    }
}

bool batched_shape_fits(const DevSys &h, int i) { return shape_slots(h, i) > 0; }

int batched_width(const DevSys &h)
{
    for (int i = 0; i < 6; ++i)
        if (batched_shape_fits(h, i)) return kBatchShapes[i][0] * 1000 + kBatchShapes[i][1];
    return 0;
}

// The automatic shape for n trajectories over the systems hs.  A CTA steps its slots in lockstep,
// so its step time grows with its slot count while the throughput of an SM levels off from about
// eight slots on: the longest trajectories, which start first from the longest-first work list,
// then set the end of the launch when there are too many slots, and the refill order of the list
// cannot balance the slots when there are too few.  The rule: the shape with the most slots on
// the GPU (slots per CTA x CTAs per SM x SMs, the slot count of the narrowest system) that still
// leaves two trajectories per slot, else the one with the fewest slots; ties go to the earlier
// entry of kAutoOrder, which puts the eight-slots-per-SM shapes first, two CTAs of four slots before one of
// eight: their barriers do not stop each other (3072 trajectories of N = 441 and uneven length: 361 against
// 387 ms; equal lengths 62.2 against 60.7 M traj-steps/s).  -1: no shape fits.
int batched_auto_shape(const std::vector<const DevSys *> &hs, int n, int sms)
{
    static const int kAutoOrder[7] = {6, 3, 4, 0, 1, 5, 2};
    int best = -1, fewest = -1;
    long long best_slots = -1, fewest_slots = 0;
    for (int k = 0; k < 7; ++k) {
        const int i = kAutoOrder[k];
        int b = 1 << 30;
        size_t smem = 0;
        for (const DevSys *h : hs) {
            size_t sm = 0;
            b = std::min(b, shape_slots(*h, i, &sm));
            smem = std::max(smem, sm);
        }
        if (hs.empty() || b <= 0) continue;
        // two CTAs of 256 threads share an SM's registers when their shared memory allows
        const int per_sm = (kBatchShapes[i][1] == 256 && smem <= 113 * 1024) ? 2 : 1;
        const long long slots = (long long)b * per_sm * sms;
        if (2 * slots <= n && slots > best_slots) {
            best_slots = slots;
            best = i;
        }
        if (fewest < 0 || slots < fewest_slots) {
            fewest_slots = slots;
            fewest = i;
        }
    }
    return best >= 0 ? best : fewest;
}

// one persistent launch over every system of the call, with the requested shape (index + 1) or
// the automatic one (batched_auto_shape)
cudaError_t run_batched(BatchMultiArgs a, const std::vector<const DevSys *> &hs, int shape, cudaStream_t st)
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (hs.empty() || (int)hs.size() > kBatchMaxSystems) return cudaErrorInvalidValue;
    auto all_fit = [&](int i) {
        for (const DevSys *h : hs)
            if (!batched_shape_fits(*h, i)) return false;
        return true;
    };
    int idx = -1;
    if (shape > 0) {
        if (shape > 7 || !all_fit(shape - 1)) return cudaErrorInvalidConfiguration;
        idx = shape - 1;
    } else {
        idx = batched_auto_shape(hs, a.n, sms);
    }
    if (idx < 0) return cudaErrorInvalidConfiguration;
    const size_t cap = shape_cap(idx);
    switch (idx) {
        case 0: return launch_batched<32, 512, 4>(a, hs, cap, sms, st);
        case 1: return launch_batched<16, 512, 4>(a, hs, cap, sms, st);
        case 2: return launch_batched<8, 256, 4>(a, hs, cap, sms, st);
        case 3: return launch_batched<8, 512, 2>(a, hs, cap, sms, st);
        case 4: return launch_batched<4, 512, 4>(a, hs, cap, sms, st);
        case 5: return launch_batched<16, 256, 4>(a, hs, cap, sms, st);
        case 6: return launch_batched<4, 256, 2>(a, hs, cap, sms, st);
        default: return cudaErrorInvalidConfiguration;
    }
}

}  // namespace mqct
