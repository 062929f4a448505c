// mp_mixed.cuh - the mixed-precision tracking engine.
//
// Same method as the FP64 path (Pollock 1988: per-axis linear velocity,
// exit time (d / v_p) ln(1 + z) / z, analytic motion, smallest exit time
// wins, hand-over to the neighbour), evaluated in local fractions
// xi in [0, 1] of the cell with velocities u = v / D (1/s) in FP32:
//   u_p = u1 + A xi, A = u2 - u1, exit distance d = 1 - xi or -xi,
//   t_a = (d / u_p) g(z), z = A d / u_p, g(z) = ln(1 + z) / z,
//   xi(t) = xi + u_p t h(A t), h(w) = (e^w - 1) / w.
// g and h are evaluated both ways and selected (no divergent branch): their
// Taylor series near 0 (|z| < 1/8, |w| < 1/2; free of the 0/0 at 0),
// otherwise logf and expf (about 1 ulp, and free of the internal branches
// of log1pf and expm1f): g = ln(u) / (u - 1) with u = fl(1 + z), exact to a
// few ulp because the rounding of 1 + z cancels (Goldberg 1991), or
// ln(u_exit / u_p) / z for z < -1/2, where the ratio, not 1 + z, keeps full
// FP32 accuracy as u_exit -> 0.
//
// The cumulative travel time is carried as an unevaluated pair of FP32
// values (a double-float number, 48-bit significand): each step adds its
// FP32 step time with Knuth's error-free two-sum, and output times and the
// stop time are compared as pairs (the host splits them once per request).
// GB300 executes FP64 at 1/64 of the FP32 rate and output events occur in a
// different step on every lane, so FP64 arithmetic there would run in
// divergent branches; the pair keeps the time to ~1e-14 relative at FP32
// cost.  FP64 is used for the values written out: travel times and global
// positions.  Compiled with FMA contraction on (results are compared with the
// FP64 oracle within stated tolerances, not bit for bit).
//
// F64T = true gives the variant in which FP64 is kept for the cumulative
// travel time (one double, compared with the FP64 output and stop times)
// and for the near-zero branch of the exit time (log1p(z) / z evaluated in
// FP64 for |z| < 1/8); everything else is as above.  It exists to measure
// what the FP32 pair and the FP32 series cost in accuracy (mp_mixed_f64t.cu,
// MP_PREC_MIXED_F64T).
#pragma once
#include <cfloat>
#include <cmath>

#include "mp_internal.h"
#include "mp_sched.cuh"

namespace mp {

template <bool F64T, bool ONE_REQ>
struct MixEngine {
    static constexpr bool ONE = ONE_REQ;
    static constexpr bool OWN_SLOTS = true;   // records wait in the lane's own slots
    // (issue bound: as many warps as fit; with FP64 time the FP64 pipe binds)
    static constexpr bool EVEN_ROUNDS = F64T;
    static constexpr int FETCH = F64T ? 4 : 16;   // steps per fetch
    // What bounds it: issue (70 % of the slots; ALU instructions take two
    // cycles each), with 32 warps an SM hiding the rest, so four blocks of 256
    // threads at 64 registers and nothing spilled.  For that the state is kept
    // small (row, column and layer come back from the cell index where a
    // position is written) and timeseries records wait in the lane's own
    // slots.  Measured on 1e6 particles, 200x200x20 cells, 50 output times:
    // persistent schedule 6.48 -> 5.70 ms (76 registers and the warp's queue
    // before; with that queue at 64 registers 5.82), static 5.48 -> 5.23 ms;
    // 2e6 particles, 400x400x40 cells, 20 times 25.1 -> 21.3 ms.  (With the
    // fetch of mp_sched.cuh: 5.26, 5.02 and 20.4 ms.)  A batch's persistent
    // kernel keeps 80 registers (the descriptors are read through a table):
    // three blocks; 240,000 particles of 24 requests 1.07 ms, at 64 registers
    // and four blocks 1.14.
    // With FP64 time (F64T) three log1p a step on the FP64 pipe bind it, as the
    // FP64 engine is bound: an idle lane costs as much as a live one, warps
    // beyond 16 an SM gain nothing, and registers are there.  So its persistent
    // kernel takes two blocks, even rounds and 4 steps a fetch (1e6 particles,
    // 50 output times 104.2 -> 101.7 ms with the constants above against these,
    // endpoints 99.3 -> 96.1; 200,000 24.3 -> 22.2 and 22.7 -> 21.2; 100,000
    // with pathlines and output times 13.3 -> 11.5).
    // Kernels with pathlines and output times take three blocks, 80 registers:
    // without a target the compiler spills at 64 (100,000 particles of ten
    // requests 1.34 -> 1.15 ms, static 1.20 -> 1.11; one request 1.06 -> 1.05;
    // with FP64 time, static, 13.5 -> 13.2).
    static constexpr int min_blocks(bool dynamic, bool ts, bool pl)
    {
        if (F64T && dynamic) return 2;
        if (ts && pl) return 3;
        return pl ? 0 : (dynamic ? (ONE ? 4 : 3) : 4);
    }
    DevField f;
    Batch b;

    // descriptor of request r of the launch (ONE: the launch has one, by value)
    __device__ __forceinline__ const Req& req(int r) const
    {
        if constexpr (ONE) return b.one;
        else return b.reqs[r];
    }


    struct State {
        int r;            // request of the particle within the launch
        int c;            // (its row, column and layer are formed where a position is written)
        float x0, x1, x2;  // local fractions in [0, 1]
        float th, tl;  // travel time as an FP32 pair th + tl (F64T: unused)
        float eh, el;  // next output time or the stop time, whichever is first (as a pair)
        double t, e;   // F64T: travel time and next event in FP64
        unsigned steps;
        unsigned long long h;
        int kn;
        int st;
        int ef;
    };

    // ---- double-float helpers (pairs with |lo| <= ulp(hi) / 2) ----
    // (nh, nl) = (th, tl) + dt, exact up to the final rounding of the low part
    __device__ __forceinline__ static void ff_add(float th, float tl, float dt, float& nh, float& nl)
    {
        const float sh = th + dt;
        const float bb = sh - th;
        const float lo = tl + ((th - (sh - bb)) + (dt - bb));
        nh = sh + lo;
        nl = lo - (nh - sh);
    }
    __device__ __forceinline__ static bool ff_ge(float ah, float al, float bh, float bl)
    {
        return ah > bh || (ah == bh && al >= bl);
    }
    // (a - b) as one FP32 value; a and b close, so the high parts cancel exactly
    __device__ __forceinline__ static float ff_diff(float ah, float al, float bh, float bl)
    {
        return (ah - bh) + (al - bl);
    }
    __device__ __forceinline__ static float2 time_pair(const DevOut& o, int kk)
    {
        return __ldg(o.times_ff + kk);
    }
    // the travel time as one FP64 value
    __device__ __forceinline__ static double time_of(const State& s)
    {
        if constexpr (F64T) return s.t;
        else return (double)s.th + (double)s.tl;
    }

    static constexpr float SMALL = 0.125f;

    // g(z) = ln(1 + z) / z, with 1 + z = u_exit / u_p: the series
    // sum_k (-z)^k / (k + 1) to degree 7 for |z| < 1/8; otherwise
    // ln(u) / (u - 1) with u = fl(1 + z), in which the rounding of 1 + z
    // cancels (Goldberg 1991), and for z < -1/2, where 1 + z itself
    // cancels, the logarithm of the ratio of the two stored velocities
    __device__ __forceinline__ static float g_log1p_over(float z, float ratio)
    {
        float ser;
        if constexpr (F64T) {
            // the near-zero branch in FP64: log1p(z) / z of the FP32 z (1 at z = 0)
            const double zd = (double)z;
            ser = (float)(zd == 0.0 ? 1.0 : log1p(zd) / zd);
        } else {
            ser = 1.0f + z * (-0.5f + z * (1.0f / 3.0f + z * (-0.25f + z * (0.2f + z * (-1.0f / 6.0f +
                                                                                  z * (1.0f / 7.0f + z * -0.125f))))));
        }
        const bool near_m1 = z < -0.5f;
        const float u = 1.0f + z;
        const float L = logf(near_m1 ? ratio : u);
        const float lg = __fdividef(L, near_m1 ? z : u - 1.0f);
        return fabsf(z) < SMALL ? ser : lg;
    }
    // h(w) = (e^w - 1) / w: sum_k w^k / (k + 1)! to degree 8 for |w| < 1/2
    // (truncation below 6e-10), otherwise the exponential (e^w - 1 then
    // loses at most a factor 2.5 to cancellation)
    __device__ __forceinline__ static float h_expm1_over(float w)
    {
        const float ser =
            1.0f + w * (0.5f + w * (1.0f / 6.0f + w * (1.0f / 24.0f + w * (1.0f / 120.0f + w * (1.0f / 720.0f +
                        w * (1.0f / 5040.0f + w * (1.0f / 40320.0f + w * (1.0f / 362880.0f))))))));
        const float ex = __fdividef(expf(w) - 1.0f, w);
        return fabsf(w) < 0.5f ? ser : ex;
    }

    template <class T>
    __device__ __forceinline__ static T sel3(int a, T x, T y, T z)
    {
        return a == 0 ? x : (a == 1 ? y : z);
    }

    // exit time along one axis in local units; branch-free around the
    // transcendental so that a warp's lanes stay converged (no-exit lanes
    // compute on harmless operands and select +inf)
    __device__ __forceinline__ static float exit_time(float u1, float u2, float A, float up, float xi, int& face)
    {
        const bool fw = up > 0.0f && u2 > 0.0f;
        const bool bw = up < 0.0f && u1 < 0.0f;
        face = fw ? 1 : (bw ? -1 : 0);
        const float d = fw ? 1.0f - xi : -xi;
        const float ue = fw ? u2 : u1;
        const float ups = face ? up : 1.0f;
        const float t1 = __fdividef(d, ups);
        const float g = g_log1p_over(A * t1, __fdividef(ue, ups));
        return face ? t1 * g : CUDART_INF_F;
    }

    __device__ __forceinline__ static float move(float A, float up, float xi, float dt)
    {
        const float s = up * dt;
        const float xn = fminf(fmaxf(xi + s * h_expm1_over(A * dt), 0.0f), 1.0f);
        return s == 0.0f ? xi : xn;
    }

    // global position = face coordinate + fraction * cell size per axis,
    // rounded step by step (no contraction) so endpoints and records agree
    // exactly
    __device__ __forceinline__ void place(int c, float x0, float x1, float x2, double& x, double& y, double& z) const
    {
        int k, i, j;
        split_cell(f, c, k, i, j);
        x = __dadd_rn(__ldg(f.xf + j), __dmul_rn((double)x0, __ldg(f.delr + j)));
        y = __dadd_rn(__ldg(f.yf + i), __dmul_rn((double)x1, __ldg(f.delc + i)));
        z = __dadd_rn(__ldg(f.zf + k), __dmul_rn((double)x2, __ldg(f.dz + k)));
    }

    __device__ __forceinline__ void record(long long q, int kk, const State& s, double x, double y, double z,
                                           int st) const
    {
        const Req& R = req(s.r);
        const DevState& in = R.in;
        const DevOut& o = R.o;
        const TrackParams& p = R.p;
        (void)in; (void)o; (void)p;
        store_record(o.ts + (long long)kk * p.n + q, x, y, z, s.c, st);
    }

    __device__ __forceinline__ void final_pos(const State& s, double& x, double& y, double& z) const
    {
        if (s.c < 0) {
            x = y = z = CUDART_NAN;
            return;
        }
        place(s.c, s.x0, s.x1, s.x2, x, y, z);
    }

    // next event as a pair: the next output time or the stop time
    __device__ __forceinline__ void next_event(State& s) const
    {
        const Req& R = req(s.r);
        const DevState& in = R.in;
        const DevOut& o = R.o;
        const TrackParams& p = R.p;
        (void)in; (void)o; (void)p;
        if constexpr (F64T) {
            double ev = p.t_stop;
            if (s.kn < p.n_times) ev = fmin(ev, __ldg(o.times + s.kn));
            s.e = ev;
            return;
        }
        float eh = p.tstop_hi, el = p.tstop_lo;
        if (s.kn < p.n_times) {
            const float2 tk = time_pair(o, s.kn);
            if (!ff_ge(tk.x, tk.y, eh, el)) { eh = tk.x; el = tk.y; }
        }
        s.eh = eh;
        s.el = el;
    }

    template <bool TS>
    __device__ __forceinline__ void load(int r, long long q, State& s) const
    {
        s.r = r;
        const Req& R = req(s.r);
        const DevState& in = R.in;
        const DevOut& o = R.o;
        const TrackParams& p = R.p;
        (void)in; (void)o; (void)p;
        s.c = in.cell[q];
        s.st = in.status[q];
        // a later flow period leaves particles that ended before it untouched
        // (decided on the stored status, before this field's cell classes)
        if (p.cont && s.st != MP_ST_ACTIVE) {
            s.st = ST_SKIP;
            return;
        }
        const double t0 = in.t[q];
        // cell-steps, hash and last face carried by a resumed particle
        s.steps = in.steps ? in.steps[q] : 0u;
        s.h = FNV_INIT;
        s.kn = 0;
        s.ef = (s.steps && in.exit_face) ? (int)in.exit_face[q] : MP_FACE_NONE;
        if (s.c >= 0 && (long long)s.c < f.ncell) {
            int k, i, j;
            split_cell(f, s.c, k, i, j);
            s.x0 = __fdiv_rn((float)in.px[q], (float)__ldg(f.delr + j));
            s.x1 = __fdiv_rn((float)in.py[q], (float)__ldg(f.delc + i));
            s.x2 = __fdiv_rn((float)in.pz[q], (float)__ldg(f.dz + k));
            s.h = (s.steps && in.hash) ? in.hash[q] : fnv_step(s.h, s.c);
            // a resumed particle may sit inside a sink cell it entered with
            // pass-through; a moving particle whose cell is not active under
            // this field (another flow period) stops there
            const int ib = __ldg(f.ibound + s.c);
            if (s.st == MP_ST_ACTIVE) {
                if (ib == 0 || ib == -1) s.st = MP_ST_BOUNDARY;
                else if (ib == 2 && sink_stops(p, f.sinkfrac, s.c)) s.st = MP_ST_SINK;
            }
        } else {
            s.c = -1;
            s.x0 = s.x1 = s.x2 = 0.0f;
            s.st = MP_ST_INVALID_RELEASE;
        }
        if (TS) {
            if (p.cont) {
                // output times up to the period start were written by the previous period
                while (s.kn < p.n_times && __ldg(o.times + s.kn) <= t0) s.kn++;
            } else {
                while (s.kn < p.n_times && __ldg(o.times + s.kn) <= t0) {
                    double x, y, z;
                    final_pos(s, x, y, z);
                    record(q, s.kn, s, x, y, z, s.st);
                    s.kn++;
                }
            }
        }
        if (s.st == MP_ST_ACTIVE && t0 >= p.t_stop) s.st = MP_ST_TIME;
        s.th = (float)t0;
        s.tl = (float)(t0 - (double)s.th);
        if constexpr (F64T) s.t = t0;
        next_event(s);
    }

    // deferred timeseries records: REC_SLOTS of each lane (slot 32 k + lane),
    // kept small, since what the block's queues take of the SM's shared
    // memory its L1 does not have for the field's records
    struct alignas(16) RecQ {
        static constexpr int N = 32 * REC_SLOTS;
        float x0[N], x1[N], x2[N], tau[N];
        int c[N];
        unsigned q[N];            // (a group of 2^32 particles would not fit the device)
        unsigned kk[N];           // output index; the top bit: status NO_EXIT, else ACTIVE
        int r[ONE ? 1 : N];
        unsigned char list[N];
    };

    // a record of output index kk at tau after the step's start
    __device__ __forceinline__ void rec_put(RecQ& Q, int slot, const State& s, long long q, int kk, float tau,
                                            bool no_exit) const
    {
        if (!ONE) Q.r[slot] = s.r;
        Q.x0[slot] = s.x0; Q.x1[slot] = s.x1; Q.x2[slot] = s.x2;
        Q.tau[slot] = tau;
        Q.q[slot] = (unsigned)q;
        Q.c[slot] = s.c;
        Q.kk[slot] = (unsigned)kk | (no_exit ? 0x80000000u : 0u);
    }

    __device__ __forceinline__ void rec_eval(const RecQ& Q, int slot) const
    {
        const Req& R = req(ONE ? 0 : Q.r[slot]);
        const DevOut& o = R.o;
        const TrackParams& p = R.p;
        const int c = Q.c[slot];
        const float tau = Q.tau[slot];
        const float4* rp = reinterpret_cast<const float4*>(f.rec32 + c);
        const float4 ra = __ldg(rp), rb = __ldg(rp + 1);
        const float Ax = ra.y - ra.x, Ay = ra.w - ra.z, Az = rb.y - rb.x;
        const float a0 = Q.x0[slot], a1 = Q.x1[slot], a2 = Q.x2[slot];
        double x, y, z;
        place(c, move(Ax, ra.x + Ax * a0, a0, tau), move(Ay, ra.z + Ay * a1, a1, tau),
              move(Az, rb.x + Az * a2, a2, tau), x, y, z);
        const unsigned kk = Q.kk[slot];
        store_record(o.ts + (long long)(kk & 0x7fffffffu) * p.n + Q.q[slot], x, y, z, c,
                     kk >> 31 ? MP_ST_NO_EXIT : MP_ST_ACTIVE);
    }

    template <bool TS>
    __device__ __forceinline__ void step(long long q, State& s, bool live, RecQ& Q, int& held) const
    {
        const Req& R = req(s.r);
        const DevState& in = R.in;
        const DevOut& o = R.o;
        const TrackParams& p = R.p;
        (void)in; (void)o; (void)p;
        enum { P_NONE, P_CROSS, P_TIME, P_NOEXIT, P_CAPTURE };
        int path = P_NONE;
        float rh = 0, rl = 0;   // the end of the step (or the stop time): output times up to it are recorded
        double rd = 0.0;        // F64T: the same
        (void)rd;
        bool due = false;
        float Ax = 0, Ay = 0, Az = 0, up0 = 0, up1 = 0, up2 = 0, tmin = 0, nh = 0, nl = 0;
        double tn = 0.0;   // F64T: the time at the end of the step
        (void)tn;
        bool ev = false;
        int f0 = 0, f1 = 0, f2 = 0, ax = -1;
        unsigned nb = 0;
        if (live) {
            if ((long long)s.steps >= p.max_steps) {
                s.st = MP_ST_STEP_CAP;
            } else if ((unsigned long long)s.c >= (unsigned long long)f.ncell) {
                atomicCAS(o.counters + COUNTER_ERR, 0ULL, (unsigned long long)q + 1ULL);
                s.st = MP_ST_INVALID_RELEASE;
            } else {
                const float4* rp = reinterpret_cast<const float4*>(f.rec32 + s.c);
                const float4 ra = __ldg(rp), rb = __ldg(rp + 1);
                const float u1x = ra.x, u2x = ra.y, u1y = ra.z, u2y = ra.w, u1z = rb.x, u2z = rb.y;
                nb = __float_as_uint(rb.z);
                Ax = u2x - u1x; Ay = u2y - u1y; Az = u2z - u1z;
                up0 = u1x + Ax * s.x0; up1 = u1y + Ay * s.x1; up2 = u1z + Az * s.x2;
                const float te0 = exit_time(u1x, u2x, Ax, up0, s.x0, f0);
                const float te1 = exit_time(u1y, u2y, Ay, up1, s.x1, f1);
                const float te2 = exit_time(u1z, u2z, Az, up2, s.x2, f2);
                tmin = CUDART_INF_F;
                if (f0 != 0 && te0 < tmin) { tmin = te0; ax = 0; }
                if (f1 != 0 && te1 < tmin) { tmin = te1; ax = 1; }
                if (f2 != 0 && te2 < tmin) { tmin = te2; ax = 2; }
                s.steps++;
                if constexpr (F64T) {
                    tn = s.t + (double)tmin;
                    ev = ax < 0 || tn >= s.e;
                } else {
                    ff_add(s.th, s.tl, tmin, nh, nl);
                    ev = ax < 0 || ff_ge(nh, nl, s.eh, s.el);
                }
                if (ev) {
                    bool past_stop;
                    if constexpr (F64T) past_stop = tn >= p.t_stop;
                    else past_stop = ff_ge(nh, nl, p.tstop_hi, p.tstop_lo);
                    if (ax < 0 && __ldg(f.ibound + s.c) == 2) path = P_CAPTURE;   // in a sink cell it passes through
                    else if (ax < 0 && !(p.t_stop < CUDART_INF)) path = P_NOEXIT;
                    else if (ax < 0 || past_stop) path = P_TIME;
                    else path = P_CROSS;
                    if (TS && path != P_CAPTURE && s.kn < p.n_times) {
                        due = true;
                        if constexpr (F64T) {
                            rd = path == P_NOEXIT ? CUDART_INF : (path == P_TIME ? p.t_stop : tn);
                        } else {
                            rh = path == P_NOEXIT ? CUDART_INF_F : (path == P_TIME ? p.tstop_hi : nh);
                            rl = path == P_NOEXIT ? 0.0f : (path == P_TIME ? p.tstop_lo : nl);
                        }
                    }
                } else {
                    path = P_CROSS;
                }
            }
        }
        if (TS) {
            // output times inside this step, t_k <= end of step, from its
            // start into the lane's slots; full slots are evaluated by the warp
            const int lane = threadIdx.x & 31;
            while (true) {
                if (due) {
                    while (true) {
                        float tau;
                        if constexpr (F64T) {
                            const double tk = __ldg(o.times + s.kn);
                            if (!(tk <= rd)) { due = false; break; }
                            tau = (float)(tk - s.t);
                        } else {
                            const float2 tk = time_pair(o, s.kn);
                            if (!ff_ge(rh, rl, tk.x, tk.y)) { due = false; break; }
                            tau = ff_diff(tk.x, tk.y, s.th, s.tl);
                        }
                        if (held == REC_SLOTS) break;
                        rec_put(Q, 32 * held + lane, s, q, s.kn, tau, path == P_NOEXIT);
                        held++;
                        s.kn++;
                        if (s.kn >= p.n_times) { due = false; break; }
                    }
                    if (!due) next_event(s);
                }
                if (!__any_sync(0xffffffffu, due)) break;
                rs_flush(*this, Q, held);
            }
        }
        if (path == P_NONE) return;
        if (path == P_CAPTURE) {
            s.st = MP_ST_SINK;
            return;
        }
        if (path == P_NOEXIT) {
            s.st = MP_ST_NO_EXIT;
            return;
        }
        if (path == P_TIME) {
            float dt;
            if constexpr (F64T) dt = (float)(p.t_stop - s.t);
            else dt = ff_diff(p.tstop_hi, p.tstop_lo, s.th, s.tl);
            s.x0 = move(Ax, up0, s.x0, dt);
            s.x1 = move(Ay, up1, s.x1, dt);
            s.x2 = move(Az, up2, s.x2, dt);
            s.th = p.tstop_hi;
            s.tl = p.tstop_lo;
            if constexpr (F64T) s.t = p.t_stop;
            s.st = MP_ST_TIME;
            return;
        }
        // the two other axes move by the analytic formula (two slots,
        // uniform across lanes), the exit axis is put on its face
        const float dt = tmin;
        const int a1 = ax == 0 ? 1 : 0, a2 = ax == 2 ? 1 : 2;
        const float n1 = move(sel3(a1, Ax, Ay, Az), sel3(a1, up0, up1, up2), sel3(a1, s.x0, s.x1, s.x2), dt);
        const float n2 = move(sel3(a2, Ax, Ay, Az), sel3(a2, up0, up1, up2), sel3(a2, s.x0, s.x1, s.x2), dt);
        const int face = ax == 0 ? f0 : (ax == 1 ? f1 : f2);
        const float onface = face > 0 ? 1.0f : 0.0f;
        s.x0 = ax == 0 ? onface : n1;
        s.x1 = ax == 1 ? onface : (ax == 0 ? n1 : n2);
        s.x2 = ax == 2 ? onface : n2;
        s.th = nh;
        s.tl = nl;
        if constexpr (F64T) s.t = tn;
        const int fidx = 2 * ax + (face > 0 ? 1 : 0);
        s.ef = fidx;
        const int cls = (int)((nb >> (2 * fidx)) & 3u);
        const int dj = ax == 0 ? face : 0, di = ax == 1 ? face : 0, dk = ax == 2 ? face : 0;
        if (cls != NB_ACTIVE &&
            !(cls == NB_SINK && !sink_stops(p, f.sinkfrac, s.c + dj + di * f.ncol + dk * f.ncol * f.nrow))) {
            s.st = cls == NB_OUTSIDE ? MP_ST_EXIT_DOMAIN : (cls == NB_BOUNDARY ? MP_ST_BOUNDARY : MP_ST_SINK);
            return;
        }
        s.c += dj + di * f.ncol + dk * f.ncol * f.nrow;
        const float entry = face > 0 ? 0.0f : 1.0f;
        s.x0 = ax == 0 ? entry : s.x0;
        s.x1 = ax == 1 ? entry : s.x1;
        s.x2 = ax == 2 ? entry : s.x2;
        s.h = fnv_step(s.h, s.c);
    }

    // the pathline point of the particle's current state
    __device__ __forceinline__ void path_point(const State& s, double& x, double& y, double& z, double& t) const
    {
        place(s.c, s.x0, s.x1, s.x2, x, y, z);
        t = time_of(s);
    }

    template <bool TS>
    __device__ __forceinline__ void finish(long long q, const State& s, unsigned long long* s_cnt) const
    {
        const Req& R = req(s.r);
        const DevState& in = R.in;
        const DevOut& o = R.o;
        const TrackParams& p = R.p;
        (void)in; (void)o; (void)p;
        const bool ok = s.c >= 0;
        const unsigned base = in.steps ? in.steps[q] : 0u;   // read before the group update
        double px = 0.0, py = 0.0, pz = 0.0, x = CUDART_NAN, y = CUDART_NAN, z = CUDART_NAN;
        if (ok) {
            int k, i, j;
            split_cell(f, s.c, k, i, j);
            px = __dmul_rn((double)s.x0, __ldg(f.delr + j));
            py = __dmul_rn((double)s.x1, __ldg(f.delc + i));
            pz = __dmul_rn((double)s.x2, __ldg(f.dz + k));
            x = __dadd_rn(__ldg(f.xf + j), px);
            y = __dadd_rn(__ldg(f.yf + i), py);
            z = __dadd_rn(__ldg(f.zf + k), pz);
        }
        o.cell[q] = s.c;
        o.x[q] = x; o.y[q] = y; o.z[q] = z;
        o.px[q] = px; o.py[q] = py; o.pz[q] = pz;
        o.t[q] = time_of(s);
        o.status[q] = (uint8_t)s.st;
        o.steps[q] = s.steps;
        o.exit_face[q] = (uint8_t)s.ef;
        o.hash[q] = s.h;
        if (p.update_group && ok) {
            in.cell[q] = s.c;
            in.px[q] = px; in.py[q] = py; in.pz[q] = pz;
            in.t[q] = time_of(s);
            in.status[q] = (uint8_t)((s.st == MP_ST_TIME || s.st == MP_ST_STEP_CAP) ? MP_ST_ACTIVE : s.st);
            if (in.steps) {
                in.steps[q] = s.steps;
                in.hash[q] = s.h;
                in.exit_face[q] = (uint8_t)s.ef;
            }
        }
        // steps taken in this launch; a particle paused at the end of a flow
        // period is counted by the period it ends in
        count_ended(*this, s.r, s.steps - base, s.st, s_cnt, p.last || !(s.st == MP_ST_TIME || s.st == MP_ST_STEP_CAP));
    }
};

// ---------------------------------------------------------------------------
// few particles: three lanes a particle
// ---------------------------------------------------------------------------

// What bounds a step of few particles: the instructions of three axes in one
// lane, about 450 a step one after the other.  As in the FP64 form, lane
// 3 g + a of a warp holds axis a of its particle g: one exit time and one
// motion a lane, the smallest time agreed by shuffles, the next cell's record
// read while the axes move, and everything but crossing into the next cell in
// one branch of the warp, in which the group's first lane writes records,
// points and ends with the axes gathered.  One step of 4864 particles 0.83 ->
// 0.42 us; 4000 particles with 20 output times, 200x200x20 cells 391 -> 195
// us (198 with the range check of the next cell in front of its load).
template <bool ONE, bool TS, bool PL>
__global__ void __launch_bounds__(32) k_track_axes_mixed(MixEngine<false, ONE> e)
{
    using E = MixEngine<false, ONE>;
    const DevField& f = e.f;
    __shared__ unsigned long long s_cnt[N_COUNTERS];
    typename E::RecQ& Q = *reinterpret_cast<typename E::RecQ*>(s_dyn);
    PathQ& P = *reinterpret_cast<PathQ*>(s_dyn + (TS ? sizeof(typename E::RecQ) : 0));
    if (threadIdx.x < N_COUNTERS) s_cnt[threadIdx.x] = 0ULL;
    window_begin(e);
    __syncwarp();
    const unsigned FULL = 0xffffffffu;
    // (lanes 30 and 31 hold no particle: they follow the first group's shuffles)
    const int lane = threadIdx.x & 31, grp = lane / 3, a = lane - 3 * grp, base = grp < AXES_PARTICLES ? 3 * grp : 0;
    const bool lead = a == 0;
    const int stride_y = f.ncol, stride_z = f.ncol * f.nrow;
    int held = 0, pcount = 0;   // held: records waiting, the same on the group's lanes, in the first one's slots
    long long q = 0;
    typename E::State s;        // x0, x1, x2: as last gathered
    s.r = 0;
    s.steps = 0;
    s.st = ST_SKIP;
    s.c = -1;
    s.x0 = s.x1 = s.x2 = 0.0f;
    s.th = s.tl = s.eh = s.el = 0.0f;
    bool live = false, ended = false, loaded = false;
    const long long g = (long long)blockIdx.x * AXES_PARTICLES + grp;
    if (grp < AXES_PARTICLES && g < e.b.n_total) {
        const int r = request_of(e, g, q);
        e.template load<TS>(r, q, s);
        live = s.st == MP_ST_ACTIVE;
        ended = !live && s.st != ST_SKIP;
        loaded = true;
    }
    if (PL)
        pl_push(e, P, pcount, s, q, lead && loaded && path_start(e, s), s.st == MP_ST_TIME ? MP_ST_ACTIVE : s.st);
    if (TS) tail_fill(e, s, q, lead && ended && !paused(e, s));
    __syncwarp();   // finish may write the group's state, which the group's other lanes load too
    if (lead && ended) e.template finish<TS>(q, s, s_cnt);
    // this lane's axis: fraction, and the cell's record of it
    float x = a == 0 ? s.x0 : (a == 1 ? s.x1 : s.x2);
    float u1 = 0.0f, u2 = 0.0f;
    unsigned nb = 0;
    auto read = [&](int c, float& v1, float& v2, unsigned& b) {
        const float* rp = reinterpret_cast<const float*>(f.rec32 + c);
        const float2 v = __ldg(reinterpret_cast<const float2*>(rp) + a);
        v1 = v.x;
        v2 = v.y;
        b = __ldg(reinterpret_cast<const unsigned*>(rp) + 6);
    };
    auto gather = [&]() {
        s.x0 = __shfl_sync(FULL, x, base);
        s.x1 = __shfl_sync(FULL, x, base + 1);
        s.x2 = __shfl_sync(FULL, x, base + 2);
    };
    if (live) read(s.c, u1, u2, nb);
    bool going = __any_sync(FULL, live);
    while (going) {
        const TrackParams& p = e.req(s.r).p;
        const bool go = live && !((long long)s.steps >= p.max_steps);
        const float A = u2 - u1;
        const float up = u1 + A * x;
        int face;
        float te = E::exit_time(u1, u2, A, up, x, face);
        if (!go) {
            face = 0;
            te = CUDART_INF_F;
        }
        const unsigned ups = __ballot_sync(FULL, face > 0);
        const float t0 = __shfl_sync(FULL, te, base), t1 = __shfl_sync(FULL, te, base + 1),
                    t2 = __shfl_sync(FULL, te, base + 2);
        int ax = -1;   // the smallest time wins, ties to the lower axis
        float tmin = CUDART_INF_F;
        if (t0 < tmin) { tmin = t0; ax = 0; }
        if (t1 < tmin) { tmin = t1; ax = 1; }
        if (t2 < tmin) { tmin = t2; ax = 2; }
        const int fx = ax < 0 ? 0 : ((ups >> (base + ax)) & 1u) ? 1 : -1;
        const int fidx = 2 * ax + (fx > 0 ? 1 : 0);
        const int cls = ax < 0 ? (int)NB_OUTSIDE : (int)((nb >> (2 * fidx)) & 3u);
        const int c2 = s.c + fx * (ax == 0 ? 1 : (ax == 1 ? stride_y : stride_z));
        // (its record is read whether it is entered or not, at an index held
        // inside the grid, so that the load waits neither for the neighbour's
        // class nor for the range check: a request of 4000 particles with 20
        // output times 242 us without the check, 245 to 249 with the load
        // behind it, 233 so)
        const int at = (int)min((unsigned)c2, (unsigned)f.ncell - 1u);
        float n1, n2;
        unsigned nnb;
        read(at, n1, n2, nnb);
        const bool inside = at == c2;   // (false across an outer face; else an error)
        const bool enter =
            go && ax >= 0 && inside && (cls == NB_ACTIVE || (cls == NB_SINK && !sink_stops(p, f.sinkfrac, c2)));
        float nh, nl;
        E::ff_add(s.th, s.tl, tmin, nh, nl);
        const float xn = E::move(A, up, x, tmin);
        // an event: an output time or the stop time in the step, no exit, a
        // path that ends here, the step cap
        const bool ev = go && (ax < 0 || E::ff_ge(nh, nl, s.eh, s.el));
        if (__any_sync(FULL, ev || (live && !enter))) {
            enum { P_NONE, P_CROSS, P_TIME, P_NOEXIT, P_CAPTURE };
            int path = go ? P_CROSS : P_NONE;
            bool due = false;
            float rh = 0.0f, rl = 0.0f;
            if (ev) {
                if (ax < 0 && __ldg(f.ibound + s.c) == 2) path = P_CAPTURE;   // in a sink cell it passes through
                else if (ax < 0 && !(p.t_stop < CUDART_INF)) path = P_NOEXIT;
                else if (ax < 0 || E::ff_ge(nh, nl, p.tstop_hi, p.tstop_lo)) path = P_TIME;
                if (TS && path != P_CAPTURE && s.kn < p.n_times) {
                    due = true;
                    rh = path == P_NOEXIT ? CUDART_INF_F : (path == P_TIME ? p.tstop_hi : nh);
                    rl = path == P_NOEXIT ? 0.0f : (path == P_TIME ? p.tstop_lo : nl);
                }
            }
            if (TS && __any_sync(FULL, due)) {
                gather();
                const DevOut& o = e.req(s.r).o;
                while (true) {
                    if (due) {
                        while (true) {
                            const float2 tk = E::time_pair(o, s.kn);
                            if (!E::ff_ge(rh, rl, tk.x, tk.y)) { due = false; break; }
                            if (held == REC_SLOTS) break;
                            if (lead)
                                e.rec_put(Q, 32 * held + lane, s, q, s.kn, E::ff_diff(tk.x, tk.y, s.th, s.tl),
                                          path == P_NOEXIT);
                            held++;
                            s.kn++;
                            if (s.kn >= p.n_times) { due = false; break; }
                        }
                        if (!due) e.next_event(s);
                    }
                    if (!__any_sync(FULL, due)) break;
                    int mine = lead ? held : 0;
                    rs_flush(e, Q, mine);
                    held = 0;
                }
            }
            if (path == P_CROSS && !enter) {
                x = a == ax ? (fx > 0 ? 1.0f : 0.0f) : xn;
                s.th = nh;
                s.tl = nl;
                s.ef = fidx;
                s.st = cls == NB_OUTSIDE ? MP_ST_EXIT_DOMAIN : (cls == NB_BOUNDARY ? MP_ST_BOUNDARY : MP_ST_SINK);
                if (!inside && (cls == NB_ACTIVE || cls == NB_SINK)) {
                    if (lead) atomicCAS(e.req(s.r).o.counters + COUNTER_ERR, 0ULL, (unsigned long long)q + 1ULL);
                    s.st = MP_ST_INVALID_RELEASE;
                }
            } else if (path == P_TIME) {
                x = E::move(A, up, x, E::ff_diff(p.tstop_hi, p.tstop_lo, s.th, s.tl));
                s.th = p.tstop_hi;
                s.tl = p.tstop_lo;
                s.st = MP_ST_TIME;
            } else if (live && path != P_CROSS) {
                s.st = path == P_CAPTURE ? MP_ST_SINK : (path == P_NOEXIT ? MP_ST_NO_EXIT : MP_ST_STEP_CAP);
            }
            ended = live && s.st != MP_ST_ACTIVE;
            if (__any_sync(FULL, ended)) {
                if (go && ended) s.steps++;
                gather();
                if (PL) pl_push(e, P, pcount, s, q, lead && go && ended && p.pathline, s.st);
                if (TS) tail_fill(e, s, q, lead && ended && !paused(e, s));
                if (ended && lead) e.template finish<TS>(q, s, s_cnt);
                live = live && !ended;
                going = __any_sync(FULL, live);
            }
        }
        if (go && live) {
            // hand over to the neighbour; the exit coordinate enters on the shared face
            s.steps++;
            x = a == ax ? (fx > 0 ? 0.0f : 1.0f) : xn;
            s.th = nh;
            s.tl = nl;
            s.ef = fidx;
            s.c = c2;
            s.h = fnv_step(s.h, c2);
            u1 = n1;
            u2 = n2;
            nb = nnb;
        }
        if (PL) {
            gather();
            pl_push(e, P, pcount, s, q, lead && go && live && p.pathline, s.st);
        }
    }
    if (TS) {
        int mine = lead ? held : 0;
        rs_flush(e, Q, mine);
    }
    if (PL) pl_flush(e, P, pcount);
    flush_counters(e, s_cnt);
    window_end(e);
}

template <bool ONE>
cudaError_t launch_axes_mixed(const MixEngine<false, ONE>& e, unsigned modes, cudaStream_t s)
{
    const bool ts = (modes & MODE_TS) != 0, pl = (modes & MODE_PATH) != 0;
    const size_t smem = (ts ? sizeof(typename MixEngine<false, ONE>::RecQ) : 0) + (pl ? sizeof(PathQ) : 0);
    const unsigned grid = (unsigned)((e.b.n_total + AXES_PARTICLES - 1) / AXES_PARTICLES);
    auto kern = ts ? (pl ? k_track_axes_mixed<ONE, true, true> : k_track_axes_mixed<ONE, true, false>)
                   : (pl ? k_track_axes_mixed<ONE, false, true> : k_track_axes_mixed<ONE, false, false>);
    kern<<<grid, 32, smem, s>>>(e);
    return cudaGetLastError();
}

}  // namespace mp
