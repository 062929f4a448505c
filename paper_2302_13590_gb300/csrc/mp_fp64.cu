// mp_fp64.cu - field records, particle release and FP64 tracking kernels.
//
// Compiled with -fmad=false: every multiply and add below rounds on its own,
// in the order written, so that the FP64 path evaluates the same IEEE
// operations as a plain double-precision statement of the method.
//
// Method (Pollock 1988, the displacement scheme the paper keeps unchanged;
// Methods, "MODPATH"): inside a cell each velocity component varies linearly
// between its two faces, v(p) = v1 + A p with A = (v2 - v1) / D, so the
// motion along each axis is p(t) = p + v_p (e^{A t} - 1) / A (p + v_p t when
// A t == 0) and the time to reach the exit face is t_a = ln(1 + z) / A with
// z = A (d / v_p) (t_a = d / v_p when z == 0); 1 / A comes with the cell.  The particle leaves through the
// face with the smallest t_a (lowest axis on ties) and is handed to the
// neighbour across it, until a stopping condition holds (Methods, "MODPATH").
#include <cfloat>
#include <cmath>
#include <type_traits>

#include "mp_internal.h"
#include "mp_sched.cuh"
#include "mp_f64math.cuh"

namespace mp {

// ---------------------------------------------------------------------------
// field records
// ---------------------------------------------------------------------------

__device__ __forceinline__ int nb_class(const DevField& f, int k, int i, int j)
{
    if (k < 0 || k >= f.nlay || i < 0 || i >= f.nrow || j < 0 || j >= f.ncol) return NB_OUTSIDE;
    const int8_t ib = f.ibound[((long long)k * f.nrow + i) * f.ncol + j];
    if (ib == 1) return NB_ACTIVE;
    if (ib == 2) return NB_SINK;
    return NB_BOUNDARY;
}

// a cell's inflow and outflow from its six face flows (+axis direction),
// face by face in the order x-, x+, y-, y+, z-, z+
__device__ double2 face_inout(const double q[6])
{
    double in = 0.0, out = 0.0;
    for (int a = 0; a < 3; ++a) {
        const double q1 = q[2 * a], q2 = q[2 * a + 1];
        if (q1 > 0.0) in += q1; else out += -q1;
        if (q2 < 0.0) in += -q2; else out += q2;
    }
    return make_double2(in, out);
}

// fraction of a cell's inflow its sink extracts; no inflow: 1
__device__ double sink_fraction(double2 io)
{
    return io.x > 0.0 ? (io.x - io.y) / io.x : 1.0;
}

// One cell a thread.  Bound by the FP64 pipe (18 divisions and 15
// conversions a cell in the plain form, about 185 instructions), not by the
// 200 bytes it moves; the divisions by a cell size share its reciprocal and
// the conversions run on the ALU: loading a 200x200x20 field from device
// arrays 436 -> 352 us.
__global__ void k_build_records(DevField f, CellF64* r64, CellF32* r32, double* sinkfrac, double2* inout,
                                const double* qx, const double* qy, const double* qz, const double* por)
{
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= f.ncell) return;
    const int ncol = f.ncol, nrow = f.nrow;
    const int j = (int)(c % ncol), i = (int)((c / ncol) % nrow), k = (int)(c / ((long long)ncol * nrow));
    unsigned long long nb = 0;
    nb |= (unsigned long long)nb_class(f, k, i, j - 1) << 0;
    nb |= (unsigned long long)nb_class(f, k, i, j + 1) << 2;
    nb |= (unsigned long long)nb_class(f, k, i - 1, j) << 4;
    nb |= (unsigned long long)nb_class(f, k, i + 1, j) << 6;
    nb |= (unsigned long long)nb_class(f, k - 1, i, j) << 8;
    nb |= (unsigned long long)nb_class(f, k + 1, i, j) << 10;
    CellF64 r{};
    CellF32 s{};
    double v2x = 0.0, v2y = 0.0, v2z = 0.0;
    const int8_t ib = f.ibound[c];
    if (ib == 1 || ib == 2) {
        const double n = por[c];
        const double dx = f.delr[j], dy = f.delc[i], dzz = f.dz[k];
        const double ax = dy * dzz, ay = dx * dzz, az = dx * dy;
        const double qx1 = qx[((long long)k * nrow + i) * (ncol + 1) + j];
        const double qx2 = qx[((long long)k * nrow + i) * (ncol + 1) + j + 1];
        const double qy1 = qy[((long long)k * (nrow + 1) + i) * ncol + j];
        const double qy2 = qy[((long long)k * (nrow + 1) + i + 1) * ncol + j];
        const double qz1 = qz[((long long)k * nrow + i) * ncol + j];
        const double qz2 = qz[((long long)(k + 1) * nrow + i) * ncol + j];
        r.v1x = qx1 / (n * ax); v2x = qx2 / (n * ax);
        r.v1y = qy1 / (n * ay); v2y = qy2 / (n * ay);
        r.v1z = qz1 / (n * az); v2z = qz2 / (n * az);
        const double yx = f.inv[j], yy = f.inv[ncol + i], yz = f.inv[ncol + nrow + k];
        const bool px = plain_divisor(dx), py = plain_divisor(dy), pz = plain_divisor(dzz);
        r.Ax = px ? div_by(v2x - r.v1x, dx, yx) : (v2x - r.v1x) / dx;
        r.Ay = py ? div_by(v2y - r.v1y, dy, yy) : (v2y - r.v1y) / dy;
        r.Az = pz ? div_by(v2z - r.v1z, dzz, yz) : (v2z - r.v1z) / dzz;
        r.iAx = r.Ax != 0.0 ? 1.0 / r.Ax : 0.0;
        r.iAy = r.Ay != 0.0 ? 1.0 / r.Ay : 0.0;
        r.iAz = r.Az != 0.0 ? 1.0 / r.Az : 0.0;
        s.u1x = px ? quot_f32(r.v1x, dx, yx) : (float)(r.v1x / dx);
        s.u2x = px ? quot_f32(v2x, dx, yx) : (float)(v2x / dx);
        s.u1y = py ? quot_f32(r.v1y, dy, yy) : (float)(r.v1y / dy);
        s.u2y = py ? quot_f32(v2y, dy, yy) : (float)(v2y / dy);
        s.u1z = pz ? quot_f32(r.v1z, dzz, yz) : (float)(r.v1z / dzz);
        s.u2z = pz ? quot_f32(v2z, dzz, yz) : (float)(v2z / dzz);
        const double q6[6] = {qx1, qx2, qy1, qy2, qz1, qz2};
        const double2 io = face_inout(q6);
        inout[c] = io;
        if (ib == 2) sinkfrac[c] = sink_fraction(io);
    } else {
        inout[c] = make_double2(0.0, 0.0);
    }
    if (ib != 2) sinkfrac[c] = 0.0;
    const double v1a[3] = {r.v1x, r.v1y, r.v1z}, v2a[3] = {v2x, v2y, v2z};
    for (int a = 0; a < 3; ++a) {
        const unsigned long long sg = (v1a[a] > 0.0 ? 1ULL : 0ULL) | (v1a[a] < 0.0 ? 2ULL : 0ULL) |
                                      (v2a[a] > 0.0 ? 4ULL : 0ULL) | (v2a[a] < 0.0 ? 8ULL : 0ULL);
        nb |= sg << (NB_SIGN + 4 * a);
    }
    r.nb = nb;
    r.fv1x = f32_rn(r.v1x); r.fv2x = f32_rn(v2x); r.fAx = f32_rn(r.Ax);
    r.fv1y = f32_rn(r.v1y); r.fv2y = f32_rn(v2y); r.fAy = f32_rn(r.Ay);
    r.fv1z = f32_rn(r.v1z); r.fv2z = f32_rn(v2z); r.fAz = f32_rn(r.Az);
    s.nb = (uint32_t)nb;
    r64[c] = r;
    r32[c] = s;
}

cudaError_t launch_build_records(const DevField& f, CellF64* rec64, CellF32* rec32, double* sinkfrac,
                                 double2* inout, const double* qx, const double* qy, const double* qz,
                                 const double* por, cudaStream_t s)
{
    if (f.ncell <= 0) return cudaSuccess;
    const int b = 256;
    const long long g = (f.ncell + b - 1) / b;
    k_build_records<<<(unsigned)g, b, 0, s>>>(f, rec64, rec32, sinkfrac, inout, qx, qy, qz, por);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// volume balance
// ---------------------------------------------------------------------------

// Maxima, counts and the sink cells' extractions of a run of cells per block;
// k_balance_total joins the runs.  Maxima and counts do not depend on the
// order; the extractions are kept in cell order (ballot and prefix counts),
// so that the host sums the few there are as a loop over the cells would.  The pass reads
// 17 B a cell; copying them to the host for such a loop took 1.6 of the 2.3 ms
// of loading a 200x200x20 field.
__device__ __forceinline__ void balance_join(BalancePart& a, const BalancePart& b)
{
    if (b.cell >= 0 && (a.cell < 0 || b.max_abs > a.max_abs || (b.max_abs == a.max_abs && b.cell < a.cell))) {
        a.max_abs = b.max_abs;
        a.cell = b.cell;
    }
    a.max_rel = fmax(a.max_rel, b.max_rel);
    if (b.first >= 0 && (a.first < 0 || b.first < a.first)) {
        a.first = b.first;
        a.r_first = b.r_first;
    }
    a.active += b.active;
    a.sinks += b.sinks;
}

__device__ __forceinline__ BalancePart balance_shfl(const BalancePart& p, int off)
{
    BalancePart q;
    q.max_abs = __shfl_down_sync(0xffffffffu, p.max_abs, off);
    q.max_rel = __shfl_down_sync(0xffffffffu, p.max_rel, off);
    q.r_first = __shfl_down_sync(0xffffffffu, p.r_first, off);
    q.cell = __shfl_down_sync(0xffffffffu, p.cell, off);
    q.first = __shfl_down_sync(0xffffffffu, p.first, off);
    q.active = __shfl_down_sync(0xffffffffu, p.active, off);
    q.sinks = __shfl_down_sync(0xffffffffu, p.sinks, off);
    return q;
}

// joins the block's parts; the result is valid in thread 0
__device__ __forceinline__ BalancePart balance_block(BalancePart p)
{
    __shared__ BalancePart s_part[32];
    for (int off = 16; off > 0; off >>= 1) {
        const BalancePart q = balance_shfl(p, off);
        if ((threadIdx.x & 31) + off < 32) balance_join(p, q);
    }
    if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = p;
    __syncthreads();
    if (threadIdx.x == 0)
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) balance_join(p, s_part[w]);
    return p;
}

__global__ void __launch_bounds__(256) k_balance(double2* inout, const int8_t* ibound, long long ncell, long long run,
                                                 BalancePart* parts)
{
    __shared__ int s_cnt[8];
    BalancePart p{0.0, 0.0, 0.0, -1, -1, 0, 0};
    const long long c0 = (long long)blockIdx.x * run, c1 = c0 + run < ncell ? c0 + run : ncell;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // the run's extractions so far, kept at the front of its part of inout:
    // 8 bytes for at most every cell that has been read, so never past it
    double* extract = reinterpret_cast<double*>(inout + c0);
    long long put = 0;
    for (long long t = c0; t < c1; t += 256) {
        const long long c = t + threadIdx.x;
        const int ib = c < c1 ? ibound[c] : 0;
        double2 io = make_double2(0.0, 0.0);
        if (ib == 1 || ib == 2) io = inout[c];
        if (ib == 1) {
            const double r = fabs(io.x - io.y);
            BalancePart q{r, 0.0, r, r == r ? c : -1, c, 1, 0};
            if (io.x > 0.0) q.max_rel = r / io.x;
            balance_join(p, q);
        }
        const unsigned m = __ballot_sync(0xffffffffu, ib == 2);
        if (lane == 0) s_cnt[warp] = __popc(m);
        __syncthreads();
        int before = 0, all = 0;
        for (int k = 0; k < 8; ++k) {
            before += k < warp ? s_cnt[k] : 0;
            all += s_cnt[k];
        }
        if (ib == 2) extract[put + before + __popc(m & ((1u << lane) - 1u))] = io.x - io.y;
        put += all;
        __syncthreads();
    }
    if (threadIdx.x == 0) p.sinks = put;
    p = balance_block(p);
    if (threadIdx.x == 0) parts[blockIdx.x] = p;
}

// joins the runs' parts (one block of BALANCE_BLOCKS threads) and leaves in
// parts[b].active how many extractions come before run b's
__global__ void __launch_bounds__(BALANCE_BLOCKS) k_balance_total(int runs, BalancePart* parts, BalancePart* total)
{
    __shared__ long long s_at[BALANCE_BLOCKS];
    const int b = threadIdx.x;
    BalancePart p{0.0, 0.0, 0.0, -1, -1, 0, 0};
    if (b < runs) p = parts[b];
    const long long mine = p.sinks;
    s_at[b] = mine;
    __syncthreads();
    for (int off = 1; off < BALANCE_BLOCKS; off <<= 1) {
        const long long v = b >= off ? s_at[b - off] : 0;
        __syncthreads();
        s_at[b] += v;
        __syncthreads();
    }
    if (b < runs) parts[b].active = s_at[b] - mine;
    p = balance_block(p);
    if (b == 0) *total = p;
}

__global__ void k_balance_sinks(const double2* inout, long long run, const BalancePart* parts, double* sinks)
{
    const double* extract = reinterpret_cast<const double*>(inout + (long long)blockIdx.x * run);
    const long long n = parts[blockIdx.x].sinks, at = parts[blockIdx.x].active;
    for (long long k = threadIdx.x; k < n; k += blockDim.x) sinks[at + k] = extract[k];
}

// runs of whole 256-cell tiles, at most BALANCE_BLOCKS of them
static long long balance_run(long long ncell)
{
    return ((ncell + 255) / 256 + BALANCE_BLOCKS - 1) / BALANCE_BLOCKS * 256;
}

cudaError_t launch_balance(double2* inout, const int8_t* ibound, long long ncell, BalancePart* parts,
                           BalancePart* total, cudaStream_t s)
{
    const long long run = balance_run(ncell);
    const int runs = (int)((ncell + run - 1) / run);
    k_balance<<<runs, 256, 0, s>>>(inout, ibound, ncell, run, parts);
    k_balance_total<<<1, BALANCE_BLOCKS, 0, s>>>(runs, parts, total);
    return cudaGetLastError();
}

cudaError_t launch_balance_sinks(const double2* inout, long long ncell, const BalancePart* parts, double* sinks,
                                 cudaStream_t s)
{
    const long long run = balance_run(ncell);
    k_balance_sinks<<<(unsigned)((ncell + run - 1) / run), 128, 0, s>>>(inout, run, parts, sinks);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// release: Philox4x32-10 (Salmon, Moraes, Dror and Shaw, SC'11)
// ---------------------------------------------------------------------------

__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k)
{
    #pragma unroll
    for (int r = 0; r < 10; ++r) {
        const unsigned hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
        const unsigned hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
        c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
        k.x += 0x9E3779B9u;
        k.y += 0xBB67AE85u;
    }
    return c;
}

__device__ __forceinline__ double unit53(unsigned a, unsigned b)
{
    const unsigned long long v = ((((unsigned long long)a) << 32) | (unsigned long long)b) >> 11;
    return (double)v * (1.0 / 9007199254740992.0);
}

// largest a in [0, n-1] with f[a] <= x; -1 if x is outside [f[0], f[n]]
__device__ __forceinline__ int locate(const double* fc, int n, double x)
{
    if (!(x >= fc[0]) || !(x <= fc[n])) return -1;
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (fc[mid] <= x) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

__device__ __forceinline__ uint8_t release_status(const DevField& f, long long c)
{
    const int8_t ib = f.ibound[c];
    return ib == 1 ? MP_ST_ACTIVE : (ib == 2 ? MP_ST_SINK : MP_ST_INVALID_RELEASE);
}

struct Box { double lo[3], hi[3]; };

// one particle of a box release: Philox counters (id, 0) and (id, 1) under
// the key `seed`, three 53-bit uniforms, the cell holding the point
__device__ __forceinline__ void release_one(const DevField& f, const DevState& st, long long q, const Box& b,
                                            unsigned long long seed, unsigned long long off)
{
    const unsigned long long id = (unsigned long long)q + off;
    const uint2 key = make_uint2((unsigned)seed, (unsigned)(seed >> 32));
    const uint4 r = philox4x32_10(make_uint4((unsigned)id, (unsigned)(id >> 32), 0u, 0u), key);
    const uint4 s = philox4x32_10(make_uint4((unsigned)id, (unsigned)(id >> 32), 1u, 0u), key);
    const double ux = unit53(r.x, r.y), uy = unit53(r.z, r.w), uz = unit53(s.x, s.y);
    const double gx = b.lo[0] + ux * (b.hi[0] - b.lo[0]);
    const double gy = b.lo[1] + uy * (b.hi[1] - b.lo[1]);
    const double gz = b.lo[2] + uz * (b.hi[2] - b.lo[2]);
    const int j = locate(f.xf, f.ncol, gx), i = locate(f.yf, f.nrow, gy), k = locate(f.zf, f.nlay, gz);
    st.t[q] = 0.0;
    if (st.steps) st.steps[q] = 0u;
    if (j < 0 || i < 0 || k < 0) {
        st.cell[q] = -1; st.px[q] = 0.0; st.py[q] = 0.0; st.pz[q] = 0.0;
        st.status[q] = MP_ST_INVALID_RELEASE;
        return;
    }
    double ox = gx - f.xf[j], oy = gy - f.yf[i], oz = gz - f.zf[k];
    ox = fmin(fmax(ox, 0.0), f.delr[j]);
    oy = fmin(fmax(oy, 0.0), f.delc[i]);
    oz = fmin(fmax(oz, 0.0), f.dz[k]);
    const long long c = ((long long)k * f.nrow + i) * f.ncol + j;
    st.cell[q] = (int32_t)c;
    st.px[q] = ox; st.py[q] = oy; st.pz[q] = oz;
    st.status[q] = release_status(f, c);
}

__global__ void k_release_box(DevField f, DevState st, long long n, Box b, unsigned long long seed,
                              unsigned long long off)
{
    const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    release_one(f, st, q, b, seed, off);
}

// Box releases of several groups in one launch: one index space over all
// of them (starts = prefix sums of the group sizes), the descriptors read
// from device memory, so a captured graph releases whatever they hold.
__global__ void k_release_boxes(DevField f, const BoxRelease* d, const long long* starts, int n_reqs,
                                long long n_total)
{
    const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= n_total) return;
    int lo = 0, hi = n_reqs - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (starts[mid] <= g) lo = mid;
        else hi = mid - 1;
    }
    const BoxRelease& r = d[lo];
    Box b;
    for (int a = 0; a < 3; ++a) { b.lo[a] = r.lo[a]; b.hi[a] = r.hi[a]; }
    release_one(f, r.st, g - starts[lo], b, r.seed, r.id_offset);
}

cudaError_t launch_release_boxes(const DevField& f, const BoxRelease* d, const long long* starts, int n_reqs,
                                 long long n_total, cudaStream_t s)
{
    if (n_total <= 0) return cudaSuccess;
    k_release_boxes<<<(unsigned)((n_total + 255) / 256), 256, 0, s>>>(f, d, starts, n_reqs, n_total);
    return cudaGetLastError();
}

__global__ void k_release_explicit(DevField f, DevState st, long long n, const int32_t* cell,
                                   const double* local, const double* t0)
{
    const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    const long long c = cell[q];
    st.t[q] = t0 ? t0[q] : 0.0;
    if (st.steps) st.steps[q] = 0u;
    if (c < 0 || c >= f.ncell) {
        st.cell[q] = -1; st.px[q] = 0.0; st.py[q] = 0.0; st.pz[q] = 0.0;
        st.status[q] = MP_ST_INVALID_RELEASE;
        return;
    }
    const int j = (int)(c % f.ncol), i = (int)((c / f.ncol) % f.nrow), k = (int)(c / ((long long)f.ncol * f.nrow));
    const double fx = fmin(fmax(local[3 * q], 0.0), 1.0);
    const double fy = fmin(fmax(local[3 * q + 1], 0.0), 1.0);
    const double fz = fmin(fmax(local[3 * q + 2], 0.0), 1.0);
    st.cell[q] = (int32_t)c;
    st.px[q] = fx * f.delr[j]; st.py[q] = fy * f.delc[i]; st.pz[q] = fz * f.dz[k];
    st.status[q] = release_status(f, c);
}

cudaError_t launch_release_box(const DevField& f, const DevState& st, long long n, const double lo[3],
                               const double hi[3], unsigned long long seed, unsigned long long id_offset,
                               cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    Box b;
    for (int a = 0; a < 3; ++a) { b.lo[a] = lo[a]; b.hi[a] = hi[a]; }
    k_release_box<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(f, st, n, b, seed, id_offset);
    return cudaGetLastError();
}

cudaError_t launch_release_explicit(const DevField& f, const DevState& st, long long n, const int32_t* cell,
                                    const double* local, const double* t0, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    k_release_explicit<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(f, st, n, cell, local, t0);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// FP64 tracking engine
// ---------------------------------------------------------------------------

// What bounds it: the FP64 pipe, 16 cycles a warp instruction for the whole
// SM (2 lanes a clock), once 16 warps are resident; with few particles the
// length of one step (one warp alone: about 1,100 issued instructions, most
// of them integer, in a chain of 25 dependent FP64 operations).  Both ask for
// the same: no FP64 operation that can be decided elsewhere, and short
// integer code around the rest.  So sign, zero and range tests take the high
// word, the FP32 truncations one funnel shift and one addition, log1p takes
// its table row from FP32, and the two motions run without branches (a rare
// flag sends a lane to the general form).  Against 64-bit tests and
// conversions and a branch in every helper: 1e6 particles, 200x200x20 cells,
// 50 output times 27.2 -> 23.5 ms; 3e4 particles, endpoints 1.19 -> 1.05 ms;
// 1000 particles, 50x50 cells 154 -> 135 us; the same bits.  (With the rounds
// and the fetch of mp_sched.cuh these now take 22.96 and 0.995 ms, and 1000
// particles go three lanes each.)
template <bool ONE_REQ>
struct F64Engine {
    static constexpr bool ONE = ONE_REQ;
    static constexpr bool OWN_SLOTS = false;   // records go through the warp's queue
    static constexpr bool EVEN_ROUNDS = true;   // more particles than lanes: rounds of even size
    static constexpr int FETCH = 8;            // steps per fetch
    // blocks of 256 threads to keep resident per SM (0: no target; the
    // kernels are FP64-pipe bound)
    static constexpr int min_blocks(bool, bool, bool) { return 0; }
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
        int c, i, j, k;
        double x0, x1, x2;   // offsets (m) from the cell's low faces
        double t;
        unsigned steps;
        unsigned cap;     // the request's step cap (its low 32 bits' range; the full one decides); 0: an
                          // offset was handed in outside its cell, and every axis is evaluated exactly
        unsigned long long h;
        int kn;
        int st;
        int ef;
        int in_sink;      // the current cell is a sink entered with pass-through
        long long tev;    // next output time or the stop time, whichever is first, as its bound_key
    };

    template <class T>
    __device__ __forceinline__ static T sel3(int a, T x, T y, T z)
    {
        return a == 0 ? x : (a == 1 ? y : z);
    }

    // size of column, row or layer a (index in f.ax) and its FP32 truncation
    __device__ __forceinline__ void axis_cell(int a, double& D, float& F) const
    {
        const double2 v = __ldg(reinterpret_cast<const double2*>(f.ax + a));
        D = v.x;
        F = __uint_as_float((unsigned)__double_as_longlong(v.y));
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

    __device__ __forceinline__ double gx(const State& s) const { return __ldg(f.xf + s.j) + s.x0; }
    __device__ __forceinline__ double gy(const State& s) const { return __ldg(f.yf + s.i) + s.x1; }
    __device__ __forceinline__ double gz(const State& s) const { return __ldg(f.zf + s.k) + s.x2; }

    __device__ __forceinline__ void final_pos(const State& s, double& x, double& y, double& z) const
    {
        const bool ok = s.c >= 0;
        x = ok ? gx(s) : CUDART_NAN;
        y = ok ? gy(s) : CUDART_NAN;
        z = ok ? gz(s) : CUDART_NAN;
    }

    // next time at which the step loop must leave its fast path
    __device__ __forceinline__ long long next_event(const State& s) const
    {
        const Req& R = req(s.r);
        const DevState& in = R.in;
        const DevOut& o = R.o;
        const TrackParams& p = R.p;
        (void)in; (void)o; (void)p;
        const double tk = s.kn < p.n_times ? __ldg(o.times + s.kn) : CUDART_INF;
        // fmin on the integer side: only the lanes with output times in the
        // step take this, and an FP64 compare would hold the whole warp's
        // FP64 pipe slot for them
        return bound_key(ge_d(tk, p.t_stop) ? p.t_stop : tk);
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
        s.x0 = in.px[q]; s.x1 = in.py[q]; s.x2 = in.pz[q];
        s.t = in.t[q];
        // cell-steps, hash and last face carried by a resumed particle
        s.steps = in.steps ? in.steps[q] : 0u;
        s.cap = p.max_steps > 0xffffffffLL ? 0xffffffffu : (unsigned)p.max_steps;
        s.h = FNV_INIT;
        s.kn = 0;
        s.ef = (s.steps && in.exit_face) ? (int)in.exit_face[q] : MP_FACE_NONE;
        s.in_sink = 0;
        if (s.c >= 0 && (long long)s.c < f.ncell) {
            split_cell(f, s.c, s.k, s.i, s.j);
            // a caller's own arrays (they come without step counts) may hold
            // offsets outside the cell, rounded ones for instance
            if (!in.steps && !(f64_inside(s.x0, __ldg(f.delr + s.j)) && f64_inside(s.x1, __ldg(f.delc + s.i)) &&
                               f64_inside(s.x2, __ldg(f.dz + s.k))))
                s.cap = 0u;
            s.h = (s.steps && in.hash) ? in.hash[q] : fnv_step(s.h, s.c);
            // a resumed particle may sit inside a sink cell it entered with
            // pass-through; a moving particle whose cell is not active under
            // this field (another flow period) stops there
            const int ib = __ldg(f.ibound + s.c);
            s.in_sink = ib == 2;
            if (s.st == MP_ST_ACTIVE) {
                if (ib == 0 || ib == -1) s.st = MP_ST_BOUNDARY;
                else if (ib == 2 && sink_stops(p, f.sinkfrac, s.c)) s.st = MP_ST_SINK;
            }
        } else {
            s.c = -1; s.i = s.j = s.k = 0;
            s.st = MP_ST_INVALID_RELEASE;
        }
        if (TS) {
            if (p.cont) {
                // output times up to the period start were written by the previous period
                while (s.kn < p.n_times && __ldg(o.times + s.kn) <= s.t) s.kn++;
            } else {
                while (s.kn < p.n_times && __ldg(o.times + s.kn) <= s.t) {
                    if (s.c >= 0) record(q, s.kn, s, gx(s), gy(s), gz(s), s.st);
                    else record(q, s.kn, s, CUDART_NAN, CUDART_NAN, CUDART_NAN, s.st);
                    s.kn++;
                }
            }
        }
        // a particle that starts at or after the stop time takes no step
        if (s.st == MP_ST_ACTIVE && s.t >= p.t_stop) s.st = MP_ST_TIME;
        s.tev = TS ? next_event(s) : bound_key(p.t_stop);
    }

    // per-warp queue of deferred timeseries records (structure of arrays)
    struct alignas(16) RecQ {
        double p0[RQ_CAP], p1[RQ_CAP], p2[RQ_CAP], t[RQ_CAP];
        long long q[RQ_CAP];
        int c[RQ_CAP], i[RQ_CAP], j[RQ_CAP], k[RQ_CAP], kk[RQ_CAP], st[RQ_CAP], r[RQ_CAP];
    };

    __device__ __forceinline__ void rec_put(RecQ& Q, int slot, const State& s, long long q, int kk, int st) const
    {
        const Req& R = req(s.r);
        const DevState& in = R.in;
        const DevOut& o = R.o;
        const TrackParams& p = R.p;
        (void)in; (void)o; (void)p;
        if (!ONE) Q.r[slot] = s.r;
        Q.p0[slot] = s.x0; Q.p1[slot] = s.x1; Q.p2[slot] = s.x2;
        Q.t[slot] = s.t;   // tau = times[kk] - t is formed in rec_eval, where all 32 lanes take it
        Q.q[slot] = q;
        Q.c[slot] = s.c; Q.i[slot] = s.i; Q.j[slot] = s.j; Q.k[slot] = s.k;
        Q.kk[slot] = kk; Q.st[slot] = st;
    }

    // the position at tau after the step's start, by the motion formula on
    // every axis (the same operations as an endpoint stop at that time)
    __device__ __forceinline__ void rec_eval(const RecQ& Q, int slot) const
    {
        const Req& R = req(ONE ? 0 : Q.r[slot]);
        const DevOut& o = R.o;
        const TrackParams& p = R.p;
        const int c = Q.c[slot], i = Q.i[slot], j = Q.j[slot], k = Q.k[slot];
        const double p0 = Q.p0[slot], p1 = Q.p1[slot], p2 = Q.p2[slot];
        const double tau = __ldg(o.times + Q.kk[slot]) - Q.t[slot];
        const double2* rp = reinterpret_cast<const double2*>(f.rec64 + c);
        const double2 r0 = __ldg(rp + 0), r1 = __ldg(rp + 1), r2 = __ldg(rp + 2), r3 = __ldg(rp + 3),
                      r4 = __ldg(rp + 4);
        const double v1x = r0.x, Ax = r0.y, iAx = r1.x, v1y = r1.y, Ay = r2.x, iAy = r2.y;
        const double v1z = r3.x, Az = r3.y, iAz = r4.x;
        const double D0 = __ldg(f.delr + j), D1 = __ldg(f.delc + i), D2 = __ldg(f.dz + k);
        const double vx = f64_vel(v1x, Ax, p0), vy = f64_vel(v1y, Ay, p1), vz = f64_vel(v1z, Az, p2);
        bool again;
        double nx = f64_move_fast(Ax, iAx, D0, vx, p0, tau, again);
        if (again) nx = f64_move(Ax, iAx, D0, vx, p0, tau);
        double ny = f64_move_fast(Ay, iAy, D1, vy, p1, tau, again);
        if (again) ny = f64_move(Ay, iAy, D1, vy, p1, tau);
        double nz = f64_move_fast(Az, iAz, D2, vz, p2, tau, again);
        if (again) nz = f64_move(Az, iAz, D2, vz, p2, tau);
        const double x = __ldg(f.xf + j) + nx, y = __ldg(f.yf + i) + ny, z = __ldg(f.zf + k) + nz;
        store_record(o.ts + (long long)Q.kk[slot] * p.n + Q.q[slot], x, y, z, c, Q.st[slot]);
    }

    // One cell-step for every lane of the warp (warp-uniform call; lanes with
    // live == false only take part in the record queue).
    template <bool TS>
    __device__ __forceinline__ void step(long long q, State& s, bool live, RecQ& Q, int& qcount) const
    {
        const Req& R = req(s.r);
        const DevState& in = R.in;
        const DevOut& o = R.o;
        const TrackParams& p = R.p;
        (void)in; (void)o; (void)p;
        enum { P_NONE, P_CROSS, P_TIME, P_NOEXIT, P_CAPTURE };
        int path = P_NONE;
        int m = 0;
        double v1x = 0, Ax = 0, v1y = 0, Ay = 0, v1z = 0, Az = 0, D0 = 1, D1 = 1, D2 = 1;
        double iAx = 0, iAy = 0, iAz = 0;
        double vp0 = 0, vp1 = 0, vp2 = 0, tmin = 0, t_end = 0;
        int f0 = 0, f1 = 0, f2 = 0, ax = -1;
        unsigned nb = 0;
        if (live) {
            const bool odd = s.steps >= s.cap;   // (off the fast path: at the cap, or its 0)
            if (odd && (long long)s.steps >= p.max_steps) {
                s.st = MP_ST_STEP_CAP;
            } else if ((unsigned)s.c >= (unsigned)f.ncell) {
                atomicCAS(o.counters + COUNTER_ERR, 0ULL, (unsigned long long)q + 1ULL);
                s.st = MP_ST_INVALID_RELEASE;
            } else {
                const double2* rp = reinterpret_cast<const double2*>(f.rec64 + s.c);
                const double2 r0 = __ldg(rp + 0), r1 = __ldg(rp + 1), r2 = __ldg(rp + 2), r3 = __ldg(rp + 3),
                              r4 = __ldg(rp + 4);
                const float4* rf = reinterpret_cast<const float4*>(rp + 5);
                const float4 g0 = __ldg(rf + 0), g1 = __ldg(rf + 1), g2 = __ldg(rf + 2);
                float F0, F1, F2;
                axis_cell(s.j, D0, F0);
                axis_cell(f.ncol + s.i, D1, F1);
                axis_cell(f.ncol + f.nrow + s.k, D2, F2);
                v1x = r0.x; Ax = r0.y; iAx = r1.x; v1y = r1.y; Ay = r2.x; iAy = r2.y;
                v1z = r3.x; Az = r3.y; iAz = r4.x;
                nb = (unsigned)__double_as_longlong(r4.y);   // (bits 0 .. 27 are in use)
                vp0 = f64_vel(v1x, Ax, s.x0);
                vp1 = f64_vel(v1y, Ay, s.x1);
                vp2 = f64_vel(v1z, Az, s.x2);
                // reachable faces, and FP32 estimates of the three exit
                // times from FP32 distances to them (the FP64 distance is
                // formed for the axes evaluated exactly)
                unsigned l0, h0, l1, h1, l2, h2;
                words(vp0, l0, h0);
                words(vp1, l1, h1);
                words(vp2, l2, h2);
                f0 = f64_face(l0, h0, nb >> NB_SIGN);
                f1 = f64_face(l1, h1, nb >> (NB_SIGN + 4));
                f2 = f64_face(l2, h2, nb >> (NB_SIGN + 8));
                bool c0, c1, c2;
                float d0 = f32_face_dist(f0, F0, s.x0, c0);
                float d1 = f32_face_dist(f1, F1, s.x1, c1);
                float d2 = f32_face_dist(f2, F2, s.x2, c2);
                if (c0 || c1 || c2) {
                    if (c0) d0 = f32_trunc(D0 - s.x0);
                    if (c1) d1 = f32_trunc(D1 - s.x1);
                    if (c2) d2 = f32_trunc(D2 - s.x2);
                }
                const float t0 = f32_estimate(d0, trunc_normal(l0, h0), g0.z, f0 > 0 ? g0.y : g0.x);
                const float t1 = f32_estimate(d1, trunc_normal(l1, h1), g1.y, f1 > 0 ? g1.x : g0.w);
                const float t2 = f32_estimate(d2, trunc_normal(l2, h2), g2.x, f2 > 0 ? g1.w : g1.z);
                const unsigned reach = (f0 ? 1u : 0u) | (f1 ? 2u : 0u) | (f2 ? 4u : 0u);
                const bool doubt = f.no_screen || odd || (f0 && !(vel_trusted(h0) && t0 < CUDART_INF_F)) ||
                                   (f1 && !(vel_trusted(h1) && t1 < CUDART_INF_F)) ||
                                   (f2 && !(vel_trusted(h2) && t2 < CUDART_INF_F));
                unsigned rest;
                const int a0 = screen(f0 ? t0 : CUDART_INF_F, f1 ? t1 : CUDART_INF_F, f2 ? t2 : CUDART_INF_F, reach,
                                      doubt, rest);
                tmin = CUDART_INF;
                if (a0 >= 0) {
                    // the exact FP64 exit time of the leading candidate (one
                    // evaluation per lane, uniform across the warp)
                    const double te = f64_exit_time_d(
                        sel3(a0, Ax, Ay, Az), sel3(a0, iAx, iAy, iAz),
                        f64_face_dist(sel3(a0, f0, f1, f2), sel3(a0, D0, D1, D2), sel3(a0, s.x0, s.x1, s.x2)),
                        sel3(a0, vp0, vp1, vp2));
                    // then the other candidates exactly (a close call; every
                    // reachable axis when the leading time is unusable): the
                    // smallest time wins, ties to the lower axis - the
                    // oracle's rule over all axes, since a non-candidate's
                    // exact time exceeds the leading one's
                    if (is_finite(te)) {
                        tmin = te;
                        ax = a0;
                    } else {
                        rest = reach & ~(1u << a0);
                    }
                    while (rest) {
                        const int a = __ffs(rest) - 1;
                        rest &= rest - 1;
                        const double t = f64_exit_time_d(
                            sel3(a, Ax, Ay, Az), sel3(a, iAx, iAy, iAz),
                            f64_face_dist(sel3(a, f0, f1, f2), sel3(a, D0, D1, D2), sel3(a, s.x0, s.x1, s.x2)),
                            sel3(a, vp0, vp1, vp2));
                        if (t < tmin || (t == tmin && a < ax)) {
                            tmin = t;
                            ax = a;
                        }
                    }
                }
                s.steps++;
                t_end = s.t + tmin;
                path = P_CROSS;
                if (ax < 0 || tkey(t_end) >= s.tev) {   // (the stop time is never before tev)
                    if (ax < 0 && s.in_sink) path = P_CAPTURE;
                    else if (ax < 0 && !(p.t_stop < CUDART_INF)) path = P_NOEXIT;
                    else if (ax < 0 || ge_d(t_end, p.t_stop)) path = P_TIME;
                    if (TS && path != P_CAPTURE) {
                        const double t_rec = path == P_NOEXIT ? CUDART_INF : (path == P_TIME ? p.t_stop : t_end);
                        int kk = s.kn;
                        // (the comparison on the integer side, as in next_event)
                        while (kk < p.n_times && ge_d(t_rec, __ldg(o.times + kk))) kk++;
                        m = kk - s.kn;
                    }
                }
            }
        }
        if (TS && __any_sync(0xffffffffu, m > 0)) {
            rq_push(*this, Q, qcount, s, q, s.kn, m, path == P_NOEXIT ? MP_ST_NO_EXIT : MP_ST_ACTIVE);
            if (m) {
                s.kn += m;
                s.tev = next_event(s);
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
            const double dt = p.t_stop - s.t;
            s.x0 = f64_move(Ax, iAx, D0, vp0, s.x0, dt);
            s.x1 = f64_move(Ay, iAy, D1, vp1, s.x1, dt);
            s.x2 = f64_move(Az, iAz, D2, vp2, s.x2, dt);
            s.t = p.t_stop;
            s.st = MP_ST_TIME;
            return;
        }
        // displacement to the exit face: the two other axes move by the
        // analytic formula (selected into two slots, uniform across lanes),
        // the exit axis is put on its face
        const double dt = tmin;
        const int a1 = ax == 0 ? 1 : 0, a2 = ax == 2 ? 1 : 2;
        const double A1 = sel3(a1, Ax, Ay, Az), iA1 = sel3(a1, iAx, iAy, iAz), E1 = sel3(a1, D0, D1, D2);
        const double A2 = sel3(a2, Ax, Ay, Az), iA2 = sel3(a2, iAx, iAy, iAz), E2 = sel3(a2, D0, D1, D2);
        const double w1 = sel3(a1, vp0, vp1, vp2), y1 = sel3(a1, s.x0, s.x1, s.x2);
        const double w2 = sel3(a2, vp0, vp1, vp2), y2 = sel3(a2, s.x0, s.x1, s.x2);
        bool again1, again2;
        double n1 = f64_move_fast(A1, iA1, E1, w1, y1, dt, again1);
        double n2 = f64_move_fast(A2, iA2, E2, w2, y2, dt, again2);
        if (again1 || again2) {
            if (again1) n1 = f64_move(A1, iA1, E1, w1, y1, dt);
            if (again2) n2 = f64_move(A2, iA2, E2, w2, y2, dt);
        }
        const int face = ax == 0 ? f0 : (ax == 1 ? f1 : f2);
        const double Dax = ax == 0 ? D0 : (ax == 1 ? D1 : D2);
        const double onface = face > 0 ? Dax : 0.0;
        s.x0 = ax == 0 ? onface : n1;
        s.x1 = ax == 1 ? onface : (ax == 0 ? n1 : n2);
        s.x2 = ax == 2 ? onface : n2;
        s.t = t_end;
        const int fidx = 2 * ax + (face > 0 ? 1 : 0);
        s.ef = fidx;
        const int cls = (int)((nb >> (2 * fidx)) & 3u);
        const int dj = ax == 0 ? face : 0, di = ax == 1 ? face : 0, dk = ax == 2 ? face : 0;
        if (cls != NB_ACTIVE &&
            !(cls == NB_SINK && !sink_stops(p, f.sinkfrac, s.c + dj + di * f.ncol + dk * f.ncol * f.nrow))) {
            s.st = cls == NB_OUTSIDE ? MP_ST_EXIT_DOMAIN : (cls == NB_BOUNDARY ? MP_ST_BOUNDARY : MP_ST_SINK);
            return;
        }
        s.in_sink = cls == NB_SINK;
        // hand over to the neighbour; the exit coordinate enters on the shared face
        s.j += dj;
        s.i += di;
        s.k += dk;
        s.c += dj + di * f.ncol + dk * f.ncol * f.nrow;
        // (the new cell's size along the exit axis, loaded by every lane:
        // one selected load instead of a branch on the direction)
        const int si = ax == 0 ? s.j : (ax == 1 ? f.ncol + s.i : f.ncol + f.nrow + s.k);
        const double entry = face < 0 ? __ldg(&f.ax[si].D) : 0.0;
        s.x0 = ax == 0 ? entry : s.x0;
        s.x1 = ax == 1 ? entry : s.x1;
        s.x2 = ax == 2 ? entry : s.x2;
        s.h = fnv_step(s.h, s.c);
    }

    // the pathline point of the particle's current state
    __device__ __forceinline__ void path_point(const State& s, double& x, double& y, double& z, double& t) const
    {
        x = gx(s);
        y = gy(s);
        z = gz(s);
        t = s.t;
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
        const double x = ok ? gx(s) : CUDART_NAN, y = ok ? gy(s) : CUDART_NAN, z = ok ? gz(s) : CUDART_NAN;
        o.cell[q] = s.c;
        o.x[q] = x; o.y[q] = y; o.z[q] = z;
        o.px[q] = s.x0; o.py[q] = s.x1; o.pz[q] = s.x2;
        o.t[q] = s.t;
        o.status[q] = (uint8_t)s.st;
        o.steps[q] = s.steps;
        o.exit_face[q] = (uint8_t)s.ef;
        o.hash[q] = s.h;
        if (p.update_group && ok) {
            in.cell[q] = s.c;
            in.px[q] = s.x0; in.py[q] = s.x1; in.pz[q] = s.x2;
            in.t[q] = s.t;
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

// What bounds a step here: a FP64 instruction occupies its SM sub-partition
// for 64 cycles whatever its active lanes, and one warp cannot overlap two of
// them (measured: two independent chains of fmas take twice one chain's time).
// So while there are no more warps than a few a sub-partition, a step takes
// its FP64 warp instructions and the integer code between them, and lanes are
// free.  Lane 3 g + a of a warp holds axis a of the warp's particle g:
// velocities, exit times and motions of the axes run in the same
// instructions, 27 FP64 ones a step instead of 37.  The axes agree on the
// smallest FP32 estimate (so that a lane that cannot win never sends the warp
// into log1p's general form), then on the smallest exact time, by shuffles;
// the next cell's record is read while the axes move; and everything but
// crossing into the next cell is one rare branch of the warp, in which the
// group's lanes each end or move their axis and its first lane writes records,
// points and ends, with the axes gathered, through the one-lane engine's own
// functions.  Every particle has its lanes from the start, so the schedules
// would give the same.  One step of 4864 particles 2.7 -> 1.7 us; 1000
// particles, 50x50 cells 135 -> 93 us; 5003 pathlines, 7x61x83 cells 449 ->
// 277 us; 10,000 particles to a stop time, 200x200x20 cells 772 -> 491 us.
// (The range check of the next cell and the signed choice of the axis came
// later: 4000 particles, endpoints 553 us before both, 545 with the choice in
// a step of its own, 549 with the check.)
// Launches of up to this many warps of ten particles on each SM take three
// lanes a particle: three warps a sub-partition (18,240 particles on 152 SMs).
// There both forms are FP64 bound at about the same time (endpoints,
// 200x200x20 cells, 329 steps the longest: 4864 particles 550 us against 880,
// 9728: 629 / 947, 19456: 1020 / 979, 38912: 2317 / 1050).
constexpr int AXES_WARPS = 12;

// one axis of a cell's record
struct AxisRec {
    double v1, A, iA, D;
    float f1, f2, fA;
    unsigned nb;
};
__device__ __forceinline__ AxisRec read_axis(const DevField& f, int c, int a, int at)
{
    const double* rp = reinterpret_cast<const double*>(f.rec64 + c);
    const float* fp = reinterpret_cast<const float*>(rp + 10) + 3 * a;
    return AxisRec{__ldg(rp + 3 * a), __ldg(rp + 3 * a + 1), __ldg(rp + 3 * a + 2), __ldg(&f.ax[at].D),
                   __ldg(fp), __ldg(fp + 1), __ldg(fp + 2), __ldg(reinterpret_cast<const unsigned*>(rp + 9))};
}

// the full position and cell indices of each particle on its three lanes
// (warp-uniform call)
template <class S>
__device__ __forceinline__ void gather_axes(S& s, double x, int ix, int base)
{
    const unsigned FULL = 0xffffffffu;
    s.x0 = __shfl_sync(FULL, x, base);
    s.x1 = __shfl_sync(FULL, x, base + 1);
    s.x2 = __shfl_sync(FULL, x, base + 2);
    s.j = __shfl_sync(FULL, ix, base);
    s.i = __shfl_sync(FULL, ix, base + 1);
    s.k = __shfl_sync(FULL, ix, base + 2);
}

template <bool ONE, bool TS, bool PL>
__global__ void __launch_bounds__(32) k_track_axes(F64Engine<ONE> e)
{
    using E = F64Engine<ONE>;
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
    const int axis_at = a == 0 ? 0 : (a == 1 ? f.ncol : f.ncol + f.nrow);
    int qcount = 0, pcount = 0;
    long long q = 0;
    typename E::State s;   // x0, x1, x2, i, j, k: as last gathered
    s.r = 0;
    s.steps = 0;
    s.st = ST_SKIP;
    s.c = -1;
    s.x0 = s.x1 = s.x2 = 0.0;
    s.i = s.j = s.k = 0;
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
    // this lane's axis: offset and index, and the cell's record of it
    double x = a == 0 ? s.x0 : (a == 1 ? s.x1 : s.x2);
    int ix = a == 0 ? s.j : (a == 1 ? s.i : s.k);
    AxisRec c{};
    c.D = 1.0;
    if (live) c = read_axis(f, s.c, a, axis_at + ix);
    const int next1 = base + (a == 2 ? 0 : a + 1), next2 = base + (a == 0 ? 2 : a - 1);
    bool going = __any_sync(FULL, live);
    // One step of the warp's particles.  False: nothing was done, the step has
    // to be made with every reachable axis's exact time (EXACT; rare, and a
    // copy of its own so that the common step carries no test for it).
    auto step = [&](auto every) -> bool {
        constexpr bool EXACT = decltype(every)::value;
        const TrackParams& p = e.req(s.r).p;
        const bool go = live && !(s.steps >= s.cap && (long long)s.steps >= p.max_steps);
        // velocity, reachable face, FP32 estimate of the time to it (as in
        // the one-lane engine; -1: not to be trusted)
        const double vp = f64_vel(c.v1, c.A, x);
        unsigned lo, hi;
        words(vp, lo, hi);
        const int face = go ? f64_face(lo, hi, c.nb >> (NB_SIGN + 4 * a)) : 0;
        const unsigned up = __ballot_sync(FULL, face > 0);
        const double d = f64_face_dist(face, c.D, x);
        float est = CUDART_INF_F;
        if (face) {
            unsigned dl, dh;
            words(d, dl, dh);
            est = f32_estimate(trunc_small(dl, dh), trunc_normal(lo, hi), c.fA, face > 0 ? c.f2 : c.f1);
            if (!(est < CUDART_INF_F) || !vel_trusted(hi) || f.no_screen) est = -1.0f;
        }
        const float em = fminf(est, fminf(__shfl_sync(FULL, est, next1), __shfl_sync(FULL, est, next2)));
        // the exact time of the axes within 2^-10 of the smallest estimate
        // (all reachable ones in doubt); the smallest wins, ties to the lower axis
        const bool use = face != 0 && (EXACT || em < 0.0f || est <= em * (1.0f + 0.0009765625f));
        const double te = f64_exit_time_d(c.A, c.iA, d, face ? vp : 1.0, use);
        words(te, lo, hi);
        const bool has = use && hi < 0x7ff00000u;   // finite, not negative
        const unsigned long long key = has ? (unsigned long long)hi << 32 | lo : 0x7ff0000000000000ULL;
        const unsigned long long k0 = __shfl_sync(FULL, key, base), k1 = __shfl_sync(FULL, key, base + 1),
                                 k2 = __shfl_sync(FULL, key, base + 2);
        int ax = -1;
        unsigned long long km = 0x7ff0000000000000ULL;
        if (k0 < km) { km = k0; ax = 0; }
        if (k1 < km) { km = k1; ax = 1; }
        if (k2 < km) { km = k2; ax = 2; }
        double tmin = __longlong_as_double((long long)km);
        if constexpr (EXACT) {   // the general choice, negative times (offsets outside the cell) among them
            const double t = use && hi_abs(hi) < 0x7ff00000u ? te : CUDART_INF;
            const double t0 = __shfl_sync(FULL, t, base), t1 = __shfl_sync(FULL, t, base + 1),
                         t2 = __shfl_sync(FULL, t, base + 2);
            ax = -1;
            tmin = CUDART_INF;
            if (t0 < tmin) { tmin = t0; ax = 0; }
            if (t1 < tmin) { tmin = t1; ax = 1; }
            if (t2 < tmin) { tmin = t2; ax = 2; }
        }
        const int fx = ax < 0 ? 0 : ((up >> (base + ax)) & 1u) ? 1 : -1;
        const int fidx = 2 * ax + (fx > 0 ? 1 : 0);
        // the neighbour across the exit face, read while the axes move
        const int cls = ax < 0 ? (int)NB_OUTSIDE : (int)((c.nb >> (2 * fidx)) & 3u);
        const int c2 = s.c + fx * (ax == 0 ? 1 : (ax == 1 ? stride_y : stride_z));
        const int ix2 = ix + (a == ax ? fx : 0);
        const bool inside = (unsigned)c2 < (unsigned)f.ncell;   // (false across an outer face; else an error)
        const bool enter =
            go && ax >= 0 && inside && (cls == NB_ACTIVE || (cls == NB_SINK && !sink_stops(p, f.sinkfrac, c2)));
        AxisRec n = c;
        if (enter) n = read_axis(f, c2, a, axis_at + ix2);
        const double t_end = s.t + tmin;
        bool again;
        double xn = f64_move_fast(c.A, c.iA, c.D, vp, x, tmin, again);
        again = again && a != ax;
        // an event: an output time or the stop time in the step, no exit, a
        // path that ends here, the step cap, a motion for the general form, a
        // candidate whose exact time is not finite (if that is the leading
        // one, the others' times are not bounded by it) or is negative: then
        // every reachable axis decides, as in the one-lane engine
        const bool open = !EXACT && use && !has;
        const bool ev = go && (ax < 0 || tkey(t_end) >= s.tev);
        if (__any_sync(FULL, open || ev || (live && (!go || !enter || again)))) {
            if (!EXACT && __any_sync(FULL, open)) return false;
            enum { P_NONE, P_CROSS, P_TIME, P_NOEXIT, P_CAPTURE };
            int path = go ? P_CROSS : P_NONE, m = 0;
            if (ev) {   // (the stop time is never before tev)
                if (ax < 0 && s.in_sink) path = P_CAPTURE;
                else if (ax < 0 && !(p.t_stop < CUDART_INF)) path = P_NOEXIT;
                else if (ax < 0 || ge_d(t_end, p.t_stop)) path = P_TIME;
                if (TS && path != P_CAPTURE) {
                    const DevOut& o = e.req(s.r).o;
                    const double t_rec = path == P_NOEXIT ? CUDART_INF : (path == P_TIME ? p.t_stop : t_end);
                    int kk = s.kn;
                    while (kk < p.n_times && ge_d(t_rec, __ldg(o.times + kk))) kk++;
                    m = kk - s.kn;
                }
            }
            if (TS && __any_sync(FULL, m > 0)) {
                gather_axes(s, x, ix, base);
                rq_push(e, Q, qcount, s, q, s.kn, lead ? m : 0, path == P_NOEXIT ? MP_ST_NO_EXIT : MP_ST_ACTIVE);
                if (m) {
                    s.kn += m;
                    s.tev = e.next_event(s);
                }
            }
            if (path == P_CROSS) {
                if (again) xn = f64_move(c.A, c.iA, c.D, vp, x, tmin);
                if (!enter) {
                    x = a == ax ? (fx > 0 ? c.D : 0.0) : xn;
                    s.t = t_end;
                    s.ef = fidx;
                    s.st = cls == NB_OUTSIDE ? MP_ST_EXIT_DOMAIN : (cls == NB_BOUNDARY ? MP_ST_BOUNDARY : MP_ST_SINK);
                    if (!inside && (cls == NB_ACTIVE || cls == NB_SINK)) {
                        if (lead) atomicCAS(e.req(s.r).o.counters + COUNTER_ERR, 0ULL, (unsigned long long)q + 1ULL);
                        s.st = MP_ST_INVALID_RELEASE;
                    }
                }
            } else if (path == P_TIME) {
                x = f64_move(c.A, c.iA, c.D, vp, x, p.t_stop - s.t);
                s.t = p.t_stop;
                s.st = MP_ST_TIME;
            } else if (live) {
                s.st = path == P_CAPTURE ? MP_ST_SINK : (path == P_NOEXIT ? MP_ST_NO_EXIT : MP_ST_STEP_CAP);
            }
            ended = live && s.st != MP_ST_ACTIVE;
            if (__any_sync(FULL, ended)) {
                if (go && ended) s.steps++;
                gather_axes(s, x, ix, base);
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
            x = a == ax ? (fx < 0 ? n.D : 0.0) : xn;
            s.t = t_end;
            s.ef = fidx;
            s.in_sink = cls == NB_SINK;
            s.c = c2;
            ix = ix2;
            s.h = fnv_step(s.h, c2);
            c = n;
        }
        if (PL) {
            gather_axes(s, x, ix, base);
            pl_push(e, P, pcount, s, q, lead && go && live && p.pathline, s.st);
        }
        return true;
    };
    while (going)
        if (!step(std::false_type{})) step(std::true_type{});
    if (TS) rec_finish(e, Q, qcount);
    if (PL) pl_flush(e, P, pcount);
    flush_counters(e, s_cnt);
    window_end(e);
}

template <bool ONE>
cudaError_t launch_axes(const F64Engine<ONE>& e, unsigned modes, cudaStream_t s)
{
    const bool ts = (modes & MODE_TS) != 0, pl = (modes & MODE_PATH) != 0;
    const size_t smem = (ts ? sizeof(typename F64Engine<ONE>::RecQ) : 0) + (pl ? sizeof(PathQ) : 0);
    const unsigned grid = (unsigned)((e.b.n_total + AXES_PARTICLES - 1) / AXES_PARTICLES);
    auto kern = ts ? (pl ? k_track_axes<ONE, true, true> : k_track_axes<ONE, true, false>)
                   : (pl ? k_track_axes<ONE, false, true> : k_track_axes<ONE, false, false>);
    kern<<<grid, 32, smem, s>>>(e);
    return cudaGetLastError();
}

// A request's endpoint arrays into the caller's: one launch for up to twelve
// copies (blockIdx.y) instead of a cudaMemcpyAsync each, which cost 34 us of
// host time and about 2 us of stream time apiece for 1000 particles.  Bound
// by launch latency below about 1e5 particles, by HBM above.  16-byte words
// where both addresses allow, 8 or 4 where a caller's slice starts between
// (the library's arrays start on 256 bytes), else single bytes.
template <class T>
__device__ __forceinline__ void copy_words(const CopyItem& c)
{
    const unsigned long long n = c.bytes / sizeof(T), step = (unsigned long long)gridDim.x * blockDim.x;
    const T* src = static_cast<const T*>(c.src);
    T* dst = static_cast<T*>(c.dst);
    unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
    for (; i + 3 * step < n; i += 4 * step) {
        const T v0 = src[i], v1 = src[i + step], v2 = src[i + 2 * step], v3 = src[i + 3 * step];
        dst[i] = v0;
        dst[i + step] = v1;
        dst[i + 2 * step] = v2;
        dst[i + 3 * step] = v3;
    }
    for (; i < n; i += step) dst[i] = src[i];
    const unsigned long long done = n * sizeof(T);
    if (blockIdx.x == 0 && threadIdx.x < c.bytes - done)
        static_cast<char*>(c.dst)[done + threadIdx.x] = static_cast<const char*>(c.src)[done + threadIdx.x];
}

__global__ void k_copy_list(const __grid_constant__ CopyList list)
{
    const CopyItem& c = list.a[blockIdx.y];
    const unsigned low = (unsigned)(reinterpret_cast<unsigned long long>(c.dst) |
                                    reinterpret_cast<unsigned long long>(c.src)) & 15u;
    if (low == 0u) copy_words<uint4>(c);
    else if ((low & 7u) == 0u) copy_words<uint2>(c);
    else if ((low & 3u) == 0u) copy_words<unsigned>(c);
    else copy_words<unsigned char>(c);
}

cudaError_t launch_copy_list(const CopyList& c, cudaStream_t s)
{
    if (c.n == 0) return cudaSuccess;
    // four words a thread; at most a few waves (12 arrays x 152 SMs)
    const unsigned long long blocks = (c.most + 256 * 64 - 1) / (256 * 64);
    k_copy_list<<<dim3((unsigned)(blocks < 608 ? blocks : 608), (unsigned)c.n), 256, 0, s>>>(c);
    return cudaGetLastError();
}

__global__ void k_zero_counters(const Req* reqs, int n)
{
    const int i = (int)(blockIdx.x * blockDim.x + threadIdx.x);
    if (i < n * N_COUNTERS) reqs[i / N_COUNTERS].o.counters[i % N_COUNTERS] = 0ULL;
}

cudaError_t launch_zero_counters(const Batch& b, cudaStream_t s)
{
    const long long words = (long long)b.n_reqs * N_COUNTERS;   // (below 2^31: fewer than 2^24 requests)
    k_zero_counters<<<(unsigned)((words + 255) / 256), 256, 0, s>>>(b.reqs, b.n_reqs);
    return cudaGetLastError();
}

// The tracking kernels keep a launch's device-time window in its first
// request's counters; a batch's other requests get a copy.
__global__ void k_spread_window(const Req* reqs, int n)
{
    const unsigned long long* src = reqs[0].o.counters + COUNTER_T_BEGIN;
    const unsigned long long t0 = src[0], t1 = src[1];
    for (int i = 1 + (int)(blockIdx.x * blockDim.x + threadIdx.x); i < n; i += (int)(gridDim.x * blockDim.x)) {
        reqs[i].o.counters[COUNTER_T_BEGIN] = t0;
        reqs[i].o.counters[COUNTER_T_END] = t1;
    }
}

cudaError_t launch_spread_window(const Batch& b, cudaStream_t s)
{
    if (b.n_reqs <= 1 || b.n_total <= 0) return cudaSuccess;
    k_spread_window<<<1, 256, 0, s>>>(b.reqs, b.n_reqs);
    return cudaGetLastError();
}

cudaError_t form_fp64(long long n, LaunchForm* out) { return form_of<F64Engine<true>>(n, AXES_WARPS, out); }

cudaError_t launch_track_fp64(const DevField& f, const Batch& b, unsigned modes, int schedule, int block, cudaStream_t s)
{
    if (b.n_total <= 0) return cudaSuccess;
    int sms = 0;
    const cudaError_t err = sm_count(&sms);
    if (err != cudaSuccess) return err;
    const bool few = few_particles(b.n_total, AXES_WARPS, sms);
    if (b.n_reqs == 1) {
        const F64Engine<true> e{f, b};
        return few ? launch_axes(e, modes, s) : launch_tracking(e, modes, schedule, block, s);
    }
    const F64Engine<false> e{f, b};
    return few ? launch_axes(e, modes, s) : launch_tracking(e, modes, schedule, block, s);
}

}  // namespace mp

namespace mp {

// ---------------------------------------------------------------------------
// field validation: bit 1 non-finite flow, bit 2 porosity outside (0, 1] in
// an active or sink cell, bit 4 ibound outside {-1, 0, 1, 2}
// ---------------------------------------------------------------------------

__global__ void k_validate(const double* qx, long long nqx, const double* qy, long long nqy, const double* qz,
                           long long nqz, const double* por, const int8_t* ib, long long ncell, unsigned* flags)
{
    const long long total = nqx + nqy + nqz + ncell;
    unsigned bad = 0;
    for (long long u = (long long)blockIdx.x * blockDim.x + threadIdx.x; u < total;
         u += (long long)gridDim.x * blockDim.x) {
        if (u < nqx) {
            if (!isfinite(qx[u])) bad |= 1u;
        } else if (u < nqx + nqy) {
            if (!isfinite(qy[u - nqx])) bad |= 1u;
        } else if (u < nqx + nqy + nqz) {
            if (!isfinite(qz[u - nqx - nqy])) bad |= 1u;
        } else {
            const long long c = u - nqx - nqy - nqz;
            const int8_t b = ib[c];
            if (b < -1 || b > 2) bad |= 4u;
            if (b == 1 || b == 2) {
                const double n = por[c];
                if (!(n > 0.0 && n <= 1.0)) bad |= 2u;
            }
        }
    }
    if (bad) atomicOr(flags, bad);
}

cudaError_t launch_validate(const double* qx, long long nqx, const double* qy, long long nqy, const double* qz,
                            long long nqz, const double* por, const int8_t* ib, long long ncell, unsigned* flags,
                            cudaStream_t s)
{
    k_validate<<<1024, 256, 0, s>>>(qx, nqx, qy, nqy, qz, nqz, por, ib, ncell, flags);
    return cudaGetLastError();
}

}  // namespace mp
