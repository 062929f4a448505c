// Checks the FP64 step's short forms (mp_f64math.cuh) against the general
// ones, bit for bit: fast_log1p against series_log1p (around every row edge,
// sqrt2 and the ends of the table too), f64_move_fast against f64_move, the
// word forms of the FP32 truncation against f32_trunc, the FP32 reciprocal
// against __frcp_rn on every significand, the time keys against the FP64
// order, the screened exit axis against all three exact times, the quotients
// and conversions of the field records against the IEEE ones.
// Prints the mismatch counts and exits non-zero on any.
#include <cstdio>

#include "mp_f64math.cuh"

using namespace mp;

__device__ __forceinline__ unsigned long long mix64(unsigned long long x)
{
    x += 0x9e3779b97f4a7c15ULL;
    x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ULL;
    x = (x ^ (x >> 27)) * 0x94d049bb133111ebULL;
    return x ^ (x >> 31);
}
__device__ __forceinline__ double unit(unsigned long long r) { return (double)(r >> 11) * 0x1.0p-53; }
// magnitudes spread over 2^lo .. 2^hi
__device__ __forceinline__ double spread(unsigned long long r, int lo, int hi)
{
    return ldexp(1.0 + unit(mix64(r)), lo + (int)(r % (unsigned)(hi - lo)));
}
__device__ __forceinline__ bool same(double a, double b)
{
    return __double_as_longlong(a) == __double_as_longlong(b) || (a != a && b != b);
}

__global__ void check(unsigned long long* bad, unsigned long long n)
{
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < n;
         i += (unsigned long long)gridDim.x * blockDim.x) {
        const unsigned long long r = mix64(i);
        // log1p: wide magnitudes of both signs, (-1, 0), (0, 16), within a
        // few rounding errors of the row edges u = (1 + f / 256) 2^e and of
        // sqrt2 2^e, and special values
        double x;
        switch (i & 7) {
        case 0: x = spread(r, -1074, 1023); break;
        case 1: x = -unit(r); break;
        case 2: x = 16.0 * unit(r); break;
        case 3: case 4: case 5: {
            const int e = (int)(r % 12) - 6;
            double u = ldexp((r >> 8) % 5 == 0 ? 1.4142135623730951 : 1.0 + (double)((r >> 16) % 256) / 256.0, e);
            u *= 1.0 + ((double)((r >> 32) % 65) - 32.0) * ((i & 7) == 3 ? 0x1.0p-53 : 0x1.0p-24);
            x = u - 1.0;
            break;
        }
        case 6: x = -spread(r, -1074, 130); break;
        default: {
            const double s[8] = {0.0, -0.0, -1.0, CUDART_INF, -CUDART_INF, CUDART_NAN, 1e40, -1e40};
            x = s[r & 7];
        }
        }
        if (!same(fast_log1p(x), series_log1p(x))) atomicAdd(bad + 0, 1ULL);
        // motion: gradients, velocities, offsets and times over wide ranges,
        // with zero gradients, velocities and times and offsets on both faces
        const double D = spread(mix64(r + 1), -20, 20);
        const unsigned long long c = mix64(r + 2);
        double pp = D * unit(mix64(r + 3));
        if (c % 7 == 0) pp = 0.0;
        if (c % 7 == 1) pp = D;
        const double v1 = (c & 1 ? 1.0 : -1.0) * spread(mix64(r + 4), -60, 10);
        double A = (c & 2 ? 1.0 : -1.0) * fabs(v1) * spread(mix64(r + 5), -40, 4) / D;
        if (c % 11 == 0) A = 0.0;
        const double iA = A != 0.0 ? 1.0 / A : 0.0;
        double vp = f64_vel(v1, A, pp), dt = (D / fabs(v1)) * spread(mix64(r + 6), -60, 6);
        if (c % 13 == 0) vp = 0.0;
        if (c % 17 == 0) dt = 0.0;
        if (c % 19 == 0) { A = spread(c, -1074, -1000); vp = spread(r, -1074, -900); }
        bool again;
        const double got = f64_move_fast(A, iA, D, vp, pp, dt, again);
        if (!again && !same(got, f64_move(A, iA, D, vp, pp, dt))) atomicAdd(bad + 1, 1ULL);
        // truncations on their domains
        unsigned lo, hi;
        const double t = (c & 4 ? 1.0 : -1.0) * spread(r, -1074, 127);
        words(t, lo, hi);
        const unsigned want = __float_as_uint(f32_trunc(t));
        if (__float_as_uint(trunc_small(lo, hi)) != want) atomicAdd(bad + 2, 1ULL);
        if (t > 0.0 && __float_as_uint(trunc_pos(lo, hi)) != want) atomicAdd(bad + 2, 1ULL);
        if (fabs(t) >= 0x1.0p-126 && __float_as_uint(trunc_normal(lo, hi)) != want) atomicAdd(bad + 2, 1ULL);
        // the FP32 reciprocal: every significand, both signs, exponents over
        // the range that d / v takes
        const float rx = __uint_as_float((unsigned)(i & 0x7fffffu) | ((7u + (unsigned)(mix64(i >> 23) % 240)) << 23) |
                                         ((unsigned)(r >> 40) << 31));
        if (__float_as_uint(rcp_rn_normal(rx)) != __float_as_uint(__frcp_rn(rx))) atomicAdd(bad + 6, 1ULL);
        // the field records' quotients and conversions against IEEE ones
        {
            const double Dd = spread(mix64(r + 40), -62, 62), yd = 1.0 / Dd;
            double v = (c & 32 ? -1.0 : 1.0) * (c % 3 ? spread(mix64(r + 41), -40, 10) : spread(mix64(r + 41), -1074, 1023));
            if (c % 5 == 0) v = Dd * (double)__uint_as_float((unsigned)(r >> 20) & 0x3fffffffu);           // near FP32 values
            if (c % 5 == 1) v = Dd * ((double)__uint_as_float(((unsigned)(r >> 20) & 0x3fffffffu) | 0x20000000u) * (1.0 + 0x1p-24));   // and middles
            if (c % 43 == 0) v = c & 64 ? 0.0 : -0.0;
            if (plain_divisor(Dd)) {
                if (!same(div_by(v, Dd, yd), v / Dd)) atomicAdd(bad + 7, 1ULL);
                if (__float_as_uint(quot_f32(v, Dd, yd)) != __float_as_uint((float)(v / Dd))) atomicAdd(bad + 7, 1ULL);
            }
            if (__float_as_uint(f32_rn(v)) != __float_as_uint((float)v)) atomicAdd(bad + 7, 1ULL);
        }
        // keys of times
        const double a = (c & 8 ? 1.0 : -1.0) * spread(mix64(r + 7), -3, 3) * (c % 23 == 0 ? 0.0 : 1.0) + 0.0;
        const double b = c % 29 == 0 ? a : (c & 16 ? 1.0 : -1.0) * spread(mix64(r + 8), -3, 3) * (c % 31 == 0 ? 0.0 : 1.0);
        if ((tkey(a) >= bound_key(b)) != (a >= b)) atomicAdd(bad + 3, 1ULL);
        // exit axis: three axes, their times from all exact evaluations and
        // from the screened ones
        float e[3];
        double te[3], vv[3], AA[3], dd[3];
        unsigned reach = 0;
        bool doubt = false;
        for (int k = 0; k < 3; ++k) {
            const unsigned long long s = mix64(r + 10 + k), g = mix64(r + 20 + k);
            const double Dk = k && s % 3 == 0 ? D : spread(s, -3, 6);
            const double pk = s % 5 == 0 ? 0.0 : (s % 5 == 1 ? Dk : Dk * unit(mix64(g)));
            const double lowv = (g & 1 ? 1.0 : -1.0) * spread(mix64(s), -8, -3) * (s % 41 == 0 ? 0x1.0p-400 : 1.0);
            const double highv = (g & 6 ? (g & 1 ? 1.0 : -1.0) : (g & 1 ? -1.0 : 1.0)) * spread(mix64(g + 1), -8, -3);
            AA[k] = s % 37 == 0 ? 0.0 : (highv - lowv) / Dk;
            vv[k] = f64_vel(lowv, AA[k], pk);
            unsigned l, h;
            words(vv[k], l, h);
            const int f = f64_face(l, h, (lowv < 0.0 ? 2u : 0u) | (highv > 0.0 ? 4u : 0u));
            if (f != ((vv[k] > 0.0 && highv > 0.0) ? 1 : (vv[k] < 0.0 && lowv < 0.0) ? -1 : 0)) atomicAdd(bad + 4, 1ULL);
            bool close;
            float fd = f32_face_dist(f, f32_trunc(Dk), pk, close);
            if (close) fd = f32_trunc(Dk - pk);
            dd[k] = f64_face_dist(f, Dk, pk);
            const float est = f32_estimate(fd, trunc_normal(l, h), (float)AA[k], (float)(f > 0 ? highv : lowv));
            doubt = doubt || (f && !(vel_trusted(h) && est < CUDART_INF_F));
            e[k] = f ? est : CUDART_INF_F;
            te[k] = CUDART_INF;
            if (f) {
                reach |= 1u << k;
                te[k] = f64_exit_time_d(AA[k], AA[k] != 0.0 ? 1.0 / AA[k] : 0.0, dd[k], vv[k]);
            }
        }
        int ax = -1;
        double tmin = CUDART_INF;
        for (int k = 0; k < 3; ++k)
            if ((reach >> k & 1u) && te[k] < tmin) { tmin = te[k]; ax = k; }
        unsigned rest;
        int got_ax = -1;
        double got_t = CUDART_INF;
        const int a0 = screen(e[0], e[1], e[2], reach, doubt, rest);
        if (a0 >= 0) {
            if (is_finite(te[a0])) { got_t = te[a0]; got_ax = a0; }
            else rest = reach & ~(1u << a0);
            while (rest) {
                const int k = __ffs(rest) - 1;
                rest &= rest - 1;
                if (te[k] < got_t || (te[k] == got_t && k < got_ax)) { got_t = te[k]; got_ax = k; }
            }
        }
        if (got_ax != ax || !same(got_t, tmin)) atomicAdd(bad + 5, 1ULL);
    }
}

int main()
{
    unsigned long long* bad = nullptr;
    if (cudaMalloc(&bad, 8 * sizeof(unsigned long long)) != cudaSuccess) return 2;
    cudaMemset(bad, 0, 8 * sizeof(unsigned long long));
    check<<<152 * 8, 128>>>(bad, 1ULL << 26);
    unsigned long long h[8] = {0};
    cudaMemcpy(h, bad, sizeof h, cudaMemcpyDeviceToHost);
    const cudaError_t e = cudaDeviceSynchronize();
    printf("%s log1p %llu move %llu trunc %llu keys %llu face %llu screen %llu rcp %llu quotients %llu\n",
           cudaGetErrorString(e), h[0], h[1], h[2], h[3], h[4], h[5], h[6], h[7]);
    cudaFree(bad);
    return (e == cudaSuccess && !(h[0] | h[1] | h[2] | h[3] | h[4] | h[5] | h[6] | h[7])) ? 0 : 1;
}
