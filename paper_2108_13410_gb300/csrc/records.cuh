// records.cuh -- angles, phase-table entries and tangents of one Trotter factor group, computed
// on the device in FP64 from the schedule and the couplings.
#pragma once
#include <cuda_runtime.h>

namespace qsim {

// ---------------------------------------------------------------------------
// Operator records built on the device from the schedule s[] and the couplings.
// A record describes one Trotter factor group: X angles per class, then the Z
// table (nA+1)(nB+1) and, for the unitary gauge, the Hadamard-basis X table.
// Every exp(i t) is stored as (u, s) = (2 sin^2(t/2), sin t) computed in FP64; for
// complex64 the float pair within +-3 ulps minimising |(1-u)^2 + s^2 - 1| is kept.
// ---------------------------------------------------------------------------
struct RecGeom {
    int n_steps, order, fsal;    // fsal: second order with merged X half-steps
    int path;                    // 1: couplings per step (cpl[k * batch + b]) with s = 1
    int batch, rec_stride;
    int nA, nB, nXA, nXB, xlut_off;
    int f32;
    int tan_off, nX0, nX1;       // tangent-form triple (0: none); X qubits per class
    double dt;
};

struct DevCouplings { double J, h, g, lambda; };

// The couplings and the schedule of a call that is short enough travel in the parameters of the
// records kernel: no copy before it, and no wait of the host for the previous call's copy (which
// held a loop over single steps at one call in flight).
constexpr int REC_INLINE = 480;
struct RecInline { double v[REC_INLINE]; };

// The float pair within +-3 ulps of (u, s) that minimises |(1 - u)^2 + s^2 - m2|, the first
// of equal ones by distance from (u, s).  With e0 the deviation of the rounded pair (FP64),
// the deviation of a neighbour is e0 + du (du - 2 (1 - u0)) + ds (ds + 2 s0) with du, ds the
// (exact) float differences, evaluated in FP32 to ~1e-14: far below the ~1e-10 that the best
// of the 49 pairs reaches, so FP64 runs once per entry instead of 49 times.  GB300 retires
// about two FP64 FMAs per clock per SM and the search in FP64 was almost all of
// k_build_records (100 us for the two factor groups of one 18-qubit step).
__device__ inline void dev_nearest_modulus(double u, double s, double m2, double *ou, double *os) {
    const float u0 = (float)u, s0 = (float)s;
    const double c0 = 1.0 - (double)u0;
    const float e0 = (float)(c0 * c0 + (double)s0 * (double)s0 - m2);
    const float ru = (float)(u - (double)u0), rs = (float)(s - (double)s0);
    const float a = -2.0f * (float)c0, b = 2.0f * s0;
    float ds[7], es[7];
    {
        float ss = s0;
        ds[3] = 0.f;
#pragma unroll
        for (int j = 2; j >= 0; --j) { ss = nextafterf(ss, -4.0f); ds[j] = ss - s0; }
        ss = s0;
#pragma unroll
        for (int j = 4; j < 7; ++j) { ss = nextafterf(ss, 4.0f); ds[j] = ss - s0; }
#pragma unroll
        for (int j = 0; j < 7; ++j) es[j] = ds[j] * (ds[j] + b);
    }
    float be = fabsf(e0), bd = 0.f, bu = 0.f, bs = 0.f;
    float uu = nextafterf(nextafterf(nextafterf(u0, -4.0f), -4.0f), -4.0f);
    for (int i = 0; i < 7; ++i, uu = nextafterf(uu, 4.0f)) {
        const float du = uu - u0;
        const float eu = e0 + du * (du + a), dd = fabsf(du - ru);
#pragma unroll
        for (int j = 0; j < 7; ++j) {
            const float e = fabsf(eu + es[j]), d = dd + fabsf(ds[j] - rs);
            if (e < be || (e == be && d < bd)) { be = e; bd = d; bu = du; bs = ds[j]; }
        }
    }
    *ou = (double)(u0 + bu); *os = (double)(s0 + bs);
}

__device__ inline void dev_unit_pair(bool f32, double t, double *ou, double *os) {
    if (!f32) {
        const double sh = sin(0.5 * t);
        *ou = 2.0 * sh * sh; *os = sin(t);
        return;
    }
    double sh, ch;
    sincos(0.5 * t, &sh, &ch);
    dev_nearest_modulus(2.0 * sh * sh, 2.0 * sh * ch, 1.0, ou, os);
}

// Careful pair of exp(i t) = (1 - u) + i s for per-step tables built inside a kernel:
// one FP64 sincos, then a 3 x 3 search over the float neighbours of s and of the u that
// makes (1 - u)^2 + s^2 = 1 for each of them, keeping the pair with the smallest
// |(1 - u)^2 + s^2 - 1| (evaluated in FP64).  complex128 tables take (u, s) as they are.
// About a tenth of dev_unit_pair's FP64 work, which matters where a table is rebuilt
// for every Trotter step inside a persistent kernel (GB300 retires about two FP64 FMAs
// per clock per SM).
template <typename R>
__device__ inline void dev_unit_pair_fast(double t, R *ou, R *os) {
    double sh, ch;
    sincos(0.5 * t, &sh, &ch);
    const double u = 2.0 * sh * sh, s = 2.0 * sh * ch;
    if (sizeof(R) == 8) { *ou = (R)u; *os = (R)s; return; }
    const bool neg = u > 1.0;           // cos t < 0: 1 - u = -sqrt(1 - s^2)
    float bu = (float)u, bs = (float)s;
    double be = 1e300;
    float sc = nextafterf((float)s, -4.0f);
    for (int i = 0; i < 3; ++i, sc = nextafterf(sc, 4.0f)) {
        const double s2 = (double)sc * (double)sc;
        const double r = sqrt(fmax(0.0, 1.0 - s2));
        const double us = neg ? 1.0 + r : s2 / (1.0 + r);
        float uc = nextafterf((float)us, -4.0f);
        for (int j = 0; j < 3; ++j, uc = nextafterf(uc, 4.0f)) {
            const double c = 1.0 - (double)uc;
            const double e = fabs(c * c + s2 - 1.0);
            if (e < be) { be = e; bu = uc; bs = sc; }
        }
    }
    *ou = (R)bu; *os = (R)bs;
}

// X angles and Z angles of factor group `op` for couplings c:
//   order 1:      op k (< N): X theta(s_k) dt, Z at s_k
//   second order: op k (<= N): X theta(s_k) dt/2 [k < N] + theta(s_{k-1}) dt/2 [k > 0],
//                 Z at s_k for k < N (the last group is the trailing X half-step)
//   path mode: step k uses H1 with couplings cpl[k * batch + b] (s = 1)
__device__ inline void dev_op_angles(const RecGeom &G, const DevCouplings *__restrict__ cpl, int b,
                                     const double *__restrict__ sv, int op, double *thx, double *zA, double *zB,
                                     bool *has_z) {
    thx[0] = thx[1] = 0.0;
    *zA = *zB = 0.0;
    *has_z = false;
    const int N = G.n_steps;
    auto cp = [&](int k) -> const DevCouplings & { return G.path ? cpl[(long long)k * G.batch + b] : cpl[b]; };
    auto sk = [&](int k) -> double { return G.path ? 1.0 : sv[k]; };
    auto add = [&](int k, double tau) {
        const double s = sk(k);
        const DevCouplings &c = cp(k);
        thx[0] += ((1.0 - s) + s * c.g) * tau;
        thx[1] += ((1.0 - s) + s * c.J) * tau;
    };
    auto zs = [&](int k) {
        const double s = sk(k);
        const DevCouplings &c = cp(k);
        *zA = s * c.h * G.dt; *zB = s * c.lambda * G.dt; *has_z = true;
    };
    if (!G.fsal) {
        add(op, G.dt);
        zs(op);
    } else {
        if (op < N) add(op, 0.5 * G.dt);
        if (op > 0) add(op - 1, 0.5 * G.dt);
        if (op < N) zs(op);
    }
}

// Tangent form of one X layer for the complex64 kernels.  In the real-rotation frame
// exp(i th X) is cos th [[1, t], [-t, 1]] with t = tan th: a butterfly a' = a + t b,
// b' = b - t a (one rounded FMA per output), and the cos th of all n0 + n1 X qubits
// multiply to one scalar C, applied once per factor group.  t is rounded to the kernel
// precision and C is computed in FP64 from the rounded t, C = (1 + t0^2)^(-n0/2)
// (1 + t1^2)^(-n1/2), so the butterflies and C together keep the norm exactly; C is
// applied through the scaled Z table (dev_scaled_pair) or, for a factor group without
// a Z layer, rounded once.  Used when |th| <= pi/4 and C >= 1/2 (the host checks;
// otherwise the (u, s) form runs).  o = [t0, t1, C, 0].
__device__ inline void dev_tan(bool f32, double th, int n, double *t, double *f) {
    double v = tan(th);
    if (f32) v = (double)(float)v;
    *t = v;
    double x = 1.0 + v * v, p = 1.0;      // (1 + t^2)^n by squaring
    for (; n; n >>= 1, x *= x)
        if (n & 1) p *= x;
    *f = p;
}

// C exp(i phi) as (u, s) with (1 - u) + i s, u = 1 - C cos phi, s = C sin phi; for
// complex64 the float pair within +-3 ulps of each component minimising
// |(1 - u)^2 + s^2 - C^2| (in double), so the modulus of every table entry is C to
// ~1e-10 relative, as the unit pairs of dev_unit_pair are 1.
__device__ inline void dev_scaled_pair(bool f32, double phi, double C, double *ou, double *os) {
    if (!f32) {
        const double sh = sin(0.5 * phi);
        *ou = (1.0 - C) + C * 2.0 * sh * sh; *os = C * sin(phi);
        return;
    }
    double sh, ch;
    sincos(0.5 * phi, &sh, &ch);
    dev_nearest_modulus((1.0 - C) + C * 2.0 * sh * sh, C * 2.0 * sh * ch, C * C, ou, os);
}

// x^n by squaring (pow costs a small pass microseconds of FP64 latency)
__device__ inline double dev_powi(double x, int n) {
    double p = 1.0;
    for (; n; n >>= 1, x *= x)
        if (n & 1) p *= x;
    return p;
}

}  // namespace qsim
