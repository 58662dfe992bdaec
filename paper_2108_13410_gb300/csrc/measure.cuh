// measure.cuh -- reductions over a state: norm, diagonal sums, X strings, overlaps, the energy
// terms and the density of states (sm_103a).
//
// All of them read the state and are bound by that where the arithmetic allows: GB300 retires
// about two FP64 operations per clock and SM, so complex64 sums run in FP32 without rounding
// error, products and sums as pairs of floats, and go to FP64 once per sixteen amplitudes.  The
// parity words of an amplitude are a tile word, a thread word and a register word (no table
// look-up per amplitude), and of an X string only one amplitude of every pair is visited.  Blocks
// write partial sums; k_finish adds them in a fixed order.
// A tile is 4096 consecutive amplitudes (registers bits 8..11, threads bits 0..7) or, for the
// X terms of the energy, one tile of an X pass (kernels.cuh).
#pragma once
#include "kernels.cuh"

namespace qsim {

// n - 2 k without a conversion instruction (quarter rate); k < 2^22.  FP64 sums take it from a
// table in shared memory: the FP64 pipe is what bounds them.
__device__ __forceinline__ float weight(const float *, float n, int k) {
    return fmaf(-2.0f, __uint_as_float(0x4b000000u | (unsigned)k) - 8388608.0f, n);
}
__device__ __forceinline__ double weight(const double *tab, double, int k) { return tab[k]; }

// tables of nA - 2 k and nB - 2 k (complex128)
template <typename R>
__device__ __forceinline__ void load_weights(R (*w)[33], int nA, int nB) {
    if (sizeof(R) == 8)
        for (int k = threadIdx.x; k < 66; k += blockDim.x) w[k / 33][k % 33] = (R)((k < 33 ? nA : nB) - 2 * (k % 33));
}
__device__ __forceinline__ float flip_sign(float x, unsigned odd) {
    return __uint_as_float(__float_as_uint(x) ^ (odd << 31));
}
__device__ __forceinline__ double flip_sign(double x, unsigned odd) {
    return __longlong_as_double(__double_as_longlong(x) ^ ((long long)odd << 63));
}

// g += s; l += the rounding error of it (complex64)
__device__ __forceinline__ void add_keep(float &g, float &l, float s) {
    const float h = __fadd_rn(g, s), b = __fsub_rn(h, g);
    l = __fadd_rn(l, __fadd_rn(__fsub_rn(g, __fsub_rn(h, b)), __fsub_rn(s, b)));
    g = h;
}
__device__ __forceinline__ void add_keep(double &g, double &, double s) { g += s; }

// A product of two amplitudes' parts, Re(conj(a) b).  complex64: without rounding error, as a sum of
// two floats: observables are small differences of sums of order one.  (With rounded products in
// runs of eight they were up to ten times further off than with one amplitude of a small state
// per FP64 addition: 18 qubits, norm 1.1e-9 against 5.1e-10, X strings 2.7e-9 against 5.4e-10; so
// 6e-16 and 1e-16.)
__device__ __forceinline__ double product(double2 a, double2 b) { return fma(a.y, b.y, a.x * b.x); }
__device__ __forceinline__ float2 product(float2 a, float2 b) {
    float h = __fmul_rn(a.x, b.x), l = __fmaf_rn(a.x, b.x, -h);
    const float q = __fmul_rn(a.y, b.y);
    l = __fadd_rn(l, __fmaf_rn(a.y, b.y, -q));
    add_keep(h, l, q);
    return make_float2(h, l);
}

// A thread's sum of products, in FP64 over runs.  complex64: two runs of eight at a time, so that
// one FP64 addition takes sixteen amplitudes (halves: the sum of two finite runs may be beyond
// FP32); l takes the parts that do not fit the runs.  complex128: one run of sixteen.
template <typename R> struct Runs;
template <> struct Runs<double> {
    typedef double T;
    double h;
    static __device__ __forceinline__ constexpr int run(int) { return 0; }
    // f += p, f += w p, f += Re(conj(a) b)
    __device__ __forceinline__ void term(double &f, double p) { f += p; }
    __device__ __forceinline__ void term(double &f, double p, double w) { f = fma(p, w, f); }
    __device__ __forceinline__ void pair(double &f, double2 a, double2 b) { f = fma(a.y, b.y, fma(a.x, b.x, f)); }
    static __device__ __forceinline__ double flip(double p, unsigned odd) { return flip_sign(p, odd); }
    __device__ __forceinline__ void add(double a, double) { h += a; }
    __device__ __forceinline__ double value() const { return h; }
};
template <> struct Runs<float> {
    typedef float2 T;
    double h;
    float l;
    static __device__ __forceinline__ constexpr int run(int r) { return r / RED_RUN; }
    __device__ __forceinline__ void term(float &f, float2 p) {
        add_keep(f, l, p.x);
        l = __fadd_rn(l, p.y);
    }
    __device__ __forceinline__ void term(float &f, float2 p, float w) {
        const float q = __fmul_rn(p.x, w);
        add_keep(f, l, q);
        l = __fadd_rn(l, __fmaf_rn(p.y, w, __fmaf_rn(p.x, w, -q)));
    }
    __device__ __forceinline__ void pair(float &f, float2 a, float2 b) { term(f, product(a, b)); }
    static __device__ __forceinline__ float2 flip(float2 p, unsigned odd) {
        return make_float2(flip_sign(p.x, odd), flip_sign(p.y, odd));
    }
    __device__ __forceinline__ void add(float a, float b) {
        float g = 0.5f * a, e = 0.f;
        add_keep(g, e, 0.5f * b);
        h += (double)g;
        l = __fmaf_rn(2.0f, e, l);
    }
    __device__ __forceinline__ double value() const { return 2.0 * h + (double)l; }
};

// Parity words of 4096-amplitude tiles: tile word from byte tables over bits 12.., thread word
// over bits 0..7, register columns over bits 8..11.
struct TileParity {
    uint32_t ta, tb;          // thread
    uint32_t ra[RB], rb[RB];  // register bits
};

__device__ __forceinline__ void load_tile_parity(TileParity &q, uint2 *tab, const uint32_t *colA, const uint32_t *colB,
                                                 int n) {
    const int t = threadIdx.x;
    for (int e = t; e < 3 * 256; e += blockDim.x) {
        uint32_t a = 0, b = 0;
        for (int j = 0; j < 8; ++j) {
            const int bit = LT + 8 * (e >> 8) + j;
            if (bit < n && ((e >> j) & 1)) { a ^= colA[bit]; b ^= colB[bit]; }
        }
        tab[e] = make_uint2(a, b);
    }
    q.ta = q.tb = 0;
#pragma unroll
    for (int j = 0; j < TB; ++j)
        if ((t >> j) & 1) { q.ta ^= colA[j]; q.tb ^= colB[j]; }
#pragma unroll
    for (int k = 0; k < RB; ++k) { q.ra[k] = colA[TB + k]; q.rb[k] = colB[TB + k]; }
}

__device__ __forceinline__ void tile_word(const uint2 *tab, long long tile, uint32_t &a, uint32_t &b) {
    const uint2 x = tab[tile & 255], y = tab[256 + ((tile >> 8) & 255)], z = tab[512 + ((tile >> 16) & 255)];
    a = x.x ^ y.x ^ z.x;
    b = x.y ^ y.y ^ z.y;
}

// partial sums [norm, sum_i p_i (nA - 2 oddA(i)), sum_i p_i (nB - 2 oddB(i)), <Z_zmask>], p = |psi|^2
// (the middle two only if SUMS, the last only if Z).  27 qubits in complex64: 0.17 ms, 0.22 with
// a Z string, 0.36 with the sums (0.16 at the measured copy rate; 0.15, 0.16 and 0.18 with rounded
// products in runs of eight); 0.66 ms with four table look-ups per amplitude and an FP64 add
// per eight amplitudes and value.  24 qubits in complex128 (FP64-bound): 0.10 ms for the norm,
// 0.31 before.
template <typename R, bool SUMS, bool Z>
__global__ void __launch_bounds__(RED_THREADS) k_reduce_diag(const typename C2<R>::T *__restrict__ psi, int n,
                                                            long long state_stride, const uint32_t *__restrict__ colA,
                                                            const uint32_t *__restrict__ colB, int nA, int nB,
                                                            unsigned long long zmask, double *__restrict__ partials) {
    using V = typename C2<R>::T;
    __shared__ uint2 tab[3 * 256];
    __shared__ R wt[2][33];
    TileParity q;
    if (SUMS) {
        load_tile_parity(q, tab, colA, colB, n);
        load_weights<R>(wt, nA, nB);
    }
    __syncthreads();
    psi += (long long)blockIdx.y * state_stride;
    const int t = threadIdx.x;
    const long long dim = 1ll << n, ntiles = n > LT ? dim >> LT : 1;
    const unsigned zt = __popc(t & (unsigned)zmask & 255u);
    Runs<R> acc[4] = {};
    for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const V *p0 = psi + (tile << LT) + t;
        V v[NR];
#pragma unroll
        for (int r = 0; r < NR; ++r)
            v[r] = n >= LT || (r << TB) + t < dim ? p0[r << TB] : mk<R>((R)0, (R)0);
        uint32_t ta = 0, tb = 0;
        if (SUMS) { tile_word(tab, tile, ta, tb); ta ^= q.ta; tb ^= q.tb; }
        const unsigned zz = zt + __popcll(((unsigned long long)tile << LT) & zmask);
        R f[2][4] = {};
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            const int k8 = Runs<R>::run(r);
            const typename Runs<R>::T p = product(v[r], v[r]);
            acc[0].term(f[k8][0], p);
            if (SUMS) {
                uint32_t a = ta, b = tb;
#pragma unroll
                for (int k = 0; k < RB; ++k)
                    if ((r >> k) & 1) { a ^= q.ra[k]; b ^= q.rb[k]; }
                acc[1].term(f[k8][1], p, weight(wt[0], (R)nA, __popc(a)));
                acc[2].term(f[k8][2], p, weight(wt[1], (R)nB, __popc(b)));
            }
            if (Z) acc[3].term(f[k8][3], Runs<R>::flip(p, (zz + __popc((unsigned)(zmask >> TB) & (unsigned)r)) & 1u));
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (k == 0 || (SUMS && k < 3) || (Z && k == 3)) acc[k].add(f[0][k], f[1][k]);
    }
    double out[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) out[k] = acc[k].value();
    block_store<4>(out, partials + ((long long)blockIdx.y * gridDim.x + blockIdx.x) * RED_NV);
}

// <X_mask> (mask != 0): twice the real part over the pairs, each visited once at its member
// with the mask's top bit clear: 0.15 ms at 27 qubits in complex64, 0.49 when every amplitude
// fetched its partner; 0.06 and 0.21 at 24 qubits in complex128.
template <typename R>
__global__ void __launch_bounds__(RED_THREADS) k_reduce_xpair(const typename C2<R>::T *__restrict__ psi, int n,
                                                             long long state_stride, unsigned long long mask, int top,
                                                             double *__restrict__ partials) {
    using V = typename C2<R>::T;
    psi += (long long)blockIdx.y * state_stride;
    const long long pairs = 1ll << (n - 1), low = (1ll << top) - 1;
    const long long stride = (long long)gridDim.x * RED_THREADS;
    Runs<R> acc = {};
    for (long long j0 = blockIdx.x * (long long)RED_THREADS + threadIdx.x; j0 < pairs; j0 += stride * RED_RUN) {
        V x[RED_RUN], y[RED_RUN];
#pragma unroll
        for (int u = 0; u < RED_RUN; ++u) {
            const long long j = j0 + u * stride;
            const long long i = ((j & ~low) << 1) | (j & low);
            x[u] = j < pairs ? psi[i] : mk<R>((R)0, (R)0);
            y[u] = j < pairs ? psi[i ^ (long long)mask] : mk<R>((R)0, (R)0);
        }
        R f = 0;
#pragma unroll
        for (int u = 0; u < RED_RUN; ++u) acc.pair(f, x[u], y[u]);
        acc.add(f, (R)0);
    }
    double out[2] = {2.0 * acc.value(), 0.0};
    block_store<2>(out, partials + ((long long)blockIdx.y * gridDim.x + blockIdx.x) * RED_NV);
}

// sum_i conj(a_i) b_i (re, im)
template <typename R>
__global__ void __launch_bounds__(RED_THREADS) k_reduce_dot(const typename C2<R>::T *__restrict__ a,
                                                           const typename C2<R>::T *__restrict__ b, int n,
                                                           long long state_stride, double *__restrict__ partials) {
    using V = typename C2<R>::T;
    a += (long long)blockIdx.y * state_stride;
    b += (long long)blockIdx.y * state_stride;
    const long long dim = 1ll << n;
    const long long stride = (long long)gridDim.x * RED_THREADS;
    Runs<R> re = {}, im = {};
    for (long long i0 = blockIdx.x * (long long)RED_THREADS + threadIdx.x; i0 < dim; i0 += stride * RED_RUN) {
        V x[RED_RUN], y[RED_RUN];
#pragma unroll
        for (int u = 0; u < RED_RUN; ++u) {
            const long long i = i0 + u * stride;
            x[u] = i < dim ? a[i] : mk<R>((R)0, (R)0);
            y[u] = i < dim ? b[i] : mk<R>((R)0, (R)0);
        }
        R f0 = 0, f1 = 0;
#pragma unroll
        for (int u = 0; u < RED_RUN; ++u) {
            re.pair(f0, x[u], y[u]);
            im.pair(f1, mk<R>(x[u].x, -x[u].y), mk<R>(y[u].y, y[u].x));
        }
        re.add(f0, (R)0);
        im.add(f1, (R)0);
    }
    double out[2] = {re.value(), im.value()};
    block_store<2>(out, partials + ((long long)blockIdx.y * gridDim.x + blockIdx.x) * RED_NV);
}

// ---------------------------------------------------------------------------
// Every term of <H> in one launch: partials [norm, sum Z_A, sum Z_B, sum X of class 0, of class
// 1, 0, 0, 0].  Blocks take roles by blockIdx.x: pass p's tiles (pairs of the pass's qubits in
// registers, through shared memory in the three stage layouts; the first pass also the
// diagonal sums), then the X strings that no tile holds (stars of the unitary gauge; below 12
// qubits all X terms, and the diagonal ones in a role of their own).  One read per pass plus
// half a read per string.  27 qubits in complex64: 0.79 ms (three reads, 0.48 at the copy rate; the
// exact diagonal sums cost the first pass its registers: 0.68 with rounded products), 1.5 with a
// diagonal pass of its own; 24 qubits with twelve stars 0.30 ms, in complex128 1.35 (FP64 pipe; 1.8
// when tiles whose partner visits a string's pairs did not skip it), 4.2 with a reduction per
// star; 18 qubits with nine stars 25 us in two launches, 150 in 24.
// EXACT (complex64): the pairs of the tiles' qubits without rounding error too, ten times their
// FP32 operations: for states of up to 20 qubits, where a call is launches and latency (at most
// 6 us more), and for the mean fields of a scan, which were reductions per qubit.  18 qubits:
// sigma^x energy 1.3e-8 -> 1e-15 from 64 bits.
// ---------------------------------------------------------------------------
constexpr int EN_NV = 8;
constexpr int EN_MASKS = 64;

struct EnergyParams {
    int n, np, gp, gm;             // qubits, passes, blocks per pass, blocks of the strings
    int nA, nB, nmasks;
    int c[4], next[4], k[4];       // passes: chunk bits, first new qubit, new qubits (first pass 12, 12, 0)
    unsigned long long cls;        // bit q: qubit q is of class 1
    unsigned long long mask[EN_MASKS];
    unsigned long long mask_cls;   // bit j: string j is of class 1
};

template <typename R, bool EXACT>
__global__ void __launch_bounds__(NT, sizeof(R) == 4 ? 3 : 2) k_energy(const typename C2<R>::T *__restrict__ psi,
                                                                    long long state_stride,
                                                                    const uint32_t *__restrict__ colA,
                                                                    const uint32_t *__restrict__ colB,
                                                                    const __grid_constant__ EnergyParams P,
                                                                    double *__restrict__ partials) {
    using V = typename C2<R>::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ uint2 tab[3 * 256];
    __shared__ double sh[NT / 32][EN_NV];
    __shared__ R wt[2][33];
    V *tile_s = reinterpret_cast<V *>(smem_raw);
    const int t = threadIdx.x;
    const int roles = P.np * P.gp;
    const int role = (int)blockIdx.x < roles ? (int)blockIdx.x / P.gp : P.np;
    psi += (long long)blockIdx.y * state_stride;
    const long long dim = 1ll << P.n, ntiles = P.n > LT ? dim >> LT : 1;
    const bool diag = role == 0 || (P.np == 0 && (int)blockIdx.x < P.gm);
    TileParity q;
    if (diag) {
        load_tile_parity(q, tab, colA, colB, P.n);
        load_weights<R>(wt, P.nA, P.nB);
    }
    __syncthreads();
    Runs<R> acc[3] = {};           // diagonal sums
    double xs[2] = {0.0, 0.0};     // X terms by class, every pair once
    // norm and diagonal sums of a tile's amplitudes
    auto diag_sums = [&](const V (&v)[NR], long long tau) {
        uint32_t ta, tb;
        tile_word(tab, tau, ta, tb);
        ta ^= q.ta; tb ^= q.tb;
        R f[2][3] = {};
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            const int k8 = Runs<R>::run(r);
            const typename Runs<R>::T p = product(v[r], v[r]);
            uint32_t a = ta, b = tb;
#pragma unroll
            for (int k = 0; k < RB; ++k)
                if ((r >> k) & 1) { a ^= q.ra[k]; b ^= q.rb[k]; }
            acc[0].term(f[k8][0], p);
            acc[1].term(f[k8][1], p, weight(wt[0], (R)P.nA, __popc(a)));
            acc[2].term(f[k8][2], p, weight(wt[1], (R)P.nB, __popc(b)));
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) acc[k].add(f[0][k], f[1][k]);
    };
    if (role < P.np) {
        const int c = P.c[role], next = P.next[role];
        auto g = [&](int j) { return j < c ? j : next + (j - c); };   // global bit of tile bit j
        const unsigned rot = role == 0 ? (1u << LT) - 1 : ((1u << LT) - 1) & ~((1u << c) - 1);
        unsigned cls = 0;
        for (int j = 0; j < LT; ++j) cls |= (unsigned)((P.cls >> g(j)) & 1) << j;
        const int mid = next - c, hi = next + P.k[role];
        long long toff = 0, rs[RB];
#pragma unroll
        for (int j = 0; j < TB; ++j)
            if ((t >> j) & 1) toff |= 1ll << g(j);
#pragma unroll
        for (int k = 0; k < RB; ++k) rs[k] = 1ll << g(TB + k);
        auto load = [&](V (&v)[NR], long long tau) {
            const V *p = psi + (((tau & ((1ll << mid) - 1)) << c) | ((tau >> mid) << hi)) + toff;
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                long long off = 0;
#pragma unroll
                for (int k = 0; k < RB; ++k)
                    if ((r >> k) & 1) off += rs[k];
                v[r] = p[off];
            }
        };
        // eight pairs of every register bit; the bits' sums add up with their rounding errors
        // kept in l0, l1 (complex64: two-sum)
        R l0 = 0, l1 = 0;
        auto pairs = [&](const V (&v)[NR], unsigned mask, unsigned cl, R &g0, R &g1) {
#pragma unroll
            for (int k = 0; k < RB; ++k) {
                if (!((mask >> k) & 1u)) continue;
                R s = 0, l = 0;
#pragma unroll
                for (int r = 0; r < NR; ++r) {
                    if ((r >> k) & 1) continue;
                    if constexpr (EXACT) {
                        const float2 p = product(v[r], v[r | (1 << k)]);
                        add_keep(s, l, p.x);
                        l += p.y;
                    } else {
                        s = fma(v[r].y, v[r | (1 << k)].y, fma(v[r].x, v[r | (1 << k)].x, s));
                    }
                }
                if ((cl >> k) & 1u) add_keep(g1, l1, s); else add_keep(g0, l0, s);
                if (EXACT) { if ((cl >> k) & 1u) l1 += l; else l0 += l; }
            }
        };
        const int tlo = t & 15, thi = t >> 4;
        V v[NR], u[NR];
        const int b0 = (int)blockIdx.x - role * P.gp;
        if (sizeof(R) == 4 && b0 < ntiles) load(u, b0);
        for (long long tau = b0; tau < ntiles; tau += P.gp) {
            if (sizeof(R) == 4) {
#pragma unroll
                for (int r = 0; r < NR; ++r) v[r] = u[r];
            } else {
                load(v, tau);
            }
            R g0 = 0, g1 = 0;
            if (role == 0) diag_sums(v, tau);
            pairs(v, rot >> 8, cls >> 8, g0, g1);
#pragma unroll
            for (int r = 0; r < NR; ++r) tile_s[swz(t | (r << TB))] = v[r];
            __syncthreads();
            // complex64: the next tile is on its way during the other two stages
            if (sizeof(R) == 4 && tau + P.gp < ntiles) load(u, tau + P.gp);
            if (rot & 15u) {
#pragma unroll
                for (int r = 0; r < NR; ++r) v[r] = tile_s[swz(r | (t << RB))];
                pairs(v, rot, cls, g0, g1);
            }
            if (rot & 0xf0u) {
#pragma unroll
                for (int r = 0; r < NR; ++r) v[r] = tile_s[swz(tlo | (r << 4) | (thi << 8))];
                pairs(v, rot >> 4, cls >> 4, g0, g1);
            }
            xs[0] += (double)g0;
            xs[1] += (double)g1;
            __syncthreads();
        }
        xs[0] += (double)l0;
        xs[1] += (double)l1;
    } else {
        const int b0 = (int)blockIdx.x - roles;
        for (long long tau = b0; tau < ntiles; tau += P.gm) {
            V v[NR];
            const long long i0 = (tau << LT) + t;
#pragma unroll
            for (int r = 0; r < NR; ++r)
                v[r] = i0 + (r << TB) < dim ? psi[i0 + (r << TB)] : mk<R>((R)0, (R)0);
            if (diag) diag_sums(v, tau);
            for (int j = 0; j < P.nmasks; ++j) {
                const long long m = (long long)P.mask[j];
                const long long top = 1ll << (63 - __clzll(m));
                if (tau & (top >> LT)) continue;     // the partner tile visits the pairs
                R f[2] = {0, 0};
                Runs<R> sum = {};
#pragma unroll
                for (int r0 = 0; r0 < NR; r0 += RED_RUN) {
                    V y[RED_RUN];
#pragma unroll
                    for (int r = 0; r < RED_RUN; ++r) {
                        const long long i = i0 + ((r0 + r) << TB);
                        y[r] = i < dim && !(i & top) ? psi[i ^ m] : mk<R>((R)0, (R)0);
                    }
#pragma unroll
                    for (int r = 0; r < RED_RUN; ++r) sum.pair(f[Runs<R>::run(r0)], v[r0 + r], y[r]);
                }
                sum.add(f[0], f[1]);
                if ((P.mask_cls >> j) & 1) xs[1] += sum.value(); else xs[0] += sum.value();
            }
        }
    }
    const double out[5] = {acc[0].value(), acc[1].value(), acc[2].value(), 2.0 * xs[0], 2.0 * xs[1]};
    const int w = t >> 5;
#pragma unroll
    for (int k = 0; k < EN_NV; ++k) {
        const double x = k < 5 ? warp_sum(out[k < 5 ? k : 0]) : 0.0;
        if ((t & 31) == 0) sh[w][k] = x;
    }
    __syncthreads();
    if (t < EN_NV) {
        double s = 0.0;
        for (int k = 0; k < NT / 32; ++k) s += sh[k][t];
        partials[((long long)blockIdx.y * gridDim.x + blockIdx.x) * EN_NV + t] = s;
    }
}

// res[b * S + v] = sum over the nblk partials [b][blk][S] (fixed order), v < nval
template <int S>
__global__ void __launch_bounds__(RED_THREADS) k_finish(const double *__restrict__ partials, int nblk, int nval,
                                                       double *__restrict__ res) {
    __shared__ double sh[RED_THREADS / 32][S];
    const int b = blockIdx.x, t = threadIdx.x;
    double acc[S];
#pragma unroll
    for (int v = 0; v < S; ++v) acc[v] = 0.0;
    for (int k = t; k < nblk; k += RED_THREADS) {
        const double *p = partials + ((long long)b * nblk + k) * S;
#pragma unroll
        for (int v = 0; v < S; ++v)
            if (v < nval) acc[v] += p[v];
    }
#pragma unroll
    for (int v = 0; v < S; ++v) {
        const double x = warp_sum(acc[v]);
        if ((t & 31) == 0) sh[t >> 5][v] = x;
    }
    __syncthreads();
    if (t < nval) {
        double s = 0.0;
        for (int w = 0; w < RED_THREADS / 32; ++w) s += sh[w][t];
        res[(long long)b * S + t] = s;
    }
}

// ---------------------------------------------------------------------------
// Density of states of Z~ = -sum_l sigma^z_l (Sec. V): weight of the amplitudes with k links
// in sigma^z = -1.  Each thread keeps its own column of bins in shared memory (no atomics) and
// adds one sum per number of links set among its register bits, products and sums in FP64 (bins
// differ by orders of magnitude).  partials[(b * gridDim.x + blk) * nbins + k].  What bounds it
// is the FP64 pipe: 2.3 operations an amplitude; the conversion instruction, of the same rate,
// is replaced by integer operations for floats that are normal or zero.  27 qubits in complex64
// 0.56 ms (1.15 with the instruction, 0.41 with product pairs in two floats, whose bins were up
// to 28 times further off; one FP64 shared-memory atomic per amplitude: 12.5), 24 qubits in
// complex128 0.09 (1.4).
// ---------------------------------------------------------------------------
// |x| of a float that is normal or zero as a double, by integer operations (the conversion
// instruction runs at the FP64 rate), and whether it is such a float
__device__ __forceinline__ double widen(float x) {
    const unsigned u = __float_as_uint(x) & 0x7fffffffu;
    return __hiloint2double((int)(u ? (u >> 3) + 0x38000000u : 0u), (int)(u << 29));
}
__device__ __forceinline__ bool widens(float x) {
    const unsigned u = __float_as_uint(x) & 0x7fffffffu;
    return u == 0u || u - 0x00800000u < 0x7f000000u;
}
__device__ __forceinline__ bool widens(float2 a) { return widens(a.x) && widens(a.y); }
__device__ __forceinline__ bool widens(double2) { return true; }
template <bool FAST> __device__ __forceinline__ double2 as_double(float2 a) {
    return FAST ? make_double2(widen(a.x), widen(a.y)) : make_double2((double)a.x, (double)a.y);
}
template <bool FAST> __device__ __forceinline__ double2 as_double(double2 a) { return a; }

// a thread's 16 amplitudes into its column of bins
template <bool FAST, bool FOLD, typename V>
__device__ __forceinline__ void dos_tile(const V (&v)[NR], double *col, unsigned reg) {
    double s[RB + 1] = {0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        const double2 a = as_double<FAST>(v[r]);
        double *bin = &col[__popc((unsigned)r & reg) * RED_THREADS];
        double &sum = FOLD ? s[(r & 1) + ((r >> 1) & 1) + ((r >> 2) & 1) + (r >> 3)] : *bin;
        sum = fma(a.y, a.y, fma(a.x, a.x, sum));
    }
    if (FOLD) {
#pragma unroll
        for (int k = 0; k <= RB; ++k) col[k * RED_THREADS] += s[k];
    }
}

template <typename R>
__global__ void __launch_bounds__(RED_THREADS) k_dos(const typename C2<R>::T *__restrict__ psi, int n,
                                                    long long state_stride, unsigned long long linkmask, int nbins,
                                                    double *__restrict__ partials) {
    using V = typename C2<R>::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *bins = reinterpret_cast<double *>(smem_raw);                   // [nbins][RED_THREADS]
    const int t = threadIdx.x;
    for (int k = 0; k < nbins; ++k) bins[k * RED_THREADS + t] = 0.0;
    psi += (long long)blockIdx.y * state_stride;
    const long long dim = 1ll << n, ntiles = n > LT ? dim >> LT : 1;
    const unsigned reg = (unsigned)(linkmask >> TB) & 15u;                 // links among the register bits
    const int kt = __popc(t & (unsigned)linkmask & 255u);
    for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const V *p0 = psi + (tile << LT) + t;
        V v[NR];
#pragma unroll
        for (int r = 0; r < NR; ++r)
            v[r] = n >= LT || (r << TB) + t < dim ? p0[r << TB] : mk<R>((R)0, (R)0);
        double *col = bins + (kt + __popcll(((unsigned long long)tile << LT) & linkmask)) * RED_THREADS + t;
        bool fast = true;
#pragma unroll
        for (int r = 0; r < NR; ++r) fast = fast && widens(v[r]);
        if (reg == 15u) { if (fast) dos_tile<true, true>(v, col, reg); else dos_tile<false, true>(v, col, reg); }
        else { if (fast) dos_tile<true, false>(v, col, reg); else dos_tile<false, false>(v, col, reg); }
    }
    __syncthreads();
    for (int k = t >> 5; k < nbins; k += RED_THREADS / 32) {
        double s = 0.0;
        for (int j = t & 31; j < RED_THREADS; j += 32) s += bins[k * RED_THREADS + j];
        s = warp_sum(s);
        if ((t & 31) == 0) partials[((long long)blockIdx.y * gridDim.x + blockIdx.x) * nbins + k] = s;
    }
}

// out[b * nval + v] = sum over nblk partials (layout [b][blk][v]), one warp per value, fixed order
__global__ void __launch_bounds__(1024) k_finish_wide(const double *__restrict__ partials, int nblk, int nval,
                                                     double *__restrict__ out) {
    const int b = blockIdx.x, lane = threadIdx.x & 31;
    for (int v = threadIdx.x >> 5; v < nval; v += 32) {
        double s = 0.0;
        for (int k = lane; k < nblk; k += 32) s += partials[((long long)b * nblk + k) * nval + v];
        s = warp_sum(s);
        if (lane == 0) out[(long long)b * nval + v] = s;
    }
}

}  // namespace qsim
