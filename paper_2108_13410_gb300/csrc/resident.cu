// resident.cu -- a whole run of Trotter factor groups in one launch for states that fit the
// chip at one tile per CTA (sm_103a).
//
// With one launch per pass a small state costs about the launch and load latency of each
// pass (8 us for the 2 MiB state of 18 qubits, on 64 of 152 SMs), whatever its arithmetic.
// Here every CTA keeps one tile of 2^M amplitudes per tile set for the whole call:
//   tile set 0: qubits 0..M-1;   tile set 1: qubits M..n-1 above a chunk of the low c =
//   2 M - n qubits (rows of 2^c amplitudes),
// takes its tile through the registers (R tile bits at a time, shared-memory transposes in
// between) and meets the other CTAs of the state only where the tile set changes: every
// amplitude is sent through a mail box in L2 and polled for by its receiver, with no barrier
// of its own (a counter barrier between storing and loading took 4200 of 7300 cycles a pass
// at 18 qubits in complex64).  States of at most 2^M amplitudes never leave their CTA.
//   gauge-Higgs (tangent-form rotations): factor group k ends on the tile set on which
//   group k + 1 begins (Eq. (8): all X-type factors commute), one exchange per group:
//       X(set 0) of group 0 | X(s) of k, Z layer of k, X(s) of k + 1, s = 1, 0, 1, ...
//   unitary gauge (Walsh-Hadamard form H D_X H, Z): two exchanges per group:
//       H(0) | [H(1) D_X H(1)] [H(0) Z H(0)] ...
// Tile size: the chip is filled with about 128 CTAs, so M grows with n (18 qubits: 2^11
// amplitudes on 128 CTAs; fewer bits per CTA would need a third tile set), except that
// complex64 rotations keep the 2^12 tiles and the stage order of the tiled passes.  What
// bounds it: the exchange (4000 of 7000 cycles a pass at 18 qubits in complex64: send, poll,
// skew), FP32 issue in double-float (12000 of 16000 cycles), the FP64 pipe up to 12 qubits.
// Measured per second-order step, one state, against one launch per pass:
//   complex64   12 qubits 3.3 / 6.7 us (gauge-Higgs), 5.2 / 11.4 (unitary gauge); 13 qubits 5.2 /
//               7.1, 7.6 / 12.3; 18 qubits 6.3 / 8.8, 7.8 / 13.5; 19 qubits 10.1 / 15.3
//   complex128  12 qubits 4.6 / 60, 8.1 / 83; 13 qubits 9.9 / 17.9, 14.7 / 23.5; 18 qubits 12.3 /
//               25.0, 17.9 / 37.6; 19 qubits 29.7 / 43.3
// Tables and rotation constants of the next pass are copied from the operator records while a
// pass runs, and the table index of each amplitude (a CTA's tiles do not change) is computed
// once per launch.
// The polls of the mail boxes are bounded (about a second), after which the error flag is set and
// every CTA leaves; the launch is cooperative, so all CTAs of a state are resident.  The named
// barriers inside a CTA have no limit: every warp reaches each of them.
#include "resident.h"

#include "df_arith.cuh"

namespace qsim {

namespace {

constexpr int RES_HEAD = 48;   // bytes of a record before its tables

// ---------------------------------------------------------------------------
// arithmetic: V in registers, S in shared and (between exchanges) in global memory,
// L a phase-table entry, T the tangent of one class
// ---------------------------------------------------------------------------
struct AF32 {
    static constexpr bool ROLLED = false, C_ALONE = true;
    typedef u64 V;
    typedef u64 S;
    typedef float2 G;                      // the caller's layout
    typedef float2 L;                      // (u, s): 8 bytes, fewer bank conflicts than packed pairs
    struct __align__(16) T { u64 p, m; };
    static __device__ __forceinline__ V zero() { return 0ull; }
    static __device__ __forceinline__ V from(S s) { return s; }
    static __device__ __forceinline__ S to(V v) { return v; }
    static __device__ __forceinline__ V first(const G *g) { const float2 x = __ldcg(g); return pk(x.x, x.y); }
    static __device__ __forceinline__ void last(G *g, V v) { __stcg(g, unpk(v)); }
    static __device__ __forceinline__ T tan(double t) { const float f = (float)t; return T{pk(f, f), pk(-f, -f)}; }
    static __device__ __forceinline__ void rot(V &a, V &b, const T &t) {
        const V x = a;
        a = fma2p(t.p, b, x);
        b = fma2p(t.m, x, b);
    }
    static __device__ __forceinline__ void had(V &a, V &b) {
        const V x = a;
        a = add2(x, b);
        b = sub2(x, b);
    }
    static __device__ __forceinline__ L entry(double u, double s) { return make_float2((float)u, (float)s); }
    static __device__ __forceinline__ void phase(V &v, const L *p) {
        const L l = *p;
        v = fma2p(pk(-l.y, l.y), swap2(v), fma2p(pk(-l.x, -l.x), v, v));
    }
    static __device__ __forceinline__ void scale(V &v, float f) { v = mul2(v, pk(f, f)); }
    static __device__ __forceinline__ void ipow(V &v, int k) { const float2 x = mul_ipow(unpk(v), k); v = pk(x.x, x.y); }
    template <int N> static __device__ __forceinline__ void tidy(V (&)[N]) {}
};

struct ADF {
    static constexpr bool ROLLED = true, C_ALONE = false;
    struct V { u64 h, l; };
    typedef ulonglong2 S;
    typedef double2 G;
    typedef DfPhase L;
    struct __align__(16) T { u64 h, l; };
    static __device__ __forceinline__ V zero() { return V{0ull, 0ull}; }
    static __device__ __forceinline__ V from(S s) { return V{s.x, s.y}; }
    static __device__ __forceinline__ S to(const V &v) { return make_ulonglong2(v.h, v.l); }
    static __device__ __forceinline__ V first(const G *g) {
        const double2 x = __ldcg(g);
        float rh, rl, ih, il;
        split_double(x.x, rh, rl);
        split_double(x.y, ih, il);
        return V{pk(rh, ih), pk(rl, il)};
    }
    static __device__ __forceinline__ void last(G *g, const V &v) { __stcg(g, df_join(v.h, v.l)); }
    static __device__ __forceinline__ T tan(double t) {
        const float a = __double2float_rn(t), b = __double2float_rn(t - (double)a);
        return T{pk(a, a), pk(b, b)};
    }
    static __device__ __forceinline__ void rot(V &a, V &b, const T &t) { df_rot_lazy(a.h, a.l, b.h, b.l, t.h, t.l); }
    static __device__ __forceinline__ void had(V &a, V &b) { df_butterfly_lazy(a.h, a.l, b.h, b.l); }
    static __device__ __forceinline__ L entry(double u, double s) {
        const double c = 1.0 - u;
        const float ch = __double2float_rn(c), cl = __double2float_rn(c - (double)ch);
        const float sh = __double2float_rn(s), sl = __double2float_rn(s - (double)sh);
        L q;
        q.ch = pk(ch, ch); q.cl = pk(cl, cl); q.sh = pk(sh, -sh); q.sl = pk(sl, -sl);
        return q;
    }
    static __device__ __forceinline__ void phase(V &v, const L *p) { df_phase(v.h, v.l, *p); }
    static __device__ __forceinline__ void scale(V &v, float f) { const u64 d = pk(f, f); v.h = mul2(v.h, d); v.l = mul2(v.l, d); }
    static __device__ __forceinline__ void ipow(V &v, int k) { df_ipow(v.h, v.l, k); }
    // |l| <= ulp(h) / 2 again, before a table product and before a store
    template <int N> static __device__ __forceinline__ void tidy(V (&v)[N]) {
#pragma unroll
        for (int r = 0; r < N; ++r) {
            const u64 nh = add2(v[r].h, v[r].l);
            v[r].l = sub2(v[r].l, sub2(nh, v[r].h));
            v[r].h = nh;
        }
    }
};

// complex64 states carried in double-float during the call
struct ADF32 : ADF {
    typedef float2 G;
    static __device__ __forceinline__ V first(const G *g) { const float2 x = __ldcg(g); return V{pk(x.x, x.y), 0ull}; }
    static __device__ __forceinline__ void last(G *g, const V &v) {
        const float2 h = unpk(v.h), l = unpk(v.l);
        __stcg(g, make_float2(h.x + l.x, h.y + l.y));
    }
};

struct AF64 {
    static constexpr bool ROLLED = false, C_ALONE = false;
    typedef double2 V;
    typedef double2 S;
    typedef double2 G;
    typedef double2 L;                     // (u, s)
    struct __align__(16) T { double t, pad; };
    static __device__ __forceinline__ V zero() { return make_double2(0.0, 0.0); }
    static __device__ __forceinline__ V from(S s) { return s; }
    static __device__ __forceinline__ S to(V v) { return v; }
    static __device__ __forceinline__ V first(const G *g) { return __ldcg(g); }
    static __device__ __forceinline__ void last(G *g, V v) { __stcg(g, v); }
    static __device__ __forceinline__ T tan(double t) { return T{t, 0.0}; }
    static __device__ __forceinline__ void rot(V &a, V &b, const T &tt) {
        const V x = a;
        const double t = tt.t;
        a.x = fma(t, b.x, x.x); a.y = fma(t, b.y, x.y);
        b.x = fma(-t, x.x, b.x); b.y = fma(-t, x.y, b.y);
    }
    static __device__ __forceinline__ void had(V &a, V &b) {
        const V x = a;
        a.x = x.x + b.x; a.y = x.y + b.y;
        b.x = x.x - b.x; b.y = x.y - b.y;
    }
    static __device__ __forceinline__ L entry(double u, double s) { return make_double2(u, s); }
    static __device__ __forceinline__ void phase(V &v, const L *p) {
        const L l = *p;
        V r;
        r.x = fma(-l.y, v.y, fma(-l.x, v.x, v.x));
        r.y = fma(l.y, v.x, fma(-l.x, v.y, v.y));
        v = r;
    }
    static __device__ __forceinline__ void scale(V &v, float f) { v.x *= (double)f; v.y *= (double)f; }
    static __device__ __forceinline__ void ipow(V &v, int k) {
        if (k & 1) v = make_double2(-v.y, v.x);
        if (k & 2) v = make_double2(-v.x, -v.y);
    }
    template <int N> static __device__ __forceinline__ void tidy(V (&)[N]) {}
};

// Exchange words: a word that holds EMPTY has not arrived yet.  EMPTY is a signalling NaN as a
// double and in its low half as a float (its high half is a quiet one), which no arithmetic
// result is; everything that is sent comes out of a butterfly or a product, and the whole word is
// compared.
constexpr u64 EMPTY = 0x7ff4dead7fa0deadull;

__device__ __forceinline__ bool arrived(u64 w) { return w != EMPTY; }
__device__ __forceinline__ bool arrived(const ulonglong2 &w) { return w.x != EMPTY && w.y != EMPTY; }
__device__ __forceinline__ bool arrived(const double2 &w) {
    return (u64)__double_as_longlong(w.x) != EMPTY && (u64)__double_as_longlong(w.y) != EMPTY;
}
__device__ __forceinline__ u64 recv(const u64 *p) {
    u64 v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ ulonglong2 recv(const ulonglong2 *p) {
    ulonglong2 v;
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ double2 recv(const double2 *p) {
    double2 v;
    asm volatile("ld.relaxed.gpu.global.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void send(u64 *p, u64 v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ void send(ulonglong2 *p, const ulonglong2 &v) {
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(v.x), "l"(v.y) : "memory");
}
__device__ __forceinline__ void send(double2 *p, const double2 &v) {
    asm volatile("st.relaxed.gpu.global.v2.f64 [%0], {%1, %2};" ::"l"(p), "d"(v.x), "d"(v.y) : "memory");
}
__device__ __forceinline__ void clear(u64 *p) { send(p, EMPTY); }
__device__ __forceinline__ void clear(ulonglong2 *p) { send(p, make_ulonglong2(EMPTY, EMPTY)); }
__device__ __forceinline__ void clear(double2 *p) { clear(reinterpret_cast<ulonglong2 *>(p)); }

__device__ __forceinline__ void copy_async16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void copy_async_wait() {
    asm volatile("cp.async.wait_all;" ::: "memory");
}
// Named barriers of a CTA.  They take converged warps (aligned forms: a split warp would count
// early, or twice), so lanes that may be apart, after a lane's fence, a copy loop or a poll that
// some lanes leave earlier, meet first.  The workers' own barrier (1) comes after straight-line
// code, except behind the poll, where receive() joins the warp.
template <int ID, int N> __device__ __forceinline__ void barrier_sync() {
    if (ID != 1) __syncwarp();
    asm volatile("bar.sync %0, %1;" ::"n"(ID), "n"(N) : "memory");
}
template <int ID, int N> __device__ __forceinline__ void barrier_arrive() {
    if (ID != 1) __syncwarp();
    asm volatile("bar.arrive %0, %1;" ::"n"(ID), "n"(N) : "memory");
}

// slot of tile amplitude l: the low four bits xor bits 4..7, so that 16 (8) consecutive
// lanes of every stage layout hit different 8-byte (16-byte) bank groups
__device__ __forceinline__ int slot(int l) { return l ^ ((l >> 4) & 15); }

// butterflies on the register bits of `mask`; bit k of `cls`: class of register bit k
template <class A, int R, bool HAD>
__device__ __forceinline__ void butterflies(typename A::V (&v)[1 << R], unsigned mask, unsigned cls,
                                            const typename A::T *tc) {
#pragma unroll
    for (int k = 0; k < R; ++k) {
        if (!((mask >> k) & 1u)) continue;
        if (HAD) {
#pragma unroll
            for (int r = 0; r < (1 << R); ++r)
                if (!((r >> k) & 1)) A::had(v[r], v[r | (1 << k)]);
        } else {
            const typename A::T t = tc[(cls >> k) & 1u];
#pragma unroll
            for (int r = 0; r < (1 << R); ++r)
                if (!((r >> k) & 1)) A::rot(v[r], v[r | (1 << k)], t);
        }
    }
}

// The registers and tile buffers of one CTA.  Stage s: registers hold tile bits base(s) ..
// base(s) + R - 1, and it rotates the bits from s R on (the top stage may overlap the one
// below).  In double-float arithmetic the stages run in a rolled loop around one copy of the
// butterflies (straight-line code for each of them ran 1.3 times slower: instruction fetch);
// the others, with a tenth of its instructions, are faster unrolled.
template <class A, int M, int R, bool HAD>
struct Worker {
    typedef typename A::V V;
    typedef typename A::S S;
    static constexpr int N = 1 << M, NTH = 1 << (M - R), NRG = 1 << R, NS = (M + R - 1) / R;
    V v[NRG];
    S *tile;                       // two buffers used in turn: one barrier per transpose
    int t, buf;

    static __host__ __device__ constexpr int base(int s) { return s * R < M - R ? s * R : M - R; }
    static __device__ __forceinline__ int pos(int t, int r, int b) {
        return (t & ((1 << b) - 1)) | (r << b) | ((t >> b) << (b + R));
    }
    __device__ __forceinline__ void sync() { barrier_sync<1, NTH>(); }
    // registers from the layout of stage SF to that of stage ST
    template <int SF, int ST> __device__ __forceinline__ void move() {
        S *p = tile + buf * N;
        buf ^= 1;
#pragma unroll
        for (int r = 0; r < NRG; ++r) p[slot(pos(t, r, base(SF)))] = A::to(v[r]);
        sync();
#pragma unroll
        for (int r = 0; r < NRG; ++r) v[r] = A::from(p[slot(pos(t, r, base(ST)))]);
    }
    template <int ST> __device__ __forceinline__ void move_down(int to) {      // from stage to + 1
        if (to == ST) move<ST + 1, ST>();
        else if constexpr (ST + 2 < NS) move_down<ST + 1>(to);
    }
    template <int ST> __device__ __forceinline__ void move_up(int to) {        // from stage to - 1
        if (to == ST) move<ST - 1, ST>();
        else if constexpr (ST + 1 < NS) move_up<ST + 1>(to);
    }
    template <int ST> __device__ __forceinline__ void to_top(int from) {       // to stage NS - 1
        if (from == ST) move<ST, NS - 1>();
        else if constexpr (ST + 2 < NS) to_top<ST + 1>(from);
    }
    // from the layout that a round ends in (stage 0, or 1 in 2^12 tiles) to its first stage
    template <int ST> __device__ __forceinline__ void to_first(int from, int to) {
        if (to == ST) { if (from) move<1, ST>(); else move<0, ST>(); }
        else if constexpr (ST + 1 < NS) to_first<ST + 1>(from, to);
    }
    template <int ST> __device__ __forceinline__ void from_top(int to) {
        if (to == ST) move<NS - 1, ST>();
        else if constexpr (ST + 2 < NS) from_top<ST + 1>(to);
    }
    template <int ST> __device__ __forceinline__ void stage(unsigned mask, unsigned cls, const typename A::T *tc) {
        butterflies<A, R, HAD>(v, (mask & ~((1u << (ST * R)) - 1)) >> base(ST), cls >> base(ST), tc);
    }
    template <int ST> __device__ __forceinline__ void down_from(int hi, int lo, unsigned mask, unsigned cls,
                                                                const typename A::T *tc) {
        if (ST <= hi && ST >= lo) {
            if constexpr (ST + 1 < NS) { if (ST != hi) move<ST + 1, ST>(); }
            stage<ST>(mask, cls, tc);
        }
        if constexpr (ST > 0) down_from<ST - 1>(hi, lo, mask, cls, tc);
    }
    template <int ST> __device__ __forceinline__ void up_from(int hi, int lo, unsigned mask, unsigned cls,
                                                              const typename A::T *tc) {
        if (ST <= hi && ST >= lo) {
            if constexpr (ST > 0) { if (ST != lo) move<ST - 1, ST>(); }
            stage<ST>(mask, cls, tc);
        }
        if constexpr (ST + 1 < NS) up_from<ST + 1>(hi, lo, mask, cls, tc);
    }
    // one round over stages hi .. lo (up = 0) or lo .. hi (up = 1); registers start in the
    // layout of its first stage and end in that of its last
    __device__ __forceinline__ void round(int up, int hi, int lo, unsigned mask, unsigned cls, const typename A::T *tc) {
        if constexpr (A::ROLLED) {
#pragma unroll 1
            for (int i = 0; i <= hi - lo; ++i) {
                const int st = up ? lo + i : hi - i;
                if (i) { if (up) move_up<1>(st); else move_down<0>(st); }
                const int b = base(st);
                butterflies<A, R, HAD>(v, (mask & ~((1u << (st * R)) - 1)) >> b, cls >> b, tc);
            }
        } else if constexpr (M == 12 && R == 4) {
            // 8..11, 0..3, 4..7 and back: the order of the tiled passes (xpass_tma.cuh), so that
            // every amplitude sees the same operations and complex64 results are the same bits
            if (up) {
                if (lo <= 1) {
                    stage<1>(mask, cls, tc);
                    if (lo == 0) {
                        move<1, 0>();
                        stage<0>(mask, cls, tc);
                        move<0, 2>();
                    } else {
                        move<1, 2>();
                    }
                }
                stage<2>(mask, cls, tc);
            } else {
                stage<2>(mask, cls, tc);
                if (lo <= 1) {
                    if (lo == 0) {
                        move<2, 0>();
                        stage<0>(mask, cls, tc);
                        move<0, 1>();
                    } else {
                        move<2, 1>();
                    }
                    stage<1>(mask, cls, tc);
                }
            }
        } else if (up) {
            up_from<0>(hi, lo, mask, cls, tc);
        } else {
            down_from<NS - 1>(hi, lo, mask, cls, tc);
        }
    }
    // the stage in whose layout a round down to stage lo ends
    static __device__ __forceinline__ int last_of(int lo) { return M == 12 && R == 4 && lo == 0 ? 1 : lo; }
};

// Resident CTAs per SM asked of the compiler: 128 registers a thread (double-float and the
// 2^12 tiles of 19 qubits, which have an SM to themselves: 168; single 2^12 tiles: two per SM).
constexpr int min_ctas(int M, int R, bool df, bool two) {
    return M == 12 ? (two ? 1 : 2) : (df ? 384 : 512) / ((1 << (M - R)) + 32);
}

// Threads 2^(M - R), then one helper warp that loads the table and the tangents of the next
// pass and takes the fence between clearing and sending (1000 cycles) off the workers' path: that
// relies on a fence covering what its thread has observed through a CTA barrier (cumulativity, as
// in a grid barrier, where one thread's fence stands for its block) and on no store of the CTA
// overtaking the barrier behind the fence; the memory model's own release pattern would have every
// sending thread fence.  blockIdx.x = group * tiles + tile of the state.  Named barriers: 1 the workers, 2 a pass has
// received and cleared (workers arrive, helper waits), 3 the next table is there and the
// clears are ordered (helper arrives, workers wait).
template <class A, int M, int R, bool HAD, bool TWO>
__global__ void __launch_bounds__((1 << (M - R)) + 32, min_ctas(M, R, sizeof(typename A::V) == 16, TWO)) k_resident(void *state_v,
                                                         const unsigned char *__restrict__ recs, void *mail_v, int *__restrict__ err_flag,
                                                         const __grid_constant__ ResParams P) {
    typedef Worker<A, M, R, HAD> W;
    typedef typename A::S S;
    typedef typename A::G G;
    typedef typename A::L L;
    constexpr int NTH = W::NTH, NRG = W::NRG, NS = W::NS, N = W::N;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ typename A::T s_t[2][2][2];   // [buffer][this group, the next][class]
    __shared__ float4 s_c[2];                // C of the group (complex64)
    __shared__ int s_ok;
    L *const lut = reinterpret_cast<L *>(smem + 2 * N * sizeof(S));   // two tables
    const int t = threadIdx.x;
    const int grp = TWO ? (int)blockIdx.x / P.tiles : (int)blockIdx.x;
    const long long T = TWO ? (int)blockIdx.x % P.tiles : 0;
    const int n_pass = HAD ? 2 * P.nops : P.nops;
    auto received = [&]() { barrier_arrive<2, NTH + 32>(); };
    auto may_send = [&]() { barrier_sync<3, NTH + 32>(); };
    // end of a state: the tables are free and every barrier-3 phase is over
    auto state_done = [&]() { barrier_sync<2, NTH + 32>(); };
    if (t == 0) s_ok = 1;
    __syncthreads();
    if (t >= NTH) {
        // ---- helper warp ----
        const int lane = t - NTH;
        for (int b = grp; b < P.batch; b += P.groups) {
            auto rec_of = [&](int op) { return recs + ((long long)op * P.batch + b) * P.rec_bytes; };
            for (int k = -1; k < n_pass; ++k) {
                if (k >= 0) {
                    barrier_sync<2, NTH + 32>();
                    if (!*(volatile int *)&s_ok) return;
                }
                if (k + 1 < n_pass) {                          // the table of pass k + 1
                    const int op = HAD ? (k + 1) >> 1 : k + 1;
                    const bool xtab = HAD && !((k + 1) & 1);
                    const int lb = (k + 1) & 1;
                    const unsigned char *r = rec_of(op);
                    const int bytes = xtab ? P.xtab_bytes : P.ztab_bytes;
                    const unsigned char *src = r + (xtab ? RES_HEAD + P.ztab_bytes : RES_HEAD);
                    unsigned char *dst = reinterpret_cast<unsigned char *>(lut) + lb * P.tab_bytes;
                    for (int i = 16 * lane; i < bytes; i += 512) copy_async16(dst + i, src + i);
                    if (!HAD && lane < 4 && op + (lane >> 1) < P.nops)
                        copy_async16(&s_t[lb][lane >> 1][lane & 1], rec_of(op + (lane >> 1)) + 16 * (lane & 1));
                    if (!HAD && lane == 4) copy_async16(&s_c[lb], r + 32);
                }
                if (TWO && lane == 0 && k >= 0) __threadfence();
                copy_async_wait();
                barrier_arrive<3, NTH + 32>();
            }
            state_done();
        }
        return;
    }
    W w;
    w.t = t;
    w.buf = 0;
    w.tile = reinterpret_cast<S *>(smem);

    // rotated tile bits [rlo, rhi) of each set, its stages lo .. hi
    const int rhi = TWO ? M : P.n;
    const unsigned mask0 = (1u << rhi) - 1, mask1 = mask0 & ~((1u << P.c) - 1);
    const int lo1 = P.c / R, hi = TWO ? NS - 1 : (P.n - 1) / R;
    const unsigned cls0 = P.cls & ((1u << M) - 1), cls1 = TWO ? (P.cls >> M) << P.c : 0u;
    const long long cm = (1ll << P.c) - 1;
    auto addr = [&](int set, long long l) -> long long {
        return !TWO || set == 0 ? (T << M) | l : (l & cm) | (T << P.c) | ((l >> P.c) << M);
    };
    // table index of this thread's amplitudes in the layout of stage `st` of a set: parity words
    // of the thread's bits and of each register bit
    auto codes = [&](uint32_t (&code)[NRG / 2], int set, int st, const uint32_t *ca, const uint32_t *cb, int nb1) {
        const int b = st * R < M - R ? st * R : M - R;
        const unsigned g0 = (unsigned)addr(set, W::pos(t, 0, b));
        uint32_t wa[NRG], wb[NRG];
        wa[0] = wb[0] = 0;
        for (int q = 0; q < P.n; ++q)
            if ((g0 >> q) & 1) { wa[0] ^= ca[q]; wb[0] ^= cb[q]; }
#pragma unroll
        for (int k = 0; k < R; ++k) {
            const int l = b + k, q = !TWO || set == 0 || l < P.c ? l : M + l - P.c;
            const uint32_t xa = ca[q], xb = cb[q];       // (zero beyond the qubits)
#pragma unroll
            for (int r = 0; r < (1 << k); ++r) { wa[r | (1 << k)] = wa[r] ^ xa; wb[r | (1 << k)] = wb[r] ^ xb; }
        }
#pragma unroll
        for (int r = 0; r < NRG; r += 2)
            code[r >> 1] = (uint32_t)(__popc(wa[r]) * nb1 + __popc(wb[r])) |
                           (uint32_t)(__popc(wa[r + 1]) * nb1 + __popc(wb[r + 1])) << 16;
    };
    // Z tables: set 0 (two sets) or the layout that a round ends in; X tables (unitary gauge)
    // on set 1 or the low layout
    uint32_t code0[NRG / 2], code1[NRG / 2];
    if (TWO) {
        codes(code0, 0, W::last_of(0), P.colA, P.colB, P.nB + 1);
        if (HAD) codes(code1, 1, W::last_of(lo1), P.xcolA, P.xcolB, P.nXB + 1);
        else codes(code1, 1, W::last_of(lo1), P.colA, P.colB, P.nB + 1);
    } else {
        codes(code0, 0, W::last_of(0), P.colA, P.colB, P.nB + 1);
        if (HAD) codes(code1, 0, W::last_of(0), P.xcolA, P.xcolB, P.nXB + 1);
    }
    const float xscale = __int_as_float((127 - P.n) << 23);   // 2^-n of the two transforms
    auto diag = [&](const uint32_t (&code)[NRG / 2], int lb) {
        A::tidy(w.v);
        const L *p = reinterpret_cast<const L *>(reinterpret_cast<const unsigned char *>(lut) + lb * P.tab_bytes);
#pragma unroll
        for (int r = 0; r < NRG; ++r) A::phase(w.v[r], p + ((code[r >> 1] >> (16 * (r & 1))) & 0xffffu));
    };
    // the group's cos factors alone, rounded once (a group without Z layer)
    auto c_scale = [&](int lb) {
        const float c = s_c[lb].x;
#pragma unroll
        for (int r = 0; r < NRG; ++r) A::scale(w.v[r], c);
    };
    auto x_scale = [&]() {
#pragma unroll
        for (int r = 0; r < NRG; ++r) A::scale(w.v[r], xscale);
    };

    int box = 0;                   // mail box of the next exchange
    bool ok = true;
    for (int b = grp; b < P.batch && ok; b += P.groups) {
        G *psi = reinterpret_cast<G *>(state_v) + ((long long)b << P.n);
        // the caller's amplitudes <-> registers in the top layout (gauge-Higgs: in the frame
        // i^popc psi)
        auto load_first = [&]() {
#pragma unroll
            for (int r = 0; r < NRG; ++r) {
                const int l = W::pos(t, r, M - R);
                const long long g = addr(0, l);
                if (TWO || g < (1ll << P.n)) {
                    w.v[r] = A::first(psi + g);
                    if (!HAD) A::ipow(w.v[r], __popcll((unsigned long long)g));
                } else {
                    w.v[r] = A::zero();
                }
            }
        };
        auto store_last = [&](int set) {
#pragma unroll
            for (int r = 0; r < NRG; ++r) {
                const int l = W::pos(t, r, M - R);
                const long long g = addr(set, l);
                if (TWO || g < (1ll << P.n)) {
                    if (!HAD) A::ipow(w.v[r], (-__popcll((unsigned long long)g)) & 3);
                    A::last(psi + g, w.v[r]);
                }
            }
        };
        load_first();
        may_send();                    // table 0
        if (!TWO) {
            // ---- one tile: the state stays in registers and shared memory ----
            const int end = W::last_of(0);
            if (hi != NS - 1) w.template from_top<0>(hi);
#pragma unroll 1
            for (int k = 0; k < n_pass; ++k) {
                received();
                if (k && hi != end) w.template to_first<1>(end, hi);
                w.round(0, hi, 0, mask0, cls0, s_t[k & 1][0]);
                if (A::C_ALONE && !HAD && k + 1 == n_pass && !P.last_z) c_scale(k & 1);
                else if (HAD && !(k & 1)) diag(code1, 0);
                else diag(code0, k & 1);
                if (HAD && !(k & 1)) x_scale();
                may_send();
            }
            A::tidy(w.v);
            if (end != NS - 1) w.template to_top<0>(end);
            store_last(0);
            state_done();
            continue;
        }
        // ---- two tile sets ----
        // Exchange through one of two mail boxes (indexed by amplitude), used in turn: send
        // the tile of one set, receive the tile of the other, clear what was received.  A
        // box is written again two exchanges later by CTAs that have received, in between,
        // what its reader sent after clearing it; the fence between clearing and sending
        // (and between receiving and sending) orders the two.
        S *const mail = reinterpret_cast<S *>(mail_v) + ((long long)grp << P.n);
        const long long box_size = (long long)P.groups << P.n;
        auto first_of = [&](int set) { return addr(set, W::pos(t, 0, M - R)); };
        // offset of register r from there (the chunk may reach into the register bits)
        auto off_of = [&](int set, int r) -> long long {
            const long long l = (long long)r << (M - R);
            return set == 0 ? l : (l & cm) | ((l >> P.c) << M);
        };
        auto receive = [&](int set) -> bool {
            S *p = mail + box * box_size + first_of(set);
            S x[NRG];
#pragma unroll
            for (int r = 0; r < NRG; ++r) x[r] = recv(p + off_of(set, r));
            const long long t0 = clock64();
            for (;;) {
                bool all = true;
#pragma unroll
                for (int r = 0; r < NRG; ++r)
                    if (!arrived(x[r])) { all = false; x[r] = recv(p + off_of(set, r)); }
                if (all) break;
                if (clock64() - t0 > P.wait) {
                    atomicOr(err_flag, 1);
                    s_ok = 0;
                    break;
                }
            }
#pragma unroll
            for (int r = 0; r < NRG; ++r) { clear(p + off_of(set, r)); w.v[r] = A::from(x[r]); }
            __syncwarp();
            w.sync();
            received();
            return *(volatile int *)&s_ok != 0;
        };
#pragma unroll 1
        for (int k = -1; k < n_pass; ++k) {
            const int set = (k + 1) & 1;
            if (k >= 0) {
                ok = receive(set);
                if (!ok) break;
                box ^= 1;
            }
            const int lo = set ? lo1 : 0;
            const unsigned mask = set ? mask1 : mask0, cls = set ? cls1 : cls0;
            const bool last = k + 1 == n_pass;
            const int lb = k & 1;
#pragma unroll 1
            for (int up = 0; up < 2; ++up) {
                if (up && (last || k < 0)) {
                    if (W::last_of(lo) != NS - 1) w.template to_top<0>(W::last_of(lo));
                    break;
                }
                w.round(up, NS - 1, lo, mask, cls, s_t[k < 0 ? 0 : lb][up]);
                if (!up && k >= 0) {
                    if (A::C_ALONE && !HAD && last && !P.last_z) c_scale(lb);
                    else if (set) diag(code1, lb);
                    else diag(code0, lb);
                    if (HAD && set) x_scale();
                }
            }
            A::tidy(w.v);
            if (k >= 0) may_send();
            if (last) {
                store_last(set);
            } else {
                S *q = mail + box * box_size + first_of(set);
#pragma unroll
                for (int r = 0; r < NRG; ++r) send(q + off_of(set, r), A::to(w.v[r]));
            }
        }
        // (a wait that gave up: the helper has left at this pass's barrier 2)
        if (ok) state_done();
    }
}

// Operator records of the resident kernel: per factor group and state two tangents and the
// group's cos factors C as a float (16 bytes each), the Z table (scaled by the group's cos factors in the tangent form) and the
// Hadamard-basis X table, entries in the kernel's own format.  Geometry as k_build_records.
template <class A, bool INLINE>
__global__ void __launch_bounds__(64) k_resident_tables(RecGeom G, const double *__restrict__ in, size_t ncpl,
                                                        const __grid_constant__ RecInline X, int op0,
                                                        unsigned char *__restrict__ recs,
                                                        const __grid_constant__ ResParams P) {
    const double *src = INLINE ? X.v : in;
    const DevCouplings *cpl = reinterpret_cast<const DevCouplings *>(src);
    const double *sv = src + 4 * ncpl;
    const long long ob = blockIdx.x;
    const int op = op0 + (int)(ob / G.batch), b = (int)(ob % G.batch);
    __shared__ double tri[2][2];        // per X class: t, (1 + t^2)^n
    double thx[2], zA, zB;
    bool has_z;
    dev_op_angles(G, cpl, b, sv, op, thx, &zA, &zB, &has_z);
    if (!P.had && threadIdx.x < 2)
        dev_tan(G.f32, thx[threadIdx.x], threadIdx.x ? G.nX1 : G.nX0, &tri[threadIdx.x][0], &tri[threadIdx.x][1]);
    __syncthreads();
    const double C = P.had ? 1.0 : 1.0 / sqrt(tri[0][1] * tri[1][1]);
    unsigned char *r = recs + ob * P.rec_bytes;
    if (!P.had && blockIdx.y == 0 && threadIdx.x < 2)
        reinterpret_cast<typename A::T *>(r)[threadIdx.x] = A::tan(tri[threadIdx.x][0]);
    if (!P.had && blockIdx.y == 0 && threadIdx.x == 2)
        *reinterpret_cast<float4 *>(r + 32) = make_float4((float)C, 0.f, 0.f, 0.f);
    const int nz = (P.nA + 1) * (P.nB + 1), nx = P.had ? (P.nXA + 1) * (P.nXB + 1) : 0;
    for (int e = blockIdx.y * 64 + threadIdx.x; e < nz + nx; e += gridDim.y * 64) {
        const bool x = e >= nz;
        const int k = x ? e - nz : e, nb1 = (x ? P.nXB : P.nB) + 1;
        const int a = k / nb1, bb = k % nb1;
        double phi, u, s;
        if (x) phi = thx[1] * (double)(P.nXA - 2 * a) + thx[0] * (double)(P.nXB - 2 * bb);
        else phi = has_z ? zA * (double)(P.nA - 2 * a) + zB * (double)(P.nB - 2 * bb) : 0.0;
        if (P.had) dev_unit_pair(G.f32, phi, &u, &s);
        else dev_scaled_pair(G.f32, phi, C, &u, &s);
        reinterpret_cast<typename A::L *>(r + RES_HEAD + (x ? P.ztab_bytes : 0))[k] = A::entry(u, s);
    }
}

__global__ void k_mail_clear(u64 *mail, long long words) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < words; i += (long long)gridDim.x * blockDim.x)
        mail[i] = EMPTY;
}

typedef void (*ResKernel)(void *, const unsigned char *, void *, int *, const ResParams);

template <class A, int M, int R>
ResKernel pick(bool had, bool two) {
    if (two) return had ? k_resident<A, M, R, true, true> : k_resident<A, M, R, false, true>;
    return had ? k_resident<A, M, R, true, false> : k_resident<A, M, R, false, false>;
}

// (two sets of rotations take 2^12 tiles)
template <int M>
ResKernel pick32(bool had, bool two) {
    if (two) return had ? k_resident<AF32, M, 4, true, true> : nullptr;
    return had ? k_resident<AF32, M, 4, true, false> : k_resident<AF32, M, 4, false, false>;
}

size_t entry_bytes(int arith) {
    return arith == RES_F32 ? sizeof(AF32::L) : arith == RES_F64 ? sizeof(AF64::L) : sizeof(ADF::L);
}

// complex64 and double-float: 16 amplitudes per thread; FP64: 2 per thread, since the FP64
// pipe (two FMAs per clock per SM) needs warps, not work per thread
ResKernel kernel_of(const ResParams &P, int *threads, size_t *smem, size_t tab_bytes) {
    const size_t lut = 2 * tab_bytes;
    const size_t N = (size_t)1 << P.M;
    if (P.arith == RES_F64) {
        *threads = 64 + 32;
        *smem = 2 * N * 16 + lut;
        return P.M == 7 ? pick<AF64, 7, 1>(P.had, P.two) : nullptr;
    }
    *threads = (int)(N >> 4) + 32;
    if (P.arith == RES_DF32) {
        *smem = 2 * N * 16 + lut;
        if (P.two || !P.had) return nullptr;
        return P.M == 9 ? k_resident<ADF32, 9, 4, true, false>
                        : P.M == 10 ? k_resident<ADF32, 10, 4, true, false> : k_resident<ADF32, 11, 4, true, false>;
    }
    if (P.arith == RES_DF) {
        *smem = 2 * N * 16 + lut;
        if (!P.two) return nullptr;
        switch (P.M) {
            case 9: return P.had ? k_resident<ADF, 9, 4, true, true> : k_resident<ADF, 9, 4, false, true>;
            case 10: return P.had ? k_resident<ADF, 10, 4, true, true> : k_resident<ADF, 10, 4, false, true>;
            case 11: return P.had ? k_resident<ADF, 11, 4, true, true> : k_resident<ADF, 11, 4, false, true>;
        }
        return nullptr;
    }
    *smem = 2 * N * 8 + lut;
    switch (P.M) {
        case 9: return pick32<9>(P.had, P.two);
        case 10: return pick32<10>(P.had, P.two);
        case 11: return pick32<11>(P.had, P.two);
        case 12: return pick<AF32, 12, 4>(P.had, P.two);
    }
    return nullptr;
}

constexpr size_t ONE_PER_SM = 116 * 1024;   // more than half of an SM's 227 KB

}  // namespace

bool resident_plan(ResParams &P, int arith, int n, int batch, int sm_count) {
    if (n > RES_MAXQ || n < 2 || batch < 1) return false;
    P.arith = arith;
    P.n = n;
    int M, lo, hi;
    if (arith == RES_F64) { lo = hi = 7; }
    else { lo = 9; hi = arith == RES_F32 ? 12 : 11; }
    const int one = arith == RES_F64 ? 7 : arith == RES_DF ? 0 : arith == RES_DF32 ? 11 : 12;   // largest single tile
    P.two = n > one;
    if (!P.two) M = n < lo ? lo : n;
    else {
        M = (n + 3) / 2;                       // a chunk of at least two qubits
        if (M < n - 7) M = n - 7;              // about 128 CTAs
        if (M < lo) M = lo;
        if (M > hi) M = hi;
        // complex64 rotations: the tiled passes' tile and order, hence their bits (2^11 tiles
        // take 5.9 instead of 6.3 us a step at 18 qubits, but round in another order, and the
        // norm of a smooth state drifts with the order: 1.1e-6 over 1500 steps)
        if (arith == RES_F32 && !P.had) M = 12;
        if (2 * M < n + 2 || M >= n) return false;
    }
    P.M = M;
    P.c = P.two ? 2 * M - n : 0;
    P.tiles = P.two ? 1 << (n - M) : 1;
    const size_t eb = entry_bytes(arith);
    P.ztab_bytes = (int)(((size_t)(P.nA + 1) * (P.nB + 1) * eb + 15) & ~(size_t)15);
    P.xtab_bytes = P.had ? (int)(((size_t)(P.nXA + 1) * (P.nXB + 1) * eb + 15) & ~(size_t)15) : 0;
    P.tab_bytes = P.ztab_bytes > P.xtab_bytes ? P.ztab_bytes : P.xtab_bytes;
    P.rec_bytes = RES_HEAD + P.ztab_bytes + P.xtab_bytes;
    int threads = 0;
    size_t smem = 0;
    // (the limit for the largest tables, 33 x 33 entries, and at least the size that one CTA
    // per SM takes below: every lattice sets the same one)
    ResKernel k = kernel_of(P, &threads, &smem, 33 * 33 * entry_bytes(arith) + 16);
    if (!k) return false;
    if (smem < ONE_PER_SM) smem = ONE_PER_SM;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    kernel_of(P, &threads, &smem, P.tab_bytes);
    // with at most one CTA per SM, none shares an SM: a CTA that does makes all wait for it
    if ((long long)P.tiles * batch <= sm_count && smem < ONE_PER_SM) smem = ONE_PER_SM;
    P.smem = smem;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, threads, smem) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    const long long room = (long long)per_sm * sm_count / P.tiles;
    if (room < 1) return false;
    P.batch = batch;
    P.wait = 2000000000ll;      // about a second
    P.groups = (int)(room < batch ? room : batch);
    if (P.groups > RES_MAX_GROUPS) P.groups = RES_MAX_GROUPS;
    return true;
}

size_t resident_mail_bytes(const ResParams &P) {
    return P.two ? ((size_t)2 * P.groups << P.n) * (P.arith == RES_F32 ? 8 : 16) : 0;
}

cudaError_t resident_mail_clear(const ResParams &P, void *mail, cudaStream_t stream) {
    k_mail_clear<<<304, 256, 0, stream>>>((u64 *)mail, (long long)(resident_mail_bytes(P) / 8));
    return cudaGetLastError();
}

template <class A>
static void launch_tables(dim3 grid, cudaStream_t stream, const RecGeom &G, const double *in, size_t ncpl, const RecInline &X,
                          bool inl, int op0, unsigned char *r, const ResParams &P) {
    if (inl) k_resident_tables<A, true><<<grid, 64, 0, stream>>>(G, in, ncpl, X, op0, r, P);
    else k_resident_tables<A, false><<<grid, 64, 0, stream>>>(G, in, ncpl, X, op0, r, P);
}

cudaError_t resident_tables(const ResParams &P, const RecGeom &G, const double *in, size_t ncpl, const RecInline &X,
                            bool inl, int op0, int nops, void *recs, int sm_count, cudaStream_t stream) {
    const int entries = (P.nA + 1) * (P.nB + 1) + (P.had ? (P.nXA + 1) * (P.nXB + 1) : 0);
    const long long blocks = (long long)nops * G.batch;
    long long gy = (entries + 63) / 64, most = 8ll * sm_count / blocks;
    if (gy > most) gy = most < 1 ? 1 : most;
    const dim3 grid((unsigned)blocks, (unsigned)gy);
    unsigned char *r = (unsigned char *)recs;
    if (P.arith == RES_F32) launch_tables<AF32>(grid, stream, G, in, ncpl, X, inl, op0, r, P);
    else if (P.arith != RES_F64) launch_tables<ADF>(grid, stream, G, in, ncpl, X, inl, op0, r, P);
    else launch_tables<AF64>(grid, stream, G, in, ncpl, X, inl, op0, r, P);
    return cudaGetLastError();
}

cudaError_t resident_launch(const ResParams &P, void *state, const void *recs, void *mail, int *err_flag,
                            cudaStream_t stream, int ctas) {
    int threads = 0;
    size_t smem = 0;
    const ResKernel k = kernel_of(P, &threads, &smem, P.tab_bytes);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(ctas ? ctas : P.tiles * P.groups));
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = P.smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = P.two ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, k, state, (const unsigned char *)recs, mail, err_flag, P);
}

}  // namespace qsim
