// xpass_df.cuh -- complex128 Walsh-Hadamard passes in double-float arithmetic (sm_103a).
//
// GB300 runs FP64 at a small fraction of its FP32 rate, so a complex128 pass written with
// FP64 butterflies is bound by the FP64 pipe far below the HBM roofline.  Here each real
// number of the state is carried as an unevaluated sum hi + lo of two floats (|lo| <=
// ulp(hi) / 2, 48 significand bits), and the passes run on the FP32 pipes with packed
// f32x2 instructions, (re, im) in one 64-bit register:
//   * sum and difference: Knuth's two-sum (two-diff) of the high parts (exact), the
//     error and the low parts summed into the low part (8 packed operations per output).
//     Within a pass the pairs are not renormalised after every butterfly (the low part
//     grows by at most the pass's number of stages times an ulp of the high part, about
//     2^-43 relative); one fast renormalisation runs before the table product and before
//     the store;
//   * product with a table entry (cos phi, sin phi) held in double-float: the rounding
//     error of the high product recovered exactly by scalar FMA (fmaf, one rounding),
//     the cross terms by packed FMA, renormalisation.  (A packed f32x2 FMA in that role
//     left the products at float precision, ~5e-8 per phase, so the exact term is not
//     taken from it.)
// Layout in HBM while a call runs ("blocked double-float"): every block of 16 amplitudes
// (256 bytes of complex128) holds the 16 high (re, im) float pairs, then the 16 low pairs.
// The first pass of a call splits the complex128 amplitudes of its tiles as it reads them and
// the last one writes them back as complex128 (against conversion kernels of their own, 27 qubits:
// one step 9.53 -> 8.51 ms, five 24.1 -> 23.1, forty 151.9 -> 151.0; what the two converting
// passes take more is about half of what the kernels took).  The high (low) halves of a tile form
// an ordinary complex64-like tile under a tensor map with doubled strides (base, base + 128
// bytes), so the pass loads a tile pair by two TMA copies and reuses the stage layouts of the
// complex64 kernel (xpass_tma.cuh).  The pass applies unnormalised Walsh-Hadamard
// butterflies on the pass's qubits (the unitary-gauge X layer H^n D_X H^n and the Z layer
// between transforms, Sec. II), optionally the diagonal table with its scale, and (MERGED)
// a second round of butterflies on the same qubits.  ROT: the gauge-Higgs form instead:
// tangent-form rotations in the real frame phi = i^popc psi (a' = a + t b, b' = b - t a,
// t = tan theta of the qubit's class in double-float, Eq. (8)), the Z layer from the
// table scaled by the group's cos factors C, C alone for a group without Z layer, the
// frame conversions on the first and last pass of a call, and (MERGED) the next factor
// group's rotations on the same qubits.
#pragma once
#include "xpass_tma.cuh"
#include "df_arith.cuh"

namespace qsim {

// fast renormalisation of every pair: |l| <= ulp(h) / 2 afterwards
__device__ __forceinline__ void df_renorm(u64 (&h)[NR], u64 (&l)[NR]) {
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        const u64 nh = add2(h[r], l[r]);
        l[r] = sub2(l[r], sub2(nh, h[r]));
        h[r] = nh;
    }
}

// unnormalised Walsh-Hadamard butterflies on the register bits of mask
__device__ __forceinline__ void df_hadamard(u64 (&h)[NR], u64 (&l)[NR], unsigned mask) {
#pragma unroll
    for (int k = 0; k < RB; ++k) {
        if (!((mask >> k) & 1u)) continue;
#pragma unroll
        for (int r = 0; r < NR; ++r)
            if (!((r >> k) & 1)) df_butterfly_lazy(h[r], l[r], h[r | (1 << k)], l[r | (1 << k)]);
    }
}

// rotations on the register bits of mask; tc[k] = {(th, th), (tl, tl)} of bit k's class
__device__ __forceinline__ void df_rotate(u64 (&h)[NR], u64 (&l)[NR], unsigned mask, const u64 (*tc)[2]) {
#pragma unroll
    for (int k = 0; k < RB; ++k) {
        if (!((mask >> k) & 1u)) continue;
        const u64 th = tc[k][0], tl = tc[k][1];
#pragma unroll
        for (int r = 0; r < NR; ++r)
            if (!((r >> k) & 1)) df_rot_lazy(h[r], l[r], h[r | (1 << k)], l[r | (1 << k)], th, tl);
    }
}

// One Walsh-Hadamard pass over a state in the blocked double-float layout: tile pairs
// (high, low) by TMA into one buffer per CTA (two CTAs per SM); the next pair's load is
// issued as soon as the current pair's last stage has been read from shared memory, and
// both halves go back by per-thread stores from registers while that load is in flight.
// RAW, bit 0: the tiles hold complex128 amplitudes (the call's first pass), bit 1: write them back as
// such (its last).  Only those two passes carry a conversion: as a branch taken at run time it
// cost every pass registers (spills of 8 to 16 bytes in the merged ones) and long calls more than
// it saved (32 qubits, 20 steps: 211.4 ms a step with conversion kernels, 215.4 with the branch,
// 209.9 so).
template <bool MERGED, bool ROT, int RAW>
__global__ void __launch_bounds__(NT, 2) k_xpass_df(float2 *__restrict__ state, const double *__restrict__ recs,
                                                    const double *__restrict__ recs2,
                                                    int rec_stride, int tiles_shift, int *__restrict__ err_flag,
                                                    const __grid_constant__ CUtensorMap tmap_h,
                                                    const __grid_constant__ CUtensorMap tmap_l,
                                                    const __grid_constant__ TmaPass P) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char *base_ptr = smem_raw + ((1024u - (smem_addr(smem_raw) & 1023u)) & 1023u);
    float2 *buf = reinterpret_cast<float2 *>(base_ptr);                  // (high, low) tile pair
    u64 *lut = reinterpret_cast<u64 *>(buf + 2 * (1 << LT));              // 4 u64 per entry
    uint2 *ptab = reinterpret_cast<uint2 *>(lut + 4 * (P.apply_z ? (P.nA + 1) * (P.nB + 1) : 0));
    __shared__ uint64_t bar;
    __shared__ int s_ok;
    __shared__ u64 s_tc[2][3][RB][2];   // ROT: per round, stage and register bit: (th, th), (tl, tl)
    __shared__ u64 s_xs[2];             // ROT: C of the group, (Ch, Ch), (Cl, Cl)

    const int t = threadIdx.x;
    const long long G = gridDim.x;
    const long long T = P.total_tiles;
    const long long first = blockIdx.x;
    const long long max_wait = 2000000000ll;
    if (t == 0) {
        mbar_init(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_ok = 1;
    }
    if (P.apply_z) {
        for (int e = t; e < 3 * 256; e += NT) {
            int byte = e >> 8, val = e & 255;
            uint32_t a = 0, b = 0;
            for (int j = 0; j < 8; ++j) {
                int bit = 8 * byte + j;
                if (bit < P.tile_bits && ((val >> j) & 1)) { a ^= P.pa_tile[bit]; b ^= P.pb_tile[bit]; }
            }
            ptab[e] = make_uint2(a, b);
        }
    }
    __syncthreads();
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");

    auto issue = [&](long long tile) {
        const int x2 = (int)(tile & ((1ll << P.mid_bits) - 1));
        const int x4 = (int)(tile >> P.mid_bits);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_arrive_expect_tx(&bar, 2 * TMA_TILE_BYTES);
        tma_load_5d(buf, &tmap_h, &bar, 0, 0, x2, 0, x4);
        tma_load_5d(buf + (1 << LT), &tmap_l, &bar, 0, 0, x2, 0, x4);
    };
    const int n_my = first < T ? (int)((T - first + G - 1) / G) : 0;
    if (t == 0 && n_my > 0) issue(first);

    const int tlo = t & 15, thi = t >> 4;
    const int a_base = swz128(t);
    int c_base[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) c_base[j] = (tlo ^ (j << 1)) | (thi << 8);
    const int b_base = t << 3, b_x = t & 7;
    // global amplitude offsets of this thread without its low four bits (global bits 0..3
    // are local bits 0..3 = tlo in the stage-C and stage-A layouts)
    long long toff_c = 0, toff_a = 0;
    uint32_t pa_t = 0, pb_t = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if ((thi >> j) & 1) toff_c += P.toff_c[4 + j];
        if ((tlo >> j) & 1) { pa_t ^= P.pa_thr[j]; pb_t ^= P.pb_thr[j]; }
        if ((thi >> j) & 1) { pa_t ^= P.pa_thr[4 + j]; pb_t ^= P.pb_thr[4 + j]; }
    }
#pragma unroll
    for (int j = 4; j < 8; ++j)
        if ((t >> j) & 1) toff_a += P.toff_a[j];
    const int nB1 = P.nB + 1;
    const int nlut = (P.nA + 1) * nB1;
    const u64 dscale = pk(P.scale, P.scale);
    const long long tmask = (1ll << tiles_shift) - 1;
    long long cur_batch = -1;

    long long tile = first;
    for (int it = 0; it < n_my; ++it, tile += G) {
        const long long batch = tile >> tiles_shift;
        if (batch != cur_batch) {
            // phase table of this batch element: (cos, sin) in double-float, packed
            __syncthreads();
            const double *rec = recs + batch * rec_stride;
            if (ROT && t < 2 * 3 * RB) {
                // round 0: this factor group (stages A, B, C); round 1 (MERGED): the next one
                const int round = t / (3 * RB), st = (t / RB) % 3, k = t % RB;
                if (round == 0 || MERGED) {
                    const double *rr = round ? recs2 + batch * rec_stride : rec;
                    const double tv = rr[P.tan_off + ((P.cls[st] >> k) & 1)];
                    const float a = __double2float_rn(tv), b = __double2float_rn(tv - (double)a);
                    s_tc[round][st][k][0] = pk(a, a);
                    s_tc[round][st][k][1] = pk(b, b);
                }
            }
            if (ROT && t == 0) {
                const double cv = rec[P.tan_off + 2];
                const float a = __double2float_rn(cv), b = __double2float_rn(cv - (double)a);
                s_xs[0] = pk(a, a);
                s_xs[1] = pk(b, b);
            }
            if (P.apply_z) {
                const int loff = ROT ? P.tan_off + 4 : P.lut_off;   // ROT: the table scaled by C
                for (int i = t; i < nlut; i += NT) {
                    const double c = 1.0 - rec[loff + 2 * i], s = rec[loff + 2 * i + 1];
                    const float ch = __double2float_rn(c), cl = __double2float_rn(c - (double)ch);
                    const float sh = __double2float_rn(s), sl = __double2float_rn(s - (double)sh);
                    u64 *q = lut + 4 * i;
                    q[0] = pk(ch, ch); q[1] = pk(cl, cl); q[2] = pk(sh, -sh); q[3] = pk(sl, -sl);
                }
            }
            cur_batch = batch;
            __syncthreads();
        }
        if (t == 0) {
            if (!mbar_wait_bounded(&bar, (uint32_t)(it & 1), max_wait)) {
                atomicOr(err_flag, 1);
                s_ok = 0;
            }
        }
        __syncthreads();
        if (!s_ok) return;

        u64 *th = reinterpret_cast<u64 *>(buf);
        u64 *tl = reinterpret_cast<u64 *>(buf + (1 << LT));
        u64 h[NR], l[NR];
        // ---- stage A: registers = local 8..11 ----
        if constexpr ((RAW & 1) != 0) {
            // complex128 amplitudes under the two maps: a block's first eight in the high tile's
            // row, the others in the low tile's; all are read before a half is written
            const ulonglong2 *src = reinterpret_cast<const ulonglong2 *>(tlo & 8 ? tl : th);
            const int unit = ((t >> 4) << 3) | ((tlo & 7) ^ ((t >> 4) & 7));
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                const ulonglong2 x = src[unit + (r << 7)];
                float rh, rl, ih, il;
                split_double(__longlong_as_double((long long)x.x), rh, rl);
                split_double(__longlong_as_double((long long)x.y), ih, il);
                h[r] = pk(rh, ih);
                l[r] = pk(rl, il);
            }
            __syncthreads();
        } else {
#pragma unroll
            for (int r = 0; r < NR; ++r) { h[r] = th[a_base + (r << TB)]; l[r] = tl[a_base + (r << TB)]; }
        }
        const int pc_tile = __popcll(tile & tmask);
        if (ROT && (P.frame & 2)) {   // psi -> phi = i^popc psi
            const int k0 = __popc(t) + pc_tile;
#pragma unroll
            for (int r = 0; r < NR; ++r) df_ipow(h[r], l[r], k0 + __popc(r));
        }
        if (ROT) df_rotate(h, l, P.rot[0], s_tc[0][0]); else df_hadamard(h, l, P.rot[0]);
#pragma unroll
        for (int r = 0; r < NR; ++r) { th[a_base + (r << TB)] = h[r]; tl[a_base + (r << TB)] = l[r]; }
        __syncthreads();
        // ---- stage B: registers = local 0..3 ----
        if (P.stage_b) {
            ulonglong2 *th2 = reinterpret_cast<ulonglong2 *>(th), *tl2 = reinterpret_cast<ulonglong2 *>(tl);
#pragma unroll
            for (int m = 0; m < NR / 2; ++m) {
                const ulonglong2 qh = th2[b_base + (m ^ b_x)], ql = tl2[b_base + (m ^ b_x)];
                h[2 * m] = qh.x; h[2 * m + 1] = qh.y;
                l[2 * m] = ql.x; l[2 * m + 1] = ql.y;
            }
            if (ROT) df_rotate(h, l, P.rot[1], s_tc[0][1]); else df_hadamard(h, l, P.rot[1]);
#pragma unroll
            for (int m = 0; m < NR / 2; ++m) {
                th2[b_base + (m ^ b_x)] = make_ulonglong2(h[2 * m], h[2 * m + 1]);
                tl2[b_base + (m ^ b_x)] = make_ulonglong2(l[2 * m], l[2 * m + 1]);
            }
            __syncthreads();
        }
        // ---- stage C: registers = local 4..7; table, scale ----
#pragma unroll
        for (int r = 0; r < NR; ++r) { h[r] = th[c_base[r & 7] + (r << 4)]; l[r] = tl[c_base[r & 7] + (r << 4)]; }
        if (!MERGED) {
            // the pair's last shared-memory read: the next pair may load
            __syncthreads();
            if (t == 0 && it + 1 < n_my) issue(tile + G);
        }
        if (ROT) df_rotate(h, l, P.rot[2], s_tc[0][2]); else df_hadamard(h, l, P.rot[2]);
        const long long mid = tile & ((1ll << P.mid_bits) - 1);
        const long long up = tile >> P.mid_bits;
        const long long gbase = (mid << P.c) + (up << (P.next + P.k));
        if (P.apply_z) {
            df_renorm(h, l);
            const long long tin = tile & tmask;
            const uint2 e0 = ptab[tin & 255], e1 = ptab[256 + ((tin >> 8) & 255)], e2 = ptab[512 + ((tin >> 16) & 255)];
            const uint32_t pa = pa_t ^ e0.x ^ e1.x ^ e2.x;
            const uint32_t pb = pb_t ^ e0.y ^ e1.y ^ e2.y;
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                const u64 *q = lut + 4 * (__popc(pa ^ P.pa_reg[r]) * nB1 + __popc(pb ^ P.pb_reg[r]));
                DfPhase ph;
                ph.ch = q[0]; ph.cl = q[1]; ph.sh = q[2]; ph.sl = q[3];
                df_phase(h[r], l[r], ph);
            }
            if (P.scale != 1.0f) {   // a power of two: exact on both parts
#pragma unroll
                for (int r = 0; r < NR; ++r) { h[r] = mul2(h[r], dscale); l[r] = mul2(l[r], dscale); }
            }
        }
        if (ROT && !P.apply_z && P.xscale) {   // C of a factor group without Z layer
            const u64 ch = s_xs[0], cl = s_xs[1];
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                u64 p, e;
                df_scale_lazy(ch, cl, h[r], l[r], p, e);
                h[r] = p; l[r] = e;
            }
        }
        if (ROT && !MERGED && (P.frame & 4)) {   // phi -> psi
            const int k0 = -(__popc(tlo) + __popc(thi) + pc_tile);
#pragma unroll
            for (int r = 0; r < NR; ++r) df_ipow(h[r], l[r], (k0 - __popc(r)) & 3);
        }
        u64 *dst;
        if (MERGED) {
            // ---- second round: stage C (in registers), B, A; store from stage A ----
            if (ROT) df_rotate(h, l, P.rot[2], s_tc[1][2]); else df_hadamard(h, l, P.rot[2]);
#pragma unroll
            for (int r = 0; r < NR; ++r) { th[c_base[r & 7] + (r << 4)] = h[r]; tl[c_base[r & 7] + (r << 4)] = l[r]; }
            __syncthreads();
            if (P.stage_b) {
                ulonglong2 *th2 = reinterpret_cast<ulonglong2 *>(th), *tl2 = reinterpret_cast<ulonglong2 *>(tl);
#pragma unroll
                for (int m = 0; m < NR / 2; ++m) {
                    const ulonglong2 qh = th2[b_base + (m ^ b_x)], ql = tl2[b_base + (m ^ b_x)];
                    h[2 * m] = qh.x; h[2 * m + 1] = qh.y;
                    l[2 * m] = ql.x; l[2 * m + 1] = ql.y;
                }
                if (ROT) df_rotate(h, l, P.rot[1], s_tc[1][1]); else df_hadamard(h, l, P.rot[1]);
#pragma unroll
                for (int m = 0; m < NR / 2; ++m) {
                    th2[b_base + (m ^ b_x)] = make_ulonglong2(h[2 * m], h[2 * m + 1]);
                    tl2[b_base + (m ^ b_x)] = make_ulonglong2(l[2 * m], l[2 * m + 1]);
                }
                __syncthreads();
            }
#pragma unroll
            for (int r = 0; r < NR; ++r) { h[r] = th[a_base + (r << TB)]; l[r] = tl[a_base + (r << TB)]; }
            __syncthreads();
            if (t == 0 && it + 1 < n_my) issue(tile + G);
            if (ROT) df_rotate(h, l, P.rot[0], s_tc[1][0]); else df_hadamard(h, l, P.rot[0]);
            if (ROT && (P.frame & 4)) {   // phi -> psi
                const int k0 = -(__popc(t) + pc_tile);
#pragma unroll
                for (int r = 0; r < NR; ++r) df_ipow(h[r], l[r], (k0 - __popc(r)) & 3);
            }
            df_renorm(h, l);
            // blocked layout: amplitude g = 16 m + j has its high pair at float2 index
            // 32 m + j and its low pair at 32 m + 16 + j
            dst = reinterpret_cast<u64 *>(state) + 2 * (gbase + toff_a) + tlo;
            if constexpr ((RAW & 2) != 0) {
                double2 *o = reinterpret_cast<double2 *>(state) + gbase + toff_a + tlo;
#pragma unroll
                for (int r = 0; r < NR; ++r) o[P.roff_a[r]] = df_join(h[r], l[r]);
            } else {
#pragma unroll
                for (int r = 0; r < NR; ++r) { dst[2 * P.roff_a[r]] = h[r]; dst[2 * P.roff_a[r] + 16] = l[r]; }
            }
        } else {
            df_renorm(h, l);
            dst = reinterpret_cast<u64 *>(state) + 2 * (gbase + toff_c) + tlo;
            if constexpr ((RAW & 2) != 0) {
                double2 *o = reinterpret_cast<double2 *>(state) + gbase + toff_c + tlo;
#pragma unroll
                for (int r = 0; r < NR; ++r) o[P.roff_c[r]] = df_join(h[r], l[r]);
            } else {
#pragma unroll
                for (int r = 0; r < NR; ++r) { dst[2 * P.roff_c[r]] = h[r]; dst[2 * P.roff_c[r] + 16] = l[r]; }
            }
        }
    }
}

}  // namespace qsim
