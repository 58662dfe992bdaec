// xpass_wide.cuh -- Walsh-Hadamard passes over tiles of 2^13 amplitudes (complex64, unitary
// gauge, one state; sm_103a).
//
// Same operator as the Walsh-Hadamard passes of k_xpass_tma / k_xpass_wl, with one more qubit per
// tile: H on the pass's qubits, optionally a diagonal table (the Hadamard-basis X layer D_X with
// its 2^-n, or the Z layer) and H again.  The passes are bound by HBM, so what counts is how many
// a step takes: tiles of 2^12 amplitudes (12 qubits, then 8 per pass) need four passes to visit
// 30 to 32 qubits and three for 22 (the sizes that lattices have there), tiles of 2^13 with rows of 64 bytes (13 qubits, then
// up to 10 per pass) three and two, i.e. 4 instead of 6 and 2 instead of 4 passes per step
// (32 qubits: 73 -> 56 ms a step, 30 qubits 18.0 -> 12.7).  Rows of 64 bytes, which only a window
// of ten qubits needs, cost 8% of the rate (plain pass 12.7 instead of 11.8 ms).
// Tile bits: the first pass 13 consecutive qubits; the others a chunk of c = 3 or 4 low qubits
// and a window of 13 - c qubits, of which the mask names the rotated ones.
//
// One CTA per SM, 32 amplitudes per thread; one more warp's first lane issues the TMA loads and
// stores over three pooled 64 KB buffers (the scheme of xpass_wl.cuh).  In the first pass two
// groups of eight warps take tiles in turn and synchronise within a group only (named barriers),
// so one group's shared-memory transposes run under the other's butterflies.  Layouts (tile bits
// in registers):
//   A: 8..12   B: 0..3, 12 (16-byte accesses)   C: 4..7, 12
// each free of bank conflicts in the swizzled tile, slot l ^ (((l >> 4) & s) << 1) with s = 7 (128-byte
// rows); rows of 64 bytes have s = 3 (the TMA xors address bits 4, 5 with bits 7, 8).
#pragma once
#include "xpass_wl.cuh"
#include "df_arith.cuh"

namespace qsim {

constexpr int WT = 13;                          // tile bits
constexpr int WR = 32;                          // amplitudes per thread
constexpr int W_GROUP = 256;                    // threads per group
constexpr int W_NBUF = 3;
constexpr int W_TILE_BYTES = (1 << WT) * 8;

struct WidePass {
    int first;                  // 13 consecutive qubits: tile coordinate in dimension 3
    int chunk;                  // 4 or 3 (first pass: 13)
    unsigned mask;              // rotated tile bits
    int round2;                 // H again after the table
    int diag;                   // apply the table
    int mid_bits;               // tile-index bits below the window
    int tile_bits;              // n - 13
    int total_tiles;
    int nA, nB, lut_off;
    float scale;
    // parity columns in the layout the table is applied in: tile bits 0..3, 8..11 and registers
    // 4..7, 12 (chunk of three: 0..2, 8..12 and registers 3..7)
    uint32_t pa_thr[8], pb_thr[8];
    uint32_t pa_reg[WR], pb_reg[WR];
    uint32_t pa_tile[24], pb_tile[24];   // parity columns of the tile-index bits
};

// butterflies of register bits of `m`
__device__ __forceinline__ void had32(u64 (&v)[WR], unsigned m) {
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        if (!((m >> k) & 1u)) continue;
#pragma unroll
        for (int r = 0; r < WR; ++r)
            if (!((r >> k) & 1)) {
                const u64 a = v[r], b = v[r | (1 << k)];
                v[r] = add2(a, b);
                v[r | (1 << k)] = sub2(a, b);
            }
    }
}

// NC consumer warps and the producer's.  MODE W_GROUPS (NC = 16): the first pass, two groups as
// in the header.  The other passes never pair amplitudes that differ in their chunk's bits, so a
// tile falls into eight slices of 1024 amplitudes and a warp takes one through both rounds with
// warp-level synchronisation only, through the slice's own shared-memory slots (the scheme of
// xpass_wl.cuh):
//   W_SLICE4 (chunk of four): slice bits 1..3; L1 registers 8..12, lanes 0, 4..7; L2 registers 4..7
//     and 12, lanes 0, 8..11; exchange slots as in xpass_wl.cuh, free of bank conflicts;
//   W_SLICE3 (chunk of three): slice bits 0..2; L1 registers 8..12, lanes 3..7; L2 registers 3..7,
//     lanes 8..12; amplitude (x, y) = (bits 3..7, bits 8..12) sits in the slot of (x ^ y, y).  A
//     slice's slots lie in half of the banks, so every access takes two wavefronts.
// Measured at 32 qubits (68.7 GB a pass, 10.1 ms at the copy rate): first pass 11.8 ms, a shared
// pass 14.0 (chunk of four), 18.5 (chunk of three); as groups of 256 threads the shared passes
// took 17 and 23 ms.  Passes over 2^12 tiles take 11.8 plain and 12.2 shared, but six a step.
enum { W_GROUPS = 0, W_SLICE4 = 1, W_SLICE3 = 2 };

template <int MODE, int NC>
__global__ void __launch_bounds__(32 * (NC + 1), 1) k_xpass_wide(const double *__restrict__ recs,
                                                                int *__restrict__ err_flag,
                                                                const __grid_constant__ CUtensorMap tmap,
                                                                const __grid_constant__ WidePass P) {
    constexpr int NTH = 32 * (NC + 1);
    extern __shared__ unsigned char smem_raw[];
    unsigned char *base_ptr = smem_raw + ((1024u - (smem_addr(smem_raw) & 1023u)) & 1023u);
    u64 *buf = reinterpret_cast<u64 *>(base_ptr);                              // W_NBUF x 8192
    float2 *lut = reinterpret_cast<float2 *>(buf + W_NBUF * (1 << WT));
    uint2 *ptab = reinterpret_cast<uint2 *>(lut + (P.diag ? (P.nA + 1) * (P.nB + 1) : 0));   // 3 x 256
    __shared__ uint64_t full[W_NBUF], done[W_NBUF];
    __shared__ int s_stamp[W_NBUF];     // tile (CTA-local index) last issued into each buffer
    __shared__ int s_abort;
    const int t = threadIdx.x, lane = t & 31;
    const int G = (int)gridDim.x, T = P.total_tiles, first = (int)blockIdx.x;
    const long long max_wait = 2000000000ll;   // SM cycles (~1 s)
    volatile int *abort_flag = &s_abort;
    volatile int *stamp = s_stamp;

    if (t == 0) {
        for (int b = 0; b < W_NBUF; ++b) { mbar_init(&full[b], 1); mbar_init(&done[b], 8); s_stamp[b] = -1; }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_abort = 0;
    }
    if (P.diag)
        for (int e = t; e < 3 * 256; e += NTH) {
            uint32_t a = 0, b = 0;
            for (int j = 0; j < 8; ++j) {
                const int bit = 8 * (e >> 8) + j;
                if (bit < P.tile_bits && ((e >> j) & 1)) { a ^= P.pa_tile[bit]; b ^= P.pb_tile[bit]; }
            }
            ptab[e] = make_uint2(a, b);
        }
    // (as in the other passes: set-up may overlap the previous kernel, reads of global memory not)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int nB1 = P.nB + 1;
    if (P.diag)
        for (int i = t; i < (P.nA + 1) * nB1; i += NTH)
            lut[i] = make_float2((float)recs[P.lut_off + 2 * i], (float)recs[P.lut_off + 2 * i + 1]);
    __syncthreads();

    const int n_my = first < T ? (T - first + G - 1) / G : 0;
    const int mid_mask = (1 << P.mid_bits) - 1;
    auto coords = [&](int j, int &x1, int &x3, int &x4) {
        const int tile = first + j * G;
        x1 = P.first ? 0 : tile & mid_mask;
        x3 = P.first ? tile : 0;
        x4 = P.first ? 0 : tile >> P.mid_bits;
    };
    auto issue_load = [&](int j) {
        int x1, x3, x4;
        coords(j, x1, x3, x4);
        const int b = j % W_NBUF;
        stamp[b] = j;
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_arrive_expect_tx(&full[b], W_TILE_BYTES);
        tma_load_5d(buf + (size_t)b * (1 << WT), &tmap, &full[b], 0, x1, 0, x3, x4);
    };

    // the diagonal table and its scale for registers in a layout with bits 4..7 and 12
    auto table = [&](u64 (&v)[WR], uint32_t pa, uint32_t pb) {
#pragma unroll
        for (int r = 0; r < WR; ++r) {
            const float2 x = cphase(unpk(v[r]), lut[__popc(pa ^ P.pa_reg[r]) * nB1 + __popc(pb ^ P.pb_reg[r])]);
            v[r] = pk(x.x, x.y);
        }
        if (P.scale != 1.0f) {
            const u64 sc = pk(P.scale, P.scale);
#pragma unroll
            for (int r = 0; r < WR; ++r) v[r] = mul2(v[r], sc);
        }
    };

    if (t >= 32 * NC) {
        // ---------------- producer ----------------
        if (lane == 0) {
            int issued = 0;
            for (; issued < W_NBUF && issued < n_my; ++issued) issue_load(issued);
            for (int j = 0; j < n_my; ++j) {
                const int b = j % W_NBUF;
                if (!mbar_wait_or_abort(&done[b], (uint32_t)((j / W_NBUF) & 1), max_wait, abort_flag)) {
                    atomicOr(err_flag, 1);
                    *abort_flag = 1;
                    break;
                }
                int x1, x3, x4;
                coords(j, x1, x3, x4);
                tma_store_5d(&tmap, buf + (size_t)b * (1 << WT), 0, x1, 0, x3, x4);
                bulk_commit();
                if (j + W_NBUF < n_my) {
                    bulk_wait_read_all();          // the store has read the buffer
                    issue_load(j + W_NBUF);
                    ++issued;
                }
            }
            // leave no copy in flight: loads that no group consumed (abort), then stores
            for (int j = issued - W_NBUF < 0 ? 0 : issued - W_NBUF; j < issued; ++j)
                mbar_wait_bounded(&full[j % W_NBUF], (uint32_t)((j / W_NBUF) & 1), max_wait);
            bulk_wait_all();
        }
        __syncwarp();
    } else if constexpr (MODE != W_GROUPS) {
        // ---------------- consumers: warp takes slices (tile, w) in turn ----------------
        const int warp = t >> 5, l0 = lane & 1, lh = lane >> 1;
        const unsigned m1 = (P.mask >> 8) & 31u, m2 = MODE == W_SLICE4 ? (P.mask >> 4) & 15u : (P.mask >> 3) & 31u;
        // parity columns of the L2 lane bits
        uint32_t pa_lane = 0, pb_lane = 0;
#pragma unroll
        for (int j = 0; j < 5; ++j)
            if ((lane >> j) & 1) {
                const int c = MODE == W_SLICE4 ? (j ? 3 + j : 0) : 3 + j;
                pa_lane ^= P.pa_thr[c]; pb_lane ^= P.pb_thr[c];
            }
        for (int item = warp; item < 8 * n_my; item += NC) {
            const int j = item >> 3, w = item & 7, b = j % W_NBUF;
            const uint32_t par = (uint32_t)((j / W_NBUF) & 1);
            int ok = 1;
            if (lane == 0) {
                const long long t0 = clock64();
                while (stamp[b] != j)
                    if (*abort_flag || clock64() - t0 > max_wait) { ok = 0; break; }
                if (ok) ok = mbar_wait_or_abort(&full[b], par, max_wait, abort_flag) ? 1 : 0;
                if (!ok) { atomicOr(err_flag, 1); *abort_flag = 1; }
            }
            if (!__shfl_sync(0xffffffffu, ok, 0)) break;
            (void)mbar_try_wait(&full[b], par);
            unsigned char *tb = reinterpret_cast<unsigned char *>(buf + (size_t)b * (1 << WT));
            // byte offsets of the lane's slots: tile (L1), exchange (L1), exchange (L2)
            const int wl = w ^ (lh & 7);
            const int base_t = MODE == W_SLICE4 ? (l0 | (wl << 1) | (lh << 4)) << 3
                                                : (w << 3) ^ (((lane >> 1) & 3) << 4) ^ (lane << 6);
            const int base_2 = MODE == W_SLICE4 ? (l0 | (wl << 1) | ((lh & 7) << 4) | (lh << 8)) << 3
                                                : base_t + (lane << 11);
            auto at_t = [&](int r) { return reinterpret_cast<u64 *>(tb + base_t + (r << 11)); };
            auto at_1 = [&](int r) {
                if (MODE == W_SLICE4)
                    return reinterpret_cast<u64 *>(tb + ((base_t ^ ((r & 7) * 0x90)) + ((r & 15) << 11)) + ((r >> 4) << 15));
                return reinterpret_cast<u64 *>(tb + (base_t ^ (((r >> 1) & 3) << 4) ^ (r << 6)) + (r << 11));
            };
            auto at_2 = [&](int r) {
                if (MODE == W_SLICE4)
                    return reinterpret_cast<u64 *>(tb + ((base_2 ^ ((r & 7) * 0x90)) + (((r >> 3) & 1) << 10)) + ((r >> 4) << 15));
                return reinterpret_cast<u64 *>(tb + (base_2 ^ (((r >> 1) & 3) << 4) ^ (r << 6)));
            };
            u64 v[WR];
#pragma unroll
            for (int r = 0; r < WR; ++r) v[r] = *at_t(r);
            had32(v, m1);
            __syncwarp();
#pragma unroll
            for (int r = 0; r < WR; ++r) *at_1(r) = v[r];
            __syncwarp();
#pragma unroll
            for (int r = 0; r < WR; ++r) v[r] = *at_2(r);
            had32(v, m2);
            if (P.diag) {
                const int tile = first + j * G;
                const uint2 e0 = ptab[tile & 255], e1 = ptab[256 + ((tile >> 8) & 255)], e2 = ptab[512 + ((tile >> 16) & 255)];
                uint32_t pa = pa_lane ^ e0.x ^ e1.x ^ e2.x, pb = pb_lane ^ e0.y ^ e1.y ^ e2.y;
#pragma unroll
                for (int q = 0; q < 3; ++q)
                    if ((w >> q) & 1) {
                        const int c = MODE == W_SLICE4 ? 1 + q : q;
                        pa ^= P.pa_thr[c]; pb ^= P.pb_thr[c];
                    }
                table(v, pa, pb);
            }
            if (P.round2) had32(v, m2);
#pragma unroll
            for (int r = 0; r < WR; ++r) *at_2(r) = v[r];
            __syncwarp();
#pragma unroll
            for (int r = 0; r < WR; ++r) v[r] = *at_1(r);
            if (P.round2) had32(v, m1);
            __syncwarp();
#pragma unroll
            for (int r = 0; r < WR; ++r) *at_t(r) = v[r];
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&done[b]);
        }
    } else {
        // ---------------- consumers: group g takes tiles g, g + 2, ... ----------------
        const int g = t / W_GROUP, u = t % W_GROUP;
        const int ulo = u & 15, uhi = u >> 4;
        auto meet = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(1 + g), "n"(W_GROUP) : "memory"); };
        // the group's barrier, true if any thread came with `bad`
        auto any_of = [&](int bad) -> bool {
            int r;
            asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.s32 q, %1, 0;\n\tbar.red.or.pred p, %2, %3, q;\n\t"
                         "selp.s32 %0, 1, 0, p;\n\t}"
                         : "=r"(r) : "r"(bad), "r"(1 + g), "n"(W_GROUP) : "memory");
            return r != 0;
        };
        uint32_t pa_t = 0, pb_t = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if ((u >> j) & 1) { pa_t ^= P.pa_thr[j]; pb_t ^= P.pb_thr[j]; }
        const int a_base = u ^ (((u >> 4) & 7) << 1);           // layout A: + (r & 15) << 8, bit 4 of r: << 12
        u64 v[WR];
        u64 *tb = buf;
        auto a_at = [&](int r) { return a_base + ((r & 15) << 8) + ((r >> 4) << 12); };
        auto c_at = [&](int r) { return (ulo ^ ((r & 7) << 1)) + ((r & 15) << 4) + (uhi << 8) + ((r >> 4) << 12); };
        auto get_a = [&]() {
#pragma unroll
            for (int r = 0; r < WR; ++r) v[r] = tb[a_at(r)];
        };
        auto put_a = [&]() {
#pragma unroll
            for (int r = 0; r < WR; ++r) tb[a_at(r)] = v[r];
        };
        auto get_c = [&]() {
#pragma unroll
            for (int r = 0; r < WR; ++r) v[r] = tb[c_at(r)];
        };
        auto put_c = [&]() {
#pragma unroll
            for (int r = 0; r < WR; ++r) tb[c_at(r)] = v[r];
        };
        // layout B in 16-byte units (128-byte rows only): read, butterflies of bits 0..3, write
        auto stage_b = [&]() {
            ulonglong2 *t2 = reinterpret_cast<ulonglong2 *>(tb);
#pragma unroll
            for (int m = 0; m < WR / 2; ++m) {
                const ulonglong2 x = t2[((u << 3) | ((m & 7) ^ (u & 7))) + ((m >> 3) << 11)];
                v[2 * m] = x.x;
                v[2 * m + 1] = x.y;
            }
            had32(v, 15u);
#pragma unroll
            for (int m = 0; m < WR / 2; ++m)
                t2[((u << 3) | ((m & 7) ^ (u & 7))) + ((m >> 3) << 11)] = make_ulonglong2(v[2 * m], v[2 * m + 1]);
        };
        for (int j = g; j < n_my; j += 2) {
            const int b = j % W_NBUF;
            const uint32_t par = (uint32_t)((j / W_NBUF) & 1);
            int ok = 1;
            if (lane == 0) {
                const long long t0 = clock64();
                while (stamp[b] != j)
                    if (*abort_flag || clock64() - t0 > max_wait) { ok = 0; break; }
                if (ok) ok = mbar_wait_or_abort(&full[b], par, max_wait, abort_flag) ? 1 : 0;
                if (!ok) { atomicOr(err_flag, 1); *abort_flag = 1; }
            }
            ok = __shfl_sync(0xffffffffu, ok, 0);
            (void)mbar_try_wait(&full[b], par);
            tb = buf + (size_t)b * (1 << WT);
            if (ok) get_a();
            if (any_of(!ok)) break;                 // the group leaves together
            // ---- round 1: A, B, C ----
            had32(v, 31u);
            put_a();
            meet();
            stage_b();
            meet();
            get_c();
            had32(v, 15u);
            if (P.diag) {
                const int tile = first + j * G;
                const uint2 e0 = ptab[tile & 255], e1 = ptab[256 + ((tile >> 8) & 255)], e2 = ptab[512 + ((tile >> 16) & 255)];
                const uint32_t pa = pa_t ^ e0.x ^ e1.x ^ e2.x, pb = pb_t ^ e0.y ^ e1.y ^ e2.y;
                table(v, pa, pb);
            }
            if (P.round2) {
                // ---- round 2: C, B, A ----
                had32(v, 15u);
                put_c();
                meet();
                stage_b();
                meet();
                get_a();
                had32(v, 31u);
                put_a();
            } else {
                put_c();
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&done[b]);
        }
    }
    __syncthreads();
}

}  // namespace qsim
