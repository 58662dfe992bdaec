// resident.h -- host interface of the resident evolution kernel (resident.cu).
#pragma once
#include <cuda_runtime.h>
#include <cstdint>

#include "records.cuh"

namespace qsim {

constexpr int RES_MAXQ = 24;

enum { RES_F32 = 0, RES_DF = 1, RES_F64 = 2, RES_DF32 = 3 };   // arithmetic

struct ResParams {
    int arith;                 // RES_F32, RES_DF32 (complex64), RES_DF, RES_F64 (complex128)
    int n, M;                  // qubits, tile bits
    int c;                     // two tile sets: chunk bits kept by the second one, 2 M - n
    int two;                   // 1: two tile sets with an exchange between them, 0: one tile per state
    int tiles;                 // CTAs per state
    int had;                   // Walsh-Hadamard passes (unitary gauge), else tangent-form rotations
    int nops, batch, groups;   // factor groups, states, states in flight
    int last_z;                // the last factor group has a Z layer
    int nA, nB, nXA, nXB;      // term counts of the two tables
    int ztab_bytes, xtab_bytes, tab_bytes;     // tables (multiples of 16), the larger one
    long long rec_bytes;       // record of one factor group and state
    size_t smem;               // dynamic shared memory per CTA
    uint32_t colA[RES_MAXQ], colB[RES_MAXQ];   // Z-layer terms containing each qubit
    uint32_t xcolA[RES_MAXQ], xcolB[RES_MAXQ]; // Hadamard-basis X terms containing each qubit
    uint32_t cls;              // bit q: qubit q is a vertex (tau^x)
    long long wait;            // limit of a poll, SM cycles
};

// Fills arith, n, M, c, two, tiles, groups and the sizes; false if the state does not fit the chip
// at one tile per resident CTA (or the kernel does not cover the size).
bool resident_plan(ResParams &P, int arith, int n, int batch, int sm_count);
// mail: resident_mail_bytes, all words empty (resident_mail_clear) before and after a launch
// that did not time out; launches that may overlap need one each.
size_t resident_mail_bytes(const ResParams &P);
cudaError_t resident_mail_clear(const ResParams &P, void *mail, cudaStream_t stream);
// Records of factor groups op0 .. op0 + nops - 1 (rec_bytes each, group-major).
cudaError_t resident_tables(const ResParams &P, const RecGeom &G, const double *in, size_t ncpl, const RecInline &X,
                            bool inl, int op0, int nops, void *recs, int sm_count, cudaStream_t stream);
// (ctas: that many of the run's CTAs only, whose polls for the others' amplitudes run out)
cudaError_t resident_launch(const ResParams &P, void *state, const void *recs, void *mail, int *err_flag,
                            cudaStream_t stream, int ctas = 0);
constexpr int RES_MAX_GROUPS = 4096;

}  // namespace qsim
