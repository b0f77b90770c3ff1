// Shared by the Ritz solve's translation units (ritz.cu, ritz_cr.cu).
#pragma once

#include "common.cuh"

namespace bbl {

constexpr int kMaxNev = 32;

// Per-segment addressing for a batch of independent T's (blockIdx.y or .z =
// segment, blockIdx.x in cluster).  The single-problem path passes d_m =
// active = nullptr and zero strides.  need: with it, a kernel runs only for the
// pairs (segment x nev + index) whose flag is set, those that the fast path could
// not certify; guess: two doubles per pair, the fast path's bracket of such a
// value (not ascending where it has none), to be checked before it is used.
struct SegArgs {
    const int* d_m;       // current order m in device memory (overrides the argument)
    const int* active;    // per-segment flag; inactive segments are skipped
    int64_t sT, sTh, sS, sWs, sTmp;
    const int* need = nullptr;
    const double* guess = nullptr;
};

// ritz_cr.cu: the lowest nev pairs by spectrum slicing and block cyclic
// reduction, into theta and S (normalised, sign convention applied); sets
// the flags of the pairs that could not be certified, clears the others, and
// writes the brackets of the former; out->need and out->guess point to both.  ws:
// per segment at least nev * ritz_cr_vec_doubles; fast: ritz_cr_bytes.
size_t ritz_cr_vec_doubles(int m, int p);
size_t ritz_cr_bytes(int m, int p, int nev, int nseg);
bool ritz_cr_supports(int m, int p);
bbl_status ritz_cr(int m, int p, int nev, int nseg, const double* Tb, double* theta, double* S, double* ws, void* fast,
                   SegArgs* out, SegArgs sa, cudaStream_t st);

}  // namespace bbl
