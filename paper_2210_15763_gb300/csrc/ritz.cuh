// Shared by the Ritz solve's translation units (ritz.cu, ritz_cr.cu).
#pragma once

#include "common.cuh"

namespace bbl {

constexpr int kMaxNev = 32;

// Per-segment addressing for a batch of independent T's (blockIdx.y or .z =
// segment, blockIdx.x in cluster).  The single-problem path passes d_m =
// active = nullptr and zero strides.  need: with it, a kernel runs only for
// segments whose flag is set (the pairs the fast path could not certify).
struct SegArgs {
    const int* d_m;       // current order m in device memory (overrides the argument)
    const int* active;    // per-segment flag; inactive segments are skipped
    int64_t sT, sTh, sS, sWs, sTmp;
    const int* need = nullptr;
};

// ritz_cr.cu: the lowest nev pairs by spectrum slicing and block cyclic
// reduction, into theta and S (normalised, sign convention applied); sets
// (*need)[seg] where a pair could not be certified, else clears it.  ws: per
// segment at least nev * ritz_cr_vec_doubles; fast: ritz_cr_bytes.
size_t ritz_cr_vec_doubles(int m, int p);
size_t ritz_cr_bytes(int m, int p, int nev, int nseg);
bool ritz_cr_supports(int m, int p);
bbl_status ritz_cr(int m, int p, int nev, int nseg, const double* Tb, double* theta, double* S, double* ws, void* fast,
                   int** need, SegArgs sa, cudaStream_t st);

}  // namespace bbl
