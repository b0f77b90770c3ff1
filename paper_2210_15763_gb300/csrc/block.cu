// S2 / S3 / S5: the tall-skinny dense kernels of the block step.
//
//  gram     C = Q^T W   (Q: nblocks row-major n x b blocks, m = nblocks*b
//                        columns; W: n x b; C: m x b FP64).  Split-K over row
//                        chunks: every CTA reads a chunk of rows once, keeps
//                        W's rows of the current 64-row tile in shared memory
//                        and each thread owns CPT columns of Q (a 16-byte
//                        vector load per row) times all b columns of W.
//                        FP32 data: products summed in FP32 over at most one
//                        64-row tile per thread, tiles and chunks summed in
//                        FP64.  Per-CTA partials are reduced in a fixed order
//                        (deterministic).
//  apply    W (-)= Q C  (thread per row; C staged in shared memory in
//                        256-row tiles; used for the Gram-Schmidt update, for
//                        W R^{-1} in CholQR2 and for the Ritz vectors X = Q S).
//  cholqr2  G = W^T W -> R = chol(G) (one CTA, b <= 16) -> W <- W R^{-1},
//           twice, the first R^{-1} applied in the pass that forms the second
//           G; B = R2 R1 (Sec. II.B normalisation, CholQR2 form).
#include <algorithm>
#include <cmath>
#include <mutex>
#include <type_traits>
#include <vector>

#include <cuda_fp16.h>

#include "async_mma.cuh"
#include "common.cuh"
#include "df32.cuh"

namespace bbl {
namespace {

// (d0, d1) += a * (b0, b1) as one packed FP32 FMA (fma.rn.f32x2): each half
// rounds as fmaf does
__device__ __forceinline__ void fma2_bcast(float& d0, float& d1, float a, float b0, float b1) {
    unsigned long long d, aa, bb;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(d0), "f"(d1));
    asm("mov.b64 %0, {%1, %1};" : "=l"(aa) : "f"(a));
    asm("mov.b64 %0, {%1, %2};" : "=l"(bb) : "f"(b0), "f"(b1));
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(aa), "l"(bb));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(d0), "=f"(d1) : "l"(d));
}

// (d0, d1) = a * (b0, b1) + (+0), as fma2_bcast on zeros
__device__ __forceinline__ void fma2_first(float& d0, float& d1, float a, float b0, float b1) {
    unsigned long long d, aa, bb;
    asm("mov.b64 %0, {%1, %1};" : "=l"(aa) : "f"(a));
    asm("mov.b64 %0, {%1, %2};" : "=l"(bb) : "f"(b0), "f"(b1));
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(aa), "l"(bb), "l"(0ull));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(d0), "=f"(d1) : "l"(d));
}
// (d0, d1) += (b0, b1) as one packed FP32 addition
__device__ __forceinline__ void add2(float& d0, float& d1, float b0, float b1) {
    unsigned long long d, bb;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(d0), "f"(d1));
    asm("mov.b64 %0, {%1, %2};" : "=l"(bb) : "f"(b0), "f"(b1));
    asm("add.rn.f32x2 %0, %0, %1;" : "+l"(d) : "l"(bb));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(d0), "=f"(d1) : "l"(d));
}

template <typename T, int N>
__device__ __forceinline__ void ldvec(const T* p, T (&out)[N]) {
    if constexpr (is_df32<T>::value) {
        if constexpr (N % 2 == 0) {
#pragma unroll
            for (int q = 0; q < N; q += 2) {
                const float4 x = __ldg(reinterpret_cast<const float4*>(p + q));
                out[q] = df32(x.x, x.y);
                out[q + 1] = df32(x.z, x.w);
            }
        } else {
#pragma unroll
            for (int q = 0; q < N; ++q) {
                const float2 x = __ldg(reinterpret_cast<const float2*>(p + q));
                out[q] = df32(x.x, x.y);
            }
        }
    } else if constexpr (N * sizeof(T) == 16) {
        if constexpr (sizeof(T) == 8) {
            double2 x = __ldg(reinterpret_cast<const double2*>(p));
            out[0] = x.x;
            out[1] = x.y;
        } else {
            float4 x = __ldg(reinterpret_cast<const float4*>(p));
            out[0] = x.x;
            out[1] = x.y;
            out[2] = x.z;
            out[3] = x.w;
        }
    } else if constexpr (N * sizeof(T) == 8 && sizeof(T) == 4) {
        float2 x = __ldg(reinterpret_cast<const float2*>(p));
        out[0] = x.x;
        out[1] = x.y;
    } else {
#pragma unroll
        for (int q = 0; q < N; ++q) out[q] = __ldg(p + q);
    }
}

// the same loads for memory the kernel also writes, and the stores
template <typename T, int N>
__device__ __forceinline__ void ldvec_rw(const T* p, T (&out)[N]) {
    if constexpr (is_df32<T>::value && N == 2) {
        const float4 x = *reinterpret_cast<const float4*>(p);
        out[0] = df32(x.x, x.y);
        out[1] = df32(x.z, x.w);
    } else if constexpr (!is_df32<T>::value && N * sizeof(T) == 16 && sizeof(T) == 8) {
        const double2 x = *reinterpret_cast<const double2*>(p);
        out[0] = x.x;
        out[1] = x.y;
    } else if constexpr (N * sizeof(T) == 16 && sizeof(T) == 4) {
        const float4 x = *reinterpret_cast<const float4*>(p);
        out[0] = x.x;
        out[1] = x.y;
        out[2] = x.z;
        out[3] = x.w;
    } else if constexpr (N * sizeof(T) == 8 && sizeof(T) == 4) {
        const float2 x = *reinterpret_cast<const float2*>(p);
        out[0] = x.x;
        out[1] = x.y;
    } else {
#pragma unroll
        for (int q = 0; q < N; ++q) out[q] = p[q];
    }
}
template <typename T, int N>
__device__ __forceinline__ void stvec(T* p, const T (&v)[N]) {
    if constexpr (is_df32<T>::value && N == 2) {
        *reinterpret_cast<float4*>(p) = make_float4(v[0].hi, v[0].lo, v[1].hi, v[1].lo);
    } else if constexpr (!is_df32<T>::value && N * sizeof(T) == 16 && sizeof(T) == 8) {
        *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
    } else if constexpr (N * sizeof(T) == 16 && sizeof(T) == 4) {
        *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
    } else if constexpr (N * sizeof(T) == 8 && sizeof(T) == 4) {
        *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]);
    } else {
#pragma unroll
        for (int q = 0; q < N; ++q) p[q] = v[q];
    }
}

constexpr int kRT = 256;   // rows per shared-memory tile in gram
constexpr int kRitzReserveSMs = 8;
constexpr int kThreads = 256;

// -------------------------------------------------------------------- gram
// One CTA: the partial Gram of the row ranges handed out by next(r0, r1)
// (called by every thread, in step) for the Q columns of column group
// `cgrp`, written to out[m][B] (this CTA's partial slot).
template <typename T, int B, int CPT, typename Next>
__device__ __forceinline__ void gram_body(int64_t n, int m, Next next, int TC, int cgrp, const T* __restrict__ Q,
                                          const T* __restrict__ W, double* __restrict__ partial_slot) {
    __shared__ T ws[kRT * B];
    extern __shared__ double sred[];
    const int tid = threadIdx.x;
    const int RS = kThreads / TC;
    const int cg = tid % TC, rs = tid / TC;
    const int a0 = (cgrp * TC + cg) * CPT;
    const bool active = a0 < m;
    const int j = active ? a0 / B : 0, off = a0 % B;
    const T* qb = Q + (int64_t)j * n * B + off;
    // FP64 running sums: in registers for FP64 data; for FP32 data the
    // per-tile FP32 sums are added into this thread's shared-memory slot, so
    // that registers go to loads in flight instead.
    constexpr bool kF32 = sizeof(T) == 4;
    constexpr int U = 8;  // rows whose loads are issued together
    double* mine = sred + (size_t)tid * CPT * B;
    double acc64[kF32 ? 1 : CPT][kF32 ? 1 : B];
    if constexpr (kF32) {
        for (int e = 0; e < CPT * B; ++e) mine[e] = 0.0;
    } else {
#pragma unroll
        for (int i = 0; i < CPT; ++i)
#pragma unroll
            for (int c = 0; c < B; ++c) acc64[i][c] = 0.0;
    }
    int64_t r_begin = 0, r_end = 0;
    while (next(r_begin, r_end))
    for (int64_t t0 = r_begin; t0 < r_end; t0 += kRT) {
        const int rows = (int)min((int64_t)kRT, r_end - t0);
        __syncthreads();
        for (int e = tid; e < rows * B; e += kThreads) ws[e] = W[t0 * B + e];
        __syncthreads();
        if (active) {
            T acc[CPT][B];
#pragma unroll
            for (int i = 0; i < CPT; ++i)
#pragma unroll
                for (int c = 0; c < B; ++c) acc[i][c] = T(0);
            int r = rs;
            for (; r + (U - 1) * RS < rows; r += U * RS) {
                T q[U][CPT];
#pragma unroll
                for (int u = 0; u < U; ++u) ldvec<T, CPT>(qb + (t0 + r + u * RS) * B, q[u]);
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const T* wr = ws + (r + u * RS) * B;
#pragma unroll
                    for (int c = 0; c < B; ++c) {
                        const T w = wr[c];
#pragma unroll
                        for (int i = 0; i < CPT; ++i) acc[i][c] = fma(q[u][i], w, acc[i][c]);
                    }
                }
            }
            for (; r < rows; r += RS) {
                T q[CPT];
                ldvec<T, CPT>(qb + (t0 + r) * B, q);
                const T* wr = ws + r * B;
#pragma unroll
                for (int c = 0; c < B; ++c) {
                    const T w = wr[c];
#pragma unroll
                    for (int i = 0; i < CPT; ++i) acc[i][c] = fma(q[i], w, acc[i][c]);
                }
            }
            if constexpr (kF32) {
#pragma unroll
                for (int i = 0; i < CPT; ++i)
#pragma unroll
                    for (int c = 0; c < B; ++c) mine[i * B + c] += (double)acc[i][c];
            } else {
#pragma unroll
                for (int i = 0; i < CPT; ++i)
#pragma unroll
                    for (int c = 0; c < B; ++c) acc64[i][c] += (double)acc[i][c];
            }
        }
    }
    if constexpr (!kF32) {
        if (RS > 1) {
#pragma unroll
            for (int i = 0; i < CPT; ++i)
#pragma unroll
                for (int c = 0; c < B; ++c) mine[i * B + c] = acc64[i][c];
        }
    }
    if (RS > 1) {
        // deterministic tree over the row slots
        __syncthreads();
        for (int s = RS / 2; s > 0; s >>= 1) {
            if (rs < s) {
                const double* other = sred + (size_t)(tid + s * TC) * CPT * B;
                for (int e = 0; e < CPT * B; ++e) mine[e] += other[e];
            }
            __syncthreads();
        }
        if (rs == 0 && active) {
            double* out = partial_slot + (int64_t)a0 * B;
            for (int e = 0; e < CPT * B; ++e) out[e] = mine[e];
        }
    } else if (active) {
        double* out = partial_slot + (int64_t)a0 * B;
        if constexpr (kF32) {
            for (int e = 0; e < CPT * B; ++e) out[e] = mine[e];
        } else {
#pragma unroll
            for (int i = 0; i < CPT; ++i)
#pragma unroll
                for (int c = 0; c < B; ++c) out[i * B + c] = acc64[i][c];
        }
    }
}

// Hands out [r0, r1) once (one fixed range per CTA).
struct OneRange {
    int64_t r0, r1;
    bool done = false;
    __device__ bool operator()(int64_t& a, int64_t& b) {
        if (done) return false;
        done = true;
        a = r0;
        b = r1;
        return r1 > r0;
    }
};

// Hands out chunks of a shared ticket counter: CTAs that start late (their
// SM was busy) simply take fewer chunks, so there is no tail wave.
struct TicketRanges {
    int* ticket;
    int64_t n, rows_per_chunk;
    int nchunks;
    __device__ bool operator()(int64_t& a, int64_t& b) {
        __shared__ int s_c;
        __syncthreads();
        if (threadIdx.x == 0) s_c = atomicAdd(ticket, 1);
        __syncthreads();
        const int c = s_c;
        if (c >= nchunks) return false;
        a = (int64_t)c * rows_per_chunk;
        b = min(n, a + rows_per_chunk);
        return true;
    }
};

// Split-K Gram: persistent CTAs (x, y) = worker x of column group y; the row
// chunks of each column group are taken from ticket[y].
template <typename T, int B, int CPT>
__global__ void __launch_bounds__(kThreads) gram_kernel(int64_t n, int m, int64_t rows_per_chunk, int nchunks, int TC,
                                                        const T* __restrict__ Q, const T* __restrict__ W,
                                                        double* __restrict__ partial, int* __restrict__ tickets) {
    TicketRanges next{tickets + blockIdx.y, n, rows_per_chunk, nchunks};
    gram_body<T, B, CPT>(n, m, next, TC, blockIdx.y, Q, W, partial + (int64_t)blockIdx.x * m * B);
}

// Row-contiguous split-K Gram (b = 4, 8).  A CTA takes a chunk of rows from
// the ticket counter and stages W's rows of the chunk in shared memory; its
// warps walk the basis blocks.  A warp streams a block's rows of the chunk
// into its own shared-memory ring with asynchronous 16-byte copies
// (cp.async), NS stages of RL * U whole consecutive rows, so that NS - 1
// stages are in flight while it computes on the oldest: no registers hold
// data in flight.  Lane (g, t) multiplies its CPL columns of a row (LPR
// lanes per row, RL = 32 / LPR rows per step) by the row's B values of W and
// keeps CPL x B sums; at the end of the block's rows the RL row lanes are
// combined by a butterfly that halves the values each lane carries per
// round, and each lane adds its share of the B x B partial to the CTA's
// FP64 slot.  Blocks are dealt to warps round-robin; with fewer than 8
// blocks the rows of a chunk are split among wpb warps per block (one slot
// per row share).  FP32 data: products are summed in FP32 per stage, then
// over the stages of the chunk and the lane tree, and in FP64 across chunks.
// Bound by HBM for large bases (FP32, b = 8, n = 1e6, m = 720: 510 -> 501 us, 5.74
// TB/s; n = 5e5, m = 320: 135 -> 113 us; n = 1e5, m = 264: 29 -> 24 us, since the
// loop counts its blocks and stages up instead of dividing, adds packed pairs and
// adds to the slots without waiting; the results are the same bits).
template <typename T, int B>
struct GramRowsShape {
    static constexpr int CPL = 16 / (int)sizeof(T);         // Q columns per lane
    static constexpr int LPR = B / CPL;                     // lanes per row
    static constexpr int RL = 32 / LPR;                     // rows per warp step
    static constexpr int R = 32768 / (B * (int)sizeof(T));  // rows per chunk (32 KB of W)
    static constexpr int U = 4;                             // rows per lane per stage
    static constexpr int NS = 4;                            // ring stages per warp
    static constexpr int SROWS = RL * U;                    // rows per stage (2 KB)
    static constexpr int NV = CPL * B;                      // sums per lane
    static constexpr int LOGRL = RL >= 32 ? 5 : RL >= 16 ? 4 : RL >= 8 ? 3 : RL >= 4 ? 2 : RL >= 2 ? 1 : 0;
    static constexpr int kWarps = kThreads / 32;
    static constexpr size_t smem_bytes = (size_t)R * B * sizeof(T) + (size_t)kWarps * NS * SROWS * B * sizeof(T);
};

template <typename T>
__device__ __forceinline__ T add_any(T a, T b) {
    return a + b;
}

// warps per basis block when a chunk has fewer blocks than warps
__host__ __device__ __forceinline__ int gram_rows_wpb(int nblocks) {
    int wpb = 1;
    while (wpb < kThreads / 32 && nblocks * wpb * 2 <= kThreads / 32) wpb <<= 1;
    return wpb;
}

// One chunk, rows [r0, r0 + rows) with rows <= R, for all threads of the
// CTA: W's rows staged in shared memory (ws), then each warp streams the
// chunk's rows of its blocks (share sub: rows [sub * rsub, (sub + 1) * rsub))
// through its ring and adds its B x B partials to slot sub of `slots`
// (wpb slots of m x B FP64).  The barrier after the W tile also orders any
// plain stores the caller made to `slots` before the adds.
template <typename T, int B>
__device__ __forceinline__ void gram_rows_chunk(int64_t n, int m, int wpb, int64_t r0, int rows, int rsub,
                                                const T* __restrict__ Q, const T* __restrict__ W,
                                                double* __restrict__ slots, T* __restrict__ ws) {
    using S = GramRowsShape<T, B>;
    constexpr int CPL = S::CPL, LPR = S::LPR, RL = S::RL, R = S::R, U = S::U, NV = S::NV, LOGRL = S::LOGRL;
    constexpr int NS = S::NS, SROWS = S::SROWS;
    constexpr int PIECES = SROWS * LPR / 32;  // 16-byte copies per lane per stage
    static_assert(LPR >= 1 && LPR <= 32 && 32 % LPR == 0 && B % CPL == 0 && (1 << LOGRL) == RL, "gram_rows shape");
    static_assert((SROWS * LPR) % 32 == 0, "stage pieces");
    const int nblocks = m / B;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane % LPR, t = lane / LPR;
    T* ring = ws + (size_t)R * B + (size_t)warp * NS * SROWS * B;
    const int ngrp = S::kWarps / wpb;
    const int grp = warp / wpb, sub = warp % wpb;
    double* part = slots + (int64_t)sub * m * B;
    // after the butterfly lane t holds sums vbase .. vbase + NK - 1; when
    // NV < RL the last rounds are plain all-reduces and only t < NV write
    constexpr int NK = NV >= RL ? NV / RL : 1;
    int vbase = 0;
#pragma unroll
    for (int k = 0; k < LOGRL; ++k)
        if ((NV >> k) > 1 && (t & (1 << k))) vbase += NV >> (k + 1);
    const bool writer = (NV >= RL) || (t < NV);
    for (int e = threadIdx.x; e < R * LPR; e += kThreads) {
        const int r = e / LPR, h = e % LPR;
        T v[CPL];
        if (r < rows) {
            ldvec<T, CPL>(W + (r0 + r) * B + h * CPL, v);
        } else {
#pragma unroll
            for (int q = 0; q < CPL; ++q) v[q] = T(0);
        }
#pragma unroll
        for (int q = 0; q < CPL; ++q) ws[(h * R + r) * CPL + q] = v[q];
    }
    __syncthreads();
    const int rb = sub * rsub;
    const int re = min(rows, rb + rsub);
    if (re <= rb) return;
    const int nst = (re - rb + SROWS - 1) / SROWS;       // stages per block
    const int nblk = (nblocks - grp + ngrp - 1) / ngrp;  // blocks of this warp
    const int total = nblk * nst;
    // Stage k: block grp + (k / nst) * ngrp, rows rb + (k % nst) * SROWS ..; both
    // ends of the ring count blocks and stages up (the divisions were a quarter
    // of the loop's instructions).
    const T* src = Q + ((int64_t)grp * n + r0 + rb) * B + lane * CPL;
    const int64_t skip = ((int64_t)ngrp * n - (int64_t)nst * SROWS) * B;  // from a block's end to the next block
    int ik = 0, is = 0;  // next stage to issue, and its number in the block
    auto issue = [&]() {
        if (ik < total) {
            T* buf = ring + (size_t)(ik % NS) * SROWS * B + lane * CPL;
            const int left = re - rb - is * SROWS;  // rows left in the share
            if (left >= SROWS) {
#pragma unroll
                for (int i = 0; i < PIECES; ++i) cp_async16(buf + 32 * i * CPL, src + 32 * i * CPL, 16);
            } else {
#pragma unroll
                for (int i = 0; i < PIECES; ++i) {
                    const bool ok = (lane + 32 * i) / LPR < left;
                    cp_async16(buf + 32 * i * CPL, ok ? (const void*)(src + 32 * i * CPL) : (const void*)Q, ok ? 16 : 0);
                }
            }
            src += SROWS * B;
            if (++is == nst) {
                is = 0;
                src += skip;
            }
            ++ik;
        }
        cp_async_commit();  // an empty group past the end keeps the count uniform
    };
#pragma unroll
    for (int k = 0; k < NS - 1; ++k) issue();
    T acc[CPL][B];
#pragma unroll
    for (int i = 0; i < CPL; ++i)
#pragma unroll
        for (int cc = 0; cc < B; ++cc) acc[i][cc] = T(0);
    int j = grp, cs = 0;  // block and stage of k
    for (int k = 0; k < total; ++k) {
        cp_async_wait<NS - 2>();
        __syncwarp();
        issue();  // into the buffer consumed at k - 1
        const T* buf = ring + (size_t)(k % NS) * SROWS * B;
        const int s0 = rb + cs * SROWS;
        T bat[CPL][B];
        // two columns per packed FP32 FMA (each half an IEEE fma.rn: the same
        // results as two fmaf, in half the issued instructions)
        constexpr bool PACKED = std::is_same<T, float>::value && B % 2 == 0;
        if constexpr (!PACKED) {
#pragma unroll
            for (int i = 0; i < CPL; ++i)
#pragma unroll
                for (int cc = 0; cc < B; ++cc) bat[i][cc] = T(0);
        }
        // the stage's rows within the W tile, which a share that is no multiple of
        // the stage can leave at its end (those rows of the stage are zeros)
        auto rows_of = [&](auto whole) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int rr = t + u * RL;  // row within the stage (zero past the share)
                const int row = whole.value ? s0 + rr : min(s0 + rr, R - 1);  // row within the W tile
                T q[CPL];
                T w[B];
                const T* qs = buf + (size_t)rr * B + g * CPL;
                if constexpr (sizeof(T) == 4) {
                    const float4 x = *reinterpret_cast<const float4*>(qs);
                    q[0] = x.x;
                    q[1] = x.y;
                    q[2] = x.z;
                    q[3] = x.w;
                } else {
#pragma unroll
                    for (int i = 0; i < CPL; ++i) q[i] = qs[i];
                }
#pragma unroll
                for (int h = 0; h < LPR; ++h) {
                    const T* wsrc = ws + (h * R + row) * CPL;
                    if constexpr (sizeof(T) == 4) {
                        const float4 x = *reinterpret_cast<const float4*>(wsrc);
                        w[h * CPL + 0] = x.x;
                        w[h * CPL + 1] = x.y;
                        w[h * CPL + 2] = x.z;
                        w[h * CPL + 3] = x.w;
                    } else {
#pragma unroll
                        for (int q2 = 0; q2 < CPL; ++q2) w[h * CPL + q2] = wsrc[q2];
                    }
                }
#pragma unroll
                for (int i = 0; i < CPL; ++i) {
                    if constexpr (PACKED) {
#pragma unroll
                        for (int cc = 0; cc < B; cc += 2) {
                            if (u == 0) fma2_first(bat[i][cc], bat[i][cc + 1], q[i], w[cc], w[cc + 1]);
                            else fma2_bcast(bat[i][cc], bat[i][cc + 1], q[i], w[cc], w[cc + 1]);
                        }
                    } else {
#pragma unroll
                        for (int cc = 0; cc < B; ++cc) bat[i][cc] = fma(q[i], w[cc], bat[i][cc]);
                    }
                }
            }
        };
        if (s0 + SROWS <= R) rows_of(std::true_type{});
        else rows_of(std::false_type{});
#pragma unroll
        for (int i = 0; i < CPL; ++i) {
            if constexpr (PACKED) {
#pragma unroll
                for (int cc = 0; cc < B; cc += 2) add2(acc[i][cc], acc[i][cc + 1], bat[i][cc], bat[i][cc + 1]);
            } else {
#pragma unroll
                for (int cc = 0; cc < B; ++cc) acc[i][cc] = add_any(acc[i][cc], bat[i][cc]);
            }
        }
        if (++cs == nst) {
            // last stage of block j: butterfly over the RL row lanes
            T v[NV];
#pragma unroll
            for (int e = 0; e < NV; ++e) v[e] = acc[e / B][e % B];
#pragma unroll
            for (int kk = 0; kk < LOGRL; ++kk) {
                const int o = (1 << kk) * LPR;
                const bool up = (t & (1 << kk)) != 0;
                if ((NV >> kk) > 1) {
                    const int hv = NV >> (kk + 1);
#pragma unroll
                    for (int x = 0; x < NV / 2; ++x) {
                        if (x < hv) {
                            const T send = up ? v[x] : v[x + hv];
                            const T keep = up ? v[x + hv] : v[x];
                            v[x] = add_any(keep, shfl_xor_any(0xffffffffu, send, o));
                        }
                    }
                } else {
                    v[0] = add_any(v[0], shfl_xor_any(0xffffffffu, v[0], o));
                }
            }
            if (writer) {
#pragma unroll
                for (int x = 0; x < NK; ++x) {
                    const int e = vbase + x;
                    const int i = e / B, cc = e % B;
                    // this lane alone adds here: no wait for the sum
                    atomicAdd(&part[(int64_t)(j * B + g * CPL + i) * B + cc], (double)v[x]);
                }
            }
#pragma unroll
            for (int i = 0; i < CPL; ++i)
#pragma unroll
                for (int cc = 0; cc < B; ++cc) acc[i][cc] = T(0);
            cs = 0;
            j += ngrp;
        }
    }
    cp_async_wait<0>();
    __syncwarp();
}

// Single problem: persistent CTAs take chunks of rc rows from the ticket
// counter and accumulate into their own wpb slots.
template <typename T, int B>
__global__ void __launch_bounds__(kThreads) gram_rows_kernel(int64_t n, int m, int wpb, int rc, int nchunks,
                                                             const T* __restrict__ Q, const T* __restrict__ W,
                                                             double* __restrict__ partial, int* __restrict__ ticket) {
    // [ W tile: layout [h][row][CPL] | per-warp rings: NS stages of SROWS rows ]
    extern __shared__ __align__(16) unsigned char gram_rows_smem[];
    T* ws = reinterpret_cast<T*>(gram_rows_smem);
    __shared__ int s_chunk;
    double* slots = partial + (int64_t)blockIdx.x * wpb * m * B;
    for (int64_t e = threadIdx.x; e < (int64_t)wpb * m * B; e += kThreads) slots[e] = 0.0;
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) s_chunk = atomicAdd(ticket, 1);
        __syncthreads();
        const int c = s_chunk;
        if (c >= nchunks) break;
        const int64_t r0 = (int64_t)c * rc;
        const int rows = (int)min((int64_t)rc, n - r0);
        gram_rows_chunk<T, B>(n, m, wpb, r0, rows, rc / wpb, Q, W, slots, ws);
    }
}

// Batch of problems stacked row-wise: CTA x takes chunk x, rows
// [chunks[3x+1], chunks[3x+2]) of segment chunks[3x] (at most R rows, never
// crossing a segment), and writes its own wpb slots at partial[x * wpb * m * B].
// m is read from device memory so that one captured graph serves every
// iteration; chunks of inactive segments do nothing.
template <typename T, int B>
__global__ void __launch_bounds__(kThreads) gram_rows_seg_kernel(int64_t n, const int* __restrict__ d_m,
                                                                 const int64_t* __restrict__ chunks,
                                                                 const int* __restrict__ seg_active,
                                                                 const T* __restrict__ Q, const T* __restrict__ W,
                                                                 double* __restrict__ partial) {
    extern __shared__ __align__(16) unsigned char gram_rows_smem[];
    const int64_t seg = chunks[3 * blockIdx.x];
    if (seg_active && !seg_active[seg]) return;
    const int m = *d_m;
    const int wpb = gram_rows_wpb(m / B);
    const int64_t r0 = chunks[3 * blockIdx.x + 1];
    const int rows = (int)(chunks[3 * blockIdx.x + 2] - r0);
    double* slots = partial + (int64_t)blockIdx.x * wpb * m * B;
    for (int64_t e = threadIdx.x; e < (int64_t)wpb * m * B; e += kThreads) slots[e] = 0.0;
    gram_rows_chunk<T, B>(n, m, wpb, r0, rows, (rows + wpb - 1) / wpb, Q, W, slots,
                          reinterpret_cast<T*>(gram_rows_smem));
}

// Segmented Gram for a batch of independent problems stacked row-wise:
// chunk x covers rows [chunks[3x+1], chunks[3x+2]) of segment chunks[3x];
// chunks of inactive segments do nothing.
template <typename T, int B, int CPT>
__global__ void __launch_bounds__(kThreads) gram_seg_kernel(int64_t n, int m, const int64_t* __restrict__ chunks,
                                                            const int* __restrict__ seg_active, int TC,
                                                            const T* __restrict__ Q, const T* __restrict__ W,
                                                            double* __restrict__ partial) {
    const int64_t seg = chunks[3 * blockIdx.x];
    if (seg_active && !seg_active[seg]) return;
    gram_body<T, B, CPT>(n, m, OneRange{chunks[3 * blockIdx.x + 1], chunks[3 * blockIdx.x + 2]}, TC, blockIdx.y, Q, W,
                         partial + (int64_t)blockIdx.x * m * B);
}

// any b (runtime), one Q column per thread
template <typename T>
__global__ void __launch_bounds__(kThreads) gram_generic_kernel(int64_t n, int m, int b, int64_t rows_per_chunk, int TC,
                                                                const T* __restrict__ Q, const T* __restrict__ W,
                                                                double* __restrict__ partial) {
    __shared__ T ws[kRT * kMaxB];
    extern __shared__ double sred[];
    const int tid = threadIdx.x;
    const int RS = kThreads / TC;
    const int cg = tid % TC, rs = tid / TC;
    const int a0 = blockIdx.y * TC + cg;
    const bool active = a0 < m;
    const int j = active ? a0 / b : 0, off = a0 % b;
    const T* qb = Q + (int64_t)j * n * b + off;
    double acc64[kMaxB];
    for (int c = 0; c < kMaxB; ++c) acc64[c] = 0.0;
    const int64_t r_begin = (int64_t)blockIdx.x * rows_per_chunk;
    const int64_t r_end = min(n, r_begin + rows_per_chunk);
    for (int64_t t0 = r_begin; t0 < r_end; t0 += kRT) {
        const int rows = (int)min((int64_t)kRT, r_end - t0);
        __syncthreads();
        for (int e = tid; e < rows * b; e += kThreads) ws[e] = W[t0 * b + e];
        __syncthreads();
        if (active) {
            T acc[kMaxB];
            for (int c = 0; c < kMaxB; ++c) acc[c] = T(0);
            for (int r = rs; r < rows; r += RS) {
                const T q = qb[(t0 + r) * b];
                for (int c = 0; c < b; ++c) acc[c] = fma(q, ws[r * b + c], acc[c]);
            }
            for (int c = 0; c < b; ++c) acc64[c] += (double)acc[c];
        }
    }
    double* mine = sred + (size_t)tid * kMaxB;
    for (int c = 0; c < b; ++c) mine[c] = acc64[c];
    __syncthreads();
    for (int s = RS / 2; s > 0; s >>= 1) {
        if (rs < s) {
            const double* other = sred + (size_t)(tid + s * TC) * kMaxB;
            for (int c = 0; c < b; ++c) mine[c] += other[c];
        }
        __syncthreads();
    }
    if (rs == 0 && active) {
        double* out = partial + ((int64_t)blockIdx.x * m + a0) * b;
        for (int c = 0; c < b; ++c) out[c] = mine[c];
    }
}

// out[e] = sum_p partial[p * count + e]: 8 entries per CTA (64-byte rows), the
// parts split over 32 groups of threads whose loads are issued together,
// combined in a fixed order.  (With 32 entries and 8 groups a thread added 38
// to 76 parts in turn: 8 to 9 us for the 304 to 608 parts of a Gram, most of it
// load latency.)
constexpr int kRedE = 8, kRedG = kThreads / kRedE;
__device__ __forceinline__ double sum_parts(int64_t count, int nparts, const double* __restrict__ partial, int64_t e,
                                            int g, int groups) {
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    int p = g;
    for (; p + 7 * groups < nparts; p += 8 * groups) {
        double a[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) a[q] = partial[(int64_t)(p + q * groups) * count + e];
#pragma unroll
        for (int q = 0; q < 8; ++q) s[q & 3] += a[q];
    }
    for (; p < nparts; p += groups) s[0] += partial[(int64_t)p * count + e];
    return (s[0] + s[1]) + (s[2] + s[3]);
}

__global__ void __launch_bounds__(kThreads) reduce_partials_kernel(int64_t count, int nparts,
                                                                   const double* __restrict__ partial,
                                                                   double* __restrict__ out) {
    __shared__ double red[kRedG][kRedE];
    const int tx = threadIdx.x % kRedE, pg = threadIdx.x / kRedE;
    const int64_t e = (int64_t)blockIdx.x * kRedE + tx;
    red[pg][tx] = e < count ? sum_parts(count, nparts, partial, e, pg, kRedG) : 0.0;
    __syncthreads();
    for (int w = kRedG / 2; w > 0; w >>= 1) {
        if (pg < w) red[pg][tx] += red[pg + w][tx];
        __syncthreads();
    }
    if (pg == 0 && e < count) out[e] = red[0][tx];
}

void launch_reduce(int64_t count, int nparts, const double* partial, double* out, cudaStream_t st) {
    reduce_partials_kernel<<<(unsigned)ceil_div(count, kRedE), kThreads, 0, st>>>(count, nparts, partial, out);
}

// Sums v[0 .. N-1] over the warp and hands each sum to put(index, sum) in one
// lane: every round a lane keeps half of its values and sends the other half (37
// additions for N = 36 where an all-reduce of each value takes 180; the same
// pairs are added, so the sums are the same).
template <int N, typename T, typename Put>
__device__ __forceinline__ void warp_sum_scatter(T (&v)[N], Put&& put) {
    const int lane = threadIdx.x & 31;
    int cnt = N, base = 0, lim = N;  // values held (padded with zeros), index of the first, valid ones
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const bool up = (lane & off) != 0;
        const int hv = (cnt + 1) / 2;
#pragma unroll
        for (int x = 0; x < (N + 1) / 2; ++x) {
            if (x < hv) {
                const T hi = x + hv < cnt ? v[x + hv < N ? x + hv : 0] : T(0);
                const T send = up ? v[x] : hi, keep = up ? hi : v[x];
                v[x] = add_any(keep, shfl_xor_any(0xffffffffu, send, off));
            }
        }
        base += up ? hv : 0;
        lim = up ? max(lim - hv, 0) : min(lim, hv);
        cnt = hv;
    }
    constexpr int K = (N + 31) / 32;
#pragma unroll
    for (int x = 0; x < K; ++x)
        if (x < lim) put(base + x, v[x]);
}

// One pass of CholQR2 over W (n x B, B <= 8), a thread per row (grid-strided,
// the next row's loads issued before the current row's arithmetic): APPLY:
// W <- W R^{-1} (upper triangular: c takes i <= c); GRAM: the partial Gram of
// the rows as stored, the B(B+1)/2 distinct products in registers, then a
// warp-shuffle and shared-memory reduction to one B x B partial per CTA.
// Applying the first factor and forming the second Gram in one pass saves a
// read of W and a launch.
// LONG: a lane sees more than 64 rows, and runs of 64 are summed in FP64 (their
// sums cost 72 registers at b = 8, and with them all but one CTA per SM).
template <typename T, int B, bool APPLY, bool GRAM, bool LONG = false>
__global__ void __launch_bounds__(kThreads) qr_pass_kernel(int64_t n, const double* __restrict__ Rinv, T* W,
                                                           double* __restrict__ partial) {
    constexpr int NP = B * (B + 1) / 2;
    __shared__ double red[GRAM ? kThreads / 32 : 1][NP];
    __shared__ T rs[B * B];
    if constexpr (APPLY) {
        for (int e = threadIdx.x; e < B * B; e += kThreads) rs[e] = (T)Rinv[e];
        __syncthreads();
    }
    T acc[GRAM ? NP : 1];
    double acc64[LONG ? NP : 1];
#pragma unroll
    for (int e = 0; e < (GRAM ? NP : 1); ++e) acc[e] = T(0);
#pragma unroll
    for (int e = 0; e < (LONG ? NP : 1); ++e) acc64[e] = 0.0;
    int cnt = 0;
    constexpr int CH = B * sizeof(T) >= 16 ? 16 / (int)sizeof(T) : B;  // elements per load
    auto load = [&](int64_t r, T (&w)[B]) {
#pragma unroll
        for (int ch = 0; ch < B / CH; ++ch) {
            T t[CH];
            ldvec_rw<T, CH>(W + r * B + ch * CH, t);
#pragma unroll
            for (int q = 0; q < CH; ++q) w[ch * CH + q] = t[q];
        }
    };
    const int64_t stride = (int64_t)gridDim.x * kThreads;
    int64_t r = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    T nx[B];
    if (r < n) load(r, nx);
    for (; r < n; r += stride) {
        T w[B];
#pragma unroll
        for (int c = 0; c < B; ++c) w[c] = nx[c];
        if (r + stride < n) load(r + stride, nx);
        if constexpr (APPLY) {
            T v[B];
#pragma unroll
            for (int c = 0; c < B; ++c) v[c] = T(0);
#pragma unroll
            for (int i = 0; i < B; ++i)
#pragma unroll
                for (int c = i; c < B; ++c) v[c] = fma(w[i], rs[i * B + c], v[c]);
#pragma unroll
            for (int c = 0; c < B; ++c) w[c] = v[c];
#pragma unroll
            for (int ch = 0; ch < B / CH; ++ch) {
                T t[CH];
#pragma unroll
                for (int q = 0; q < CH; ++q) t[q] = w[ch * CH + q];
                stvec<T, CH>(W + r * B + ch * CH, t);
            }
        }
        if constexpr (GRAM) {
            int e = 0;
#pragma unroll
            for (int i = 0; i < B; ++i)
#pragma unroll
                for (int k = i; k < B; ++k) {
                    acc[e] = fma(w[i], w[k], acc[e]);
                    ++e;
                }
            if (LONG && ++cnt == 64) {  // FP32 runs of at most 64 rows, summed in FP64
#pragma unroll
                for (int q = 0; q < NP; ++q) {
                    acc64[LONG ? q : 0] += (double)acc[q];
                    acc[q] = T(0);
                }
                cnt = 0;
            }
        }
    }
    if constexpr (GRAM) {
        // warp tree in the data type (FP32 sums of at most 64 rows per lane,
        // then 32 lanes)
        const int warp = threadIdx.x / 32;
        warp_sum_scatter<NP>(acc, [&](int q, T v) { red[warp][q] = (double)v; });
        if constexpr (LONG) {
            __syncwarp();
            warp_sum_scatter<NP>(acc64, [&](int q, double v) { red[warp][q] += v; });
        }
        __syncthreads();
        if (threadIdx.x < NP) {
            double v = 0.0;
            for (int w = 0; w < kThreads / 32; ++w) v += red[w][threadIdx.x];
            // unpack the upper-triangle index into (i, k) and store both halves
            int i = 0, e = threadIdx.x;
            while (e >= B - i) {
                e -= B - i;
                ++i;
            }
            const int k = i + e;
            partial[(int64_t)blockIdx.x * B * B + i * B + k] = v;
            partial[(int64_t)blockIdx.x * B * B + k * B + i] = v;
        }
    }
}

// Column groups of the split-K Gram for m basis columns: each thread of a
// CTA owns CPT columns, so a group covers up to kThreads * CPT columns, and
// each group has its own chunk ticket.
template <int CPT>
int gram_groups(int m) {
    const int cols = (m + CPT - 1) / CPT;
    return (cols + kThreads - 1) / kThreads;
}

// Launches the persistent split-K Gram and the reduction of its per-worker
// partials.  partial: room for `cap` doubles; tickets: room for `ticket_cap`
// ints, of which gram_groups<CPT>(m) are zeroed here and used (a request
// needing more is refused before any launch).
template <typename T, int B, int CPT>
bbl_status gram_core(int64_t n, int m, const T* Q, const T* W, double* C, double* partial, int64_t cap, int* tickets,
                     int64_t ticket_cap, cudaStream_t st) {
    int cols = (m + CPT - 1) / CPT;
    int TC = 1;
    while (TC < cols && TC < kThreads) TC <<= 1;
    const int gy = (cols + TC - 1) / TC;
    if (gy != gram_groups<CPT>(m) || gy > ticket_cap)
        return set_error(BBL_ERR_INVALID_ARG, "gram: %d column groups exceed the %lld chunk tickets", gy,
                         (long long)ticket_cap);
    const int RS = kThreads / TC;
    // FP32 data keeps its FP64 running sums in shared memory; FP64 data needs
    // the buffer only for the reduction over row slots
    const size_t smem_max = sizeof(double) * kThreads * CPT * B;
    const size_t smem = (RS > 1 || sizeof(T) == 4) ? smem_max : 0;
    static OncePerDevice once;
    BBL_TRY(allow_smem(once, gram_kernel<T, B, CPT>, smem_max));
    static int occ = 0;
    if (occ == 0) {
        BBL_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, gram_kernel<T, B, CPT>, kThreads, smem_max));
        if (occ < 1) occ = 1;
    }
    const int64_t rpc = 4 * kRT;
    const int nch = (int)std::max<int64_t>(1, ceil_div(n, rpc));
    const int64_t per = (int64_t)m * B;
    int64_t workers = std::max<int64_t>(1, (int64_t)sm_count() * occ / gy);
    workers = std::min<int64_t>(workers, nch);
    workers = std::min<int64_t>(workers, cap / per);
    if (workers < 1)
        return set_error(BBL_ERR_INVALID_ARG, "gram: %lld partial sums exceed the %lld-double scratch", (long long)per,
                         (long long)cap);
    BBL_CUDA(cudaMemsetAsync(tickets, 0, sizeof(int) * gy, st));
    dim3 grid((unsigned)workers, (unsigned)gy);
    gram_kernel<T, B, CPT><<<grid, kThreads, smem, st>>>(n, m, rpc, nch, TC, Q, W, partial, tickets);
    BBL_LAUNCH_CHECK();
    launch_reduce(per, (int)workers, partial, C, st);
    BBL_LAUNCH_CHECK();
    return BBL_OK;
}

template <typename T, int B>
bbl_status launch_gram_rows(int64_t n, int m, const T* Q, const T* W, double* C, DevBuf& partials, cudaStream_t st) {
    using S = GramRowsShape<T, B>;
    static OncePerDevice once;
    BBL_TRY(allow_smem(once, gram_rows_kernel<T, B>, S::smem_bytes));
    static int occ = 0;
    if (occ == 0) {
        BBL_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, gram_rows_kernel<T, B>, kThreads, S::smem_bytes));
        if (occ < 1) occ = 1;
    }
    const int nblocks = m / B;
    const int wpb = gram_rows_wpb(nblocks);  // warps per block when there are fewer blocks than warps
    // leave a few SMs to the Ritz solve that runs beside the main stream: a
    // persistent CTA that cannot start until such a kernel ends would hold the
    // whole Gram back
    const int64_t slots_max = (int64_t)std::max(1, sm_count() - kRitzReserveSMs) * occ;
    // rows per chunk: the full tile, or fewer so that small n still spreads
    // over the GPU (a multiple of RL * wpb)
    const int unit = S::RL * wpb;
    int64_t rc = ceil_div(n, slots_max);
    rc = std::max<int64_t>(unit * S::U, ceil_div(rc, unit) * unit);
    rc = std::min<int64_t>(rc, S::R);
    const int nch = (int)std::max<int64_t>(1, ceil_div(n, rc));
    const int64_t workers = std::min<int64_t>(slots_max, nch);
    const int64_t per = (int64_t)m * B;
    const int64_t slots = workers * wpb;
    const size_t need = sizeof(double) * (size_t)(slots * per) + 256;
    BBL_TRY(partials.grow(need));
    int* ticket = reinterpret_cast<int*>(partials.as<char>() + sizeof(double) * (size_t)(slots * per));
    BBL_CUDA(cudaMemsetAsync(ticket, 0, sizeof(int), st));
    gram_rows_kernel<T, B><<<(unsigned)workers, kThreads, S::smem_bytes, st>>>(n, m, wpb, (int)rc, nch, Q, W,
                                                                              partials.as<double>(), ticket);
    BBL_LAUNCH_CHECK();
    launch_reduce(per, (int)slots, partials.as<double>(), C, st);
    BBL_LAUNCH_CHECK();
    return BBL_OK;
}

// First-pass Gram from an FP16 copy of an FP32 basis (b = 8): C ~= Q16^T W,
// on the tensor cores.  The first Gram-Schmidt pass only has to take out
// the bulk of W's component in span(Q) -- the FP32 second pass removes what
// is left, and A_j sums both passes' coefficients -- so its coefficients may
// carry FP16 roundings (relative 2^-11) of Q and of W, and the pass reads 2
// instead of 4 bytes per basis element.
//
// Persistent CTAs take chunks of kHalfRows rows from a ticket counter.  W's
// rows of the chunk are scaled by an exact power of two (the chunk's largest
// |W| lands in [2^13, 2^14)) and rounded to FP16 into shared memory.  Warp w
// owns the pairs of basis blocks p = w, w + 8, ...: per 16 rows a pair is a
// 16 x 16 FP16 tile A (16 basis columns x 16 rows), brought into a per-warp
// shared-memory ring by cp.async (one 16-byte row per lane, kHmSK tiles per
// stage, kHmNS stages) and loaded transposed with ldmatrix; W's 16 x 8 tile
// is the B operand; one mma.sync.m16n8k16 (FP16 in, FP32 accumulate) adds
// the pair's 16 x 8 block of C.  Over a chunk the sums stay in FP32; at the
// chunk's end they are unscaled (exactly) and added to the CTA's FP64 slot
// (m x 8), reduced over the CTAs afterwards.
constexpr int kHalfRows = 1024;
constexpr int kHmSK = 2;   // 16-row tiles per ring stage
constexpr int kHmNS = 3;   // ring stages per warp
constexpr int kHmWarps = kThreads / 32;

__device__ __forceinline__ void ldsm_x4_trans(unsigned& r0, unsigned& r1, unsigned& r2, unsigned& r3, const void* p) {
    const unsigned a = (unsigned)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(a));
}
__device__ __forceinline__ void ldsm_x2_trans(unsigned& r0, unsigned& r1, const void* p) {
    const unsigned a = (unsigned)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];\n" : "=r"(r0), "=r"(r1) : "r"(a));
}
template <bool GROUPED>
__global__ void __launch_bounds__(kThreads) gram_half_kernel(int64_t n, int m, int nitems, int groups,
                                                             const __half* __restrict__ Q, const float* __restrict__ W,
                                                             double* __restrict__ partial, int* __restrict__ ticket) {
    constexpr int B = 8;
    constexpr int STAGE = kHmSK * 32 * B;  // halves per ring stage (kHmSK tiles of 32 rows of 16 bytes)
    __shared__ __align__(16) __half ws[kHalfRows * B];
    __shared__ __align__(16) __half ring[kHmWarps][kHmNS][STAGE];
    __shared__ float s_max[kHmWarps];
    __shared__ int s_chunk;
    const int nblocks = m / B;
    const int npairs = (nblocks + 1) / 2;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, tig = lane & 3;
    double* part = partial + (int64_t)blockIdx.x * m * B;
    for (int e = threadIdx.x; e < m * B; e += kThreads) part[e] = 0.0;
    const int per_group = GROUPED ? (npairs + groups - 1) / groups : npairs;  // pairs of an item
    constexpr int NST = kHalfRows / 16 / kHmSK;  // stages per pair per chunk
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) s_chunk = atomicAdd(ticket, 1);
        __syncthreads();
        const int item = s_chunk;
        if (item >= nitems) break;
        // an item is a chunk and a group of its pairs
        const int c = GROUPED ? item / groups : item;
        const int p0 = GROUPED ? (item - c * groups) * per_group + warp : warp;
        const int p1 = GROUPED ? min(npairs, p0 - warp + per_group) : npairs;
        const int mypairs = p0 < p1 ? (p1 - p0 + kHmWarps - 1) / kHmWarps : 0;
        const int64_t r0 = (int64_t)c * kHalfRows;
        const int rows = (int)min((int64_t)kHalfRows, n - r0);
        // the chunk's largest |W| -> power-of-two scale
        float mx = 0.f;
        for (int e = threadIdx.x; e < rows * B; e += kThreads) mx = fmaxf(mx, fabsf(W[r0 * B + e]));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (lane == 0) s_max[warp] = mx;
        __syncthreads();
        mx = 0.f;
#pragma unroll
        for (int w = 0; w < kHmWarps; ++w) mx = fmaxf(mx, s_max[w]);
        int ex = 0;
        if (mx > 0.f) frexpf(mx, &ex);
        const float scale = ldexpf(1.f, 14 - ex);
        const double unscale = ldexp(1.0, ex - 14);
        for (int e = threadIdx.x; e < kHalfRows * B; e += kThreads)
            ws[e] = __float2half_rn(e < rows * B ? W[r0 * B + e] * scale : 0.f);
        __syncthreads();
        const int total = mypairs * NST;
        // ring stage k: pair p0 + (k / NST) * kHmWarps, rows (k % NST) * 16 * kHmSK ..
        // lane L copies row (L & 15) of block 2p + (L >> 4) for each tile u
        auto issue = [&](int k) {
            if (k < total) {
                const int p = p0 + (k / NST) * kHmWarps;
                const int j = 2 * p + (lane >> 4);
                __half* buf = ring[warp][k % kHmNS];
#pragma unroll
                for (int u = 0; u < kHmSK; ++u) {
                    const int rr = (k % NST) * 16 * kHmSK + u * 16 + (lane & 15);
                    const bool ok = j < nblocks && rr < rows;
                    cp_async16(buf + (u * 32 + lane) * B, ok ? (const void*)(Q + ((int64_t)j * n + r0 + rr) * B)
                                                             : (const void*)Q, ok ? 16 : 0);
                }
            }
            cp_async_commit();
        };
#pragma unroll
        for (int k = 0; k < kHmNS - 1; ++k) issue(k);
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
        // ldmatrix row addresses: A, matrix q = lane >> 3 (rows 0-7 / 8-15 of blocks 0 / 1), row lane & 7
        const int a_row = ((lane >> 3) & 1) * 16 + (lane >> 4) * 8 + (lane & 7);
        const int b_row = ((lane >> 3) & 1) * 8 + (lane & 7);
        for (int k = 0; k < total; ++k) {
            cp_async_wait<kHmNS - 2>();
            __syncwarp();
            issue(k + kHmNS - 1);  // into the stage consumed at k - 1
            const __half* buf = ring[warp][k % kHmNS];
#pragma unroll
            for (int u = 0; u < kHmSK; ++u) {
                unsigned a[4], bq[2];
                ldsm_x4_trans(a[0], a[1], a[2], a[3], buf + (u * 32 + a_row) * B);
                const int kk = (k % NST) * kHmSK + u;  // 16-row tile of the chunk
                ldsm_x2_trans(bq[0], bq[1], ws + (kk * 16 + b_row) * B);
                mma_16816(acc, a, bq[0], bq[1]);
            }
            if ((k % NST) == NST - 1) {
                // the pair's sums over this chunk: rows g (block 2p) and g + 8 (block 2p + 1), columns 2 tig, 2 tig + 1
                const int p = p0 + (k / NST) * kHmWarps;
                const int j0 = 2 * p, j1 = 2 * p + 1;
                double* o0 = part + ((int64_t)j0 * B + g) * B + 2 * tig;
                o0[0] += (double)acc[0] * unscale;
                o0[1] += (double)acc[1] * unscale;
                if (j1 < nblocks) {
                    double* o1 = part + ((int64_t)j1 * B + g) * B + 2 * tig;
                    o1[0] += (double)acc[2] * unscale;
                    o1[1] += (double)acc[3] * unscale;
                }
                acc[0] = acc[1] = acc[2] = acc[3] = 0.f;
            }
        }
        cp_async_wait<0>();
    }
}

bbl_status launch_gram_half(int64_t n, int m, const __half* Q, const float* W, double* C, DevBuf& partials,
                            cudaStream_t st) {
    static int occ = 0;
    if (occ == 0) {
        BBL_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, gram_half_kernel<false>, kThreads, 0));
        if (occ < 1) occ = 1;
    }
    const int64_t slots_max = (int64_t)std::max(1, sm_count() - kRitzReserveSMs) * occ;
    const int nch = (int)std::max<int64_t>(1, ceil_div(n, kHalfRows));
    // fewer chunks than SMs: a chunk's pairs are split into groups of at least one
    // pair per warp (n = 1e5, 60 blocks: 48.4 us, in three groups 32.9; with more
    // chunks than that the groups' partial sums cost more)
    const int npairs = (m / 8 + 1) / 2;
    int64_t groups = 1;
    if (nch < sm_count()) groups = std::max<int64_t>(1, std::min<int64_t>(ceil_div(slots_max, nch), npairs / kHmWarps));
    const int64_t workers = std::min<int64_t>(slots_max, nch * groups);
    const int64_t per = (int64_t)m * 8;
    const size_t need = sizeof(double) * (size_t)(workers * per) + 256;
    BBL_TRY(partials.grow(need));
    int* ticket = reinterpret_cast<int*>(partials.as<char>() + sizeof(double) * (size_t)(workers * per));
    BBL_CUDA(cudaMemsetAsync(ticket, 0, sizeof(int), st));
    const auto kernel = groups > 1 ? gram_half_kernel<true> : gram_half_kernel<false>;
    kernel<<<(unsigned)workers, kThreads, 0, st>>>(n, m, (int)(nch * groups), (int)groups, Q, W, partials.as<double>(),
                                                   ticket);
    BBL_LAUNCH_CHECK();
    launch_reduce(per, (int)workers, partials.as<double>(), C, st);
    BBL_LAUNCH_CHECK();
    return BBL_OK;
}

__global__ void f32_to_f16_kernel(int64_t count, const float* __restrict__ in, __half* __restrict__ out) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < count; e += (int64_t)gridDim.x * blockDim.x)
        out[e] = __float2half_rn(in[e]);
}

template <typename T, int B, int CPT>
bbl_status launch_gram(int64_t n, int m, const T* Q, const T* W, double* C, DevBuf& partials, cudaStream_t st) {
    const int64_t per = (int64_t)m * B;
    const int64_t cap = per * (int64_t)sm_count() * 8;        // enough for any occupancy
    const int64_t gy = gram_groups<CPT>(m);                   // one ticket per column group
    const size_t ticket_bytes = 256 * (size_t)ceil_div(gy * (int64_t)sizeof(int), 256);
    const size_t need = sizeof(double) * (size_t)cap + ticket_bytes;
    BBL_TRY(partials.grow(need));
    int* tickets = reinterpret_cast<int*>(partials.as<char>() + sizeof(double) * (size_t)cap);
    return gram_core<T, B, CPT>(n, m, Q, W, C, partials.as<double>(), cap, tickets,
                                (int64_t)(ticket_bytes / sizeof(int)), st);
}

template <typename T>
bbl_status launch_gram_generic(int64_t n, int m, int b, const T* Q, const T* W, double* C, DevBuf& partials,
                               cudaStream_t st) {
    int TC = 1;
    while (TC < m && TC < kThreads) TC <<= 1;
    const int gy = (m + TC - 1) / TC;
    int64_t target = std::max<int64_t>(1, (152 * 2) / gy);
    int64_t rpc = std::max<int64_t>(kRT * 4, ceil_div(n, target));
    rpc = ceil_div(rpc, kRT) * kRT;
    const int64_t nch = std::max<int64_t>(1, ceil_div(n, rpc));
    const size_t need = sizeof(double) * (size_t)nch * m * b;
    BBL_TRY(partials.grow(need));
    const size_t smem = sizeof(double) * kThreads * kMaxB;
    static OncePerDevice once;
    BBL_TRY(allow_smem(once, gram_generic_kernel<T>, smem));
    dim3 grid((unsigned)nch, (unsigned)gy);
    gram_generic_kernel<T><<<grid, kThreads, smem, st>>>(n, m, b, rpc, TC, Q, W, partials.as<double>());
    BBL_LAUNCH_CHECK();
    const int64_t count = (int64_t)m * b;
    launch_reduce(count, (int)nch, partials.as<double>(), C, st);
    BBL_LAUNCH_CHECK();
    return BBL_OK;
}

template <typename T>
bbl_status gram_typed(int64_t n, int b, int m, const T* Q, const T* W, double* C, DevBuf& partials, cudaStream_t st) {
    switch (b) {
        case 1: return launch_gram<T, 1, 1>(n, m, Q, W, C, partials, st);
        case 2: return launch_gram<T, 2, 2>(n, m, Q, W, C, partials, st);
        case 4: return launch_gram_rows<T, 4>(n, m, Q, W, C, partials, st);
        case 8: return launch_gram_rows<T, 8>(n, m, Q, W, C, partials, st);
        case 16:  // (FP64: on the tensor cores, tc64.cu)
            if constexpr (!std::is_same<T, double>::value) return launch_gram<T, 16, 2>(n, m, Q, W, C, partials, st);
            [[fallthrough]];
        default: return launch_gram_generic<T>(n, m, b, Q, W, C, partials, st);
    }
}

// -------------------------------------------------------------------- apply
// W[r][c] (SUB ? -= : =) sum_a Q[r][a] C[a][c], c < kc.  Q: nblocks blocks of
// n x B; C: m x kc FP64 row-major; W: n x kc (type TO).  TA: accumulation type.
constexpr int kKT = 256;
// One CTA: rows r = row0 + threadIdx.x (r < row_end) of W (-)= Q C.
template <typename T, int B, int KCT, bool SUB, typename TA, typename TO>
__device__ __forceinline__ void apply_body(int64_t n, int m, int kc, int64_t row0, int64_t row_end, const T* Q,
                                           const double* __restrict__ C, TO* W) {
    constexpr int KM = KCT > 0 ? KCT : kMaxB;
    // FP32 sums into an FP64 result: FP32 within a tile of kKT columns, FP64
    // across tiles
    constexpr bool kTiled = sizeof(TA) == 4 && !is_df32<TA>::value && sizeof(TO) == 8;
    __shared__ TA cs[kKT * KM];
    const int tid = threadIdx.x;
    const int64_t r = row0 + tid;
    const int64_t rlim = row_end;
    TA acc[KM];
    double acc64[kTiled ? KM : 1];
#pragma unroll
    for (int c = 0; c < KM; ++c) acc[c] = TA(0);
    if constexpr (kTiled) {
#pragma unroll
        for (int c = 0; c < KM; ++c) acc64[c] = 0.0;
    }
    for (int a0 = 0; a0 < m; a0 += kKT) {
        const int rows = min(kKT, m - a0);
        __syncthreads();
        for (int e = tid; e < rows * KM; e += kThreads) {
            const int a = e / KM, c = e % KM;
            cs[e] = (c < kc) ? (TA)C[(int64_t)(a0 + a) * kc + c] : TA(0);
        }
        __syncthreads();
        if (r < rlim) {
#pragma unroll 4
            for (int jb = 0; jb < rows; jb += B) {
                const int j = (a0 + jb) / B;
                T q[B];
                if constexpr (B * sizeof(T) >= 16) {
                    constexpr int CH = 16 / (int)sizeof(T);
#pragma unroll
                    for (int ch = 0; ch < B / CH; ++ch) {
                        T t[CH];
                        ldvec<T, CH>(Q + (int64_t)j * n * B + r * B + ch * CH, t);
#pragma unroll
                        for (int q2 = 0; q2 < CH; ++q2) q[ch * CH + q2] = t[q2];
                    }
                } else {
                    ldvec<T, B>(Q + (int64_t)j * n * B + r * B, q);
                }
                const TA* cr = cs + jb * KM;
#pragma unroll
                for (int i = 0; i < B; ++i) {
                    const TA qi = (TA)q[i];
#pragma unroll
                    for (int c = 0; c < KM; ++c) acc[c] = fma(qi, cr[i * KM + c], acc[c]);
                }
            }
        }
        if constexpr (kTiled) {
#pragma unroll
            for (int c = 0; c < KM; ++c) {
                acc64[c] += (double)acc[c];
                acc[c] = TA(0);
            }
        }
    }
    if (r < rlim) {
#pragma unroll
        for (int c = 0; c < KM; ++c) {
            if (c < kc) {
                TO* w = W + r * kc + c;
                if constexpr (kTiled) {
                    if (SUB) *w = (TO)((double)(*w) - acc64[c]);
                    else *w = (TO)acc64[c];
                } else {
                    if (SUB) *w = (TO)((TA)(*w) - acc[c]);
                    else *w = (TO)acc[c];
                }
            }
        }
    }
}

template <typename T, int B, int KCT, bool SUB, typename TA, typename TO>
__global__ void __launch_bounds__(kThreads) apply_kernel(int64_t n, int m, int kc, const T* Q, const double* __restrict__ C,
                                                         TO* W) {
    apply_body<T, B, KCT, SUB, TA, TO>(n, m, kc, (int64_t)blockIdx.x * kThreads, n, Q, C, W);
}

// Segmented apply: CTA x handles rows [ctas[3x+1], ctas[3x+2]) (at most 256)
// of segment s = ctas[3x], with that segment's coefficients C + s*cstride and
// m = ms[s * ms_stride] basis columns (ms_stride 0: one shared count; ms NULL:
// m_all); inactive segments skip.
template <typename T, int B, int KCT, bool SUB, typename TA, typename TO>
__global__ void __launch_bounds__(kThreads) apply_seg_kernel(int64_t n, int m_all, const int* __restrict__ ms,
                                                             int ms_stride, int kc,
                                                             const int64_t* __restrict__ ctas,
                                                             const int* __restrict__ seg_active, const T* Q,
                                                             const double* __restrict__ C, int64_t cstride, TO* W) {
    const int64_t seg = ctas[3 * blockIdx.x];
    if (seg_active && !seg_active[seg]) return;
    const int m = ms ? ms[seg * ms_stride] : m_all;
    apply_body<T, B, KCT, SUB, TA, TO>(n, m, kc, ctas[3 * blockIdx.x + 1], ctas[3 * blockIdx.x + 2], Q,
                                       C + seg * cstride, W);
}

// any b (runtime)
template <typename T, bool SUB, typename TA, typename TO>
__global__ void __launch_bounds__(kThreads) apply_generic_kernel(int64_t n, int m, int b, int kc, const T* Q,
                                                                 const double* __restrict__ C, TO* W) {
    __shared__ TA cs[kKT * kMaxB];
    const int tid = threadIdx.x;
    const int64_t r = (int64_t)blockIdx.x * kThreads + tid;
    TA acc[kMaxB];
    for (int c = 0; c < kMaxB; ++c) acc[c] = TA(0);
    const int kt = (kKT / b) * b;
    for (int a0 = 0; a0 < m; a0 += kt) {
        const int rows = min(kt, m - a0);
        __syncthreads();
        for (int e = tid; e < rows * kc; e += kThreads) cs[e] = (TA)C[(int64_t)a0 * kc + e];
        __syncthreads();
        if (r < n) {
            for (int a = 0; a < rows; ++a) {
                const int ga = a0 + a;
                const TA q = (TA)Q[(int64_t)(ga / b) * n * b + r * b + ga % b];
                for (int c = 0; c < kc; ++c) acc[c] = fma(q, cs[a * kc + c], acc[c]);
            }
        }
    }
    if (r < n) {
        for (int c = 0; c < kc; ++c) {
            TO* w = W + r * kc + c;
            if (SUB) *w = (TO)((TA)(*w) - acc[c]);
            else *w = (TO)acc[c];
        }
    }
}

// First-pass update of the FP32 stage, b = 8, with the older blocks read
// from the FP16 copy: W -= sum_j Q_j C_j.  In Lanczos the first pass's
// coefficients of the blocks older than the two newest are of the order of
// the lost orthogonality (about 1e-7 of ||W|| in FP32): the FP16 rounding
// of those blocks (2^-12 relative) changes W by about 2^-12 of that, far
// below W's own FP32 rounding, and a rounding of their coefficients is a
// change of the coefficients only (it stays in span(Q), and the second
// pass removes it).  So the older blocks' product runs on the tensor cores
// straight from the FP16 copy (mma.sync m16n8k16, FP16 in, FP32
// accumulate): C's rows of those blocks are scaled by one power of two s
// (the largest entry to [2^13, 2^14)) and rounded to FP16, and the sum is
// multiplied by 1/s.  The newest blocks (jsplit and up), whose coefficients
// are A_j and B_{j-1}^T, are FP32 FMA products with C rounded to FP32, as
// in the FP32 update.

// B fragments of the older blocks' product, per block pair q (blocks 2q,
// 2q + 1 < jsplit, the second zero past it) and lane (g = lane / 4, t = lane
// % 4): {C rows 16q + 2t, +1 | C rows 16q + 8 + 2t, +1}, column g, times s,
// in FP16 pairs (low half = lower row); scale[0] = 1/s.  One CTA.
__global__ void __launch_bounds__(256) half_old_prep_kernel(int jsplit, const double* __restrict__ C,
                                                            uint2* __restrict__ frag, float* __restrict__ scale) {
    __shared__ double smax[256];
    double mx = 0.0;
    for (int e = threadIdx.x; e < jsplit * 64; e += 256) mx = fmax(mx, fabs(C[e]));
    smax[threadIdx.x] = mx;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w) smax[threadIdx.x] = fmax(smax[threadIdx.x], smax[threadIdx.x + w]);
        __syncthreads();
    }
    mx = smax[0];
    int ex = 0;
    if (mx > 0.0) (void)frexp(mx, &ex);  // mx = f 2^ex, f in [0.5, 1)
    // max * sc in [2^13, 2^14); coefficients below 2^-100 (negligible) keep
    // sc = 2^114, so that sc and 1/sc stay finite and normal in FP32
    ex = ex < -100 ? -100 : ex;
    const double sc = (mx > 0.0) ? ldexp(1.0, 14 - ex) : 1.0;
    if (threadIdx.x == 0) scale[0] = (float)(1.0 / sc);
    const int npo = (jsplit + 1) >> 1;
    for (int e = threadIdx.x; e < npo * 32; e += 256) {
        const int q = e >> 5, lane = e & 31, g = lane >> 2, t = lane & 3;
        const int ra = 16 * q + 2 * t, rb = 16 * q + 8 + 2 * t;
        const bool two = 2 * q + 1 < jsplit;
        const __half2 b0 = __floats2half2_rn((float)(C[ra * 8 + g] * sc), (float)(C[(ra + 1) * 8 + g] * sc));
        const __half2 b1 = two ? __floats2half2_rn((float)(C[rb * 8 + g] * sc), (float)(C[(rb + 1) * 8 + g] * sc))
                               : __floats2half2_rn(0.f, 0.f);
        frag[e] = make_uint2(*reinterpret_cast<const unsigned*>(&b0), *reinterpret_cast<const unsigned*>(&b1));
    }
}

// One warp per 16-row tile.  A fragments of the older blocks come straight
// from global memory (each 4-byte load of a warp covers 8 rows x 16 bytes
// of one block: one 128-byte line).
template <int U, bool AHEAD>
__global__ void __launch_bounds__(256) apply_half_old_kernel(int64_t n, int nblocks, int jsplit,
                                                             const __half* __restrict__ Q16,
                                                             const float* __restrict__ Q,
                                                             const double* __restrict__ C,
                                                             const uint2* __restrict__ frag,
                                                             const float* __restrict__ scale, float* __restrict__ W) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int64_t tile = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t r0 = tile * 16;
    if (r0 >= n) return;
    const int64_t ra = r0 + g, rb = r0 + g + 8;
    const bool oka = ra < n, okb = rb < n;
    const unsigned* Q16w = reinterpret_cast<const unsigned*>(Q16);  // two halves per word
    float d[4] = {0.f, 0.f, 0.f, 0.f};
    const int npo = (jsplit + 1) >> 1;
    // groups of U block pairs; AHEAD: two in turn, a group's loads issued before the
    // products of the group before it, else all loads of a group before its products
    struct Group {
        unsigned a[U][4], b[U][2];
    };
    auto load = [&](int q0, Group& x) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int q = q0 + u;
            const bool on = q < npo;
            const int j0 = on ? 2 * q : 0;
            const int j1 = (on && 2 * q + 1 < nblocks) ? 2 * q + 1 : j0;  // past the basis: b1 is zero
            x.a[u][0] = (on && oka) ? __ldg(Q16w + (((int64_t)j0 * n + ra) * 8 + 2 * t) / 2) : 0u;
            x.a[u][1] = (on && okb) ? __ldg(Q16w + (((int64_t)j0 * n + rb) * 8 + 2 * t) / 2) : 0u;
            x.a[u][2] = (on && oka) ? __ldg(Q16w + (((int64_t)j1 * n + ra) * 8 + 2 * t) / 2) : 0u;
            x.a[u][3] = (on && okb) ? __ldg(Q16w + (((int64_t)j1 * n + rb) * 8 + 2 * t) / 2) : 0u;
            const uint2 f = on ? __ldg(frag + q * 32 + lane) : make_uint2(0u, 0u);
            x.b[u][0] = f.x;
            x.b[u][1] = f.y;
        }
    };
    auto products = [&](int q0, const Group& x) {
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (q0 + u < npo) mma_16816(d, x.a[u], x.b[u][0], x.b[u][1]);
    };
    Group g0;
    if constexpr (AHEAD) {
        Group g1;
        if (npo > 0) load(0, g0);
        for (int q0 = 0; q0 < npo; q0 += 2 * U) {
            if (q0 + U < npo) load(q0 + U, g1);
            products(q0, g0);
            if (q0 + 2 * U < npo) load(q0 + 2 * U, g0);
            products(q0 + U, g1);
        }
    } else {
        for (int q0 = 0; q0 < npo; q0 += U) {
            load(q0, g0);
            products(q0, g0);
        }
    }
    const float inv = npo > 0 ? __ldg(scale) : 0.f;
    // acc[row][col]: rows ra / rb, columns 2t, 2t + 1
    float acc[2][2] = {{d[0] * inv, d[1] * inv}, {d[2] * inv, d[3] * inv}};
    for (int j = jsplit; j < nblocks; ++j) {
        float cj[8][2];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            cj[i][0] = (float)__ldg(C + (8 * j + i) * 8 + 2 * t);
            cj[i][1] = (float)__ldg(C + (8 * j + i) * 8 + 2 * t + 1);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int64_t rr = h ? rb : ra;
            if (rr < n) {
                const float4 x0 = __ldg(reinterpret_cast<const float4*>(Q + ((int64_t)j * n + rr) * 8));
                const float4 x1 = __ldg(reinterpret_cast<const float4*>(Q + ((int64_t)j * n + rr) * 8 + 4));
                const float qv[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    acc[h][0] = fmaf(qv[i], cj[i][0], acc[h][0]);
                    acc[h][1] = fmaf(qv[i], cj[i][1], acc[h][1]);
                }
            }
        }
    }
    if (oka) {
        float2* w = reinterpret_cast<float2*>(W + ra * 8 + 2 * t);
        const float2 v = *w;
        *w = make_float2(v.x - acc[0][0], v.y - acc[0][1]);
    }
    if (okb) {
        float2* w = reinterpret_cast<float2*>(W + rb * 8 + 2 * t);
        const float2 v = *w;
        *w = make_float2(v.x - acc[1][0], v.y - acc[1][1]);
    }
}

// Update of the float-float polish, b = 8: W -= sum_j Q_j C_j with the
// blocks older than jsplit read from the FP32 copy of the basis (the high
// parts) with FP32 products and sums, the newer ones from the float-float
// basis with float-float products.  The older blocks' coefficients are the
// lost orthogonality and the FP32 first-pass Gram's error, so their FP32
// products (2^-24 relative) change W far below its float-float rounding;
// their bytes halve and their arithmetic is one FMA per product.
__global__ void __launch_bounds__(kThreads) apply_df32_f32old_kernel(int64_t n, int m, int jsplit,
                                                                     const float* __restrict__ Q32,
                                                                     const df32* __restrict__ Q,
                                                                     const double* __restrict__ C, df32* W) {
    constexpr int B = 8;
    __shared__ df32 cs[kKT * B];
    const int tid = threadIdx.x;
    const int64_t r = (int64_t)blockIdx.x * kThreads + tid;
    float a32[B];
    df32 adf[B];
#pragma unroll
    for (int c = 0; c < B; ++c) {
        a32[c] = 0.f;
        adf[c] = df32(0.f);
    }
    for (int a0 = 0; a0 < m; a0 += kKT) {
        const int rows = min(kKT, m - a0);
        __syncthreads();
        for (int e = tid; e < rows * B; e += kThreads) cs[e] = df32(C[(int64_t)a0 * B + e]);
        __syncthreads();
        if (r < n) {
            for (int jb = 0; jb < rows; jb += B) {
                const int j = (a0 + jb) / B;
                const df32* cr = cs + jb * B;
                if (j < jsplit) {
                    const float4 x0 = __ldg(reinterpret_cast<const float4*>(Q32 + ((int64_t)j * n + r) * B));
                    const float4 x1 = __ldg(reinterpret_cast<const float4*>(Q32 + ((int64_t)j * n + r) * B + 4));
                    const float q[B] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
#pragma unroll
                    for (int i = 0; i < B; ++i)
#pragma unroll
                        for (int c = 0; c < B; ++c) a32[c] = fmaf(q[i], cr[i * B + c].hi, a32[c]);
                } else {
                    df32 q[B];
                    ldvec<df32, B>(Q + ((int64_t)j * n + r) * B, q);
#pragma unroll
                    for (int i = 0; i < B; ++i)
#pragma unroll
                        for (int c = 0; c < B; ++c) adf[c] = dfm::fma(q[i], cr[i * B + c], adf[c]);
                }
            }
        }
    }
    if (r < n) {
#pragma unroll
        for (int c = 0; c < B; ++c) {
            df32* w = W + r * B + c;
            *w = *w - (adf[c] + df32(a32[c]));
        }
    }
}

template <typename T, bool SUB, typename TA, typename TO>
bbl_status apply_typed(int64_t n, int b, int m, int kc, const T* Q, const double* C, TO* W, cudaStream_t st) {
    const unsigned grid = (unsigned)ceil_div(n, kThreads);
    const bool same = (kc == b);
    if (same) {
        switch (b) {
            case 1: apply_kernel<T, 1, 1, SUB, TA, TO><<<grid, kThreads, 0, st>>>(n, m, kc, Q, C, W); break;
            case 2: apply_kernel<T, 2, 2, SUB, TA, TO><<<grid, kThreads, 0, st>>>(n, m, kc, Q, C, W); break;
            case 4: apply_kernel<T, 4, 4, SUB, TA, TO><<<grid, kThreads, 0, st>>>(n, m, kc, Q, C, W); break;
            case 8: apply_kernel<T, 8, 8, SUB, TA, TO><<<grid, kThreads, 0, st>>>(n, m, kc, Q, C, W); break;
            case 16:  // (the FP64 update: on the tensor cores, tc64.cu)
                if constexpr (!(SUB && std::is_same<T, double>::value)) {
                    apply_kernel<T, 16, 16, SUB, TA, TO><<<grid, kThreads, 0, st>>>(n, m, kc, Q, C, W);
                    break;
                }
                [[fallthrough]];
            default: apply_generic_kernel<T, SUB, TA, TO><<<grid, kThreads, 0, st>>>(n, m, b, kc, Q, C, W);
        }
    } else {
        switch (b) {
            case 1: apply_kernel<T, 1, 0, SUB, TA, TO><<<grid, kThreads, 0, st>>>(n, m, kc, Q, C, W); break;
            case 2: apply_kernel<T, 2, 0, SUB, TA, TO><<<grid, kThreads, 0, st>>>(n, m, kc, Q, C, W); break;
            case 4: apply_kernel<T, 4, 0, SUB, TA, TO><<<grid, kThreads, 0, st>>>(n, m, kc, Q, C, W); break;
            case 8: apply_kernel<T, 8, 0, SUB, TA, TO><<<grid, kThreads, 0, st>>>(n, m, kc, Q, C, W); break;
            case 16:  // (FP64 Ritz vectors: tc64.cu)
                if constexpr (!std::is_same<T, double>::value) {
                    apply_kernel<T, 16, 0, SUB, TA, TO><<<grid, kThreads, 0, st>>>(n, m, kc, Q, C, W);
                    break;
                }
                [[fallthrough]];
            default: apply_generic_kernel<T, SUB, TA, TO><<<grid, kThreads, 0, st>>>(n, m, b, kc, Q, C, W);
        }
    }
    BBL_LAUNCH_CHECK();
    return BBL_OK;
}

// -------------------------------------------------------------------- Cholesky of the b x b Gram
// status bits: 1 = non-finite Gram.  mask[i] = 1 for deflated columns.

// 1 / d for d in 2^-959 .. 2^957, rounded as the division rounds it but for one
// case in about 2^39: an FP32 seed on the mantissa and two Newton steps, the last
// from an error below 2^-45 (four FP64 instructions in a chain; an FP64 instruction
// occupies its scheduler for 64 cycles here, and the division takes about ten).
__device__ __forceinline__ double recip(double d) {
    const int hi = __double2hiint(d), ex = hi >> 20;
    const double m = __hiloint2double(hi - (ex - 1023) * (1 << 20), __double2loint(d));
    double y = (double)__frcp_rn((float)m);
    y = fma(y, fma(-m, y, 1.0), y);
    y = fma(y, fma(-m, y, 1.0), y);
    return __hiloint2double(__double2hiint(y) - (ex - 1023) * (1 << 20), __double2loint(y));
}

constexpr int kCholThreads = 256;
constexpr int kCholParts = 128;  // most partial Grams one CTA adds itself (two FP64 additions per cycle)

// G = L D L^T with deflation, right-looking by one warp, whose lanes keep the
// entries of G's Schur complement and of L^{-1} in registers: a step is one
// reciprocal, one product and one update deep.  (The left-looking form with a
// square root and divisions in the chain took 15 us at b = 8 by a warp and 14 us
// by one thread per segment, this one about 8.)
struct CholShared {
    double G[kMaxB * kMaxB];
    double L[kMaxB * kMaxB];      // row k: D[k] L[.][k]
    double Z[kMaxB * kMaxB];      // row k of L^{-1}
    double row[2][2][kMaxB];      // row k of the Schur complement and of L^{-1}
    double scaled[kMaxB];         // row k times a power of two
    double d[kMaxB], root[kMaxB]; // D (0 for deflated columns) and its square roots
    int deflated[kMaxB];
};

__device__ __forceinline__ void chol_core(int b, double thresh2, int relative, CholShared& sh, int& cnt, int& bad) {
    const int lane = threadIdx.x & 31, bb = b * b;
    constexpr int E = kMaxB * kMaxB / 32;
    double a[E], z[E];
    int ei[E], ec[E];
    bad = 0;
#pragma unroll
    for (int x = 0; x < E; ++x) {
        const int q = lane + 32 * x;
        ei[x] = q < bb ? q / b : -1;
        ec[x] = q < bb ? q - ei[x] * b : 0;
        a[x] = q < bb ? sh.G[q] : 0.0;
        z[x] = ei[x] == ec[x] ? 1.0 : 0.0;
        if (!isfinite(a[x])) bad = 1;
    }
    bad = __any_sync(0xffffffffu, bad);
    if (relative) {
        double gmax = 0.0;
        for (int q = 0; q < b; ++q) gmax = fmax(gmax, sh.G[q * b + q]);
        thresh2 *= gmax;
    }
    cnt = 0;
#pragma unroll
    for (int x = 0; x < E; ++x)
        if (ei[x] == 0) {
            sh.row[0][0][ec[x]] = a[x];
            sh.row[0][1][ec[x]] = z[x];
        }
    __syncwarp();
    for (int k = 0; k < b; ++k) {
        const double* ra = sh.row[k & 1][0];
        const double* rz = sh.row[k & 1][1];
        const double d = ra[k];
        const int defl = !(d > thresh2) || bad;
        cnt += defl;
        const double* rl = ra;
        double y = 0.0;
        const int ex = __double2hiint(d) >> 20;
        if (!defl) {
            if ((unsigned)ex - 64u <= 1916u) {
                y = recip(d);
            } else {  // far pivots: they and their row by a power of two
                const double f = __hiloint2double((ex < 64 ? 1623 : 423) << 20, 0);
                if (lane < b) sh.scaled[lane] = ra[lane] * f;
                __syncwarp();
                rl = sh.scaled;
                y = recip(d * f);
            }
        }
        if (lane == 0) {
            sh.deflated[k] = defl;
            sh.d[k] = defl ? 0.0 : d;
        }
        if (lane < b) {
            sh.L[k * b + lane] = lane < k || defl ? 0.0 : ra[lane];
            sh.Z[k * b + lane] = lane > k || defl ? 0.0 : rz[lane];
        }
#pragma unroll
        for (int x = 0; x < E; ++x) {
            if (32 * x < bb && ei[x] > k) {
                const double l = rl[ei[x]] * y;
                if (!defl && ec[x] >= ei[x]) a[x] = fma(-l, ra[ec[x]], a[x]);
                if (!defl && ec[x] <= k) z[x] = fma(-l, rz[ec[x]], z[x]);
                if (ei[x] == k + 1) {
                    sh.row[(k + 1) & 1][0][ec[x]] = a[x];
                    sh.row[(k + 1) & 1][1][ec[x]] = z[x];
                }
            }
        }
        __syncwarp();
    }
    if (lane < b) sh.root[lane] = sqrt(sh.d[lane]);
    __syncwarp();
}

// entry e of R = D^{1/2} L^T and of R^{-1}: zero rows (columns) for deflated columns
// (one division each: L scaled by the root, after the reciprocal, rounds twice more)
__device__ __forceinline__ double chol_R(const CholShared& sh, int b, int e) {
    const int i = e / b, c = e - i * b;
    if (c <= i || sh.deflated[i]) return c == i ? sh.root[i] : 0.0;
    return sh.L[e] / sh.root[i];
}
__device__ __forceinline__ double chol_Rinv(const CholShared& sh, int b, int e) {
    const int i = e / b, c = e % b;
    return c >= i && !sh.deflated[c] ? sh.Z[c * b + i] / sh.root[c] : 0.0;
}

// sh.G = the sum of nparts partial b x b Grams, by all kCholThreads threads
__device__ __forceinline__ void chol_gram(int b, int nparts, const double* __restrict__ partial, double* red,
                                          CholShared& sh) {
    const int tid = threadIdx.x, bb = b * b;
    const int groups = kCholThreads / bb, e = tid % bb, g = tid / bb;  // groups of bb threads add the parts
    red[tid] = g < groups ? sum_parts(bb, nparts, partial, e, g, groups) : 0.0;
    __syncthreads();
    if (tid < bb) {
        double s = red[tid];
        for (int q = 1; q < groups; ++q) s += red[tid + q * bb];
        sh.G[tid] = s;
    }
    __syncthreads();
}

// The Cholesky step of CholQR2 by one CTA: G = the sum of nparts partial b x b
// Grams, R = chol(G) with deflation and R^{-1}, and, with Bout, B = R R1.
__global__ void __launch_bounds__(kCholThreads) chol_kernel(int b, int nparts, const double* __restrict__ partial,
                                                            double thresh2, int relative, double* __restrict__ R,
                                                            double* __restrict__ Rinv, int* __restrict__ ndefl,
                                                            int* __restrict__ mask, int* __restrict__ status,
                                                            const double* __restrict__ R1, double* __restrict__ Bout) {
    __shared__ CholShared sh;
    __shared__ double red[kCholThreads];
    const int tid = threadIdx.x, bb = b * b;
    chol_gram(b, nparts, partial, red, sh);
    if (tid < 32) {
        int cnt, bad;
        chol_core(b, thresh2, relative, sh, cnt, bad);
        if (tid == 0) {
            if (ndefl) *ndefl += cnt;
            if (bad && status) atomicOr(status, 1);
        }
    }
    __syncthreads();
    if (tid < bb) {
        red[tid] = R[tid] = chol_R(sh, b, tid);
        Rinv[tid] = chol_Rinv(sh, b, tid);
    }
    __syncthreads();
    if (Bout && tid < bb) {
        const int i = tid / b, c = tid % b;
        double s = 0.0;
        for (int l = i; l <= c; ++l) s += red[i * b + l] * R1[l * b + c];
        Bout[tid] = s;
    }
    if (mask && tid < b) mask[tid] = sh.deflated[tid];
}

// A CTA per segment: G = the sum of the segment's partial Grams (slots of b x b,
// `per` for each of its chunks), then its Cholesky by one warp with threshold
// thresh2[s].
__global__ void __launch_bounds__(kCholThreads) chol_seg_kernel(int b, const double* __restrict__ partial,
                                                                const int* __restrict__ seg_chunk_ptr, int per,
                                                                const double* __restrict__ thresh2, int relative,
                                                                double* __restrict__ R, double* __restrict__ Rinv,
                                                                int* __restrict__ ndefl, int* __restrict__ mask,
                                                                int* __restrict__ status,
                                                                const int* __restrict__ active) {
    __shared__ CholShared sh;
    __shared__ double red[kCholThreads];
    const int s = blockIdx.x, tid = threadIdx.x, lane = tid, bb = b * b;
    if (active && !active[s]) return;
    const int64_t o = (int64_t)s * bb;
    const int p0 = seg_chunk_ptr[s] * per, p1 = seg_chunk_ptr[s + 1] * per;
    chol_gram(b, p1 - p0, partial + (int64_t)p0 * bb, red, sh);
    if (tid >= 32) return;
    int cnt, bad;
    chol_core(b, thresh2 ? thresh2[s] : 0.0, relative, sh, cnt, bad);
    for (int e = lane; e < bb; e += 32) {
        R[o + e] = chol_R(sh, b, e);
        Rinv[o + e] = chol_Rinv(sh, b, e);
    }
    if (mask && lane < b) mask[(int64_t)s * b + lane] = sh.deflated[lane];
    if (lane == 0) {
        if (ndefl) ndefl[s] += cnt;
        if (bad && status) atomicOr(status + s, 1);
    }
}

}  // namespace

// -------------------------------------------------------------------- internal API
void reduce_partials(int64_t count, int nparts, const double* partial, double* out, cudaStream_t st) {
    launch_reduce(count, nparts, partial, out, st);
}

int gram_worker_sms() { return std::max(1, sm_count() - kRitzReserveSMs); }

bbl_status gram(int64_t n, int b, int nblocks, int dtype, const void* Q, const void* W, double* C, DevBuf& partials,
                cudaStream_t st) {
    const int m = nblocks * b;
    if (dtype == BBL_FP64 && tc64_gram_supports(n, b, m))
        return gram_tc64(n, b, m, static_cast<const double*>(Q), static_cast<const double*>(W), C, partials, st);
    if (dtype == BBL_FP64)
        return gram_typed<double>(n, b, m, static_cast<const double*>(Q), static_cast<const double*>(W), C, partials, st);
    if (dtype == kDF32)
        return gram_typed<df32>(n, b, m, static_cast<const df32*>(Q), static_cast<const df32*>(W), C, partials, st);
    return gram_typed<float>(n, b, m, static_cast<const float*>(Q), static_cast<const float*>(W), C, partials, st);
}

// C ~= Q16^T W for b = 8: Q16 the FP16 copy of an FP32 basis of nblocks blocks
bbl_status gram_half(int64_t n, int nblocks, const void* Q16, const float* W, double* C, DevBuf& partials,
                     cudaStream_t st) {
    return launch_gram_half(n, nblocks * 8, static_cast<const __half*>(Q16), W, C, partials, st);
}

// FP16 copy (round to nearest) of count FP32 values
bbl_status to_half(int64_t count, const float* in, void* out, cudaStream_t st) {
    f32_to_f16_kernel<<<152 * 8, 256, 0, st>>>(count, in, static_cast<__half*>(out));
    BBL_LAUNCH_CHECK();
    return BBL_OK;
}

bbl_status update(int64_t n, int b, int nblocks, int dtype, const void* Q, const double* C, void* W, cudaStream_t st) {
    const int m = nblocks * b;
    if (dtype == BBL_FP64 && tc64_update_supports(b, m))
        return update_tc64(n, b, m, b, static_cast<const double*>(Q), C, static_cast<double*>(W), true, st);
    if (dtype == BBL_FP64)
        return apply_typed<double, true, double, double>(n, b, m, b, static_cast<const double*>(Q), C,
                                                         static_cast<double*>(W), st);
    if (dtype == kDF32)
        return apply_typed<df32, true, df32, df32>(n, b, m, b, static_cast<const df32*>(Q), C, static_cast<df32*>(W),
                                                   st);
    return apply_typed<float, true, float, float>(n, b, m, b, static_cast<const float*>(Q), C, static_cast<float*>(W),
                                                  st);
}

bbl_status update_half_old(int64_t n, int nblocks, int nnew, const void* Q16, const float* Q, const double* C,
                           float* W, DevBuf& work, cudaStream_t st) {
    const int jsplit = nblocks > nnew ? nblocks - nnew : 0;
    const int npo = (jsplit + 1) >> 1;
    BBL_TRY(work.grow(sizeof(uint2) * (size_t)npo * 32 + 256));
    uint2* frag = work.as<uint2>();
    float* scale = reinterpret_cast<float*>(work.as<char>() + sizeof(uint2) * (size_t)npo * 32);
    if (npo > 0) {
        half_old_prep_kernel<<<1, 256, 0, st>>>(jsplit, C, frag, scale);
        BBL_LAUNCH_CHECK();
    }
    const int64_t warps = ceil_div(n, (int64_t)16);
    // With 48 warps per SM and more, few registers and two pairs ahead: n = 1e6, 90
    // blocks 275 -> 261 us, n = 5e5, 45 blocks 89 -> 80 (3 ahead 278 and 89, 4 ahead 305
    // and 104: the registers cost more warps than the loads in flight bring).  With
    // fewer, eight pairs at once: n = 9000, 90 blocks 10.1 us, two ahead 11.1; n = 6e4
    // 25.0 and 26.3; n = 1e5, 60 blocks 27.0 and 27.3.
    const auto kernel = warps >= (int64_t)sm_count() * 48 ? apply_half_old_kernel<2, true> : apply_half_old_kernel<8, false>;
    kernel<<<(unsigned)ceil_div(warps * 32, 256), 256, 0, st>>>(n, nblocks, jsplit, static_cast<const __half*>(Q16), Q, C,
                                                                frag, scale, W);
    BBL_LAUNCH_CHECK();
    return BBL_OK;
}

bbl_status update_df32_f32old(int64_t n, int nblocks, int nnew, const float* Q32, const void* Q, const double* C,
                             void* W, cudaStream_t st) {
    const int jsplit = nblocks > nnew ? nblocks - nnew : 0;
    apply_df32_f32old_kernel<<<(unsigned)ceil_div(n, kThreads), kThreads, 0, st>>>(
        n, nblocks * 8, jsplit, Q32, static_cast<const df32*>(Q), C, static_cast<df32*>(W));
    BBL_LAUNCH_CHECK();
    return BBL_OK;
}

bbl_status ritz_vectors(int64_t n, int b, int nblocks, int dtype, const void* Q, int k, const double* S, double* X,
                        cudaStream_t st) {
    const int m = nblocks * b;
    if (dtype == BBL_FP64 && tc64_update_supports(b, m))
        return update_tc64(n, b, m, k, static_cast<const double*>(Q), S, X, false, st);
    if (dtype == BBL_FP64)
        return apply_typed<double, false, double, double>(n, b, m, k, static_cast<const double*>(Q), S, X, st);
    if (dtype == kDF32)
        return apply_typed<df32, false, df32, double>(n, b, m, k, static_cast<const df32*>(Q), S, X, st);
    // FP32 blocks: FP32 products and sums (the vectors carry FP32 accuracy
    // anyway), FP64 output
    return apply_typed<float, false, float, double>(n, b, m, k, static_cast<const float*>(Q), S, X, st);
}

// One pass over W for b in {1, 2, 4, 8}: W <- W Rinv (Rinv not NULL), then with
// gram the partial Grams of the result; *nparts of them in partials.
template <typename T, int B>
bbl_status launch_qr_pass(int64_t n, const double* Rinv, T* W, bool gram, DevBuf& partials, int* nparts,
                          cudaStream_t st) {
    const int grid = (int)std::min<int64_t>(152 * 4, std::max<int64_t>(1, ceil_div(n, kThreads)));
    if (gram) {
        BBL_TRY(partials.grow(sizeof(double) * (size_t)grid * B * B));
        *nparts = grid;
        const bool lng = n > (int64_t)64 * grid * kThreads;
        double* out = partials.as<double>();
        if (Rinv && lng) qr_pass_kernel<T, B, true, true, true><<<grid, kThreads, 0, st>>>(n, Rinv, W, out);
        else if (Rinv) qr_pass_kernel<T, B, true, true><<<grid, kThreads, 0, st>>>(n, Rinv, W, out);
        else if (lng) qr_pass_kernel<T, B, false, true, true><<<grid, kThreads, 0, st>>>(n, Rinv, W, out);
        else qr_pass_kernel<T, B, false, true><<<grid, kThreads, 0, st>>>(n, Rinv, W, out);
    } else {
        const int g2 = (int)std::min<int64_t>(152 * 8, std::max<int64_t>(1, ceil_div(n, kThreads)));
        qr_pass_kernel<T, B, true, false><<<g2, kThreads, 0, st>>>(n, Rinv, W, nullptr);
    }
    BBL_LAUNCH_CHECK();
    return BBL_OK;
}

template <typename T>
bbl_status qr_pass_typed(int64_t n, int b, const double* Rinv, T* W, bool want_gram, DevBuf& partials,
                         int* nparts, cudaStream_t st) {
    switch (b) {
        case 1: return launch_qr_pass<T, 1>(n, Rinv, W, want_gram, partials, nparts, st);
        case 2: return launch_qr_pass<T, 2>(n, Rinv, W, want_gram, partials, nparts, st);
        case 4: return launch_qr_pass<T, 4>(n, Rinv, W, want_gram, partials, nparts, st);
        case 8: return launch_qr_pass<T, 8>(n, Rinv, W, want_gram, partials, nparts, st);
        default: break;
    }
    // other b: the general update; the caller forms the Gram (nparts 0)
    if (Rinv) BBL_TRY((apply_typed<T, false, T, T>(n, b, b, b, W, Rinv, W, st)));
    *nparts = 0;
    return BBL_OK;
}

// small: >= 8*b*b doubles + 4*b ints.  B (device, b x b) receives R2 R1.
bbl_status cholqr2_dev(int64_t n, int b, int dtype, void* W, double* B, double defl_abs2, int* d_ndefl, int* d_mask,
                       DevBuf& partials, DevBuf& small, cudaStream_t st) {
    const size_t need = sizeof(double) * 8 * kMaxB * kMaxB + sizeof(int) * 4 * kMaxB;
    if (small.bytes < need) BBL_TRY(small.alloc(need));
    double* G = small.as<double>();
    double* R1 = G + kMaxB * kMaxB;
    double* R1i = R1 + kMaxB * kMaxB;
    double* R2 = R1i + kMaxB * kMaxB;
    double* R2i = R2 + kMaxB * kMaxB;
    int* status = reinterpret_cast<int*>(G + 8 * kMaxB * kMaxB);
    const int relative = defl_abs2 < 0 ? 1 : 0;
    const double t1 = relative ? -defl_abs2 : defl_abs2;
    // W <- W Rinv (if given), then the Gram of W (if wanted): its partial sums, or
    // G itself (many partial sums are added by more than one CTA)
    const double* gsum = nullptr;
    int nparts = 0;
    auto pass = [&](const double* Rinv, bool want_gram) -> bbl_status {
        if (dtype == BBL_FP64)
            BBL_TRY(qr_pass_typed<double>(n, b, Rinv, static_cast<double*>(W), want_gram, partials, &nparts, st));
        else if (dtype == kDF32)
            BBL_TRY(qr_pass_typed<df32>(n, b, Rinv, static_cast<df32*>(W), want_gram, partials, &nparts, st));
        else
            BBL_TRY(qr_pass_typed<float>(n, b, Rinv, static_cast<float*>(W), want_gram, partials, &nparts, st));
        if (!want_gram) return BBL_OK;
        if (nparts == 0) {
            BBL_TRY(gram(n, b, 1, dtype, W, W, G, partials, st));
            nparts = 1;
            gsum = G;
        } else if (nparts > kCholParts) {
            launch_reduce((int64_t)b * b, nparts, partials.as<double>(), G, st);
            BBL_LAUNCH_CHECK();
            nparts = 1;
            gsum = G;
        } else {
            gsum = partials.as<double>();
        }
        return BBL_OK;
    };
    BBL_TRY(pass(nullptr, true));
    chol_kernel<<<1, kCholThreads, 0, st>>>(b, nparts, gsum, t1, relative, R1, R1i, d_ndefl, d_mask, status, nullptr,
                                            nullptr);
    BBL_LAUNCH_CHECK();
    BBL_TRY(pass(R1i, true));
    // second pass: columns of Q1 have norm ~1; a pivot below 1e-6 means the
    // first pass produced no usable direction (it was deflated or lost).
    chol_kernel<<<1, kCholThreads, 0, st>>>(b, nparts, gsum, 1e-6, 0, R2, R2i, nullptr, nullptr, status, R1, B);
    BBL_LAUNCH_CHECK();
    return pass(R2i, false);
}

// -------------------------------------------------------------------- segmented (batched) forms
// A batch of independent problems is stacked row-wise: segment s owns rows
// [off[s], off[s+1]) of every n_tot x b block.  Work tables are built once
// on the host: gram chunks (seg, r0, r1) never cross a segment, apply CTAs
// (seg, r0, r1) cover at most 256 rows of one segment.  The current number of
// basis columns may be read from device memory (d_m), so that one captured
// graph serves every iteration.
namespace {

// C[s] = sum of segment s's partial slots (rows_slots: the row-contiguous
// kernel's wpb slots per chunk, else one): 32 entries per CTA, the slots split
// over 8 groups of threads and combined in a fixed order.  (One thread per entry
// adding all slots in turn took 11.6 us for the 40 slots of an FP64 segment of 2e4
// rows and 4.9 us in FP32.)
__global__ void __launch_bounds__(256) reduce_seg_kernel(int m_max, int b, const int* __restrict__ d_m,
                                                         const int* __restrict__ seg_chunk_ptr,
                                                         const int* __restrict__ active,
                                                         const double* __restrict__ partial, double* __restrict__ C,
                                                         int rows_slots) {
    __shared__ double red[8][32];
    const int s = blockIdx.y;
    if (active && !active[s]) return;
    const int m = d_m ? *d_m : m_max;
    const int per = rows_slots ? gram_rows_wpb(m / b) : 1;
    const int64_t count = (int64_t)m * b;
    const int x = threadIdx.x & 31, g = threadIdx.x >> 5;
    const int64_t e = (int64_t)blockIdx.x * 32 + x;
    if (e - x >= count) return;  // the whole CTA
    const int p0 = seg_chunk_ptr[s] * per, p1 = seg_chunk_ptr[s + 1] * per;
    red[g][x] = e < count ? sum_parts(count, p1 - p0, partial + (int64_t)p0 * count, e, g, 8) : 0.0;
    __syncthreads();
    if (g == 0 && e < count) {
        double v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = red[q][x];
        C[(int64_t)s * m_max * b + e] = ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
    }
}

template <typename T, int B>
bbl_status launch_gram_rows_seg(int64_t n, const int* d_m, const T* Q, const T* W, const int64_t* chunks, int nchunks,
                                const int* active, double* partial, cudaStream_t st) {
    using S = GramRowsShape<T, B>;
    static OncePerDevice once;
    BBL_TRY(allow_smem(once, gram_rows_seg_kernel<T, B>, S::smem_bytes));
    gram_rows_seg_kernel<T, B><<<(unsigned)nchunks, kThreads, S::smem_bytes, st>>>(n, d_m, chunks, active, Q, W,
                                                                                   partial);
    BBL_LAUNCH_CHECK();
    return BBL_OK;
}

template <typename T, int B, int CPT>
__global__ void __launch_bounds__(kThreads) gram_seg_dyn_kernel(int64_t n, const int* __restrict__ d_m,
                                                                const int64_t* __restrict__ chunks,
                                                                const int* __restrict__ seg_active,
                                                                const T* __restrict__ Q, const T* __restrict__ W,
                                                                double* __restrict__ partial) {
    const int64_t seg = chunks[3 * blockIdx.x];
    if (seg_active && !seg_active[seg]) return;
    const int m = *d_m;
    const int cols = (m + CPT - 1) / CPT;
    int TC = 1;
    while (TC < cols && TC < kThreads) TC <<= 1;
    if ((int)blockIdx.y * TC * CPT >= m) return;
    gram_body<T, B, CPT>(n, m, OneRange{chunks[3 * blockIdx.x + 1], chunks[3 * blockIdx.x + 2]}, TC, blockIdx.y, Q, W,
                         partial + (int64_t)blockIdx.x * m * B);
}

template <typename T, int B, int CPT>
bbl_status launch_gram_seg(int64_t n, int m_max, const int* d_m, const T* Q, const T* W, const int64_t* chunks,
                           int nchunks, const int* active, double* partial, cudaStream_t st) {
    const int cols = (m_max + CPT - 1) / CPT;
    const int gy = (cols + kThreads - 1) / kThreads;
    static OncePerDevice once;
    BBL_TRY(allow_smem(once, gram_seg_dyn_kernel<T, B, CPT>, sizeof(double) * kThreads * CPT * B));
    dim3 grid((unsigned)nchunks, (unsigned)gy);
    gram_seg_dyn_kernel<T, B, CPT><<<grid, kThreads, sizeof(double) * kThreads * CPT * B, st>>>(n, d_m, chunks, active,
                                                                                                Q, W, partial);
    BBL_LAUNCH_CHECK();
    return BBL_OK;
}

template <typename T, bool SUB, typename TA, typename TO, int B>
bbl_status launch_apply_seg(int64_t n, int kc, const int* ms, int mss, const int64_t* ctas, int nctas,
                            const int* active, const T* Q, const double* C, int64_t cstride, TO* W, cudaStream_t st) {
    if (kc == B)
        apply_seg_kernel<T, B, B, SUB, TA, TO><<<nctas, kThreads, 0, st>>>(n, 0, ms, mss, kc, ctas, active, Q, C,
                                                                          cstride, W);
    else
        apply_seg_kernel<T, B, 0, SUB, TA, TO><<<nctas, kThreads, 0, st>>>(n, 0, ms, mss, kc, ctas, active, Q, C,
                                                                          cstride, W);
    BBL_LAUNCH_CHECK();
    return BBL_OK;
}

template <typename T, bool SUB, typename TA, typename TO>
bbl_status apply_seg_typed(int64_t n, int b, int kc, const int* ms, int mss, const int64_t* ctas, int nctas,
                           const int* active, const T* Q, const double* C, int64_t cstride, TO* W, cudaStream_t st) {
    switch (b) {
        case 1: return launch_apply_seg<T, SUB, TA, TO, 1>(n, kc, ms, mss, ctas, nctas, active, Q, C, cstride, W, st);
        case 2: return launch_apply_seg<T, SUB, TA, TO, 2>(n, kc, ms, mss, ctas, nctas, active, Q, C, cstride, W, st);
        case 4:  // (FP64 updates of 4 and 8 columns: tc64.cu)
            if constexpr (!(SUB && std::is_same<T, double>::value))
                return launch_apply_seg<T, SUB, TA, TO, 4>(n, kc, ms, mss, ctas, nctas, active, Q, C, cstride, W, st);
            break;
        case 8:
            if constexpr (!(SUB && std::is_same<T, double>::value))
                return launch_apply_seg<T, SUB, TA, TO, 8>(n, kc, ms, mss, ctas, nctas, active, Q, C, cstride, W, st);
            break;
        case 16: return launch_apply_seg<T, SUB, TA, TO, 16>(n, kc, ms, mss, ctas, nctas, active, Q, C, cstride, W, st);
        default: break;
    }
    return set_error(BBL_ERR_UNSUPPORTED, "batched: b=%d (supported: 1, 2, 4, 8, 16)", b);
}

}  // namespace

int gram_seg_chunk_rows(int b, int dtype) {
    if (dtype == BBL_FP64) {
        if (b == 4 || b == 8) return tc64_seg_chunk_rows();  // within the row kernel's tile
    } else if (dtype == BBL_FP32) {
        if (b == 4) return GramRowsShape<float, 4>::R;
        if (b == 8) return GramRowsShape<float, 8>::R;
        if (b == 16) return GramRowsShape<float, 16>::R;
    }
    return 0;
}

bbl_status gram_seg(int64_t n, int b, int m_max, const int* d_m, int dtype, const void* Q, const void* W,
                    const int64_t* chunks, int nchunks, const int* seg_chunk_ptr, int nseg, const int* active,
                    double* partial, double* C, cudaStream_t st) {
    // against a whole basis the FP64 products run on the tensor cores; the self
    // Gram of one block (m_max = b) fills too little of a tile of 16 columns
    const bool tc = dtype == BBL_FP64 && tc64_seg_supports(b) && m_max >= 32;
    const int rows_slots = !tc && gram_seg_chunk_rows(b, dtype) > 0 ? 1 : 0;
    if (tc) {
        BBL_TRY(gram_tc64_seg(n, b, d_m, static_cast<const double*>(Q), static_cast<const double*>(W), chunks, nchunks,
                              active, partial, st));
    } else if (rows_slots) {
        if (dtype == BBL_FP64) {
            auto q = static_cast<const double*>(Q);
            auto w = static_cast<const double*>(W);
            if (b == 4) BBL_TRY((launch_gram_rows_seg<double, 4>(n, d_m, q, w, chunks, nchunks, active, partial, st)));
            else BBL_TRY((launch_gram_rows_seg<double, 8>(n, d_m, q, w, chunks, nchunks, active, partial, st)));
        } else {
            auto q = static_cast<const float*>(Q);
            auto w = static_cast<const float*>(W);
            if (b == 4) BBL_TRY((launch_gram_rows_seg<float, 4>(n, d_m, q, w, chunks, nchunks, active, partial, st)));
            else if (b == 8) BBL_TRY((launch_gram_rows_seg<float, 8>(n, d_m, q, w, chunks, nchunks, active, partial, st)));
            else BBL_TRY((launch_gram_rows_seg<float, 16>(n, d_m, q, w, chunks, nchunks, active, partial, st)));
        }
    } else if (dtype == BBL_FP64) {
        auto q = static_cast<const double*>(Q);
        auto w = static_cast<const double*>(W);
        switch (b) {
            case 1: BBL_TRY((launch_gram_seg<double, 1, 1>(n, m_max, d_m, q, w, chunks, nchunks, active, partial, st))); break;
            case 2: BBL_TRY((launch_gram_seg<double, 2, 2>(n, m_max, d_m, q, w, chunks, nchunks, active, partial, st))); break;
            case 16: BBL_TRY((launch_gram_seg<double, 16, 2>(n, m_max, d_m, q, w, chunks, nchunks, active, partial, st))); break;
            default: return set_error(BBL_ERR_UNSUPPORTED, "batched: b=%d", b);
        }
    } else {
        auto q = static_cast<const float*>(Q);
        auto w = static_cast<const float*>(W);
        switch (b) {
            case 1: BBL_TRY((launch_gram_seg<float, 1, 1>(n, m_max, d_m, q, w, chunks, nchunks, active, partial, st))); break;
            case 2: BBL_TRY((launch_gram_seg<float, 2, 2>(n, m_max, d_m, q, w, chunks, nchunks, active, partial, st))); break;
            default: return set_error(BBL_ERR_UNSUPPORTED, "batched: b=%d", b);
        }
    }
    if (!C) return BBL_OK;  // the caller takes the partial sums
    dim3 g((unsigned)ceil_div((int64_t)m_max * b, 32), (unsigned)nseg);
    reduce_seg_kernel<<<g, 256, 0, st>>>(m_max, b, d_m, seg_chunk_ptr, active, partial, C, rows_slots);
    BBL_LAUNCH_CHECK();
    return BBL_OK;
}

bbl_status apply_seg(int64_t n, int b, int kc, const int* ms, int ms_stride, int dtype, const void* Q, const double* C,
                     int64_t cstride, void* W, bool sub, bool f64_out, const int64_t* ctas, int nctas, const int* active,
                     cudaStream_t st) {
    if (dtype == BBL_FP64) {
        auto q = static_cast<const double*>(Q);
        if (sub && tc64_seg_supports(b))  // (kc is b)
            return update_tc64_seg(n, b, ms, ms_stride, ctas, nctas, active, q, C, cstride, static_cast<double*>(W), st);
        if (sub) return apply_seg_typed<double, true, double, double>(n, b, kc, ms, ms_stride, ctas, nctas, active, q, C, cstride,
                                                                      static_cast<double*>(W), st);
        return apply_seg_typed<double, false, double, double>(n, b, kc, ms, ms_stride, ctas, nctas, active, q, C, cstride,
                                                              static_cast<double*>(W), st);
    }
    auto q = static_cast<const float*>(Q);
    if (f64_out)
        return apply_seg_typed<float, false, double, double>(n, b, kc, ms, ms_stride, ctas, nctas, active, q, C, cstride,
                                                             static_cast<double*>(W), st);
    if (sub) return apply_seg_typed<float, true, float, float>(n, b, kc, ms, ms_stride, ctas, nctas, active, q, C, cstride,
                                                               static_cast<float*>(W), st);
    return apply_seg_typed<float, false, float, float>(n, b, kc, ms, ms_stride, ctas, nctas, active, q, C, cstride,
                                                       static_cast<float*>(W), st);
}

// partial: of gram_seg with m_max = b and no C
bbl_status chol_seg(int b, int dtype, int nseg, const double* partial, const int* seg_chunk_ptr, const double* thresh2,
                    int relative, double* R, double* Rinv, int* ndefl, int* mask, int* status, const int* active,
                    cudaStream_t st) {
    const int per = gram_seg_chunk_rows(b, dtype) > 0 ? gram_rows_wpb(1) : 1;
    chol_seg_kernel<<<(unsigned)nseg, kCholThreads, 0, st>>>(b, partial, seg_chunk_ptr, per, thresh2, relative, R, Rinv,
                                                             ndefl, mask, status, active);
    BBL_LAUNCH_CHECK();
    return BBL_OK;
}

}  // namespace bbl

// -------------------------------------------------------------------- C ABI
extern "C" {

bbl_status bbl_block_reorth(int64_t n, int b, int nblocks, bbl_dtype dtype, const void* basis, void* W, double* coeff,
                            int passes, void* stream) {
    using namespace bbl;
    if (n < 1 || b < 1 || b > kMaxB || nblocks < 1 || passes < 1 || passes > 2 || !basis || !W)
        return set_error(BBL_ERR_INVALID_ARG, "block_reorth: bad arguments");
    if (dtype != BBL_FP64 && dtype != BBL_FP32) return set_error(BBL_ERR_INVALID_ARG, "block_reorth: bad dtype");
    if (!aligned16(basis) || !aligned16(W)) return set_error(BBL_ERR_INVALID_ARG, "block_reorth: pointers must be 16-byte aligned");
    cudaStream_t st = as_stream(stream);
    DevBuf partials(st), cbuf(st);
    const int m = nblocks * b;
    double* C = coeff;
    if (!C) {
        BBL_TRY(cbuf.alloc(sizeof(double) * m * b));
        C = cbuf.as<double>();
    }
    for (int p = 0; p < passes; ++p) {
        double* Cp = coeff ? coeff + (size_t)p * m * b : C;
        BBL_TRY(gram(n, b, nblocks, dtype, basis, W, Cp, partials, st));
        BBL_TRY(update(n, b, nblocks, dtype, basis, Cp, W, st));
    }
    BBL_CUDA(cudaStreamSynchronize(st));
    return BBL_OK;
}

bbl_status bbl_cholqr2(int64_t n, int b, bbl_dtype dtype, void* W, double* B, double defl_abs, int* n_deflated,
                       void* stream) {
    using namespace bbl;
    if (n < 1 || b < 1 || b > kMaxB || !W || !B) return set_error(BBL_ERR_INVALID_ARG, "cholqr2: bad arguments");
    if (dtype != BBL_FP64 && dtype != BBL_FP32) return set_error(BBL_ERR_INVALID_ARG, "cholqr2: bad dtype");
    if (!aligned16(W)) return set_error(BBL_ERR_INVALID_ARG, "cholqr2: W must be 16-byte aligned");
    if (defl_abs < 0) return set_error(BBL_ERR_INVALID_ARG, "cholqr2: defl_abs < 0");
    cudaStream_t st = as_stream(stream);
    DevBuf partials(st), small(st), cnt(st);
    BBL_TRY(cnt.alloc(sizeof(int)));
    BBL_CUDA(cudaMemsetAsync(cnt.p, 0, sizeof(int), st));
    BBL_TRY(small.alloc(sizeof(double) * 8 * kMaxB * kMaxB + sizeof(int) * 4 * kMaxB));
    BBL_CUDA(cudaMemsetAsync(small.p, 0, small.bytes, st));
    BBL_TRY(cholqr2_dev(n, b, dtype, W, B, defl_abs * defl_abs, cnt.as<int>(), nullptr, partials, small, st));
    int h[2] = {0, 0};
    BBL_CUDA(cudaMemcpyAsync(&h[0], cnt.p, sizeof(int), cudaMemcpyDeviceToHost, st));
    BBL_CUDA(cudaMemcpyAsync(&h[1], reinterpret_cast<char*>(small.p) + sizeof(double) * 8 * kMaxB * kMaxB,
                             sizeof(int), cudaMemcpyDeviceToHost, st));
    BBL_CUDA(cudaStreamSynchronize(st));
    if (n_deflated) *n_deflated = h[0];
    if (h[1]) return set_error(BBL_ERR_NUMERICAL, "cholqr2: non-finite Gram matrix");
    return BBL_OK;
}

bbl_status bbl_ritz_vectors(int64_t n, int b, int nblocks, bbl_dtype dtype, const void* basis, int k, const double* S,
                            double* X, void* stream) {
    using namespace bbl;
    if (n < 1 || b < 1 || b > kMaxB || nblocks < 1 || k < 1 || k > kMaxB || !basis || !S || !X)
        return set_error(BBL_ERR_INVALID_ARG, "ritz_vectors: bad arguments");
    if (!aligned16(basis)) return set_error(BBL_ERR_INVALID_ARG, "ritz_vectors: basis must be 16-byte aligned");
    BBL_TRY(ritz_vectors(n, b, nblocks, dtype, basis, k, S, X, as_stream(stream)));
    BBL_CUDA(cudaStreamSynchronize(as_stream(stream)));
    return BBL_OK;
}

}  // extern "C"

// -------------------------------------------------------------------- allocation-free Gram
// For callers that must not allocate device memory: for example a process
// whose device memory is already handed out by a framework's caching
// allocator under a fixed budget, or a latency-critical loop that cannot
// afford the implicit device synchronisation of cudaFree.  The per-chunk
// partial sums of the Gram product live in a fixed file-scope device array
// instead of a cudaMalloc'ed buffer.  Every device that loads this library
// holds the array (8 MiB) until the process exits.
namespace bbl {
namespace {

constexpr int64_t kNoAllocScratchDoubles = int64_t(1) << 20;  // 8 MiB: chunk tickets + FP64 partial sums
// The front of the array holds one chunk ticket (int) per column group of the
// Gram.  2048 doubles hold 4096 tickets, more than any request within the
// limit below needs (b = 1: m <= 2^20 - 2048 columns in groups of 256 give at
// most 4088; larger b have fewer groups); the rest holds the partial sums.
constexpr int64_t kNoAllocTicketDoubles = 2048;
constexpr int64_t kNoAllocPartialDoubles = kNoAllocScratchDoubles - kNoAllocTicketDoubles;
__device__ __align__(256) double g_noalloc_gram_scratch[kNoAllocScratchDoubles];

constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mutex;
double* g_noalloc_addr[kMaxDevices] = {};

// Device address of the scratch array for the current device.  Host code
// only holds a host-side stand-in for the array's name, so the address is
// looked up once per device with that device current.
bbl_status noalloc_scratch(double** out) {
    int dev = 0;
    BBL_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) return set_error(BBL_ERR_UNSUPPORTED, "block_gram_noalloc: device %d", dev);
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_addr[dev]) {
        void* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_gram_scratch);
        if (e != cudaSuccess || !p)
            return set_error(BBL_ERR_CUDA, "block_gram_noalloc: cudaGetSymbolAddress failed: %s", cudaGetErrorString(e));
        g_noalloc_addr[dev] = static_cast<double*>(p);
    }
    *out = g_noalloc_addr[dev];
    return BBL_OK;
}

template <typename T, int B, int CPT>
bbl_status launch_gram_fixed(int64_t n, int m, const T* Q, const T* W, double* C, double* scratch, cudaStream_t st) {
    // the front of the array holds the chunk tickets (the ones a call uses
    // are zeroed by that call), the rest the per-worker partial sums
    const int64_t per_worker = (int64_t)m * B;
    if (per_worker > kNoAllocPartialDoubles)
        return set_error(BBL_ERR_INVALID_ARG,
                         "block_gram_noalloc: nblocks*b*b = %lld exceeds the fixed scratch of %lld doubles",
                         (long long)per_worker, (long long)kNoAllocPartialDoubles);
    return gram_core<T, B, CPT>(n, m, Q, W, C, scratch + kNoAllocTicketDoubles, kNoAllocPartialDoubles,
                                reinterpret_cast<int*>(scratch),
                                kNoAllocTicketDoubles * (int64_t)(sizeof(double) / sizeof(int)), st);
}

template <typename T>
bbl_status gram_fixed_typed(int64_t n, int b, int m, const T* Q, const T* W, double* C, double* scratch,
                            cudaStream_t st) {
    constexpr bool F = sizeof(T) == 4;
    switch (b) {
        case 1: return launch_gram_fixed<T, 1, 1>(n, m, Q, W, C, scratch, st);
        case 2: return launch_gram_fixed<T, 2, 2>(n, m, Q, W, C, scratch, st);
        case 4: return launch_gram_fixed<T, 4, F ? 4 : 2>(n, m, Q, W, C, scratch, st);
        case 8: return launch_gram_fixed<T, 8, F ? 4 : 2>(n, m, Q, W, C, scratch, st);
        case 16: return launch_gram_fixed<T, 16, 2>(n, m, Q, W, C, scratch, st);
        default:
            return set_error(BBL_ERR_UNSUPPORTED, "block_gram_noalloc: b=%d (supported: 1, 2, 4, 8, 16)", b);
    }
}

}  // namespace
}  // namespace bbl

extern "C" bbl_status bbl_block_gram_noalloc(int64_t n, int b, int nblocks, bbl_dtype dtype, const void* basis,
                                             const void* W, double* C, void* stream) {
    using namespace bbl;
    if (n < 1 || b < 1 || b > kMaxB || nblocks < 1 || !basis || !W || !C)
        return set_error(BBL_ERR_INVALID_ARG, "block_gram_noalloc: bad arguments");
    if (dtype != BBL_FP64 && dtype != BBL_FP32) return set_error(BBL_ERR_INVALID_ARG, "block_gram_noalloc: bad dtype");
    if (!aligned16(basis) || !aligned16(W))
        return set_error(BBL_ERR_INVALID_ARG, "block_gram_noalloc: pointers must be 16-byte aligned");
    double* scratch = nullptr;
    BBL_TRY(noalloc_scratch(&scratch));
    cudaStream_t st = as_stream(stream);
    const int m = nblocks * b;
    if (dtype == BBL_FP64)
        BBL_TRY(gram_fixed_typed<double>(n, b, m, static_cast<const double*>(basis), static_cast<const double*>(W), C,
                                         scratch, st));
    else
        BBL_TRY(gram_fixed_typed<float>(n, b, m, static_cast<const float*>(basis), static_cast<const float*>(W), C,
                                        scratch, st));
    BBL_CUDA(cudaStreamSynchronize(st));
    return BBL_OK;
}

// -------------------------------------------------------------------- pivot overlap diagnostic
// How much of each converged eigenvector lies in the span of the pivot block
// (Sec. II.B: the pivot must overlap the wanted eigenvectors; Sec. III.A:
// states the pivot misses come late or as intruders).
namespace bbl {
namespace {

constexpr int kOvRows = 64;

// partial[cta][a*k + i] = sum over the CTA's rows r of Q[r][a] X[r][i]
// (thread t < b*k owns the pair a = t / k, i = t % k; row tiles of Q and X
// are staged in shared memory).
__global__ void __launch_bounds__(256) cross_gram_kernel(int64_t n, int b, int k, const double* __restrict__ Q,
                                                         const double* __restrict__ X, double* __restrict__ partial) {
    __shared__ double qs[kOvRows * kMaxB];
    __shared__ double xs[kOvRows * kMaxB];
    const int t = threadIdx.x;
    const int a = t / k, i = t - (t / k) * k;
    double s = 0.0;
    for (int64_t r0 = (int64_t)blockIdx.x * kOvRows; r0 < n; r0 += (int64_t)gridDim.x * kOvRows) {
        const int rows = (int)min((int64_t)kOvRows, n - r0);
        __syncthreads();
        for (int e = t; e < rows * b; e += blockDim.x) qs[e] = Q[r0 * b + e];
        for (int e = t; e < rows * k; e += blockDim.x) xs[e] = X[r0 * k + e];
        __syncthreads();
        if (t < b * k)
            for (int r = 0; r < rows; ++r) s = fma(qs[r * b + a], xs[r * k + i], s);
    }
    if (t < b * k) partial[(int64_t)blockIdx.x * b * k + t] = s;
}

}  // namespace
}  // namespace bbl

extern "C" bbl_status bbl_pivot_overlap(int64_t n, int b, const double* P, int k, const double* X, double* overlap,
                                        void* stream) {
    using namespace bbl;
    if (n < 1 || b < 1 || b > kMaxB || k < 1 || k > kMaxB || !P || !X || !overlap)
        return set_error(BBL_ERR_INVALID_ARG, "pivot_overlap: bad arguments (b, k in 1..%d)", kMaxB);
    cudaStream_t st = as_stream(stream);
    DevBuf Q(st), Xd(st), partials(st), small(st), cnt(st), part(st), C(st);
    BBL_TRY(Q.alloc(sizeof(double) * n * b));
    BBL_CUDA(cudaMemcpyAsync(Q.p, P, sizeof(double) * n * b, cudaMemcpyDefault, st));
    const double* Xp = X;
    if (!is_device_pointer(X)) {
        BBL_TRY(Xd.alloc(sizeof(double) * n * k));
        BBL_CUDA(cudaMemcpyAsync(Xd.p, X, sizeof(double) * n * k, cudaMemcpyHostToDevice, st));
        Xp = Xd.as<double>();
    }
    // Q = orth(P) by CholQR2; a column dependent on the others to 1e-10 of
    // the largest column norm is dropped (a zero column of Q)
    BBL_TRY(cnt.alloc(sizeof(int)));
    BBL_CUDA(cudaMemsetAsync(cnt.p, 0, sizeof(int), st));
    BBL_TRY(small.alloc(sizeof(double) * 8 * kMaxB * kMaxB + sizeof(int) * 4 * kMaxB));
    BBL_CUDA(cudaMemsetAsync(small.p, 0, small.bytes, st));
    DevBuf Bm(st);
    BBL_TRY(Bm.alloc(sizeof(double) * kMaxB * kMaxB));
    BBL_TRY(cholqr2_dev(n, b, BBL_FP64, Q.p, Bm.as<double>(), -1e-20, cnt.as<int>(), nullptr, partials, small, st));
    const int grid = (int)std::min<int64_t>(152 * 4, ceil_div(n, kOvRows));
    BBL_TRY(part.alloc(sizeof(double) * (size_t)grid * b * k));
    BBL_TRY(C.alloc(sizeof(double) * b * k));
    cross_gram_kernel<<<grid, 256, 0, st>>>(n, b, k, Q.as<double>(), Xp, part.as<double>());
    BBL_LAUNCH_CHECK();
    launch_reduce((int64_t)b * k, grid, part.as<double>(), C.as<double>(), st);
    BBL_LAUNCH_CHECK();
    std::vector<double> h(b * k);
    int bad = 0;
    BBL_CUDA(cudaMemcpyAsync(h.data(), C.p, sizeof(double) * b * k, cudaMemcpyDeviceToHost, st));
    BBL_CUDA(cudaMemcpyAsync(&bad, reinterpret_cast<char*>(small.p) + sizeof(double) * 8 * kMaxB * kMaxB, sizeof(int),
                             cudaMemcpyDeviceToHost, st));
    BBL_CUDA(cudaStreamSynchronize(st));
    if (bad) return set_error(BBL_ERR_NUMERICAL, "pivot_overlap: non-finite pivot Gram matrix");
    for (int i = 0; i < k; ++i) {
        double s = 0.0;
        for (int a = 0; a < b; ++a) s += h[a * k + i] * h[a * k + i];
        overlap[i] = std::sqrt(s);
    }
    return BBL_OK;
}
