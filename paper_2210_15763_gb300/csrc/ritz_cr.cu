// S4, the fast path of the Ritz solve: the lowest nev eigenpairs of the band
// matrix T (Eq. 12) without a recurrence over its m rows for the vectors.
//
// A sequential band factorisation is a chain of m dependent row steps: on
// one CTA per eigenvalue the float-float LU with its three triangular solves
// took 1.71 ms and the one-CTA bisection 1.31 ms at m = 728, p = 8, nev = 8,
// with 8 of 152 SMs busy.  The kernels here take 0.15 ms for the same pairs
// (prep 6, slices 29 + 30, vec 79 us; the whole call 6.5 -> 0.20 to 0.26 ms), bound by
// the latency of their dependent steps:
//
//  1. slice   counts the eigenvalues below many shifts at once (Sylvester
//             inertia of T - sigma I, FP32): two rounds of shifts spread over
//             the SMs, first over the Gershgorin interval, then inside each
//             wanted eigenvalue's bracket.  A shift is two threads: one
//             eliminates from the top, one from the bottom, and the P x P
//             Schur complement in the middle adds both (the chain is m/2
//             rows); one warp per scheduler, so a row step costs its
//             latency.  Brackets are 1e-6 to 4e-6 of the spectrum wide.
//  2. vec     one CTA per eigenvalue: block cyclic reduction of T - sigma0 I
//             (blocks of 8 or 16 rows; a block is eliminated with a warp, log2
//             (m / 8) levels) in FP32 at a shift just below the bracket,
//             three inverse iterations, then corrections x -= (T - sigma0 I)^-1
//             (T x - theta x) whose residual and Rayleigh quotient are FP64:
//             each divides the error by the FP32 solve's relative error or
//             (theta - sigma0) / gap, whichever is worse, until the residual
//             is at FP64 rounding.  The reduction's negative pivots count the
//             eigenvalues below sigma0.  FP32 is enough there: over Lanczos
//             bands and random ones (m up to 1920, p 1 to 16) the pairs came out
//             to 1e-15 of the spectrum, as accurate as FP64 LAPACK's.
//
// A pair is accepted when the reduction counts exactly i eigenvalues below
// sigma0, the value lies in its bracket, the bracket holds one eigenvalue
// and the FP64 residual is at most 1e-15 of the Gershgorin bound.  Otherwise
// (degenerate or nearly degenerate values, extreme pivots, non-finite
// input) its need flag is set and the sequential kernels of ritz.cu compute the
// pair as before, from the bracket found here.
#include <algorithm>

#include "ritz.cuh"

namespace bbl {
namespace {

constexpr int kSliceThreads = 128;
constexpr int kSliceShifts = 64;     // per CTA: 2 warps from the top, 2 from the bottom
constexpr int kPrepThreads = 1024;
constexpr int kVecThreads = 1024;
constexpr int kVecWarps = kVecThreads / 32;
constexpr size_t kSmemMax = 220 * 1024;
// 4096 x 512 shifts narrow a bracket to 1e-6 of the spectrum in two launches
// of at most 64 CTAs (8 wanted values), one warp per scheduler; below that FP32
// counts are no longer those of T
constexpr int kMaxNs1 = 4096, kNs2 = 512;
constexpr int kSolvesF32 = 3;        // inverse iterations before the FP64 corrections
constexpr int kMaxCorr = 8;          // FP64 corrections with one factorisation
constexpr int kMaxTries = 3;         // factorisations (shifts) per eigenvalue
constexpr float kAccepted = 1e-15f;  // residual of an accepted pair, relative to the Gershgorin bound

// Shifts of the first round: one problem spreads over the GPU; many segments
// share it (the second round then resolves 512 times finer).
int first_shifts(int nseg) { return nseg <= 4 ? kMaxNs1 : 1024; }

// What the first round found out about a segment.  All values below are
// those of T times 2^-e, which puts the largest |entry| into [1, 2).
struct Hdr {
    float lo, hi;  // Gershgorin interval
    float scale;   // max(|lo|, |hi|)
    int e;
    int ok;        // finite and not zero
};

// One wanted eigenvalue's bracket after the first round.
struct Bracket1 {
    float a, b;
    int cb;  // eigenvalues below b
};

struct Lay {  // fast-path workspace
    Hdr* hdr;          // nseg
    int* need;         // nseg x nev
    double* guess;     // nseg x nev x 2
    Bracket1* br;      // nseg x nev
    int* c1;           // nseg x kMaxNs1
    int* c2;           // nseg x nev x kNs2
    float* band;       // nseg x band_stride: the scaled band in FP32
    int64_t band_stride;
};

__host__ __device__ inline int slice_width(int p) { return p <= 1 ? 1 : p <= 2 ? 2 : p <= 4 ? 4 : p <= 8 ? 8 : 16; }
__host__ __device__ inline int padded_rows(int m, int P) { return m > P + 1 ? m : P + 1; }

size_t round256(size_t x) { return (x + 255) & ~size_t(255); }

size_t layout(int m, int p, int nev, int nseg, void* base, Lay* l) {
    char* q = static_cast<char*>(base);
    const int P = slice_width(p);
    const size_t bs = ((size_t)padded_rows(m, P) * (P + 1) + 3) & ~size_t(3);
    const size_t o1 = round256(sizeof(Hdr) * nseg);
    const size_t og = o1 + round256(sizeof(int) * (size_t)nseg * nev);
    const size_t o2 = og + round256(sizeof(double) * 2 * (size_t)nseg * nev);
    const size_t o3 = o2 + round256(sizeof(Bracket1) * (size_t)nseg * nev);
    const size_t o4 = o3 + round256(sizeof(int) * (size_t)nseg * kMaxNs1);
    const size_t o5 = o4 + round256(sizeof(int) * (size_t)nseg * nev * kNs2);
    if (l) {
        l->hdr = reinterpret_cast<Hdr*>(q);
        l->need = reinterpret_cast<int*>(q + o1);
        l->guess = reinterpret_cast<double*>(q + og);
        l->br = reinterpret_cast<Bracket1*>(q + o2);
        l->c1 = reinterpret_cast<int*>(q + o3);
        l->c2 = reinterpret_cast<int*>(q + o4);
        l->band = reinterpret_cast<float*>(q + o5);
        l->band_stride = (int64_t)bs;
    }
    return o5 + round256(sizeof(float) * bs * nseg);
}

// v * 2^-e rounded to FP32, by integer operations (FP64 instructions issue
// at 1/64 of the FP32 rate); below 2^-126 it is zero.  |v| 2^-e < 2.
__device__ __forceinline__ float scaled_f32(double v, int e) {
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    const int ex = (int)((hi >> 20) & 0x7ff) - 1023 - e + 127;
    if (ex <= 0) return 0.0f;
    unsigned bits = ((unsigned)ex << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29);
    bits += (lo >> 28) & 1u;
    return __uint_as_float(bits | (hi & 0x80000000u));
}

__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// entry (r, r - d) exists: inside the band and the matrix
__device__ __forceinline__ bool in_band(int r, int d, int p) { return d <= p && d <= r; }

// The scaled band in FP32 (rows of P + 1 entries, columns past p zero; rows
// m .. mp - 1 are padding, decoupled, with a large diagonal), its Gershgorin
// interval, and need = 0 (1 if a band is not finite).  One CTA per segment: done once, the slices and
// the reduction then copy FP32 rows.
__global__ void __launch_bounds__(kPrepThreads) prep_kernel(int m, int p, int P, int nev, const double* __restrict__ Tg,
                                                            Hdr* __restrict__ hdr, int* __restrict__ need,
                                                            double* __restrict__ guess,
                                                            float* __restrict__ band, int64_t band_stride,
                                                            SegArgs sa) {
    __shared__ unsigned s_mx;
    __shared__ float s_red[2][kPrepThreads / 32];
    const int seg = blockIdx.x, tid = threadIdx.x;
    if (sa.active && !sa.active[seg]) return;
    if (sa.d_m) m = *sa.d_m;
    Tg += seg * sa.sT;
    band += seg * band_stride;
    const int mp = padded_rows(m, P), P1 = P + 1, p1 = p + 1;
    if (tid == 0) s_mx = 0;
    __syncthreads();
    unsigned mx = 0;
#pragma unroll 4
    for (int x = tid; x < m * p1; x += kPrepThreads) {
        const unsigned h = (unsigned)__double2hiint(Tg[x]) & 0x7fffffffu;
        if (x % p1 <= x / p1) mx = max(mx, h);  // entries left of the matrix are not part of it
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    if ((tid & 31) == 0) atomicMax(&s_mx, mx);
    __syncthreads();
    const int e = (int)(s_mx >> 20) - 1023;  // the largest |entry| is in [2^e, 2^(e+1))
    const bool ok = e > -1023 && e < 1024;
    float lo = 3e38f, hi = -3e38f;
    if (ok) {
#pragma unroll 4
        for (int x = tid; x < mp * P1; x += kPrepThreads) {
            const int r = x / P1, d = x - r * P1;
            float v = 0.0f;
            if (r < m) {
                if (in_band(r, d, p)) v = scaled_f32(Tg[(int64_t)r * p1 + d], e);
            } else if (d == 0) {
                v = 1e30f;
            }
            band[x] = v;
        }
        __syncthreads();
        for (int r = tid; r < m; r += kPrepThreads) {
            float off = 0.0f;
            for (int d = 1; d <= p; ++d) {
                off += fabsf(band[r * P1 + d]);
                if (r + d < m) off += fabsf(band[(r + d) * P1 + d]);
            }
            lo = fminf(lo, band[r * P1] - off);
            hi = fmaxf(hi, band[r * P1] + off);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    if ((tid & 31) == 0) {
        s_red[0][tid >> 5] = lo;
        s_red[1][tid >> 5] = hi;
    }
    __syncthreads();
    if (tid == 0) {
        for (int w = 0; w < kPrepThreads / 32; ++w) {
            lo = fminf(lo, s_red[0][w]);
            hi = fmaxf(hi, s_red[1][w]);
        }
        const float s = fmaxf(fabsf(lo), fabsf(hi));
        Hdr h;
        h.lo = lo - 1e-5f * s;
        h.hi = hi + 1e-5f * s;
        h.scale = fmaxf(fabsf(h.lo), fabsf(h.hi));
        h.e = e;
        h.ok = ok ? 1 : 0;
        hdr[seg] = h;
    }
    if (tid < nev) {
        need[seg * nev + tid] = ok ? 0 : 1;
        guess[2 * (seg * nev + tid)] = guess[2 * (seg * nev + tid) + 1] = 0.0;  // no bracket
    }
}

// copy of the prepared band into shared memory
__device__ __forceinline__ void stage_band(const float* __restrict__ g, int count, float* __restrict__ band) {
    const float4* s = reinterpret_cast<const float4*>(g);
    float4* d = reinterpret_cast<float4*>(band);
#pragma unroll 8
    for (int x = threadIdx.x; x < (count + 3) / 4; x += blockDim.x) d[x] = s[x];
}

// `steps` rows of the LDL^T of T - sigma I from the top (BOT: from the
// bottom, the matrix read in reversed order) by one thread, the lower
// triangle of the (P+1) x (P+1) active window in its registers; returns the
// negative pivots and leaves the window in E.
template <int P, bool BOT>
__device__ __forceinline__ int eliminate(const float* __restrict__ band, int mp, int steps, float sigma, float pivmin,
                                         float (&E)[P + 1][P + 1]) {
    constexpr int P1 = P + 1;
    // entry (R, R - d) of the matrix or of its reversal
    auto at = [&](int R, int d) { return BOT ? band[(mp - 1 - R) * P1 + d * (P1 + 1)] : band[R * P1 + d]; };
#pragma unroll
    for (int r = 0; r < P1; ++r)
#pragma unroll
        for (int c = 0; c <= r; ++c) {
            E[r][c] = at(r, r - c);
            if (r == c) E[r][c] -= sigma;
        }
    int neg = 0;
    float nx[P1];  // the row that enters the window at the end of the step, loaded a step ahead
#pragma unroll
    for (int c = 0; c < P1; ++c) nx[c] = at(min(P1, mp - 1), P - c);
    for (int k = 0; k < steps; ++k) {
        float d = E[0][0];
        if (fabsf(d) < pivmin) d = -pivmin;
        neg += d < 0.0f ? 1 : 0;
        const float rd = rcp_approx(d);
        float l[P1], e0[P1];
#pragma unroll
        for (int r = 1; r < P1; ++r) {
            e0[r] = E[r][0];
            l[r] = e0[r] * rd;
        }
#pragma unroll
        for (int r = 1; r < P1; ++r)
#pragma unroll
            for (int c = 1; c <= r; ++c) E[r - 1][c - 1] = fmaf(-l[r], e0[c], E[r][c]);
#pragma unroll
        for (int c = 0; c < P1; ++c) E[P][c] = nx[c];
        E[P][P] -= sigma;
        const int R = min(k + 1 + P1, mp - 1);  // (past the last row: outside the part that is used)
#pragma unroll
        for (int c = 0; c < P1; ++c) nx[c] = at(R, P - c);
    }
    return neg;
}

// Eigenvalues below sigma for the 64 shifts of a CTA: warps 0, 1 from the
// top, 2, 3 from the bottom; count valid in warps 0 and 1.
template <int P>
__device__ __forceinline__ int count_two_sided(const float* __restrict__ band, int mp, float sigma, float pivmin,
                                               float* __restrict__ xch /* 2 x (P(P+1)/2 + 1) x 32 */) {
    constexpr int P1 = P + 1, NT = P * P1 / 2;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int h = (mp - P) / 2;
    float* mine = xch + (warp & 1) * (NT + 1) * 32 + lane;
    float E[P1][P1];
    int neg;
    if (warp >= 2) {
        neg = eliminate<P, true>(band, mp, mp - h - P, sigma, pivmin, E);
        // window row r of the bottom part is row P - 1 - r of the middle block
        int q = 0;
#pragma unroll
        for (int r = 0; r < P; ++r)
#pragma unroll
            for (int c = 0; c <= r; ++c) mine[32 * q++] = E[P - 1 - c][P - 1 - r];
        mine[32 * NT] = __int_as_float(neg);
    } else {
        neg = eliminate<P, false>(band, mp, h, sigma, pivmin, E);
    }
    __syncthreads();
    if (warp < 2) {
        int q = 0;
#pragma unroll
        for (int r = 0; r < P; ++r)
#pragma unroll
            for (int c = 0; c <= r; ++c) {
                const float a = band[(h + r) * P1 + (r - c)] - (r == c ? sigma : 0.0f);
                E[r][c] += mine[32 * q++] - a;
            }
        neg += __float_as_int(mine[32 * NT]);
#pragma unroll
        for (int k = 0; k < P; ++k) {
            float d = E[k][k];
            if (fabsf(d) < pivmin) d = -pivmin;
            neg += d < 0.0f ? 1 : 0;
            const float rd = rcp_approx(d);
#pragma unroll
            for (int r = k + 1; r < P; ++r) {
                const float l = E[r][k] * rd;
#pragma unroll
                for (int c = k + 1; c <= r; ++c) E[r][c] = fmaf(-l, E[c][k], E[r][c]);
            }
        }
    }
    return neg;
}

// sample t of ns inside (a, b)
__device__ __forceinline__ float sample(float a, float b, int t, int ns) {
    return a + (b - a) * ((float)(t + 1) / (float)(ns + 1));
}

// last sample with at most i eigenvalues below it and the first with more
// (-1 and ns where there is none); all threads of the CTA
__device__ void find_bracket(const int* __restrict__ counts, int ns, int i, int& tl, int& th) {
    __shared__ int s_tl, s_th;
    if (threadIdx.x == 0) {
        s_tl = -1;
        s_th = ns;
    }
    __syncthreads();
    int l = -1, h = ns;
    const int4* c4 = reinterpret_cast<const int4*>(counts);  // ns is a multiple of 4
#pragma unroll 8
    for (int q = threadIdx.x; q < ns / 4; q += blockDim.x) {
        const int4 c = c4[q];
        const int v[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (v[k] <= i) l = max(l, 4 * q + k);
            else h = min(h, 4 * q + k);
        }
    }
    l = __reduce_max_sync(0xffffffffu, l);
    h = __reduce_min_sync(0xffffffffu, h);
    if ((threadIdx.x & 31) == 0) {
        atomicMax(&s_tl, l);
        atomicMin(&s_th, h);
    }
    __syncthreads();
    tl = s_tl;
    th = s_th;
    __syncthreads();
}

template <int P>
constexpr size_t slice_extra() {
    return sizeof(float) * 2 * (P * (P + 1) / 2 + 1) * 32;
}

// First round: 64 shifts of the Gershgorin interval per CTA.
template <int P>
__global__ void __launch_bounds__(kSliceThreads) slice_first_kernel(int m, int ns1, const Hdr* __restrict__ hdr,
                                                                    const float* __restrict__ gband,
                                                                    int64_t band_stride, int* __restrict__ c1,
                                                                    SegArgs sa) {
    extern __shared__ __align__(16) float sl_smem[];
    const int seg = blockIdx.y;
    if (sa.active && !sa.active[seg]) return;
    if (sa.d_m) m = *sa.d_m;
    const Hdr h = hdr[seg];
    if (!h.ok) return;
    const int mp = padded_rows(m, P);
    float* xch = sl_smem;
    float* band = sl_smem + slice_extra<P>() / sizeof(float);
    stage_band(gband + seg * band_stride, mp * (P + 1), band);
    __syncthreads();
    const int t = blockIdx.x * kSliceShifts + (threadIdx.x & 63);
    const int neg = count_two_sided<P>(band, mp, sample(h.lo, h.hi, t, ns1), 1e-7f * h.scale, xch);
    if (threadIdx.x < 64) c1[(int64_t)seg * kMaxNs1 + t] = neg;
}

// Second round: 64 shifts per CTA inside eigenvalue blockIdx.y's bracket.
template <int P>
__global__ void __launch_bounds__(kSliceThreads) slice_second_kernel(int m, int nev, int ns1,
                                                                     const Hdr* __restrict__ hdr,
                                                                     const float* __restrict__ gband,
                                                                     int64_t band_stride,
                                                                     const int* __restrict__ c1,
                                                                     Bracket1* __restrict__ br, int* __restrict__ c2,
                                                                     SegArgs sa) {
    extern __shared__ __align__(16) float sl_smem[];
    const int i = blockIdx.y, seg = blockIdx.z;
    if (sa.active && !sa.active[seg]) return;
    if (sa.d_m) m = *sa.d_m;
    if (i >= min(nev, m)) return;
    const Hdr h = hdr[seg];
    if (!h.ok) return;
    c1 += (int64_t)seg * kMaxNs1;
    const int mp = padded_rows(m, P);
    float* xch = sl_smem;
    float* band = sl_smem + slice_extra<P>() / sizeof(float);
    stage_band(gband + seg * band_stride, mp * (P + 1), band);
    int tl, th;
    find_bracket(c1, ns1, i, tl, th);
    if (tl > th) {  // FP32 counts out of order near the value: both samples are in the bracket
        const int q = tl;
        tl = th - 1;
        th = q + 1;
    }
    const float a = tl >= 0 ? sample(h.lo, h.hi, tl, ns1) : h.lo;
    const float b = th < ns1 ? sample(h.lo, h.hi, th, ns1) : h.hi;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        Bracket1 q;
        q.a = a;
        q.b = b;
        q.cb = th < ns1 ? c1[th] : m;
        br[seg * nev + i] = q;
    }
    const int t = blockIdx.x * kSliceShifts + (threadIdx.x & 63);
    const int neg = count_two_sided<P>(band, mp, sample(a, b, t, kNs2), 1e-7f * h.scale, xch);
    if (threadIdx.x < 64) c2[((int64_t)seg * nev + i) * kNs2 + t] = neg;
}

// ------------------------------------------------------------------ block cyclic reduction
// Blocks of BS rows, J of them (padding rows decoupled).  Level s = 1, 2, 4,
// ...: the remaining blocks are the multiples of s; the odd multiples j are
// eliminated.  D[j]: the diagonal block, then its inverse; L[j]: the coupling
// to the block on the left; Wl[j], Wr[j]: D^-1 times the couplings to the
// left and right neighbour at j's elimination.  Row-major blocks.
template <int BS>
struct CrMat {
    float *D, *L, *Wl, *Wr;
};

// N consecutive floats (N a multiple of 2, the address a multiple of 4 min(N, 4) bytes)
template <int N>
__device__ __forceinline__ void load_part(const float* __restrict__ p, float (&v)[N]) {
    if constexpr (N % 4 == 0) {
#pragma unroll
        for (int q = 0; q < N; q += 4) {
            const float4 x = *reinterpret_cast<const float4*>(p + q);
            v[q] = x.x;
            v[q + 1] = x.y;
            v[q + 2] = x.z;
            v[q + 3] = x.w;
        }
    } else {
#pragma unroll
        for (int q = 0; q < N; q += 2) {
            const float2 x = *reinterpret_cast<const float2*>(p + q);
            v[q] = x.x;
            v[q + 1] = x.y;
        }
    }
}
template <int N>
__device__ __forceinline__ void store_part(float* __restrict__ p, const float (&v)[N]) {
    if constexpr (N % 4 == 0) {
#pragma unroll
        for (int q = 0; q < N; q += 4) *reinterpret_cast<float4*>(p + q) = make_float4(v[q], v[q + 1], v[q + 2], v[q + 3]);
    } else {
#pragma unroll
        for (int q = 0; q < N; q += 2) *reinterpret_cast<float2*>(p + q) = make_float2(v[q], v[q + 1]);
    }
}

// In-place inversion of a symmetric block by BS sweeps (natural order),
// one warp: lane l holds entries (l / LPR, CPL * (l % LPR) + 0 .. CPL - 1).
// Returns the number of negative pivots.
template <int BS>
__device__ __forceinline__ int invert_block(float* __restrict__ D, float pivmin) {
    constexpr int LPR = 32 / BS, CPL = BS / LPR;
    const int lane = threadIdx.x & 31;
    const int r = lane / LPR, q = lane % LPR;
    float a[CPL];
    load_part<CPL>(D + r * BS + q * CPL, a);
    int neg = 0;
#pragma unroll
    for (int k = 0; k < BS; ++k) {
        const int kq = k / CPL, kc = k % CPL;
        float piv = __shfl_sync(0xffffffffu, a[kc], k * LPR + kq);
        const float col = __shfl_sync(0xffffffffu, a[kc], r * LPR + kq);
        float row[CPL];
#pragma unroll
        for (int c = 0; c < CPL; ++c) row[c] = __shfl_sync(0xffffffffu, a[c], k * LPR + q);
        if (fabsf(piv) < pivmin) piv = -pivmin;
        neg += piv < 0.0f ? 1 : 0;
        const float r0 = rcp_approx(piv);
        const float rp = r0 * fmaf(-piv, r0, 2.0f);
        const float l = col * rp;
#pragma unroll
        for (int c = 0; c < CPL; ++c) {
            const bool kcol = q == kq && c == kc;
            float v = fmaf(-l, row[c], a[c]);
            if (r == k) v = kcol ? -rp : row[c] * rp;
            else if (kcol) v = l;
            a[c] = v;
        }
    }
#pragma unroll
    for (int c = 0; c < CPL; ++c) a[c] = -a[c];
    store_part<CPL>(D + r * BS + q * CPL, a);
    return neg;
}

// acc += A B (MODE 0), A B^T (1) or A^T B (2) for the lane's entries of a
// BS x BS product of row-major blocks
template <int BS, int MODE>
__device__ __forceinline__ void block_mul(const float* __restrict__ A, const float* __restrict__ B,
                                          float (&acc)[BS * BS / 32]) {
    constexpr int LPR = 32 / BS, CPL = BS / LPR;
    const int lane = threadIdx.x & 31;
    const int r = lane / LPR, c0 = (lane % LPR) * CPL;
    float x[BS];
    if constexpr (MODE != 2) load_part<BS>(A + r * BS, x);
    else {
#pragma unroll
        for (int k = 0; k < BS; ++k) x[k] = A[k * BS + r];
    }
    if constexpr (MODE == 1) {
#pragma unroll
        for (int c = 0; c < CPL; ++c) {
            float y[BS];
            load_part<BS>(B + (c0 + c) * BS, y);
#pragma unroll
            for (int k = 0; k < BS; ++k) acc[c] = fmaf(x[k], y[k], acc[c]);
        }
    } else {
#pragma unroll
        for (int k = 0; k < BS; ++k) {
            float y[CPL];
            load_part<CPL>(B + k * BS + c0, y);
#pragma unroll
            for (int c = 0; c < CPL; ++c) acc[c] = fmaf(x[k], y[c], acc[c]);
        }
    }
}

template <int BS>
__device__ __forceinline__ void block_store(float* __restrict__ D, float (&v)[BS * BS / 32], float sign) {
    constexpr int LPR = 32 / BS, CPL = BS / LPR;
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int c = 0; c < CPL; ++c) v[c] *= sign;
    store_part<CPL>(D + (lane / LPR) * BS + (lane % LPR) * CPL, v);
}

// Factors the matrix in M; returns (to thread 0's warp via *s_neg) the number
// of negative pivots.  All threads.
template <int BS>
__device__ void cr_factor(const CrMat<BS>& M, int J, float pivmin, int* s_neg) {
    constexpr int BB = BS * BS, CPL = BB / 32;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int neg = 0;
    for (int s = 1; s < J; s <<= 1) {
        for (int j = s + 2 * s * warp; j < J; j += 2 * s * kVecWarps) {
            float* Dj = M.D + (int64_t)j * BB;
            neg += invert_block<BS>(Dj, pivmin);
            __syncwarp();
            float w[CPL] = {};
            block_mul<BS, 0>(Dj, M.L + (int64_t)j * BB, w);
            block_store<BS>(M.Wl + (int64_t)j * BB, w, 1.0f);
            if (j + s < J) {
                float v[CPL] = {};
                block_mul<BS, 1>(Dj, M.L + (int64_t)(j + s) * BB, v);
                block_store<BS>(M.Wr + (int64_t)j * BB, v, 1.0f);
            }
        }
        __syncthreads();
        for (int r = 2 * s * warp; r < J; r += 2 * s * kVecWarps) {
            const int j = r - s, j2 = r + s;
            float u[CPL] = {}, nl[CPL] = {};
            if (j >= 0) {
                block_mul<BS, 0>(M.L + (int64_t)r * BB, M.Wr + (int64_t)j * BB, u);
                block_mul<BS, 0>(M.L + (int64_t)r * BB, M.Wl + (int64_t)j * BB, nl);
            }
            if (j2 < J) block_mul<BS, 2>(M.L + (int64_t)j2 * BB, M.Wl + (int64_t)j2 * BB, u);
            __syncwarp();
            constexpr int LPR = 32 / BS, CP = BS / LPR;
            float* Dr = M.D + (int64_t)r * BB + (lane / LPR) * BS + (lane % LPR) * CP;
            float dv[CPL];
            load_part<CPL>(Dr, dv);
#pragma unroll
            for (int c = 0; c < CPL; ++c) dv[c] -= u[c];
            store_part<CPL>(Dr, dv);
            if (j >= 0) block_store<BS>(M.L + (int64_t)r * BB, nl, -1.0f);
        }
        __syncthreads();
    }
    if (warp == 0) neg += invert_block<BS>(M.D, pivmin);
    if (lane == 0 && neg) atomicAdd(s_neg, neg);
    __syncthreads();
}

// F <- (T - sigma I)^-1 F from the factored M.  All threads.
template <int BS>
__device__ void cr_solve(const CrMat<BS>& M, int J, float* __restrict__ F) {
    constexpr int BB = BS * BS, LPR = 32 / BS;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tc = lane % BS, tk = lane / BS;     // transposed product: column, first row
    const int r = lane / LPR, q = lane % LPR;     // plain product: row, part
    int top = 1;
    for (int s = 1; s < J; s <<= 1) {
        for (int b = 2 * s * warp; b < J; b += 2 * s * kVecWarps) {
            float t = 0.0f;
            if (b - s >= 0) {
                const float* W = M.Wr + (int64_t)(b - s) * BB;
                const float* f = F + (b - s) * BS;
#pragma unroll
                for (int k = tk; k < BS; k += LPR) t = fmaf(W[k * BS + tc], f[k], t);
            }
            if (b + s < J) {
                const float* W = M.Wl + (int64_t)(b + s) * BB;
                const float* f = F + (b + s) * BS;
#pragma unroll
                for (int k = tk; k < BS; k += LPR) t = fmaf(W[k * BS + tc], f[k], t);
            }
#pragma unroll
            for (int o = BS; o < 32; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            if (tk == 0) F[b * BS + tc] -= t;
        }
        __syncthreads();
        top = s;
    }
    auto row_dot = [&](const float* W, const float* f) {
        float t = 0.0f;
#pragma unroll
        for (int k = 0; k < BS / LPR; ++k) t = fmaf(W[r * BS + q * (BS / LPR) + k], f[q * (BS / LPR) + k], t);
        return t;
    };
    auto reduce_row = [&](float t) {
#pragma unroll
        for (int o = 1; o < LPR; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        return t;
    };
    if (warp == 0) {
        const float t = reduce_row(row_dot(M.D, F));
        __syncwarp();
        if (q == 0) F[r] = t;
    }
    __syncthreads();
    if (J == 1) return;
    for (int s = top; s >= 1; s >>= 1) {
        for (int j = s + 2 * s * warp; j < J; j += 2 * s * kVecWarps) {
            float t = row_dot(M.D + (int64_t)j * BB, F + j * BS) -
                      row_dot(M.Wl + (int64_t)j * BB, F + (j - s) * BS);
            if (j + s < J) t -= row_dot(M.Wr + (int64_t)j * BB, F + (j + s) * BS);
            t = reduce_row(t);
            __syncwarp();
            if (q == 0) F[j * BS + r] = t;
        }
        __syncthreads();
    }
}

// sums over the CTA; every thread gets the same values (two barriers)
template <int N, typename T>
__device__ __forceinline__ void block_sum(T (&v)[N], T* red /* kVecWarps x N */) {
    static_assert(kVecWarps == 32, "the second stage is one value per lane");
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int q = 0; q < N; ++q) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
    if (lane == 0) {
#pragma unroll
        for (int q = 0; q < N; ++q) red[warp * N + q] = v[q];
    }
    __syncthreads();
    if constexpr (sizeof(T) == 4) {
#pragma unroll
        for (int q = 0; q < N; ++q) v[q] = red[lane * N + q];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int q = 0; q < N; ++q) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
        __syncthreads();
    } else {  // FP64: one warp adds (every warp would issue the same FP64 instructions)
        if (warp == 0) {
#pragma unroll
            for (int q = 0; q < N; ++q) v[q] = red[lane * N + q];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int q = 0; q < N; ++q) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
            __syncwarp();
            if (lane == 0) {
#pragma unroll
                for (int q = 0; q < N; ++q) red[q] = v[q];
            }
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < N; ++q) v[q] = red[q];
        __syncthreads();
    }
}

template <int BS>
__host__ __device__ constexpr size_t vec_mat_floats(int J) {
    return (size_t)4 * J * BS * BS;
}
// the vector (FP64) and the right-hand side (FP32)
template <int BS>
__host__ __device__ constexpr size_t vec_vectors_bytes(int J) {
    return (size_t)J * BS * (sizeof(double) + sizeof(float));
}

template <int BS>
__global__ void __launch_bounds__(kVecThreads) vec_kernel(int m, int p, int nev, const double* __restrict__ Tg,
                                                          int mats_in_smem, const Hdr* __restrict__ hdr,
                                                          const Bracket1* __restrict__ br, const int* __restrict__ c2,
                                                          const float* __restrict__ band, int64_t band_stride,
                                                          double* __restrict__ ws, int64_t ws_stride,
                                                          double* __restrict__ theta, double* __restrict__ S,
                                                          int* __restrict__ need, double* __restrict__ guess,
                                                          SegArgs sa) {
    constexpr int BB = BS * BS;
    extern __shared__ __align__(16) unsigned char vk_smem[];
    __shared__ double red64[kVecWarps];
    __shared__ float red[kVecWarps * 3];
    __shared__ int s_neg, s_idx;
    __shared__ unsigned long long s_key;
    const int i = blockIdx.x, seg = blockIdx.y, tid = threadIdx.x;
    if (sa.active && !sa.active[seg]) return;
    if (sa.d_m) m = *sa.d_m;
    if (i >= min(nev, m)) return;
    const Hdr h = hdr[seg];
    if (!h.ok) return;
    Tg += seg * sa.sT;
    theta += seg * sa.sTh;
    S += seg * sa.sS;
    band += seg * band_stride;
    const int J = (m + BS - 1) / BS, p1 = p + 1, P1 = slice_width(p) + 1;
    double* x = reinterpret_cast<double*>(vk_smem);
    float* F = reinterpret_cast<float*>(x + (size_t)J * BS);
    float* mats = mats_in_smem ? F + (size_t)J * BS
                               : reinterpret_cast<float*>(ws + seg * sa.sWs + (int64_t)i * ws_stride);
    CrMat<BS> M;
    M.D = mats;
    M.L = M.D + (size_t)J * BB;
    M.Wl = M.L + (size_t)J * BB;
    M.Wr = M.Wl + (size_t)J * BB;
    // the bracket, and whether it holds one eigenvalue
    const Bracket1 bk = br[seg * nev + i];
    const int* cc = c2 + ((int64_t)seg * nev + i) * kNs2;
    int tl, th;
    find_bracket(cc, kNs2, i, tl, th);
    if (tl > th) {
        const int t = tl;
        tl = th - 1;
        th = t + 1;
    }
    const float lo = tl >= 0 ? sample(bk.a, bk.b, tl, kNs2) : bk.a;
    const float hi = th < kNs2 ? sample(bk.a, bk.b, th, kNs2) : bk.b;
    bool single = th < kNs2 || bk.cb == i + 1;
    for (int t = th; t < min(th + 3, kNs2); ++t) single = single && cc[t] == i + 1;
    const float margin = 2e-6f * h.scale;
    const float pivmin = 1e-10f * h.scale;
    const double sc = ldexp(1.0, -h.e);
    // value in the scaled units; close enough at the start that the residual
    // y - val x carries the Rayleigh quotient's correction in FP32
    double val = 0.5 * ((double)lo + (double)hi);
    // The sequential kernels leave 2e-15 to 4e-15 with their float-float factors
    // (p = 1, 2, 4, 8) and 1e-16 to 3e-16 with FP64 ones, so there the corrections go on
    // until the residual stalls (30 random bands per p: at most 4.6e-16 and 2.3e-16).
    const float done = p == 1 || p == 2 || p == 4 || p == 8 ? 4e-16f : 0.0f;
    bool good = false, near_val = false;  // near_val: x and val are a pair to 1e-6
    for (int tries = 0; tries < kMaxTries && single && !good; ++tries) {
        // FP32 counts are those of a matrix within about 5e-7 of T: below the
        // bracket (or the value) by four times that, the count is i
        const float sigma = near_val ? (float)val - margin : lo - (float)(1 + tries) * margin;
        if (tid == 0) s_neg = 0;
        // T - sigma I in blocks
#pragma unroll 2
        for (int e = tid; e < J * BB; e += kVecThreads) {
            const int j = e / BB, r = (e % BB) / BS, c = e % BS;
            const int R = j * BS + r;
            float d = 0.0f, l = 0.0f;
            if (R >= m) {
                d = r == c ? 4.0f * h.scale : 0.0f;
            } else {
                const int C = j * BS + c;
                if (r == c) {
                    d = (float)(Tg[(int64_t)R * p1] * sc - (double)sigma);
                } else if (C < m) {
                    const int a = max(R, C), o = a - min(R, C);
                    if (o <= p) d = band[a * P1 + o];
                }
                const int o = BS + r - c;  // row R, column C - BS
                if (j > 0 && o <= p) l = band[R * P1 + o];
            }
            M.D[e] = d;
            M.L[e] = l;
        }
        if (!near_val) {
            // pseudo-random start (splitmix-style hash of (index, try, row))
            for (int r = tid; r < J * BS; r += kVecThreads) {
                uint64_t z = ((uint64_t)i + 1 + 64 * tries) * 0x9E3779B97F4A7C15ull + (uint64_t)r + 0x632BE59BD9B4E019ull;
                z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
                z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
                z ^= z >> 31;
                F[r] = r < m ? (float)(z >> 40) * 0x1.0p-23f - 1.0f : 0.0f;
            }
        }
        __syncthreads();
        cr_factor<BS>(M, J, pivmin, &s_neg);
        const bool counted = s_neg == i;
        __syncthreads();
        if (!counted) continue;
        if (!near_val) {
            val = 0.5 * ((double)lo + (double)hi);
            for (int it = 0; it < kSolvesF32; ++it) {
                cr_solve<BS>(M, J, F);
                // back to O(1): an exact power of two from the largest entry
                unsigned mx = 0;
                for (int r = tid; r < m; r += kVecThreads) mx = max(mx, __float_as_uint(F[r]) & 0x7fffffffu);
                mx = __reduce_max_sync(0xffffffffu, mx);
                if (tid == 0) s_idx = 0;
                __syncthreads();
                if ((tid & 31) == 0) atomicMax(&s_idx, (int)mx);
                __syncthreads();
                const int ex = (s_idx >> 23) - 127;
                const float f = ex >= -126 && ex <= 126 ? __uint_as_float((unsigned)(127 - ex) << 23) : 1.0f;
                for (int r = tid; r < J * BS; r += kVecThreads) F[r] *= f;
                __syncthreads();
            }
            for (int r = tid; r < J * BS; r += kVecThreads) x[r] = (double)F[r];
            __syncthreads();
        }
        // corrections with FP64 residuals r = T x - val x; val moves by the FP32
        // quotient x.r / x.x, exact enough as r shrinks
        float prev = 0.0f;
        for (int it = 0; it < kMaxCorr; ++it) {
            float v[3] = {0.0f, 0.0f, 0.0f};
            for (int r = tid; r < m; r += kVecThreads) {
                const double xr = x[r];
                const double* row = Tg + (int64_t)r * p1;
                double t = row[0] * xr;
                const int dl = min(p, r), du = min(p, m - 1 - r);
                for (int d = 1; d <= dl; ++d) t = fma(row[d], x[r - d], t);
                for (int d = 1; d <= du; ++d) t = fma(row[(int64_t)d * (p + 2)], x[r + d], t);
                const float rf = (float)fma(t, sc, -val * xr), xf = (float)xr;
                F[r] = rf;
                v[0] = fmaf(xf, rf, v[0]);
                v[1] = fmaf(xf, xf, v[1]);
                const float rs = rf * 0x1.0p+30f;
                v[2] = fmaf(rs, rs, v[2]);
            }
            block_sum<3>(v, red);
            const float dval = v[0] / v[1];
            const float rel = sqrtf(v[2] / v[1]) * 0x1.0p-30f / h.scale;  // relative residual
            val += (double)dval;
            near_val = rel <= 1e-6f;
            if (!(rel < 1e30f)) break;  // not a number
            // at FP64 rounding, or no longer falling by 4: judged by its size
            if (rel <= done || (it > 0 && rel > 0.25f * prev)) {
                good = rel <= kAccepted;
                break;
            }
            prev = rel;
            for (int r = tid; r < J * BS; r += kVecThreads) F[r] = r < m ? fmaf(-dval, (float)x[r], F[r]) : 0.0f;
            __syncthreads();
            cr_solve<BS>(M, J, F);
            for (int r = tid; r < m; r += kVecThreads) x[r] -= (double)F[r];
            __syncthreads();
        }
        // the value the count speaks of: the first above sigma, in the bracket
        good = good && val > (double)sigma && val <= (double)hi + (double)margin;
        near_val = near_val && !good && val > (double)lo - (double)margin && val <= (double)hi + (double)margin;
    }
    if (!good) {
        if (tid == 0) {
            need[seg * nev + i] = 1;
            guess[2 * (seg * nev + i)] = ldexp((double)lo - 1e-6 * h.scale, h.e);
            guess[2 * (seg * nev + i) + 1] = ldexp((double)hi + 1e-6 * h.scale, h.e);
        }
        return;
    }
    // unit vector; the first entry of largest magnitude is positive
    double nrm[1] = {0.0};
    unsigned long long key = 0;
    for (int r = tid; r < m; r += kVecThreads) {
        nrm[0] = fma(x[r], x[r], nrm[0]);
        key = max(key, (unsigned long long)__double_as_longlong(x[r]) & 0x7fffffffffffffffull);
    }
    if (tid == 0) {
        s_key = 0;
        s_idx = 0x7fffffff;
    }
    block_sum<1>(nrm, red64);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) key = max(key, __shfl_xor_sync(0xffffffffu, key, o));
    if ((tid & 31) == 0) atomicMax(&s_key, key);
    if (tid == 0) red64[0] = 1.0 / sqrt(nrm[0]);
    __syncthreads();
    key = s_key;
    for (int r = tid; r < m; r += kVecThreads)
        if (((unsigned long long)__double_as_longlong(x[r]) & 0x7fffffffffffffffull) == key) atomicMin(&s_idx, r);
    __syncthreads();
    const double inv = x[s_idx] < 0.0 ? -red64[0] : red64[0];
    for (int r = tid; r < m; r += kVecThreads) S[(int64_t)r * nev + i] = x[r] * inv;
    if (tid == 0) theta[i] = ldexp(val, h.e);
}

}  // namespace

size_t ritz_cr_vec_doubles(int m, int p) {
    const size_t BS = p <= 8 ? 8 : 16;
    return ((size_t)m + BS - 1) / BS * BS * BS * 2;
}

namespace {

template <int P>
bbl_status launch_slices(int m, int nev, int nseg, const Lay& l, SegArgs sa, cudaStream_t st) {
    const int ns1 = first_shifts(nseg);
    const size_t sm = slice_extra<P>() + sizeof(float) * (size_t)((padded_rows(m, P) * (P + 1) + 3) & ~3);
    static OncePerDevice first_once, second_once;
    BBL_TRY(allow_smem(first_once, slice_first_kernel<P>, kSmemMax));
    BBL_TRY(allow_smem(second_once, slice_second_kernel<P>, kSmemMax));
    slice_first_kernel<P><<<dim3(ns1 / kSliceShifts, nseg), kSliceThreads, sm, st>>>(m, ns1, l.hdr, l.band,
                                                                                    l.band_stride, l.c1, sa);
    BBL_LAUNCH_CHECK();
    slice_second_kernel<P><<<dim3(kNs2 / kSliceShifts, nev, nseg), kSliceThreads, sm, st>>>(
        m, nev, ns1, l.hdr, l.band, l.band_stride, l.c1, l.br, l.c2, sa);
    BBL_LAUNCH_CHECK();
    return BBL_OK;
}

template <int BS>
bbl_status launch_vec(int m, int p, int nev, int nseg, const double* Tb, double* theta, double* S, double* ws,
                      const Lay& l, SegArgs sa, cudaStream_t st) {
    const int J = (m + BS - 1) / BS;
    const size_t vecs = vec_vectors_bytes<BS>(J), mats = sizeof(float) * vec_mat_floats<BS>(J);
    const int in_smem = vecs + mats <= kSmemMax ? 1 : 0;
    static OncePerDevice once;
    BBL_TRY(allow_smem(once, vec_kernel<BS>, kSmemMax));
    vec_kernel<BS><<<dim3(nev, nseg), kVecThreads, vecs + (in_smem ? mats : 0), st>>>(
        m, p, nev, Tb, in_smem, l.hdr, l.br, l.c2, l.band, l.band_stride, ws, (int64_t)ritz_cr_vec_doubles(m, p), theta, S,
        l.need, l.guess, sa);
    BBL_LAUNCH_CHECK();
    return BBL_OK;
}

}  // namespace

size_t ritz_cr_bytes(int m, int p, int nev, int nseg) { return layout(m, p, nev, nseg, nullptr, nullptr); }

// the FP32 band and the vectors fit in shared memory
bool ritz_cr_supports(int m, int p) {
    const int P = slice_width(p), BS = p <= 8 ? 8 : 16;
    const size_t band = sizeof(float) * ((size_t)padded_rows(m, P) * (P + 1) + 4) + sizeof(float) * 2 * (P * (P + 1) / 2 + 1) * 32;
    const size_t vecs = (size_t)((m + BS - 1) / BS) * BS * (sizeof(double) + sizeof(float));
    return band <= kSmemMax && vecs <= kSmemMax;
}

bbl_status ritz_cr(int m, int p, int nev, int nseg, const double* Tb, double* theta, double* S, double* ws, void* fast,
                   SegArgs* out, SegArgs sa, cudaStream_t st) {
    Lay l;
    layout(m, p, nev, nseg, fast, &l);
    out->need = l.need;
    out->guess = l.guess;
    prep_kernel<<<nseg, kPrepThreads, 0, st>>>(m, p, slice_width(p), nev, Tb, l.hdr, l.need, l.guess, l.band, l.band_stride, sa);
    BBL_LAUNCH_CHECK();
    switch (slice_width(p)) {
        case 1: BBL_TRY(launch_slices<1>(m, nev, nseg, l, sa, st)); break;
        case 2: BBL_TRY(launch_slices<2>(m, nev, nseg, l, sa, st)); break;
        case 4: BBL_TRY(launch_slices<4>(m, nev, nseg, l, sa, st)); break;
        case 8: BBL_TRY(launch_slices<8>(m, nev, nseg, l, sa, st)); break;
        default: BBL_TRY(launch_slices<16>(m, nev, nseg, l, sa, st)); break;
    }
    if (p <= 8) return launch_vec<8>(m, p, nev, nseg, Tb, theta, S, ws, l, sa, st);
    return launch_vec<16>(m, p, nev, nseg, Tb, theta, S, ws, l, sa, st);
}

}  // namespace bbl
