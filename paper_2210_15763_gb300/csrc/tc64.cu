// FP64 Gram and update of the Gram-Schmidt passes on the tensor cores, to
// FP64 accuracy (splitting after Ozaki, Ogita, Oishi, Rump 2012 in the FP16
// tensor-core form of Mukunoki, Ozaki, Ogita, Imamura 2020).
//
// GB300's FP64 pipes (1.06 TFLOP/s measured) bind C = Q^T W and W -= Q C at
// 16 operations per 8-byte basis element (b = 8): 12 times the time HBM needs.
// Here an FP64 number becomes an integer of 64 bits relative to a power of
// two near its row's (or column's) largest entry, cut into eight digits of 8
// bits; a digit with its sign is an FP16 number, and a product of two digit
// matrices is exact in the tensor cores' FP32 sums as long as these stay
// below 2^24.  Digit products i, j of one order o = i + j share an
// accumulator: 36 products give the orders 0..7.  Orders 0..4 move to 64-bit
// integers after every 64 terms (at most 64 (1023 * 128 + 3 * 255 * 128 + 255 * 256) <
// 1.13 * 2^24, and above 2^24 only where the first digits are large); orders 5..7
// weigh 2^-40 and less, where FP32 rounding is below 2^-62.  The basis is cut in
// sign and magnitude (the first digit has two spare bits, so a line may outgrow
// its first entries fourfold); the other operand, cut once per CTA, into balanced
// digits -128..127 of the rounded value, so that the dropped orders (below 2^-62 of
// the largest products) have random signs instead of the products' own.
//
// What the cut loses is measured against a line's largest entry, and a sum whose
// own terms are all far below that (a basis column with one large entry opposite
// a zero, a row that is tiny where the coefficients are large) would lose bits that
// FP64 sums keep.  So each sum certifies itself: one more product, of the leading
// digits' magnitudes, gives Sigma, which is at most twice sum |q||w| in units of
// 2^96 of the (56-bit) integers' product.  What is dropped and truncated is at most
// 2^50.5 per term, and about 2^46.5 with a random sign: 2^51 over 512 terms.  From
// Sigma = 128 on, sum |q||w| of 2^102 and more, that is 4 x 2^-53 of it over 512 terms
// (3 N x 2^-53 for N terms if all signs agree; the bound of an FP64 sum in sequence
// is N x 2^-53).  A sum below, or with an operand that is not finite, is formed
// again by FP64 FMA, which also treats infinities and numbers below the digits'
// range as FP64 does.  In a Lanczos run that is about one sum in 10^5 (the update
// counts |W|, by which its difference rounds, towards Sigma).  The largest error
// of any sum, relative to its sum of magnitudes, on orthonormal bases (n = 2e4, b = 4,
// 360 columns; n = 2e5, b = 8, 400): Gram 9.1e-17 and 1.1e-16, update 5.8e-17 and
// 7.4e-17; FP64 FMA kernels 1.3e-16 and 1.8e-16, 1.9e-16 and 2.8e-16; 56-bit
// integers without the check 9.2e-17 and 1.2e-16, 6.1e-16 and 6.1e-16.
//
// Digits are cut by integer instructions in registers from a ring of
// asynchronous copies.  At n = 6e5, b = 8, 90 blocks (3.5 GB, 0.51 ms at the copy
// rate) the Gram takes 1.23 ms and the update 1.20 ms (with 56 bits and no check
// 1.09 and 1.12).  What bounds them is the latency of the cutting at four warps per
// scheduler (integer pipe about half, tensor pipe a third active, DRAM a third of
// the copy rate).
#include <algorithm>
#include <cstdint>

#include <cuda_fp16.h>

#include "async_mma.cuh"
#include "common.cuh"

namespace bbl {
namespace {

constexpr int kT = 256;            // threads per CTA
constexpr int kWarps = kT / 32;
constexpr int kDig = 8;            // digits of 8 bits
constexpr int kOrd = 8;            // orders summed (of the products' 15)
constexpr int kExact = 5;          // orders kept exactly
constexpr float kCertified = 128.0f;  // a sum's Sigma from which the digits' error is that of FP64 sums
constexpr int kOver = 2;           // bits by which an entry may exceed its line's scale (the first digit's spare bits)
constexpr int kMaxRows = 448;      // Gram: rows per CTA (two CTAs per SM by their shared memory)
constexpr int kMaxCols = 512;      // update: coefficient rows staged at once
constexpr int kEmin = 100;         // smallest exponent field used for a scale
constexpr int kRing = 3;           // steps of a warp in its shared-memory ring
constexpr int kStepBytes = 2048;   // 16 x 16 basis entries

struct Acc {
    float f[kOrd][4];   // order sums
    long long h[4];     // exact sums of the first orders, in units of order 4
    float c[4];         // Sigma, in units of the present scales
    __device__ __forceinline__ Acc() {
        clear();
#pragma unroll
        for (int e = 0; e < 4; ++e) c[e] = 0.0f;
    }
    __device__ __forceinline__ void clear() {  // the sums, not Sigma
#pragma unroll
        for (int o = 0; o < kOrd; ++o)
#pragma unroll
            for (int e = 0; e < 4; ++e) f[o][e] = 0.0f;
#pragma unroll
        for (int e = 0; e < 4; ++e) h[e] = 0;
    }
    __device__ __forceinline__ void to_int() {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int i1 = __float2int_rn(f[1][e]), i2 = __float2int_rn(f[2][e]), i3 = __float2int_rn(f[3][e]);
            const long long up = (long long)i1 * (1 << 24) + h[e];
            const long long low = (long long)i3 * (1 << 8) + ((long long)i2 * (1 << 16) + __float2int_rn(f[4][e]));
            h[e] = up + low + (long long)__float2int_rn(f[0][e]) * (1ll << 32);
        }
#pragma unroll
        for (int o = 0; o < kExact; ++o)
#pragma unroll
            for (int e = 0; e < 4; ++e) f[o][e] = 0.0f;
    }
    // the sum over the orders in units of order 4 (call to_int before)
    __device__ __forceinline__ double value(int e) const {
        const float L = fmaf(fmaf(f[7][e], 0x1p-8f, f[6][e]), 0x1p-8f, f[5][e]);
        return fma((double)L, 0x1p-8, (double)h[e]);
    }
};

// exponent field of a double's high word, in place (bits 20..30)
__device__ __forceinline__ int exp_bits(double v) { return __double2hiint(v) & 0x7ff00000; }

// 2^e, e clamped to the normal range
__device__ __forceinline__ double pow2(int e) {
    e = max(-1022, min(1023, e));
    return __hiloint2double((e + 1023) << 20, 0);
}

// v * 2^e: the exponent field moved by integer arithmetic where v and the
// result are normal, else by two exact powers of two
__device__ __forceinline__ double scale_by(double v, int e) {
    const int hi = __double2hiint(v), ex = (hi >> 20) & 0x7ff;
    if (ex > 0 && ex < 0x7ff && ex + e > 0 && ex + e < 0x7ff) return __hiloint2double(hi + e * (1 << 20), __double2loint(v));
    const int h = e / 2;
    return v * pow2(h) * pow2(e - h);
}

// The right shift that cuts an entry's mantissa (left-aligned as below) to the
// scale of exponent field E, plus 2048 for a negative entry: modulo 2048 it is
// at most 31 for entries down to 2^-29 of the scale, and its bits 5..10 tell
// smaller entries and entries above the scale by more than kOver bits.
// It is the high word of (E + kOver) 2^32 + 2^32 - 1 - hi 2^12, one multiply-add.
__device__ __forceinline__ unsigned shift_word(int E, double v) {
    unsigned s;
    asm("{.reg .b64 t, c; .reg .b32 l; mov.b64 c, {%1, %2}; mad.wide.s32 t, %3, -4096, c; mov.b64 {l, %0}, t;}"
        : "=r"(s)
        : "r"(0xffffffffu), "r"(E + kOver), "r"(__double2hiint(v)));
    return s;
}

// the mantissa times 2^5 (its leading bit at 57 = 55 + kOver)
__device__ __forceinline__ void aligned_mantissa(double v, unsigned& yl, unsigned& yh) {
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    // products, not shifts: the integer ALU is the busiest pipe, the multiplier idles
    unsigned c;
    asm("{.reg .b64 t; mul.wide.u32 t, %2, 32; mov.b64 {%0, %1}, t;}" : "=r"(yl), "=r"(c) : "r"(lo));
    yh = ((hi * 32u + c) & 0x01ffffffu) | 0x02000000u;
}

// The magnitude of v relative to the exponent field E: floor(|v| 2^(55 - (E
// - 1023))), below 2^56 if v's exponent field is at most E, in .x, .y, and the
// next eight bits in the top of .z; s = shift_word with bits 5..10 clear.
__device__ __forceinline__ uint3 magnitude(double v, unsigned s) {
    unsigned yl, yh;
    aligned_mantissa(v, yl, yh);
    return make_uint3(__funnelshift_r(yl, yh, s), __funnelshift_r(yh, 0u, s), __funnelshift_r(0u, yl, s));
}

// the same for any s with v at most kOver bits above the scale
__device__ __forceinline__ uint3 magnitude_any(double v, unsigned s) {
    unsigned yl, yh;
    aligned_mantissa(v, yl, yh);
    s &= 0x7ffu;
    if (s >= 96) return make_uint3(0u, 0u, 0u);
    if (s >= 64) return make_uint3(0u, 0u, yh >> (s - 64));
    if (s >= 32) return make_uint3(yh >> (s - 32), 0u, __funnelshift_r(yl, yh, s - 32));
    return make_uint3(__funnelshift_r(yl, yh, s), yh >> s, __funnelshift_r(0u, yl, s));
}

__device__ __forceinline__ unsigned fma_f16x2(unsigned a, unsigned b, unsigned c) {
    unsigned r;
    asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
    return r;
}
// Two magnitudes and the high words that carry their signs: digit i
// (0 = most significant) of both as a pair of signed FP16 numbers.  The integer
// ALU is the busiest pipe, and per pair of digits this takes one and a half byte
// permutations (one interleaves two entries' bytes, one each puts two of them
// below the exponent of 1024) and one FMA.
struct Pair {
    unsigned w0, w12, w34, w56;  // interleaved: 1024 + digit 0; digits 2, 1; 4, 3; 6, 5
    unsigned last;               // digit 7
    unsigned sg, off;            // +-1 and -+1024 as FP16 pairs
    template <bool ANY>
    __device__ __forceinline__ void set(double a, double b, unsigned sa, unsigned sb) {
        const uint3 x = ANY ? magnitude_any(a, sa) : magnitude(a, sa);
        const uint3 y = ANY ? magnitude_any(b, sb) : magnitude(b, sb);
        const unsigned s = __byte_perm((unsigned)__double2hiint(a), (unsigned)__double2hiint(b), 0x7430) & 0x80008000u;
        sg = s | 0x3c003c00u;
        off = s ^ 0xe400e400u;
        w0 = __byte_perm(x.y, y.y, 0x7632) | 0x64006400u;  // the bits from 48 on: up to ten
        w12 = __byte_perm(x.y, y.y, 0x5140);
        w34 = __byte_perm(x.x, y.x, 0x7362);
        w56 = __byte_perm(x.x, y.x, 0x5140);
        last = fma_f16x2((__byte_perm(x.z, y.z, 0x7733) & 0x00ff00ffu) | 0x64006400u, sg, off);
    }
    template <int I>
    __device__ __forceinline__ unsigned digit() const {
        if constexpr (I == 7) return last;
        if constexpr (I == 0) return fma_f16x2(w0, sg, off);
        const unsigned w = I < 3 ? w12 : I < 5 ? w34 : w56;
        return fma_f16x2(__byte_perm(w, 0x64646464u, I % 2 ? 0x4342 : 0x4140), sg, off);
    }
    __device__ __forceinline__ unsigned lead() const {  // digit 0 without its sign
        unsigned r;
        asm("add.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(w0), "r"(0xe400e400u));
        return r;
    }
};

template <int I>
__device__ __forceinline__ void mma_digit(Acc& acc, const Pair (&p)[4], const uint2 (&b)[kDig]) {
    const unsigned a[4] = {p[0].digit<I>(), p[1].digit<I>(), p[2].digit<I>(), p[3].digit<I>()};
#pragma unroll
    for (int j = 0; j < kDig && I + j < kOrd; ++j) mma_16816(acc.f[I + j], a, b[j].x, b[j].y);
}

// 16 terms: pairs p (fragment registers 0..3 of A), B's digits at frag[j * 32 + lane]
__device__ __forceinline__ void mma_step(Acc& acc, const Pair (&p)[4], const uint2* __restrict__ frag, int lane) {
    uint2 b[kDig];
#pragma unroll
    for (int j = 0; j < kDig; ++j) b[j] = frag[j * 32 + lane];
    mma_digit<7>(acc, p, b);
    const unsigned a[4] = {p[0].lead(), p[1].lead(), p[2].lead(), p[3].lead()};
    mma_16816(acc.c, a, b[0].x & 0x7fff7fffu, b[0].y & 0x7fff7fffu);
    mma_digit<0>(acc, p, b);
    mma_digit<1>(acc, p, b);
    mma_digit<2>(acc, p, b);
    mma_digit<3>(acc, p, b);
    mma_digit<4>(acc, p, b);
    mma_digit<5>(acc, p, b);
    mma_digit<6>(acc, p, b);
}

// r = round(|v| 2^(63 - (E - 1023))) with v's sign in balanced digits -128 .. 127
// (the first -256 .. 256, the last -128 .. 128); E at least v's exponent field.  The
// first seven come in unsigned fields: plus 128 in each of the low six bytes of q
// and 384 in the bits above.
constexpr unsigned long long kBalance = 0x0180808080808080ull;
struct Balanced {
    unsigned long long q;
    int last;
};
__device__ __forceinline__ Balanced balanced(double v, int E) {
    const unsigned hi = (unsigned)__double2hiint(v);
    const int ex = (int)(hi >> 20) & 0x7ff;
    if (ex == 0) return {kBalance, 0};  // zero (or denormal)
    // the mantissa with its leading bit at 63, then rounded to the place
    const unsigned lo = (unsigned)__double2loint(v);
    unsigned long long r =
        ((unsigned long long)__funnelshift_l(lo, (hi & 0xfffffu) | 0x100000u, 11) << 32) | (lo << 11);
    const int d = E - ex;
    if (d > 0) r = ((r >> min(d - 1, 63)) + 1) >> 1;
    if (d > 64) r = 0;
    const unsigned long long h = (r + 128) >> 8;  // (no carry out: eleven bits below the mantissa are zero)
    const int last = (int)(signed char)(r & 255u);
    const bool neg = (hi >> 31) != 0;
    return {neg ? kBalance - h : kBalance + h, neg ? -last : last};
}

// B's digits of one lane: terms x[0], x[1] and x[2], x[3] of its column,
// exponent field E of the column's scale
__device__ __forceinline__ void store_frag(uint2* __restrict__ frag, int lane, const double (&x)[4], int E) {
    Balanced q[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) q[i] = balanced(x[i], E);
#pragma unroll
    for (int j = 0; j < kDig; ++j) {
        const int sh = 8 * (kDig - 2 - j);
        const unsigned mask = j == 0 ? 0x3ffu : 0xffu;
        unsigned w[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const Balanced &p0 = q[2 * h], &p1 = q[2 * h + 1];
            const unsigned lo = j < 7 ? (unsigned)(p0.q >> max(sh, 0)) & mask : (unsigned)(p0.last + 128);
            const unsigned hi = j < 7 ? (unsigned)(p1.q >> max(sh, 0)) & mask : (unsigned)(p1.last + 128);
            const unsigned b = 0x64006400u | lo | (hi << 16);  // 1024 + 128 (or 384) + digit
            asm("add.rn.f16x2 %0, %1, %2;" : "=r"(w[h]) : "r"(b), "r"(j == 0 ? 0xe580e580u : 0xe480e480u));
        }
        frag[j * 32 + lane] = make_uint2(w[0], w[1]);
    }
}

// the field by which a column's entry counts towards its scale: its exponent, 1
// for a denormal number (0 stands for a column of zeros)
__device__ __forceinline__ int scale_field(double v) {
    const int e = exp_bits(v);
    return e == 0 && v != 0.0 ? 1 << 20 : e;
}

// The A operand's scales: a lane's registers 0 and 2 belong to line g (a basis
// column in the Gram, a row in the update), 1 and 3 to line g + 8.  E0, E1:
// the exponent fields of the two scales, shared by the four lanes of a line.
// x: the lane's eight entries, pairs (0,1) (2,3) (4,5) (6,7) of registers 0..3.
struct LineScale {
    int E0 = 0, E1 = 0;
    unsigned nz0 = 0, nz1 = 0;  // not zero: the lane has seen entries that are not zero
    // shift words of the entries; for the whole warp: 0 if all are at most 31 (no
    // entry is zero, none above its scale by more than kOver bits), else 1
    __device__ __forceinline__ unsigned cut(const double (&x)[8], unsigned (&s)[8]) {
        unsigned bits = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            s[k] = shift_word((k & 2) ? E1 : E0, x[k]);
            bits |= s[k] & 0x7e0u;
        }
        if (__any_sync(0xffffffffu, bits)) return 1;
        nz0 = nz1 = 1u;
        return 0;
    }
    // whether an entry of the warp exceeds its scale by more than kOver bits
    __device__ __forceinline__ bool over(const double (&x)[8]) const {
        bool far = false;
#pragma unroll
        for (int k = 0; k < 8; ++k)
            far = far || (int)(((unsigned)__double2hiint(x[k]) >> 20) & 0x7ffu) > ((k & 2) ? E1 : E0) + kOver;
        return __any_sync(0xffffffffu, far);
    }
    __device__ __forceinline__ void seen(const double (&x)[8]) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const unsigned any = ((unsigned)__double2hiint(x[k]) << 1) | (unsigned)__double2loint(x[k]);
            if (k & 2) nz1 |= any;
            else nz0 |= any;
        }
    }
    __device__ __forceinline__ void raise(const double (&x)[8]) {
        int m0 = max(max(exp_bits(x[0]), exp_bits(x[1])), max(exp_bits(x[4]), exp_bits(x[5])));
        int m1 = max(max(exp_bits(x[2]), exp_bits(x[3])), max(exp_bits(x[6]), exp_bits(x[7])));
#pragma unroll
        for (int o = 1; o <= 2; o <<= 1) {
            m0 = max(m0, __shfl_xor_sync(0xffffffffu, m0, o));
            m1 = max(m1, __shfl_xor_sync(0xffffffffu, m1, o));
        }
        E0 = limit(max(m0 >> 20, E0));
        E1 = limit(max(m1 >> 20, E1));
    }
    // a zero's shift word is E + kOver modulo 2048: E stays below 2048 - kOver
    // (finite entries above are within kOver bits), or is 0x7ff, whose sums are NaN
    static __device__ __forceinline__ int limit(int E) { return E >= 0x7ff ? 0x7ff : max(kEmin, min(E, 0x7fd)); }
};

// 2^-d, d >= 0 (0 from d = 127 on)
__device__ __forceinline__ float down2(int d) { return d < 127 ? __int_as_float((127 - d) << 23) : 0.0f; }

// One step of 16 terms; flush() moves the accumulators to the sums at the old
// scales (nothing before the first step).  settle: 64 terms since the last move to
// integers, which is done here, between the cutting and the products: right after
// the products it waits for the tensor cores (n = 6e5, b = 8, m = 720: update 1251 us,
// here 1213).
template <typename Flush>
__device__ __forceinline__ void step(Acc& acc, LineScale& sc, const double (&x)[8], const uint2* __restrict__ frag,
                                     int lane, bool settle, Flush&& flush) {
    unsigned s[8];
    Pair p[4];
    const bool first = sc.E0 == 0;
    unsigned how = first ? 1u : sc.cut(x, s);
    if (how && (first || sc.over(x))) {
        if (!first) flush();
        const int e0 = sc.E0, e1 = sc.E1;
        sc.raise(x);
        const float d0 = down2(sc.E0 - e0), d1 = down2(sc.E1 - e1);
        acc.c[0] *= d0;
        acc.c[1] *= d0;
        acc.c[2] *= d1;
        acc.c[3] *= d1;
        how = sc.cut(x, s);  // (on ordinary data the first step goes on like the others)
    }
    if (how == 0) {
#pragma unroll
        for (int r = 0; r < 4; ++r) p[r].template set<false>(x[2 * r], x[2 * r + 1], s[2 * r], s[2 * r + 1]);
    } else {
        sc.seen(x);
#pragma unroll
        for (int r = 0; r < 4; ++r) p[r].template set<true>(x[2 * r], x[2 * r + 1], s[2 * r], s[2 * r + 1]);
    }
    if (settle) acc.to_int();
    mma_step(acc, p, frag, lane);
}

// the fields of the lane's lines as the sums 0, 1 and 2, 3 see them, 0 for a line of zeros
__device__ __forceinline__ void line_fields(const LineScale& sc, int (&E)[2]) {
    unsigned n0 = sc.nz0, n1 = sc.nz1;
#pragma unroll
    for (int o = 1; o <= 2; o <<= 1) {
        n0 |= __shfl_xor_sync(0xffffffffu, n0, o);
        n1 |= __shfl_xor_sync(0xffffffffu, n1, o);
    }
    E[0] = n0 ? sc.E0 : 0;
    E[1] = n1 ? sc.E1 : 0;
}

// Which of the lane's four sums (bit e) the digits do not certify: a line and a
// column that are not zero (fields not 0) with too small a Sigma, or one that is
// not finite.
__device__ __forceinline__ unsigned uncertified(const float (&c)[4], const int (&E)[2], int field0, int field1) {
    unsigned bad = 0;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int line = E[e >> 1], field = (e & 1) ? field1 : field0;
        if ((line != 0 && field != 0 && !(c[e] >= kCertified)) || line >= 0x7ff || field >= 0x7ff) bad |= 1u << e;
    }
    return bad;
}

// The sums (bits of bad: sum e of this lane is that of line g + 8 (e / 2) and column 2t
// + e % 2) formed again in FP64: term(line, column, k) gives a's and b's entry of
// term k < terms.  A few sums are shared by the warp's lanes one after the other
// (about 20 FP64 instructions each for 450 terms); of many, each lane forms its own.
template <typename Term, typename Put>
__device__ __forceinline__ void again(unsigned bad, int terms, Term&& term, Put&& put) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    if (__reduce_add_sync(0xffffffffu, __popc(bad)) > 48) {
        double sum[4] = {0.0, 0.0, 0.0, 0.0};
        if (bad) {
            for (int k = 0; k < terms; ++k) {
                double a[2], b[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) term(g + 8 * h, 2 * t + h, k, a[h], b[h]);
#pragma unroll
                for (int e = 0; e < 4; ++e) sum[e] = fma(a[e >> 1], b[e & 1], sum[e]);
            }
        }
#pragma unroll
        for (int e = 0; e < 4; ++e)
            if (bad >> e & 1) put(e, sum[e]);
        return;
    }
#pragma unroll
    for (int e = 0; e < 4; ++e)
        for (unsigned left = __ballot_sync(0xffffffffu, bad >> e & 1); left; left &= left - 1) {
            const int who = __ffs(left) - 1;
            double sum = 0.0;
            for (int k0 = lane; k0 < terms; k0 += 128) {  // four terms' loads at once
                double a[4], b[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    a[u] = b[u] = 0.0;
                    if (k0 + 32 * u < terms) term((who >> 2) + 8 * (e >> 1), 2 * (who & 3) + (e & 1), k0 + 32 * u, a[u], b[u]);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) sum = fma(a[u], b[u], sum);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
            if (lane == who) put(e, sum);
        }
}

__device__ __forceinline__ double not_a_number() { return __longlong_as_double(0x7ff8000000000000ll); }

// v: the sum over orders in units of order 4 (2^64); the scales of A and B are
// 2^(EA - 1078) and 2^(EB - 1078).  An entry that is not finite has the field
// 0x7ff: its line's (column's) sums are NaN.
__device__ __forceinline__ double unscale(double v, int ea, int eb) {
    if (ea >= 0x7ff || eb >= 0x7ff) return not_a_number();
    return scale_by(v, 64 + ea + eb - 2156);
}

// The sums of a Gram item (basis columns j0 .. j0 + 15, rows from r on, columns
// c0 .. c0 + 7 of W) and of an update (16 rows from r on, below row_end) that the
// digits do not certify: results at res[32 e] of the lane.  Lines and columns past
// the operands' are zeros.  Kept out of line: the hot kernels' code stays short.
template <int B>
__device__ __noinline__ void again_gram(unsigned bad, int terms, int64_t n, int m, int j0, int64_t r, int c0,
                                        const double* __restrict__ Q, const double* __restrict__ W, double* res) {
    again(bad, terms,
          [&](int line, int c, int k, double& a, double& b) {
              const int j = j0 + line;
              a = j < m ? Q[((int64_t)(j / B) * n + r + k) * B + j % B] : 0.0;
              b = c0 + c < B ? W[(r + k) * B + c0 + c] : 0.0;
          },
          [&](int e, double v) { res[32 * e] = v; });
}
template <int B>
__device__ __noinline__ void again_update(unsigned bad, int m, int64_t n, int kc, int64_t r, int64_t row_end, int c0,
                                          const double* Q, const double* __restrict__ C, double* res) {
    again(bad, m,
          [&](int line, int c, int k, double& a, double& b) {
              a = r + line < row_end ? Q[((int64_t)(k / B) * n + r + line) * B + k % B] : 0.0;
              b = c0 + c < kc ? C[(int64_t)k * kc + c0 + c] : 0.0;
          },
          [&](int e, double v) { res[32 * e] = v; });
}

// -------------------------------------------------------------------- C = Q^T W
// Persistent CTAs take chunks of rc rows from a ticket counter: columns c0 ..
// c0 + 7 of W (n x B) against all m basis columns.  W's digits of a chunk are
// staged as B fragments; a warp's items are (tile of 16 basis columns, one of
// `parts` shares of the chunk's steps).  A warp copies its tile's next steps
// (16 rows, 2 KB) into its ring with cp.async, so that no register holds data
// in flight; terms 2t, 2t+1, 2t+8, 2t+9 of a step are its rows t, t+4, t+8, t+12,
// which with the swizzle below makes the fragment reads conflict-free.  An
// item's sums are added to its CTA's slot (m x B); the slots are summed
// afterwards in a fixed order (adding every chunk's sums straight to C cost two
// to three times the FP64 kernels' rounding error).
template <int B>
__device__ __forceinline__ int swizzle(int row, int q) {  // 16-byte chunk q of a row of B entries
    return B == 16 ? q ^ (2 * (row & 3)) : B == 8 ? q ^ (row & 2) : q;
}

// Shares of a chunk's steps per tile: with fewer tiles than warps the idle
// warps take shares (a warp then has one item at most).
__host__ __device__ inline int gram_parts(int ntiles) {
    int p = 1;
    while (ntiles * p * 2 <= kWarps) p *= 2;
    return p;
}

// Basis tiles tile0 .. tile0 + ntiles - 1 (16 columns each) of rows [r0, r0 +
// rows) (at most kMaxRows) and columns c0 .. c0 + 7 of W: added to slot (m x B).
// All threads, after a barrier that follows the last use of smem and the zeroing
// of slot and ew.
template <int B>
__device__ __forceinline__ void gram_chunk(int64_t n, int m, int tile0, int ntiles, int parts, int64_t r0, int rows,
                                           int c0,
                                           const double* __restrict__ Q, const double* __restrict__ W,
                                           double* __restrict__ slot, unsigned char* smem, int* ew,
                                           double (*sums)[128]) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    unsigned char* ring = smem + warp * kRing * kStepBytes;
    uint2* frag = reinterpret_cast<uint2*>(smem + kWarps * kRing * kStepBytes);
    const int g = lane >> 2, t = lane & 3;
    const bool col = c0 + g < B;
    const int items = ntiles * parts;
    // a step of a tile in the ring: block-major, then rows of B entries
    constexpr int CPR = B / 2;                       // 16-byte chunks per row
    constexpr int CPB = 16 * CPR;                    // chunks per block (B = 2, 4, 8, 16: 16 .. 128)
    const int ob = (g / B) * 16 * B * 8;             // line g's block, and line g + 8's
    const int ob8 = ((g + 8) / B) * 16 * B * 8;
    const int og = g % B, og8 = (g + 8) % B;
    const int steps = (rows + 15) / 16;
    // the columns' scales, then the digits: a warp per step, a lane's four rows of column c0 + g
    constexpr int SW = (kMaxRows / 16 + kWarps - 1) / kWarps;
    {
        double xw[SW][4];
        int mx = 0;
#pragma unroll
        for (int k = 0; k < SW; ++k)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int r = 16 * (warp + k * kWarps) + t + 4 * i;
                xw[k][i] = (col && r < rows) ? __ldg(W + (r0 + r) * B + c0 + g) : 0.0;
                mx = max(mx, scale_field(xw[k][i]));
            }
#pragma unroll
        for (int o = 1; o <= 2; o <<= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (t == 0 && mx) atomicMax(&ew[g], mx >> 20);
        __syncthreads();
        const int eg = max(ew[g], kEmin);
#pragma unroll
        for (int k = 0; k < SW; ++k)
            if (warp + k * kWarps < steps) store_frag(frag + (warp + k * kWarps) * kDig * 32, lane, xw[k], eg);
    }
    __syncthreads();
    const int per = (steps + parts - 1) / parts;
    for (int w = warp; w < items; w += kWarps) {
        const int tile = tile0 + w / parts, part = w % parts;
        const int s0 = part * per, s1 = min(steps, s0 + per);
        if (s0 >= s1) continue;
        const int j0 = 16 * tile / B, nblk = (m - 16 * tile) / B;  // first block and blocks left
        const bool whole = nblk * B >= 16;
        const double* p = Q + ((int64_t)j0 * n + r0) * B;
        auto issue = [&](int s) {
            if (s < s1) {
                unsigned char* buf = ring + (s % kRing) * kStepBytes;
                const bool full = whole && 16 * s + 16 <= rows;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int e = lane + 32 * i;
                    const int j = e / CPB, r = (e % CPB) / CPR, q = e % CPR;
                    void* dst = buf + (j * CPB + r * CPR + swizzle<B>(r, q)) * 16;
                    const double* src = p + (int64_t)j * n * B + (16 * s + r) * B + 2 * q;
                    if (full) cp_async16(dst, src);
                    else cp_async16(dst, (j < nblk && 16 * s + r < rows) ? src : Q, j < nblk && 16 * s + r < rows ? 16 : 0);
                }
            }
            cp_async_commit();
        };
#pragma unroll
        for (int k = 0; k < kRing - 1; ++k) issue(s0 + k);
        Acc acc;
        LineScale sc;
        double* mine = sums[warp] + lane;
#pragma unroll
        for (int e = 0; e < 4; ++e) mine[32 * e] = 0.0;
        auto flush = [&]() {
            acc.to_int();
#pragma unroll
            for (int e = 0; e < 4; ++e)
                mine[32 * e] += unscale(acc.value(e), (e & 2) ? sc.E1 : sc.E0, max(ew[2 * t + (e & 1)], kEmin));
            acc.clear();
        };
        for (int s = s0; s < s1; ++s) {
            cp_async_wait<kRing - 2>();
            __syncwarp();
            issue(s + kRing - 1);  // into the buffer of step s - 1
            const unsigned char* buf = ring + (s % kRing) * kStepBytes;
            double x[8];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int r = t + 4 * i;
                const int k = (i >> 1) * 4 + (i & 1);  // register 0 / 2 of line g, 1 / 3 of line g + 8
                x[k] = *reinterpret_cast<const double*>(buf + ob + r * B * 8 + swizzle<B>(r, og >> 1) * 16 + (og & 1) * 8);
                x[k + 2] = *reinterpret_cast<const double*>(buf + ob8 + r * B * 8 + swizzle<B>(r, og8 >> 1) * 16 + (og8 & 1) * 8);
            }
            step(acc, sc, x, frag + s * kDig * 32, lane, s != s0 && ((s - s0) & 3) == 0, flush);
        }
        cp_async_wait<0>();
        __syncwarp();
        flush();
        int E[2];
        line_fields(sc, E);
        const unsigned bad = uncertified(acc.c, E, ew[2 * t], ew[2 * t + 1]);
        if (__any_sync(0xffffffffu, bad)) {
            again_gram<B>(bad, min(16 * s1, rows) - 16 * s0, n, m, 16 * tile, r0 + 16 * s0, c0, Q, W, mine);
        }
        if (parts == 1) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int a = 16 * tile + g + ((e & 2) ? 8 : 0), c = c0 + 2 * t + (e & 1);
                // this tile's only writer; an add that returns nothing is not waited for
                if (a < m && c < B) atomicAdd(slot + (int64_t)a * B + c, mine[32 * e]);
            }
        }
    }
    if (parts > 1) {  // the shares in order
        __syncthreads();
        for (int e = tid; e < items / parts * 128; e += kT) {
            const int tile = e / 128, q = e % 128, l = q & 31;
            double v = 0.0;
            for (int p = 0; p < parts && p * ((steps + parts - 1) / parts) < steps; ++p) v += sums[tile * parts + p][q];
            const int a = 16 * (tile0 + tile) + (l >> 2) + ((q & 64) ? 8 : 0), c = c0 + 2 * (l & 3) + ((q & 32) ? 1 : 0);
            if (a < m && c < B) slot[(int64_t)a * B + c] += v;
        }
    }
}

template <int B>
__global__ void __launch_bounds__(kT, 2) gram_tc64_kernel(int64_t n, int m, int rc, int nchunks, int per_group,
                                                          int ngroups, int parts,
                                                          const double* __restrict__ Q, const double* __restrict__ W,
                                                          double* __restrict__ partial, int* __restrict__ tickets) {
    extern __shared__ __align__(16) unsigned char tc_smem[];
    __shared__ int ew[8];
    __shared__ double sums[kWarps][128];  // an item's sums
    __shared__ int s_chunk;
    const int tid = threadIdx.x, c0 = blockIdx.y * 8;
    double* slot = partial + (int64_t)blockIdx.x * m * B;
    for (int e = tid; e < m * B; e += kT)
        if (e % B >= c0 && e % B < c0 + 8) slot[e] = 0.0;
    for (;;) {
        __syncthreads();
        if (tid == 0 && tickets) s_chunk = atomicAdd(tickets + blockIdx.y, 1);
        if (tid < 8) ew[tid] = 0;
        __syncthreads();
        const int chunk = tickets ? s_chunk : blockIdx.x;  // no tickets: one chunk per CTA
        if (chunk >= nchunks) break;
        // chunk = a range of rc rows and a group of per_group tiles
        const int range = ngroups > 1 ? chunk / ngroups : chunk;
        const int t0 = (chunk - range * ngroups) * per_group;
        const int64_t r0 = (int64_t)range * rc;
        gram_chunk<B>(n, m, t0, min(per_group, (m + 15) / 16 - t0), parts, r0, (int)min((int64_t)rc, n - r0), c0, Q, W,
                      slot, tc_smem, ew, sums);
        if (!tickets) break;
    }
}

// Batch of problems stacked row-wise: CTA x takes chunk x, rows [chunks[3x+1],
// chunks[3x+2]) of segment chunks[3x] (at most kMaxRows, never crossing a segment),
// into its own slot at partial[x * m * B]; m is read from device memory, chunks
// of inactive segments do nothing.
template <int B>
__global__ void __launch_bounds__(kT, 2) gram_tc64_seg_kernel(int64_t n, const int* __restrict__ d_m,
                                                              const int64_t* __restrict__ chunks,
                                                              const int* __restrict__ seg_active,
                                                              const double* __restrict__ Q,
                                                              const double* __restrict__ W,
                                                              double* __restrict__ partial) {
    extern __shared__ __align__(16) unsigned char tc_smem[];
    __shared__ int ew[8];
    __shared__ double sums[kWarps][128];
    const int64_t seg = chunks[3 * blockIdx.x];
    if (seg_active && !seg_active[seg]) return;
    const int m = *d_m;
    const int64_t r0 = chunks[3 * blockIdx.x + 1];
    const int rows = (int)(chunks[3 * blockIdx.x + 2] - r0);
    double* slot = partial + (int64_t)blockIdx.x * m * B;
    for (int e = threadIdx.x; e < m * B; e += kT) slot[e] = 0.0;
    if (threadIdx.x < 8) ew[threadIdx.x] = 0;
    __syncthreads();
    gram_chunk<B>(n, m, 0, (m + 15) / 16, gram_parts((m + 15) / 16), r0, rows, 0, Q, W, slot, tc_smem, ew, sums);
}

// -------------------------------------------------------------------- W (-)= Q C
// W[r][c0 .. c0 + 7] (SUB ? -= : =) sum_a Q[r][a] C[a][c], row stride kc of C
// and W.  A warp takes 16 rows; the digits of up to kMaxCols rows of C are
// staged as B fragments (in one go, kept over the CTA's row groups, when they
// are all of C).
// One group of rows from row0 on (16 per row tile, `tiles` of them by ks warps
// each, below row_end); staged: C's digits are in smem from an earlier group.  All threads.
template <int B, bool SUB>
__device__ __forceinline__ void update_group(int64_t n, int m, int kc, int ks, int tiles, int c0, int64_t row0,
                                             int64_t row_end,
                                             bool& staged, const double* Q, const double* __restrict__ C, double* W,
                                             unsigned char* smem, int* ew) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    double2* ring = reinterpret_cast<double2*>(smem + warp * kRing * kStepBytes) + lane;
    uint2* frag = reinterpret_cast<uint2*>(smem + kWarps * kRing * kStepBytes);
    const int g = lane >> 2, t = lane & 3;
    const bool col = c0 + g < kc;
    const int sub = warp % ks;  // ks warps share a tile of 16 rows, each a share of the steps
    // (a warp without a tile works on rows past the end)
    const int64_t rt = warp / ks < tiles ? row0 + (warp / ks) * 16 : row_end, ra = rt + g, rb = ra + 8;
    double out[4] = {0.0, 0.0, 0.0, 0.0};
    Acc acc;
    LineScale sc;
    for (int k0 = 0; k0 < m; k0 += kMaxCols) {
        const int cols = min(kMaxCols, m - k0), steps = (cols + 15) / 16;
        if (!staged) {
            // the columns' scales grow from one staged piece of C to the next, as the lines' do
            __syncthreads();
            const int f0 = max(ew[2 * t], kEmin), f1 = max(ew[2 * t + 1], kEmin);
            __syncthreads();
            if (k0 == 0 && tid < 8) ew[tid] = 0;
            __syncthreads();
            int mx = 0;
            for (int s = warp; s < steps; s += kWarps)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int a = 16 * s + 2 * t + (i & 1) + 8 * (i >> 1);
                    if (col && a < cols) mx = max(mx, scale_field(C[(int64_t)(k0 + a) * kc + c0 + g]));
                }
#pragma unroll
            for (int o = 1; o <= 2; o <<= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            if (t == 0 && mx) atomicMax(&ew[g], mx >> 20);
            __syncthreads();
            const int eg = max(ew[g], kEmin);
            for (int s = warp; s < steps; s += kWarps) {
                double x[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int a = 16 * s + 2 * t + (i & 1) + 8 * (i >> 1);
                    x[i] = (col && a < cols) ? C[(int64_t)(k0 + a) * kc + c0 + g] : 0.0;
                }
                store_frag(frag + s * kDig * 32, lane, x, eg);
            }
            __syncthreads();
            const float d0 = down2(max(ew[2 * t] - f0, 0)), d1 = down2(max(ew[2 * t + 1] - f1, 0));
            acc.c[0] *= d0;
            acc.c[2] *= d0;
            acc.c[1] *= d1;
            acc.c[3] *= d1;
            staged = m <= kMaxCols;
        }
        // registers 0, 1: columns 2t, 2t+1 of rows g, g+8; 2, 3: columns 2t+8,
        // 2t+9.  A lane copies its own 16-byte pairs into its ring and reads them back.
        const int per = (steps + ks - 1) / ks, s0 = sub * per, s1 = min(steps, s0 + per);
        const bool rows_in = row0 + (warp / ks) * 16 + 16 <= row_end && warp / ks < tiles;
        auto issue = [&](int s) {
            if (s < s1) {
                const bool full = rows_in && k0 + 16 * s + 16 <= m;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int a = k0 + 16 * s + 8 * (i >> 1) + 2 * t;
                    const int64_t r = (i & 1) ? rb : ra;
                    const double* src = Q + ((int64_t)(a / B) * n + r) * B + a % B;
                    double2* dst = ring + (s % kRing) * 128 + i * 32;
                    if (full) cp_async16(dst, src);
                    else cp_async16(dst, (a < m && r < row_end) ? src : Q, a < m && r < row_end ? 16 : 0);
                }
            }
            cp_async_commit();
        };
#pragma unroll
        for (int k = 0; k < kRing - 1; ++k) issue(s0 + k);
        auto flush = [&]() {
            acc.to_int();
#pragma unroll
            for (int e = 0; e < 4; ++e)
                out[e] += unscale(acc.value(e), (e & 2) ? sc.E1 : sc.E0, max(ew[2 * t + (e & 1)], kEmin));
            acc.clear();
        };
        for (int s = s0; s < s1; ++s) {
            cp_async_wait<kRing - 2>();
            double x[8];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const double2 v = ring[(s % kRing) * 128 + i * 32];
                x[2 * i] = v.x;
                x[2 * i + 1] = v.y;
            }
            issue(s + kRing - 1);  // into the buffer of step s - 1
            step(acc, sc, x, frag + s * kDig * 32, lane, s != s0 && ((s - s0) & 3) == 0, flush);
        }
        cp_async_wait<0>();
        if (s0 < s1) flush();
    }
    int E[2];
    line_fields(sc, E);
    if (ks > 1) {  // the shares' sums, Sigmas and fields through the rings, which nobody uses any more
        struct Share {
            double out[4];
            float c[4];
            int E[2];
        };
        Share* shares = reinterpret_cast<Share*>(smem);
        __syncthreads();
        Share& own = shares[tid];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            own.out[e] = out[e];
            own.c[e] = acc.c[e];
        }
        own.E[0] = E[0];
        own.E[1] = E[1];
        __syncthreads();
        if (sub == 0) {
            for (int q = 1; q < ks; ++q) {
                const Share& o = shares[tid + 32 * q];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int top = max(E[h], o.E[h]);
                    const float a = down2(top - E[h]), b = down2(top - o.E[h]);
                    E[h] = top;
#pragma unroll
                    for (int e = 2 * h; e < 2 * h + 2; ++e) {
                        acc.c[e] = acc.c[e] * a + o.c[e] * b;
                        out[e] += o.out[e];
                    }
                }
            }
        }
        __syncthreads();
        if (sub != 0) return;
    }
    unsigned bad = uncertified(acc.c, E, ew[2 * t], ew[2 * t + 1]);
    if (__any_sync(0xffffffffu, bad)) {
        if (SUB) {  // the difference rounds by |W| as well, which counts towards Sigma
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int64_t r = (e & 2) ? rb : ra;
                const int c = 2 * t + (e & 1), line = E[e >> 1], field = max(ew[c], kEmin);
                if ((bad >> e & 1) && line < 0x7ff && field < 0x7ff && r < row_end && c0 + c < kc &&
                    acc.c[e] + scale_by(fabs(W[r * kc + c0 + c]), 2156 - 96 - line - field) >= kCertified)
                    bad &= ~(1u << e);
            }
        }
        double* res = reinterpret_cast<double*>(smem + warp * kRing * kStepBytes) + lane;  // the warp's ring, free now
#pragma unroll
        for (int e = 0; e < 4; ++e) res[32 * e] = out[e];
        again_update<B>(bad, m, n, kc, rt, row_end, c0, Q, C, res);
#pragma unroll
        for (int e = 0; e < 4; ++e) out[e] = res[32 * e];
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int64_t r = (e & 2) ? rb : ra;
        const int c = c0 + 2 * t + (e & 1);
        if (r < row_end && c < kc) {
            double* w = W + r * kc + c;
            *w = SUB ? *w - out[e] : out[e];
        }
    }
}

template <int B, bool SUB>
__global__ void __launch_bounds__(kT, 2) update_tc64_kernel(int64_t n, int m, int kc, int ks, int tiles, const double* Q,
                                                            const double* __restrict__ C, double* W) {
    extern __shared__ __align__(16) unsigned char tc_smem[];
    __shared__ int ew[8];
    const int rows = 16 * tiles;
    bool staged = false;
    for (int64_t row0 = (int64_t)blockIdx.x * rows; row0 < n; row0 += (int64_t)gridDim.x * rows)
        update_group<B, SUB>(n, m, kc, ks, tiles, blockIdx.y * 8, row0, n, staged, Q, C, W, tc_smem, ew);
}

// Segmented: CTA x updates rows [ctas[3x+1], ctas[3x+2]) of segment s = ctas[3x]
// with that segment's coefficients C + s * cstride and m = ms[s * ms_stride]
// columns; inactive segments skip.
template <int B>
__global__ void __launch_bounds__(kT, 2) update_tc64_seg_kernel(int64_t n, const int* __restrict__ ms, int ms_stride,
                                                                const int64_t* __restrict__ ctas,
                                                                const int* __restrict__ seg_active, const double* Q,
                                                                const double* __restrict__ C, int64_t cstride,
                                                                double* W) {
    extern __shared__ __align__(16) unsigned char tc_smem[];
    __shared__ int ew[8];
    const int64_t seg = ctas[3 * blockIdx.x];
    if (seg_active && !seg_active[seg]) return;
    const int m = ms[seg * ms_stride];
    const int64_t r1 = ctas[3 * blockIdx.x + 2];
    bool staged = false;
    for (int64_t row0 = ctas[3 * blockIdx.x + 1]; row0 < r1; row0 += 16 * kWarps)
        update_group<B, true>(n, m, B, 1, kWarps, 0, row0, r1, staged, Q, C + seg * cstride, W, tc_smem, ew);
}

constexpr int kFragBytes = kDig * 32 * (int)sizeof(uint2);  // a step's B fragments
constexpr int kRingBytes = kWarps * kRing * kStepBytes;

template <int B>
bbl_status launch_gram(int64_t n, int m, const double* Q, const double* W, double* C, DevBuf& partials, cudaStream_t st) {
    static OncePerDevice once;
    BBL_TRY(allow_smem(once, gram_tc64_kernel<B>, kRingBytes + kMaxRows / 16 * kFragBytes));
    constexpr int NH = (B + 7) / 8;
    // One chunk per resident CTA where that gives at least 64 rows, at most the
    // staged kMaxRows, else chunks of equal size for several rounds; with fewer
    // rows the tiles are split into groups of
    // one per warp, which take more rows each (an item's end, its FP64
    // conversions, costs as much as three steps).  n = 2e4, b = 4, m = 400: 36.7 us
    // in one group, 33.4 in four; m = 200: 21.2 and 21.0 (with 56-bit splits; now 36.4 and 22.3).
    const int64_t resident = (int64_t)2 * gram_worker_sms();
    const int ntiles = (m + 15) / 16;
    int64_t groups = (ntiles + kWarps - 1) / kWarps;
    groups = std::max<int64_t>(std::min<int64_t>(groups, kMaxRows * resident / std::max<int64_t>(n, 1)), 1);
    const int per_group = (int)ceil_div(ntiles, groups);
    groups = ceil_div(ntiles, per_group);
    const int64_t rounds = ceil_div(ceil_div(n * groups, resident), kMaxRows);
    const int64_t rc = std::max<int64_t>(ceil_div(ceil_div(n * groups, resident * rounds), 16) * 16, 64);
    const int64_t chunks = ceil_div(n, rc) * groups;
    const int64_t ctas = std::min<int64_t>(chunks, resident);
    const int64_t per = (int64_t)m * B;
    BBL_TRY(partials.grow(sizeof(double) * (size_t)(ctas * per) + 256));
    int* tickets = nullptr;
    if (chunks > ctas) {
        tickets = reinterpret_cast<int*>(partials.as<double>() + ctas * per);
        BBL_CUDA(cudaMemsetAsync(tickets, 0, sizeof(int) * NH, st));
    }
    gram_tc64_kernel<B><<<dim3((unsigned)ctas, NH), kT, kRingBytes + (size_t)(rc / 16) * kFragBytes, st>>>(
        n, m, (int)rc, (int)chunks, per_group, (int)groups, gram_parts(per_group), Q, W, partials.as<double>(), tickets);
    BBL_LAUNCH_CHECK();
    reduce_partials(per, (int)ctas, partials.as<double>(), C, st);
    BBL_LAUNCH_CHECK();
    return BBL_OK;
}

template <int B, bool SUB>
bbl_status launch_update(int64_t n, int m, int kc, const double* Q, const double* C, double* W, cudaStream_t st) {
    static OncePerDevice once;
    BBL_TRY(allow_smem(once, update_tc64_kernel<B, SUB>, kRingBytes + kMaxCols / 16 * kFragBytes));
    const int64_t rtiles = ceil_div(n, 16);
    const int cols = std::min(m, kMaxCols), steps = (cols + 15) / 16;
    const int64_t ny = (kc + 7) / 8;
    // few rows: up to eight warps share a row tile's steps, so that the SMs' 16
    // warps have work
    int ks = 1;
    while (ks < kWarps && rtiles * ks * 2 <= (int64_t)sm_count() * 2 * kWarps && steps >= ks * 4) ks <<= 1;
    int tiles = kWarps / ks;
    // between one and two CTAs per SM: fewer tiles each, so that every SM has two
    // (n = 2e4, m = 200: 5 tiles, 250 CTAs, 26.2 us; with 8 five of the 152 SMs had
    // two CTAs, 27.1 us, with 56-bit splits; now 28.5)
    const int64_t total = ceil_div(rtiles, tiles) * ny;
    if (ks == 1 && total > sm_count() && total < (int64_t)2 * sm_count()) tiles = (int)ceil_div(rtiles * ny, (int64_t)2 * sm_count());
    const int64_t groups = ceil_div(rtiles, tiles);
    const dim3 grid((unsigned)std::min<int64_t>(groups, (int64_t)sm_count() * 8), (unsigned)((kc + 7) / 8));
    update_tc64_kernel<B, SUB><<<grid, kT, kRingBytes + (size_t)steps * kFragBytes, st>>>(n, m, kc, ks, tiles, Q, C, W);
    BBL_LAUNCH_CHECK();
    return BBL_OK;
}

}  // namespace

// Measured against the FP64 FMA kernels (us, FMA / split): the split is faster from
// 16 columns on with b = 8 (n = 1e6: Gram 332 / 115, update 217 / 117; m = 80: 1592 / 329,
// 1052 / 270; n = 2000: 10.4 / 6.1, 11.5 / 6.1) and b = 16; with one block (m = 8) half of each
// tile is padding.  With b = 4 the Gram from 16 on (n = 1e6: 177 / 114; n = 3e4: 10.8 / 10.8), for
// few rows from 40 on (n = 4000, m = 24: 6.3 / 7.5, 40: 8.6 / 8.0), the update from 32 on
// (n = 1e6, m = 16: 115 / 158, 28: 184 / 177, 32: 219 / 186; n = 3e4, m = 32: 11.2 / 10.5).  With b = 2
// the Gram from 32 on (n = 4000: 23.5 / 7.7), for many rows, where the FMA kernel is full, from 48
// on (n = 1e6, m = 32: 132 / 154, 40: 246 / 254, 48: 251 / 233; n = 2e5, m = 32: 39.3 / 38.0).  With b = 1,
// and in the update b = 2, the FMA kernels have no more than two products per entry.
bool tc64_gram_supports(int64_t n, int b, int m) {
    if (b == 2) return m >= (n <= 400000 ? 32 : 48);
    if (b == 4) return m >= (n < 10000 ? 40 : 16);
    return (b == 8 || b == 16) && m >= 16;
}
bool tc64_update_supports(int b, int m) { return (b == 4 && m >= 32) || ((b == 8 || b == 16) && m >= 16); }

namespace {

template <int B>
bbl_status launch_gram_seg(int64_t n, const int* d_m, const double* Q, const double* W, const int64_t* chunks,
                           int nchunks, const int* active, double* partial, cudaStream_t st) {
    constexpr int kSmem = kRingBytes + kMaxRows / 16 * kFragBytes;
    static OncePerDevice once;
    BBL_TRY(allow_smem(once, gram_tc64_seg_kernel<B>, kSmem));
    gram_tc64_seg_kernel<B><<<(unsigned)nchunks, kT, kSmem, st>>>(n, d_m, chunks, active, Q, W, partial);
    BBL_LAUNCH_CHECK();
    return BBL_OK;
}

template <int B>
bbl_status launch_update_seg(int64_t n, const int* ms, int ms_stride, const int64_t* ctas, int nctas, const int* active,
                             const double* Q, const double* C, int64_t cstride, double* W, cudaStream_t st) {
    constexpr int kSmem = kRingBytes + kMaxCols / 16 * kFragBytes;
    static OncePerDevice once;
    BBL_TRY(allow_smem(once, update_tc64_seg_kernel<B>, kSmem));
    update_tc64_seg_kernel<B><<<(unsigned)nctas, kT, kSmem, st>>>(n, ms, ms_stride, ctas, active, Q, C, cstride, W);
    BBL_LAUNCH_CHECK();
    return BBL_OK;
}

}  // namespace

bool tc64_seg_supports(int b) { return b == 4 || b == 8; }
int tc64_seg_chunk_rows() { return kMaxRows; }

bbl_status gram_tc64_seg(int64_t n, int b, const int* d_m, const double* Q, const double* W, const int64_t* chunks,
                         int nchunks, const int* active, double* partial, cudaStream_t st) {
    if (b == 4) return launch_gram_seg<4>(n, d_m, Q, W, chunks, nchunks, active, partial, st);
    return launch_gram_seg<8>(n, d_m, Q, W, chunks, nchunks, active, partial, st);
}

bbl_status update_tc64_seg(int64_t n, int b, const int* ms, int ms_stride, const int64_t* ctas, int nctas,
                           const int* active, const double* Q, const double* C, int64_t cstride, double* W,
                           cudaStream_t st) {
    if (b == 4) return launch_update_seg<4>(n, ms, ms_stride, ctas, nctas, active, Q, C, cstride, W, st);
    return launch_update_seg<8>(n, ms, ms_stride, ctas, nctas, active, Q, C, cstride, W, st);
}

bbl_status gram_tc64(int64_t n, int b, int m, const double* Q, const double* W, double* C, DevBuf& partials,
                     cudaStream_t st) {
    switch (b) {
        case 2: return launch_gram<2>(n, m, Q, W, C, partials, st);
        case 4: return launch_gram<4>(n, m, Q, W, C, partials, st);
        case 8: return launch_gram<8>(n, m, Q, W, C, partials, st);
        default: return launch_gram<16>(n, m, Q, W, C, partials, st);
    }
}

bbl_status update_tc64(int64_t n, int b, int m, int kc, const double* Q, const double* C, double* W, bool sub,
                       cudaStream_t st) {
    switch (b) {
        case 4: return sub ? launch_update<4, true>(n, m, kc, Q, C, W, st) : launch_update<4, false>(n, m, kc, Q, C, W, st);
        case 8: return sub ? launch_update<8, true>(n, m, kc, Q, C, W, st) : launch_update<8, false>(n, m, kc, Q, C, W, st);
        default: return sub ? launch_update<16, true>(n, m, kc, Q, C, W, st) : launch_update<16, false>(n, m, kc, Q, C, W, st);
    }
}

}  // namespace bbl
