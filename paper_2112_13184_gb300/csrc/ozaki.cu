// Emulated-FP64 GEMM on the GB300 tensor cores (tcgen05 + TMEM + TMA).
//
// Each FP64 operand row (of A) or column (of B) is scaled by a power of two
// 2^e with max|x| <= 2^e and cut into s signed 8-bit digits,
//     x = 2^(e-8) * sum_t a_t 2^(-8t),   a_0 in [-256,256], a_t in [-128,127],
// computed with integer operations on the FP64 bit pattern (the FP64 pipe of
// GB300 is slow).  The scaled digits at_t = a_t 2^(-8t) are exact in BF16.
// C = A B is then the sum of BF16 slice products at_t * bt_u, accumulated
// on the tensor cores in FP32 over K-chunks of 256 and read out of TMEM
// after every chunk:
//   level 0 (t+u = 0) and level 1 (t+u = 1) are integer-valued (in units of
//   1 and 2^-8); over one chunk they stay below 2^24 units and are exact;
//   all pairs with 2 <= t+u <= s-1 carry a weight <= 2^-16 and share one
//   FP32 accumulator, restarted every chunk so that the tensor cores'
//   rounding does not grow with the magnitude accumulated over K;
//   pairs with t+u >= s are dropped (same order as the slicing error).
// Every chunk's S0 (level 0), S1 (level 1) and F (the rest) are added to one
// int64 per entry, Z = 2^28 S0 + 2^20 S1 + round(2^28 F), and C = 2^(eA+eB-44)
// Z.  Error: the slicing, 2^(2-8s) max|row| max|col| K, plus the tensor
// cores' FP32 rounding of the levels >= 2 within a chunk, measured at about
// 2^-36 max|row| max|col| K; so 5 slices reach ~1e-11 relative per unit K
// and a 6th adds nothing.  Split-BF16 accumulated in FP32 over all of K
// cannot go below ~2^-24.
#include <cooperative_groups.h>
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <mutex>

#include "internal.h"

namespace cg = cooperative_groups;

namespace ctm {
namespace oz {

constexpr int BM = 128;          // rows per CTA (one TMEM lane per row)
constexpr int BK = 32;           // K per pipeline stage (64 bytes: one SW64 row)
constexpr int CHUNK_KB = 8;      // k-blocks per exact chunk (K = 256)
constexpr int EPI_WARPS = 12;    // 3 warps per TMEM lane quarter
constexpr int THREADS = (EPI_WARPS + 2) * 32;  // + producer warp + MMA warp
constexpr int MAX_S = 6;

// A strided multi-index view: index i = (i_0, ..., i_{n-1}) in row-major
// order over dims, offset = sum_a i_a * stride[a].  Used to read operands as
// permuted views of larger tensors and to write results into permuted
// layouts, so that no FP64 permutation pass is needed.
struct View {
    int n;
    int dim[4];
    long long stride[4];
};
__host__ __device__ __forceinline__ long long view_offset(const View& v, long long i) {
    long long off = 0;
#pragma unroll
    for (int a = 3; a >= 0; --a) {
        if (a < v.n) {
            const long long q = i / v.dim[a];
            off += (i - q * v.dim[a]) * v.stride[a];
            i = q;
        }
    }
    return off;
}

// 32-bit decomposition (all view extents here are below 2^31)
__device__ __forceinline__ long long view_offset32(const View& v, unsigned i) {
    long long off = 0;
#pragma unroll
    for (int a = 3; a >= 0; --a) {
        if (a < v.n) {
            const unsigned dm = (unsigned)v.dim[a];
            const unsigned q = i / dm;
            off += (long long)(i - q * dm) * v.stride[a];
            i = q;
        }
    }
    return off;
}

// walks a view's indices in order, one add per step (carry on wrap)
struct Odometer {
    int idx[4];
    long long off;
    __device__ __forceinline__ void init(const View& v, unsigned i) {
        off = 0;
#pragma unroll
        for (int a = 3; a >= 0; --a) {
            idx[a] = 0;
            if (a < v.n) {
                const unsigned dm = (unsigned)v.dim[a];
                const unsigned q = i / dm;
                idx[a] = (int)(i - q * dm);
                off += (long long)idx[a] * v.stride[a];
                i = q;
            }
        }
    }
    __device__ __forceinline__ void step(const View& v) {
#pragma unroll
        for (int a = 3; a >= 0; --a) {
            if (a < v.n) {
                off += v.stride[a];
                if (++idx[a] < v.dim[a]) return;
                off -= (long long)v.dim[a] * v.stride[a];
                idx[a] = 0;
            }
        }
    }
};

// v * 2^k for finite v, through the exponent field when the result stays
// normal (the common case), else by ldexp
__device__ __forceinline__ double scale_pow2(double v, int k) {
    const long long b = __double_as_longlong(v);
    const int e = (int)((b >> 52) & 0x7ff);
    if (v == 0.0) return v;
    if (e > 0 && e + k > 0 && e + k < 2047) return __longlong_as_double(b + ((long long)k << 52));
    return ldexp(v, k);
}

// Z * 2^E outside the normal FP64 range (rare): kept out of line so that its
// FP64 conversion and scaling are not if-converted into every element
__device__ __noinline__ double i64_ldexp_slow(long long Z, int E) {
    return ldexp((double)Z, E);
}

// Z * 2^E as an FP64 number (round to nearest even) with integer operations
// only: GB300's FP64 pipe is too slow to spend on every output element.
__device__ __forceinline__ double i64_ldexp(long long Z, int E) {
    if (Z == 0) return 0.0;
    const unsigned long long neg = Z < 0 ? 1ull : 0ull;
    unsigned long long m = neg ? (0ull - (unsigned long long)Z) : (unsigned long long)Z;
    int sh = (64 - __clzll((long long)m)) - 53;  // bits beyond a 53-bit mantissa
    unsigned long long mant;
    if (sh > 0) {
        const unsigned long long rem = m & ((1ull << sh) - 1), half = 1ull << (sh - 1);
        mant = m >> sh;
        if (rem > half || (rem == half && (mant & 1ull))) {
            ++mant;
            if (mant >> 53) {
                mant >>= 1;
                ++sh;
            }
        }
    } else {
        mant = m << (-sh);
    }
    const int be = E + sh + 52 + 1023;  // value = mant 2^(E+sh), mant in [2^52, 2^53)
    if (be <= 0 || be >= 2047) return i64_ldexp_slow(Z, E);  // outside the normal range
    return __longlong_as_double((long long)((neg << 63) | ((unsigned long long)be << 52) | (mant & ((1ull << 52) - 1))));
}

// C = 2^(eA+eB-16) (S0 + S1/256 + F): with F kept to 2^-28 of an S0 unit (below
// 2^-44 of max|row| max|col|), Z = 2^28 S0 + 2^20 S1 + round(2^28 F) is an
// exact int64 (one K chunk: |Z| < 2^53; 64 chunks: < 2^59) and C = Z
// 2^(eA+eB-44).  S0 and S1/256 are whole-numbered FP32 accumulators; F, below
// 2^9 per chunk, is split by two magic additions of 1.5 2^23 into 6 and 22
// fractional bits: no conversion of it (an FP32 -> int64 conversion issues on
// the FP64 pipe, 64 cycles a warp; FP32 -> int32 on the 16-lane one).
// fixed_add_w takes the integer weights as kernel arguments: as literals the
// compiler turns the 32 x 32 + 64 multiply-adds of the FMA pipe into shifts and
// adds on the half-rate integer pipe, which bounds the short products'
// epilogue (262144 x 192 x 64: 171 -> 159 us).  The long products' one is short
// of registers instead and keeps the literals (8192 x 128 x 8192: 261 us, 290
// with arguments).
struct Weights {
    int w20, w22, w28, one;
};
__device__ __forceinline__ long long mad_wide(int a, int b, long long c) {
    long long d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
}
__device__ __forceinline__ long long fixed_add_w(const Weights& w, long long Z, float a0, float a1, float F) {
    const float h = fmaf(F, 64.0f, 12582912.0f);
    const float r = fmaf(F, 64.0f, 12582912.0f - h);  // F 2^6 minus its rounding, exact
    const float h2 = fmaf(r, 4194304.0f, 12582912.0f);
    Z = mad_wide(__float_as_int(h2) - 0x4B400000, w.one, Z);
    Z = mad_wide(__float_as_int(h) - 0x4B400000, w.w22, Z);
    Z = mad_wide(__float2int_rn(a1 * 256.0f), w.w20, Z);
    return mad_wide(__float2int_rn(a0), w.w28, Z);
}
__device__ __forceinline__ long long fixed_add(long long Z, float a0, float a1, float F) {
    const float h = fmaf(F, 64.0f, 12582912.0f);
    const float r = fmaf(F, 64.0f, 12582912.0f - h);
    const float h2 = fmaf(r, 4194304.0f, 12582912.0f);
    const int i1 = __float_as_int(h) - 0x4B400000, i2 = __float_as_int(h2) - 0x4B400000;
    Z += i2;
    Z += (long long)i1 * (1 << 22);
    Z += (long long)__float2int_rn(a1 * 256.0f) * (1 << 20);
    Z += (long long)__float2int_rn(a0) * (1 << 28);
    return Z;
}
// exponents of rows with an infinity or a NaN (1025) become one that leaves
// the FP64 range from any finite partner
constexpr int BAD_EXP = 100000;
__device__ __forceinline__ int safe_exp(int e) { return e > 1024 ? BAD_EXP : e; }
// Z 2^E where |Z| < 2^53 (exact: a left shift only; SHORT: known to hold) and
// the result is normal or zero; else `bad` is set and the value is
// meaningless.  No branch: a branch per entry kept the entries of a block from
// overlapping.
template <bool SHORT>
__device__ __forceinline__ double z_scaled_fast(long long Z, int E, bool& bad) {
    const long long sg = Z >> 63;
    const unsigned long long m = (unsigned long long)((Z ^ sg) - sg);
    const unsigned mh = (unsigned)(m >> 32), ml = (unsigned)m;
    const int c = mh ? __clz((int)mh) : 32 + __clz((int)ml);
    const unsigned be = (unsigned)(E + 1085 - c);  // exponent field of m 2^E minus 1: the implicit bit adds 1
    bad = bad || be >= 2046u || (!SHORT && c < 11);
    const unsigned long long mant = m << ((c - 11) & 63);  // implicit bit at 52
    const unsigned hi = (unsigned)(mant >> 32) + (m ? be << 20 : 0u) + ((unsigned)sg & 0x80000000u);
    return __hiloint2double((int)hi, (int)(unsigned)mant);
}
// larger |Z| (sums of several chunks), results outside the normal range,
// non-finite operands
__device__ __noinline__ double z_scaled_slow(long long Z, int E) {
    if (E > BAD_EXP / 2) return __longlong_as_double(0x7ff8000000000000ll);
    return i64_ldexp(Z, E);
}
__device__ __forceinline__ double z_scaled(long long Z, int E) {
    bool bad = false;
    const double v = z_scaled_fast<false>(Z, E, bad);
    return bad ? z_scaled_slow(Z, E) : v;
}

__device__ __noinline__ double f32_ldexp_slow(float f, int E) { return ldexp((double)f, E); }

// f 2^E as an FP64 number for an FP32 f (the accumulator of the FP32-
// accumulated modes), built from the bit pattern: the exponent is rebiased
// and the 23-bit significand widened, integer instructions only.
__device__ __forceinline__ double f32_scaled(float f, int E) {
    const unsigned b = __float_as_uint(f);
    const int ex = (int)((b >> 23) & 0xff);
    if (ex == 0) return 0.0;                                      // zero or FP32 denormal
    if (ex == 255) return __longlong_as_double(0x7ff8000000000000ll);  // Inf/NaN accumulator
    const int be = ex - 127 + 1023 + E;
    if (be <= 0 || be >= 2047) return f32_ldexp_slow(f, E);       // outside the normal FP64 range
    return __longlong_as_double((long long)(((unsigned long long)(b >> 31) << 63) |
                                            ((unsigned long long)be << 52) |
                                            ((unsigned long long)(b & 0x7fffffu) << 29)));
}

// ---------------------------------------------------------------------------
// slicing
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long abs_bits(double x) {
    return (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
}
__device__ __forceinline__ unsigned long long umax64(unsigned long long a, unsigned long long b) {
    return a > b ? a : b;
}
// row_exponent of the bit pattern of max|x| (integer operations only)
__device__ __forceinline__ int row_exponent_bits(unsigned long long mb) {
    if ((mb & 0x7fffffffffffffffull) == 0) return 0;
    const int E = (int)((mb >> 52) & 0x7ff);
    return E == 0 ? -1022 : E - 1022;
}
// exponent e with max|x| < 2^e (0 for an all-zero row; 1025 when the row
// holds an infinity or a NaN, which the products turn into NaN outputs)
__device__ __forceinline__ int row_exponent(double mx) {
    if (mx == 0.0) return 0;
    const int E = (int)((__double_as_longlong(mx) >> 52) & 0x7ff);
    return E == 0 ? -1022 : E - 1022;
}

// Signed base-256 digits of Y = round(x * 2^(8s - e)), |x| < 2^e, held as the
// bytes of one biased integer: with B = sum_{t=1}^{s-1} 128 * 256^(s-1-t), the
// balanced recurrence Y' = floor((Y + 128) / 256), d = Y - 256 Y' (d in
// [-128, 127]) is what long division of Z = Y + B gives, so that digit t >= 1
// is byte s-1-t of Z minus 128 and d_0 = Z >> 8(s-1) carries the sign and the
// top: one 64-bit addition instead of s dependent shift-and-subtract steps.
// The slicers are then bound by memory, not by integer issue (~30
// instructions per element instead of ~100): the warm sweep at d=3, D=8,
// chi=128 went from 763 to 545 ms with the column slicers below.
__host__ __device__ constexpr unsigned long long digit_bias(int s) {
    unsigned long long b = 0;
    for (int t = 1; t < s; ++t) b = (b << 8) | 128ull;
    return b;
}
// Z from the FP64 bit pattern b of x; base = 1075 - 8s + e.  x = mant
// 2^(ex-1075), so Y = mant >> (base - ex) rounded half away from zero, and
// |x| < 2^e makes that a right shift by at least 53 - 8 MAX_S > 0 bits.
__device__ __forceinline__ unsigned long long digit_bytes(unsigned long long b, int base, unsigned long long bias) {
    const unsigned hi = (unsigned)(b >> 32);
    const int ex0 = (int)((hi >> 20) & 0x7ff);
    const int ex = max(ex0, 1);
    const unsigned mh = (hi & 0xfffffu) | (ex0 ? 0x100000u : 0u);  // denormals have no implicit bit
    const unsigned long long mant = ((unsigned long long)mh << 32) | (unsigned)b;
    const int sh = min(base - ex, 55);  // mant < 2^53: everything from 54 on gives 0
    const unsigned long long y = ((mant >> (sh - 1)) + 1ull) >> 1;
    const unsigned long long m = (unsigned long long)((long long)b >> 63);
    return (y ^ m) - m + bias;
}

// A small int as an FP32 without a conversion instruction: 1.5 2^23 + d has
// the bit pattern 0x4B400000 + d for |d| < 2^22, so one FP32 subtraction
// recovers d exactly.
__device__ __forceinline__ float small_int_f32(int d) {
    return __int_as_float(0x4B400000 + d) - 12582912.0f;
}

// BF16 pair of digit t >= 1 of two elements (a in the low half): `w` holds
// their digit bytes u = d + 128 in bits 0-7 and 16-23.  With u = 128 h + l, l < 128:
// (128 + l) 2^(-8t) is a BF16 whose 7 mantissa bits are l, (256 - 128 h)
// 2^(-8t) one whose lowest exponent bit is !h, and their difference, exact in
// BF16, is d 2^(-8t): two logic operations and one packed subtraction for
// two digits, no conversion instruction.
__device__ __forceinline__ unsigned digit_pair(unsigned w, int t) {
    const unsigned kv = (unsigned)(134 - 8 * t) << 7, kc = (unsigned)(135 - 8 * t) << 7;
    const unsigned v = (w & 0x007f007fu) | (kv * 0x10001u);
    const unsigned c = (w & 0x00800080u) ^ (kc * 0x10001u);
    const __nv_bfloat162 d = __hsub2(*reinterpret_cast<const __nv_bfloat162*>(&v),
                                     *reinterpret_cast<const __nv_bfloat162*>(&c));
    return *reinterpret_cast<const unsigned*>(&d);
}
__device__ __forceinline__ unsigned bf2_bits(float a, float b) {
    const __nv_bfloat162 p = __floats2bfloat162_rn(a, b);  // a in the low half (lower address)
    return *reinterpret_cast<const unsigned*>(&p);
}
// Slice t of two elements with digit integers za, zb as a BF16 pair (the byte
// index depends on s, the powers of two on t).
__device__ __forceinline__ unsigned slice_of_pair(unsigned long long za, unsigned long long zb, int s, int t) {
    if (t == 0)  // |d_0| <= 256: exact in BF16
        return bf2_bits(small_int_f32((int)((long long)za >> (8 * (s - 1)))),
                        small_int_f32((int)((long long)zb >> (8 * (s - 1)))));
    const int byte = s - 1 - t;  // below 4 but for t = 1 of 6 slices
    const unsigned a = byte < 4 ? (unsigned)za : (unsigned)(za >> 32);
    const unsigned b = byte < 4 ? (unsigned)zb : (unsigned)(zb >> 32);
    // byte of a to bits 0-7, byte of b to bits 16-23
    return digit_pair(__byte_perm(a, b, (byte & 3) | ((4 + (byte & 3)) << 8)), t);
}

// Per-row maxima of operands whose rows are not contiguous in k, as bit
// patterns that have the exponent of max|x| and are zero only where it is (all
// that row_exponent_bits asks for): lane = row, a warp takes 32 rows x
// `krange` k, combined with atomicMax (non-negative doubles order like
// integers).  PLAIN: one K stride.  Bound by HBM: three integer instructions an
// element on its two words and 16 loads in flight per lane.  (8 loads and an
// odometer step for each: 147 us for the 537 MB of 8192 x 8192, about 85 now;
// a whole 8192 x 16 x 8192 product 548 -> 484.)
template <bool PLAIN>
__global__ void __launch_bounds__(128) k_rowmax_cols(const double* __restrict__ X, int R, int K, View rv, View kv,
                                                     int kranges, int krange, unsigned long long* __restrict__ maxbits) {
    dep_wait(X, maxbits);
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    const int rg = w / kranges, kr = w - rg * kranges;
    const int r = rg * 32 + lane;
    const int k0 = kr * krange;
    if (r >= R || k0 >= K) return;
    const int k1 = min(K, k0 + krange);
    const int2* xr = reinterpret_cast<const int2*>(X) + view_offset32(rv, (unsigned)r);
    int hi = 0, lo = 0;
    int k = k0;
    auto take = [&](const int2* v) {
#pragma unroll
        for (int u = 0; u < 16; ++u) {
            hi = max(hi, v[u].y & 0x7fffffff);
            lo |= v[u].x;
        }
    };
    if (PLAIN) {
        const long long cs = kv.stride[0];
        xr += k0 * cs;
        for (; k + 16 <= k1; k += 16, xr += 16 * cs) {
            int2 v[16];
#pragma unroll
            for (int u = 0; u < 16; ++u) v[u] = __ldg(xr + u * cs);
            take(v);
        }
        for (; k < k1; ++k, xr += cs) {
            const int2 v = __ldg(xr);
            hi = max(hi, v.y & 0x7fffffff);
            lo |= v.x;
        }
    } else {
        Odometer od;
        od.init(kv, (unsigned)k0);
        for (; k < k1; k += 16) {
            int2 v[16];
#pragma unroll
            for (int u = 0; u < 16; ++u) {
                v[u] = k + u < k1 ? __ldg(xr + od.off) : make_int2(0, 0);
                if (k + u + 1 < k1) od.step(kv);
            }
            take(v);
        }
    }
    atomicMax(maxbits + r, (unsigned long long)hi << 32 | (lo != 0));
}

// round(x 2^(nbits - e)) as an integer, |x| <= 2^e (integer operations on the
// FP64 bit pattern, as in digit_bytes)
__device__ __forceinline__ long long scaled_round(double x, int e, int nbits) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    int ex = (int)((b >> 52) & 0x7ff);
    unsigned long long mant = b & ((1ull << 52) - 1);
    if (ex == 0) ex = 1;
    else mant |= 1ull << 52;
    const int shift = ex - 1075 + nbits - e;
    long long Y;
    if (mant == 0) Y = 0;
    else if (shift >= 0) Y = (long long)(mant << shift);
    else {
        const int sh = -shift;
        Y = sh >= 54 ? 0 : (long long)((mant + (1ull << (sh - 1))) >> sh);
    }
    return (b >> 63) ? -Y : Y;
}

// TF32 slices for 3xTF32: round(x 2^(22 - e)) = 2048 d0 + d1 with d1 in
// [-1024, 1023] and |d0| <= 2048; slice 0 = d0, slice 1 = d1 2^-11, each
// with at most 11 significant bits (exact in TF32), stored as FP32
// [2][R][K4].  One thread per row and 4 consecutive k (one 16-byte store per
// slice); general strided views; row maxima from k_rowmax_cols.
__global__ void k_split_tf32(const double* __restrict__ X, int R, int K, int K4, View rv, View kv,
                             const unsigned long long* __restrict__ maxbits, float* __restrict__ out,
                             int* __restrict__ ex) {
    dep_wait(X, maxbits, out, ex);
    const long long tid = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const int nq = K4 / 4;
    const long long r = tid / nq;
    const int kq = (int)(tid - r * nq);
    if (r >= R) return;
    const int e = row_exponent(__longlong_as_double((long long)maxbits[r]));
    if (kq == 0) ex[r] = e;
    const long long roff = view_offset32(rv, (unsigned)r);
    float s0[4], s1[4];
    const float lo_scale = __int_as_float((127 - 11) << 23);  // 2^-11
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int k = 4 * kq + u;
        const double x = k < K ? X[roff + view_offset32(kv, (unsigned)k)] : 0.0;
        const int y = (int)scaled_round(x, e, 22);  // |y| <= 2^22
        const int hi = (y + 1024) >> 11;
        s0[u] = small_int_f32(hi);
        s1[u] = small_int_f32(y - (hi << 11)) * lo_scale;
    }
    const size_t plane = (size_t)R * K4;
    float* o = out + (size_t)r * K4 + 4 * kq;
    *reinterpret_cast<float4*>(o) = make_float4(s0[0], s0[1], s0[2], s0[3]);
    *reinterpret_cast<float4*>(o + plane) = make_float4(s1[0], s1[1], s1[2], s1[3]);
}

// slice t of eight consecutive values (16 bytes per slice) from their digit integers
__device__ __forceinline__ void slice8_pack(const unsigned long long* z, int s, uint4* q) {
#pragma unroll
    for (int t = 0; t < MAX_S; ++t)
        if (t < s)
            q[t] = make_uint4(slice_of_pair(z[0], z[1], s, t), slice_of_pair(z[2], z[3], s, t),
                              slice_of_pair(z[4], z[5], s, t), slice_of_pair(z[6], z[7], s, t));
}

// K contiguous, rows at stride rs, K8 <= 4 * 8 * TPR: TPR threads per row,
// each holding up to four 8-wide chunks (chunk c = j + i TPR) in registers,
// so X is read once.  VEC: rows start on 16 bytes (16-byte loads).
template <int TPR, bool VEC>
__global__ void __launch_bounds__(256) k_split_rows_reg(const double* __restrict__ X, int R, int K, int K8,
                                                       long long rs, int s, __nv_bfloat16* __restrict__ out,
                                                       int* __restrict__ ex) {
    dep_wait(X, out, ex);
    constexpr int RPB = 256 / TPR;
    __shared__ unsigned long long red[8];
    const int g = threadIdx.x / TPR, j = threadIdx.x % TPR;
    const int r = blockIdx.x * RPB + g;
    const bool live = r < R;
    // the row is held as FP64 bit patterns: kept as doubles, every value
    // cost one FP64-pipe instruction (GB300 issues those at 2 lanes per
    // clock per SM), and nothing here needs FP64 arithmetic
    const unsigned long long* xr =
        reinterpret_cast<const unsigned long long*>(X) + (live ? (long long)r * rs : 0);
    const int nch = K8 >> 3;
    unsigned long long v[4][8];
    unsigned long long mb = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int c = j + i * TPR;
        const int k0 = c * 8;
        if (VEC && live && c < nch && k0 + 8 <= K) {
            const ulonglong2* p2 = reinterpret_cast<const ulonglong2*>(xr + k0);
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const ulonglong2 w = __ldcs(p2 + h);
                v[i][2 * h] = w.x;
                v[i][2 * h + 1] = w.y;
            }
        } else {
#pragma unroll
            for (int u = 0; u < 8; ++u) v[i][u] = (live && c < nch && k0 + u < K) ? __ldcs(xr + k0 + u) : 0ull;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) mb = umax64(mb, v[i][u] & 0x7fffffffffffffffull);
    }
    if (TPR <= 32) {
#pragma unroll
        for (int o = TPR / 2; o > 0; o >>= 1) mb = umax64(mb, __shfl_xor_sync(0xffffffffu, mb, o));
    } else {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mb = umax64(mb, __shfl_xor_sync(0xffffffffu, mb, o));
        const int w = threadIdx.x >> 5;
        if ((threadIdx.x & 31) == 0) red[w] = mb;
        __syncthreads();
        constexpr int WPR = TPR / 32;  // warps per row
        mb = 0;
#pragma unroll
        for (int q = 0; q < WPR; ++q) mb = umax64(mb, red[g * WPR + q]);
    }
    if (!live) return;
    const int e = row_exponent_bits(mb);
    if (j == 0) ex[r] = e;
    const size_t plane = (size_t)R * K8;
    const int base = 1075 - 8 * s + e;
    const unsigned long long bias = digit_bias(s);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int c = j + i * TPR;
        if (c < nch) {
            uint4 q[MAX_S];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[i][u] = digit_bytes(v[i][u], base, bias);
            slice8_pack(v[i], s, q);
            __nv_bfloat16* dst = out + (size_t)r * K8 + (size_t)c * 8;
#pragma unroll
            for (int t = 0; t < MAX_S; ++t)
                if (t < s) *reinterpret_cast<uint4*>(dst + t * plane) = q[t];
        }
    }
}

// K contiguous but longer than the register-resident kernel takes (or read
// through a view): row maxima by (row, 1024-wide K range), then one thread
// per eight consecutive k.  A one-warp-per-row form left a 9 x 1M operand (the
// two-site density matrix at chi = 128) to nine warps.
constexpr int ROWS_KRANGE = 1024;
__global__ void __launch_bounds__(256) k_rowmax_rows(const double* __restrict__ X, int R, int K, View rv, View kv,
                                                    int kranges, unsigned long long* __restrict__ maxbits) {
    dep_wait(X, maxbits);
    const long long w = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    const long long r = w / kranges;
    if (r >= R) return;
    const int k0 = (int)(w - r * kranges) * ROWS_KRANGE, k1 = min(K, k0 + ROWS_KRANGE);
    const double* xr = X + view_offset32(rv, (unsigned)r);
    unsigned long long mb = 0;
    for (int k = k0 + lane; k < k1; k += 32)
        mb = umax64(mb, abs_bits(xr[kv.n == 1 ? (long long)k : view_offset32(kv, (unsigned)k)]));
    for (int o = 16; o > 0; o >>= 1) mb = umax64(mb, __shfl_xor_sync(0xffffffffu, mb, o));
    if (lane == 0) atomicMax(maxbits + r, mb);
}
__global__ void __launch_bounds__(256) k_split_rows_long(const double* __restrict__ X, int R, int K, int K8, View rv,
                                                        View kv, int s,
                                                        const unsigned long long* __restrict__ maxbits,
                                                        __nv_bfloat16* __restrict__ out, int* __restrict__ ex) {
    dep_wait(X, maxbits, out, ex);
    const int nch = K8 >> 3;
    const long long tid = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const long long r = tid / nch;
    const int c = (int)(tid - r * nch);
    if (r >= R) return;
    const int e = row_exponent_bits(maxbits[r]);
    if (c == 0) ex[r] = e;
    const unsigned long long* xr =
        reinterpret_cast<const unsigned long long*>(X) + view_offset32(rv, (unsigned)r);
    const int base = 1075 - 8 * s + e;
    const unsigned long long bias = digit_bias(s);
    unsigned long long z[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const int k = c * 8 + u;
        z[u] = k < K ? __ldcs(xr + (kv.n == 1 ? (long long)k : view_offset32(kv, (unsigned)k))) : 0ull;
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) z[u] = digit_bytes(z[u], base, bias);
    uint4 q[MAX_S];
    slice8_pack(z, s, q);
    const size_t plane = (size_t)R * K8;
    __nv_bfloat16* dst = out + (size_t)r * K8 + (size_t)c * 8;
#pragma unroll
    for (int t = 0; t < MAX_S; ++t)
        if (t < s) *reinterpret_cast<uint4*>(dst + t * plane) = q[t];
}

// Slices of 32 rows (lane = row) x 32 consecutive k from k0, given the digit
// integers z of the lane's row, through this warp's shared-memory tile so that
// four lanes write one row's 64 contiguous bytes in one store instruction:
// lanes that each wrote 16 bytes of a different row left half-written
// sectors that L2 filled from DRAM (1.5x the bytes each way).  One slice at
// a time: the tile is 2.5 KB per warp whatever the number of slices.
__device__ __forceinline__ void store_tile32(const unsigned long long* z, int s, uint4 (*tile)[5], int lane, int r0,
                                             int R, int k0, int kend, int K8, size_t plane,
                                             __nv_bfloat16* __restrict__ out) {
#pragma unroll
    for (int t = 0; t < MAX_S; ++t) {
        if (t >= s) break;
        unsigned p[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) p[u] = slice_of_pair(z[2 * u], z[2 * u + 1], s, t);
#pragma unroll
        for (int c = 0; c < 4; ++c) tile[lane][c] = make_uint4(p[4 * c], p[4 * c + 1], p[4 * c + 2], p[4 * c + 3]);
        __syncwarp();
        // lane -> (row rr = j * 8 + lane / 4, 16-byte chunk c = lane % 4)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int rr = j * 8 + (lane >> 2), c = lane & 3;
            if (r0 + rr < R && k0 + 8 * c < kend)
                *reinterpret_cast<uint4*>(out + t * plane + (size_t)(r0 + rr) * K8 + k0 + 8 * c) = tile[rr][c];
        }
        __syncwarp();
    }
}
// 32 consecutive k of the lane's row as bit patterns (0 beyond K)
template <bool PLAIN>
__device__ __forceinline__ void load32(const unsigned long long* xr, bool live, int k0, int K, const View& kv,
                                       unsigned long long* v) {
    if (PLAIN) {
        const long long cs = kv.stride[0];
#pragma unroll
        for (int u = 0; u < 32; ++u) v[u] = (live && k0 + u < K) ? __ldg(xr + (long long)(k0 + u) * cs) : 0ull;
    } else {
        Odometer od;
        od.init(kv, (unsigned)min(k0, K - 1));
#pragma unroll
        for (int u = 0; u < 32; ++u) {
            v[u] = (live && k0 + u < K) ? __ldg(xr + od.off) : 0ull;
            if (k0 + u + 1 < K) od.step(kv);
        }
    }
}

// Operands read along their rows' contiguous direction (lane = row): one
// warp per 32 rows x kspan k (kspan a multiple of 32), row maxima from
// k_rowmax_cols.  PLAIN: one K stride.  Bound by HBM; warps of 64 k at most
// and 16 of them on an SM keep the last wave short: 8192 x 16 x 8192 485 -> 477
// us, 5000 x 16 x 6000 265 -> 245 against 256 k and 12 warps.
constexpr int COLS_SPAN = 64;
template <bool PLAIN>
__global__ void __launch_bounds__(64, 8) k_split_cols(const double* __restrict__ X, int R, int K, int K8, View rv, View kv,
                                                  int s, const unsigned long long* __restrict__ maxbits,
                                                  __nv_bfloat16* __restrict__ out, int* __restrict__ ex, int kspan,
                                                  int kgroups) {
    dep_wait(X, maxbits, out, ex);
    __shared__ uint4 tile[2][32][5];  // +1 uint4 per row against bank conflicts
    const int wid = (int)((blockIdx.x * (size_t)blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    const int rg = wid / kgroups, kg = wid - rg * kgroups;
    if (rg * 32 >= R) return;
    const int r0 = rg * 32, r = r0 + lane;
    const bool live = r < R;
    const int e = live ? row_exponent_bits(maxbits[r]) : 0;
    if (live && kg == 0) ex[r] = e;
    const unsigned long long* xr =
        reinterpret_cast<const unsigned long long*>(X) + (live ? view_offset32(rv, (unsigned)r) : 0);
    const size_t plane = (size_t)R * K8;
    const int base = 1075 - 8 * s + e;
    const unsigned long long bias = digit_bias(s);
    const int kend = min(K8, (kg + 1) * kspan);
    for (int k0 = kg * kspan; k0 < kend; k0 += 32) {
        unsigned long long v[32];
        load32<PLAIN>(xr, live, k0, K, kv, v);
#pragma unroll
        for (int u = 0; u < 32; ++u) v[u] = digit_bytes(v[u], base, bias);
        store_tile32(v, s, tile[threadIdx.x >> 5], lane, r0, R, k0, kend, K8, plane, out);
    }
}

// The same in one launch: a cluster of CTAs takes 32 rows, each of its warps
// 32 k at a time.  The warps agree on the row maxima (a maximum for each CTA,
// pushed to every other through distributed shared memory) and slice; the last
// 32 k a warp read stay in registers, so that K up to 512 times the cluster's
// CTAs is read once.  What bounds small operands is the integer work of
// slicing on few SMs, the launches of the long form (clear, maxima, slices)
// and its second read; large ones HBM, and there one CTA of 16 warps per SM,
// with its loads and its slicing one after the other, loses to the long form.
constexpr int COLS_ONE_MAX = 1536;
constexpr int COLS_ONE_WARPS = 16;
template <bool PLAIN>
__global__ void __launch_bounds__(32 * COLS_ONE_WARPS) k_split_cols_one(const double* __restrict__ X, int R, int K, int K8,
                                                                       View rv, View kv, int s,
                                                                       __nv_bfloat16* __restrict__ out,
                                                                       int* __restrict__ ex) {
    dep_wait(X, out, ex);
    __shared__ uint4 tile[COLS_ONE_WARPS][32][5];
    __shared__ unsigned long long red[COLS_ONE_WARPS][32], all[16][32];  // of the warps; of the cluster's CTAs
    cg::cluster_group cl = cg::this_cluster();
    const int w = threadIdx.x >> 5, nw = blockDim.x >> 5, lane = threadIdx.x & 31;
    const int nc = (int)cl.num_blocks(), c = (int)cl.block_rank();
    if (nc > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    const int r0 = (int)(blockIdx.x / nc) * 32, r = r0 + lane;
    const bool live = r < R;
    const unsigned long long* xr =
        reinterpret_cast<const unsigned long long*>(X) + (live ? view_offset32(rv, (unsigned)r) : 0);
    const int step = nc * nw * 32;
    unsigned long long v[32];
    unsigned long long mb = 0;
    int k0 = (c * nw + w) * 32, last = -1;
    for (; k0 < K8; k0 += step) {
        load32<PLAIN>(xr, live, k0, K, kv, v);
#pragma unroll
        for (int u = 0; u < 32; ++u) mb = umax64(mb, v[u] & 0x7fffffffffffffffull);
        last = k0;
    }
    red[w][lane] = mb;
    __syncthreads();
    if (nc > 1) {
        // every CTA of the cluster runs before its shared memory is written to
        asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
        if (w < nc) {
            mb = 0;
            for (int i = 0; i < nw; ++i) mb = umax64(mb, red[i][lane]);
            for (int i = w; i < nc; i += nw) cl.map_shared_rank(&all[0][0], i)[c * 32 + lane] = mb;
        }
        cl.sync();
    }
    mb = 0;
    const int n = nc > 1 ? nc : nw;
    for (int i = 0; i < n; ++i) mb = umax64(mb, nc > 1 ? all[i][lane] : red[i][lane]);
    const int e = row_exponent_bits(mb);
    if (live && w == 0 && c == 0) ex[r] = e;
    const size_t plane = (size_t)R * K8;
    const int base = 1075 - 8 * s + e;
    const unsigned long long bias = digit_bias(s);
    for (k0 = last; k0 >= 0; k0 -= step) {
        if (k0 != last) load32<PLAIN>(xr, live, k0, K, kv, v);
#pragma unroll
        for (int u = 0; u < 32; ++u) v[u] = digit_bytes(v[u], base, bias);
        store_tile32(v, s, tile[w], lane, r0, R, k0, K8, K8, plane, out);
    }
}

// ---------------------------------------------------------------------------
// PTX helpers: mbarrier, TMA, tcgen05
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// try_wait with a suspend-time hint: the thread sleeps in hardware until the
// phase completes or ~20 us pass, instead of spinning on issue slots
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity), "r"(20000u)
        : "memory");
    return ok != 0;
}
// Bounded wait: gives up after `limit` cycles (about 1 s at the default
// 2e9), or at once when another thread has already given up, recording the
// failure in *err.
constexpr long long WAIT_LIMIT_CYCLES = 2000000000ll;
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, int* err,
                                          long long limit = WAIT_LIMIT_CYCLES) {
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity)) {
        if (*(volatile int*)err) return false;
        if (clock64() - t0 > limit) {
            atomicCAS(err, 0, 1);
            return false;
        }
    }
    return true;
}

// Failure-detection check of the bounded wait above: thread 0 waits on an
// mbarrier of count 1.  With `arrive` set, thread 32 arrives on it (the wait
// completes); without, nothing ever arrives and the wait must give up after
// `limit` cycles, set *err and return, leaving the context usable.
__global__ void k_wait_probe(long long limit, int arrive, int* err) {
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (threadIdx.x == 32 && arrive) mbar_arrive(&bar);
    if (threadIdx.x == 0) mbar_wait(&bar, 0u, err, limit);
}

__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int c0, int c1, int c2,
                                            uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_u32(dst)),
        "l"((uint64_t)map), "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                       uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void tc_mma_tf32(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                            uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void tc_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                     smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ void tc_ld16(uint32_t taddr, uint32_t* r) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}
__device__ __forceinline__ void tc_ld8(uint32_t taddr, uint32_t* r) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
        : "r"(taddr));
}
// four doubles to a 32-byte aligned address: a whole sector per lane
__device__ __forceinline__ void st_global4(double* p, const double* v) {
    asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p), "d"(v[0]), "d"(v[1]), "d"(v[2]), "d"(v[3])
                 : "memory");
}
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Shared-memory matrix descriptor of a K-major, 64-byte-swizzled tile
// (rows of 64 bytes, 8-row groups 512 bytes apart).
__device__ __forceinline__ uint64_t sw64_desc(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFF);
    d |= (uint64_t)1 << 16;                 // leading byte offset (unused for swizzled K-major)
    d |= (uint64_t)(512 >> 4) << 32;        // stride byte offset: 8 rows x 64 B
    d |= (uint64_t)1 << 46;                 // descriptor version
    d |= (uint64_t)4 << 61;                 // SWIZZLE_64B
    return d;
}


// one thread of a converged warp (the same one at every call)
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}
// tc_mma on descriptors given by their low words (address, leading offset)
__device__ __forceinline__ void tc_mma_lo(uint32_t d_tmem, uint32_t alo, uint32_t blo, uint32_t hi, uint32_t idesc,
                                          uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
        "mov.b64 da, {%1, %3};\n\tmov.b64 db, {%2, %3};\n\t"
        "setp.ne.b32 p, %5, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p;\n\t}" ::"r"(d_tmem),
        "r"(alo), "r"(blo), "r"(hi), "r"(idesc), "r"(accumulate)
        : "memory");
}
// All slice products of one 32-wide k-block, S slices: level 0 and level 1 into
// their accumulators, the rest into the third; keep = 0 restarts the three.
// Straight-line code on constant offsets from the two tile addresses: issued
// from loops over runtime slice indices an MMA took 137 cycles whatever its
// width, so ~100 at N = 144 and 75 at N = 64.  Level by level: the FP32
// rounding of the third accumulator follows the order.  (A slice by A slice with
// the operand kept in the collector buffer was 4-10% faster, and its rounding
// moved observables of small emulated runs by up to 4e-10.)
template <int S, int BN>
__device__ __forceinline__ void issue_levels(uint32_t tmem, uint32_t sa, uint32_t sb, uint32_t idesc, uint32_t keep) {
    constexpr uint64_t top = (uint64_t)(512 >> 4) << 32 | (uint64_t)1 << 46 | (uint64_t)4 << 61;  // as sw64_desc
    constexpr uint32_t hi = (uint32_t)(top >> 32);
    const uint32_t a0 = (sa >> 4) | (1u << 16), b0 = (sb >> 4) | (1u << 16);
#pragma unroll
    for (int h = 0; h < 2; ++h) {  // two K=16 halves, 32 bytes apart in the 64-byte row
        const uint32_t k0 = h ? 1u : keep;
#pragma unroll
        for (int L = 0; L < S; ++L)
#pragma unroll
            for (int t = 0; t <= L; ++t) {
                const int u = L - t;
                const uint32_t d = tmem + (L < 2 ? L : 2) * BN;
                const uint32_t a = a0 + t * (BM * 4) + 2 * h, b = b0 + u * (BN * 4) + 2 * h;
                tc_mma_lo(d, a, b, hi, idesc, t == 0 && u <= 2 ? k0 : 1u);
            }
    }
}

// ---------------------------------------------------------------------------
// slice GEMM
// ---------------------------------------------------------------------------
struct GemmArgs {
    int M, N;             // logical output size
    int nkb;              // 32-wide k-blocks in K
    int kb_per_split;     // k-blocks per blockIdx.z
    int s;                // slices per operand
    int stages;
    uint32_t a_bytes, stage_bytes;
    const int* eA;        // row exponents of A (M)
    const int* eB;        // column exponents of B (N)
    int direct;           // 1: write C; 0: write split-K partials
    double alpha, beta;
    double* C;
    View out_r, out_c;    // C offset of (m, n) = view(out_r, m) + view(out_c, n)
    Weights w;            // of the int64 sums' parts
    int plain;            // alpha = 1 and beta = 0
    int vec;              // 4 or 2: aligned groups of so many columns are contiguous; else 1
    long long* PZ;        // split-K partials [z][Mpad][Npad]
    int Mpad, Npad;
    int m_tiles, n_tiles;
    int* err;
    long long wait_limit; // cycles before a bounded wait gives up
};

// Eight consecutive output columns from n8 of the lane's row m: built from
// their int64 sums and stored (crow: the row's output address, ea = row
// exponent - 44; every lane of the warp calls).
template <bool SHORT>
__device__ __forceinline__ void emit8(const GemmArgs& g, const long long* Z, int ea, int m, int n8, double* crow,
                                      int lane) {
    // the columns are the same for every lane: lane j works out column j's
    // offset and exponent once
    const int nl = n8 + (lane & 7);
    const unsigned coff_l = nl < g.N ? (unsigned)view_offset32(g.out_c, (unsigned)nl) : 0u;
    const int eb_l = nl < g.N ? safe_exp(g.eB[nl]) : 0;
    double v[8];
    bool bad = false;
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = z_scaled_fast<SHORT>(Z[j], ea + __shfl_sync(0xffffffffu, eb_l, j), bad);
    if (__any_sync(0xffffffffu, bad)) {
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = z_scaled(Z[j], ea + __shfl_sync(0xffffffffu, eb_l, j));
    }
    const bool row = m < g.M;
    // alpha = 1, beta = 0 (every product of the sweep): no FP64 arithmetic at
    // all; the branches are uniform, so nothing is issued under a predicate
    if (g.plain && n8 + 8 <= g.N) {
        if (g.vec == 4) {
            const unsigned c0 = __shfl_sync(0xffffffffu, coff_l, 0), c4 = __shfl_sync(0xffffffffu, coff_l, 4);
            if (row) {
                st_global4(crow + c0, v);
                st_global4(crow + c4, v + 4);
            }
        } else if (g.vec == 2) {
#pragma unroll
            for (int j = 0; j < 8; j += 2) {
                const unsigned c = __shfl_sync(0xffffffffu, coff_l, j);
                if (row) *reinterpret_cast<double2*>(crow + c) = make_double2(v[j], v[j + 1]);
            }
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const unsigned c = __shfl_sync(0xffffffffu, coff_l, j);
                if (row) crow[c] = v[j];
            }
        }
        return;
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const unsigned c = __shfl_sync(0xffffffffu, coff_l, j);
        if (!row || n8 + j >= g.N) continue;
        double* cp = crow + c;
        if (g.plain) {
            *cp = v[j];
        } else {
            const double w = v[j] * g.alpha;
            *cp = g.beta == 0.0 ? w : fma(g.beta, *cp, w);
        }
    }
}

// MODE 0: exact-level emulated FP64 (above).  MODE 1: split-BF16 -- the same
// BF16 digit slices, every product of levels <= s-1 accumulated in one FP32
// accumulator over all of K.  MODE 2: 3xTF32 -- two TF32 slices (base-2^11
// digits), hi*hi + hi*lo + lo*hi on kind::tf32 into one FP32 accumulator.
// Modes 1 and 2 run without split-K and read TMEM once per tile.
template <int NB16, int MODE>
__global__ void __launch_bounds__(THREADS, 1)
    k_oz_gemm(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const GemmArgs g) {
    constexpr int BN = 16 * NB16;
    constexpr int NBG = (NB16 + 2) / 3;  // 16-column blocks per epilogue warp
    constexpr int NACC = MODE == 0 ? 3 : 1;  // TMEM accumulators of BN columns
    constexpr uint32_t TMEM_COLS = (NACC * BN <= 32) ? 32 : (NACC * BN <= 64) ? 64 : (NACC * BN <= 128) ? 128
                                   : (NACC * BN <= 256) ? 256 : 512;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t* sbase = smem_raw + (base - raw);
    uint64_t* full = (uint64_t*)(sbase + (size_t)g.stages * g.stage_bytes);
    uint64_t* empty = full + g.stages;
    uint64_t* acc_full = empty + g.stages;
    uint64_t* acc_empty = acc_full + 1;
    uint64_t* drain = acc_full + 2;
    uint32_t* tmem_slot = (uint32_t*)(drain + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // Direct output: a persistent grid strides over the m_tiles x n_tiles
    // tiles, n fastest (CTAs running together share A tiles through L2), and
    // the stage ring and the accumulator hand-off run on across tiles, so one
    // tile's epilogue overlaps the next tile's loads and MMAs.  Split-K
    // partials: one tile per CTA (blockIdx x: m, y: n, z: split).
    const int ntiles = g.direct ? g.m_tiles * g.n_tiles : 1;
    const int t_first = g.direct ? (int)blockIdx.x : 0, t_step = g.direct ? (int)gridDim.x : 1;
    auto tile_m0 = [&](int t) { return (g.direct ? t / g.n_tiles : (int)blockIdx.x) * BM; };
    auto tile_n0 = [&](int t) { return (g.direct ? t % g.n_tiles : (int)blockIdx.y) * BN; };
    const int kb0 = g.direct ? 0 : (int)blockIdx.z * g.kb_per_split;
    const int kb1 = min(g.nkb, kb0 + g.kb_per_split);
    const int nkb = kb1 - kb0;
    const int nchunks = (nkb + CHUNK_KB - 1) / CHUNK_KB;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 32) {
        for (int st = 0; st < g.stages; ++st) {
            mbar_init(&full[st], 1);
            mbar_init(&empty[st], 1);
        }
        mbar_init(acc_full, 1);
        mbar_init(acc_empty, EPI_WARPS);
        mbar_init(drain, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    dep_wait();  // the operands and the outputs are touched from here on only

    if (warp == EPI_WARPS) {
        // ---------------- TMA producer ----------------
        if (lane == 0) {
            int issued = 0;
            bool ok = true;
            for (int t = t_first; t < ntiles && ok; t += t_step) {
                const int m0 = tile_m0(t), n0 = tile_n0(t);
                for (int i = 0; i < nkb; ++i) {
                    const int st = issued % g.stages;
                    const uint32_t ph = (uint32_t)(issued / g.stages) & 1u;
                    if (!mbar_wait(&empty[st], ph ^ 1u, g.err, g.wait_limit)) {
                        ok = false;
                        break;
                    }
                    uint8_t* sa = sbase + (size_t)st * g.stage_bytes;
                    mbar_expect_tx(&full[st], g.stage_bytes);
                    const int kc = (kb0 + i) * (MODE == 2 ? BK / 2 : BK);  // 64 bytes of K per stage
                    tma_load_3d(sa, &tmA, kc, m0, 0, &full[st]);
                    tma_load_3d(sa + g.a_bytes, &tmB, kc, n0, 0, &full[st]);
                    ++issued;
                }
            }
            if (*(volatile int*)g.err) {
                // let the copies still in flight land before the CTA exits
                for (int i = max(0, issued - g.stages); i < issued; ++i) {
                    const long long t0 = clock64();
                    while (!mbar_try_wait(&full[i % g.stages], (uint32_t)(i / g.stages) & 1u) &&
                           clock64() - t0 < g.wait_limit) {
                    }
                }
            }
        }
    } else if (warp == EPI_WARPS + 1) {
        // ---------------- MMA issuer ----------------
        // the warp stays converged and elects the issuing thread per k-block:
        // addresses then live in uniform registers
        {
            // D format F32 (1); A and B both BF16 (1) under kind::f16, both TF32 (2) under kind::tf32
            constexpr uint32_t fmt = MODE == 2 ? 2u : 1u;
            const uint32_t idesc = (1u << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)(BN >> 3) << 17) |
                                   ((uint32_t)(BM >> 4) << 24);
            int it = 0, cc = 0;  // k-blocks and accumulator chunks issued so far, over all tiles
            bool ok = true;
            for (int t = t_first; t < ntiles && ok; t += t_step)
            for (int i = 0; i < nkb; ++i, ++it) {
                const int st = it % g.stages;
                const uint32_t ph = (uint32_t)(it / g.stages) & 1u;
                const bool first = MODE == 0 ? (i % CHUNK_KB) == 0 : i == 0;
                const bool last = MODE == 0 ? ((i % CHUNK_KB) == CHUNK_KB - 1 || i == nkb - 1) : i == nkb - 1;
                bool go = !(first && cc > 0) || mbar_wait(acc_empty, (uint32_t)(cc - 1) & 1u, g.err, g.wait_limit);
                go = go && mbar_wait(&full[st], ph, g.err, g.wait_limit);
                if (!__all_sync(0xffffffffu, go)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t sa = base + (uint32_t)st * g.stage_bytes;
                const uint32_t sb = sa + g.a_bytes;
                if (elect_one()) {
                    if (MODE != 0) {
                        // two 32-byte K halves (16 BF16 or 8 TF32 each); every level
                        // <= s-1 into the one FP32 accumulator
                        for (int h = 0; h < 2; ++h) {
                            bool f1 = first && h == 0;
                            for (int L = 0; L < g.s; ++L)
                                for (int t2 = 0; t2 <= L; ++t2) {
                                    const uint64_t ad = sw64_desc(sa + t2 * (BM * 64) + h * 32);
                                    const uint64_t bd = sw64_desc(sb + (L - t2) * (BN * 64) + h * 32);
                                    if (MODE == 2) tc_mma_tf32(tmem, ad, bd, idesc, f1 ? 0u : 1u);
                                    else tc_mma(tmem, ad, bd, idesc, f1 ? 0u : 1u);
                                    f1 = false;
                                }
                        }
                    } else {
                        const uint32_t keep = first ? 0u : 1u;  // the FP32 levels restart every chunk too
                        switch (g.s) {
                            case 2: issue_levels<2, BN>(tmem, sa, sb, idesc, keep); break;
                            case 3: issue_levels<3, BN>(tmem, sa, sb, idesc, keep); break;
                            case 4: issue_levels<4, BN>(tmem, sa, sb, idesc, keep); break;
                            case 5: issue_levels<5, BN>(tmem, sa, sb, idesc, keep); break;
                            default: issue_levels<6, BN>(tmem, sa, sb, idesc, keep); break;
                        }
                    }
                    tc_commit(&empty[st]);
                    if (last) tc_commit(acc_full);
                }
                __syncwarp();
                if (last) ++cc;
            }
            // every MMA issued by this warp completes before TMEM is freed
            if (elect_one()) {
                tc_commit(drain);
                const long long t0 = clock64();
                while (!mbar_try_wait(drain, 0u) && clock64() - t0 < g.wait_limit) {
                }
            }
            __syncwarp();
        }
    } else if (MODE != 0) {
        // ---------------- epilogue of the FP32-accumulated modes ----------------
        const int q = warp & 3, grp = warp >> 2;
        const uint32_t lane_addr = tmem + ((uint32_t)(q * 32) << 16);
        const bool unit_alpha = g.alpha == 1.0, zero_beta = g.beta == 0.0;
        constexpr int dbits = MODE == 2 ? 11 : 8;  // digit width of the slices
        int cc = 0;
        for (int t = t_first; t < ntiles; t += t_step, ++cc) {
            const int m0 = tile_m0(t), n0 = tile_n0(t);
            const int m = m0 + q * 32 + lane;
            const int ea = m < g.M ? g.eA[m] : 0;
            if (!mbar_wait(acc_full, (uint32_t)cc & 1u, g.err, g.wait_limit)) break;
            tc_fence_after();
            float F[NBG][16];
#pragma unroll
            for (int jb = 0; jb < NBG; ++jb) {
                const int b = grp + 3 * jb;
                if (b >= NB16) continue;
                uint32_t r[16];
                tc_ld16(lane_addr + b * 16, r);
                tc_wait_ld();
#pragma unroll
                for (int j = 0; j < 16; ++j) F[jb][j] = __uint_as_float(r[j]);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acc_empty);
#pragma unroll
            for (int jb = 0; jb < NBG; ++jb) {
                const int b = grp + 3 * jb;
                if (b >= NB16) continue;
                const int nl = n0 + b * 16 + (lane & 15);
                const long long coff_l = nl < g.N ? view_offset32(g.out_c, (unsigned)nl) : 0;
                const int eb_l = nl < g.N ? g.eB[nl] : 0;
                double* crow = g.C + (m < g.M ? view_offset32(g.out_r, (unsigned)m) : 0);
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const long long coff = __shfl_sync(0xffffffffu, coff_l, j);
                    const int eb = __shfl_sync(0xffffffffu, eb_l, j);
                    const int n = n0 + b * 16 + j;
                    if (m >= g.M || n >= g.N) continue;
                    double v = f32_scaled(F[jb][j], ea + eb - 2 * dbits);
                    if (ea > 1024 || eb > 1024) v = __longlong_as_double(0x7ff8000000000000ll);  // non-finite operand
                    double* cp = crow + coff;
                    // uniform branch: no FP64 arithmetic issued when alpha = 1, beta = 0
                    if (unit_alpha && zero_beta) *cp = v;
                    else *cp = zero_beta ? v * g.alpha : fma(g.beta, *cp, v * g.alpha);
                }
            }
        }
    } else {
        // ---------------- epilogue: warps 0..11 ----------------
        // Three warps per TMEM lane quarter share the tile's 8-column blocks.
        // Every chunk's three accumulators are added to one int64 per entry;
        // the last chunk's TMEM is released as soon as it is read, so that the
        // next tile's MMAs run while this tile's results are built and stored.
        // (Held as two int32 and one FP32 sum, 144 columns took more registers
        // than there are: the spills cost a K = 8192 product ~16000 cycles per
        // chunk beside 25000 of MMAs.)
        const int q = warp & 3, grp = warp >> 2;
        const uint32_t lane_addr = tmem + ((uint32_t)(q * 32) << 16);
        constexpr int NB8 = 2 * NB16, NC = (NB8 + 2) / 3;  // 8-column blocks, most per warp
        int cc = 0;  // accumulator chunks drained so far, over all tiles
        bool ok = true;
        for (int t = t_first; t < ntiles && ok; t += t_step) {
            const int m0 = tile_m0(t), n0 = tile_n0(t);
            const int m = m0 + q * 32 + lane;
            const int ea = (g.direct && m < g.M) ? safe_exp(g.eA[m]) - 44 : 0;
            long long Z[NC][8];
#pragma unroll
            for (int jb = 0; jb < NC; ++jb)
#pragma unroll
                for (int j = 0; j < 8; ++j) Z[jb][j] = 0;
            for (int c = 0; c < nchunks; ++c, ++cc) {
                if (!mbar_wait(acc_full, (uint32_t)cc & 1u, g.err, g.wait_limit)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
#pragma unroll
                for (int jb = 0; jb < NC; ++jb) {
                    const int b = grp + 3 * jb;
                    if (b >= NB8) continue;
                    uint32_t r0[8], r1[8], r2[8];
                    tc_ld8(lane_addr + b * 8, r0);
                    tc_ld8(lane_addr + BN + b * 8, r1);
                    if (g.s > 2) tc_ld8(lane_addr + 2 * BN + b * 8, r2);
                    tc_wait_ld();
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        Z[jb][j] = fixed_add(Z[jb][j], __uint_as_float(r0[j]), __uint_as_float(r1[j]),
                                             g.s > 2 ? __uint_as_float(r2[j]) : 0.0f);
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(acc_empty);
            }
            if (!ok) break;
            if (g.direct) {
                double* crow = g.C + (m < g.M ? view_offset32(g.out_r, (unsigned)m) : 0);
#pragma unroll
                for (int jb = 0; jb < NC; ++jb) {
                    const int b = grp + 3 * jb;
                    if (b < NB8) emit8<false>(g, Z[jb], ea, m, n0 + b * 8, crow, lane);
                }
            } else {
#pragma unroll
                for (int jb = 0; jb < NC; ++jb) {
                    const int b = grp + 3 * jb;
                    if (b >= NB8) continue;
                    longlong2* row = reinterpret_cast<longlong2*>(
                        g.PZ + ((size_t)blockIdx.z * g.Mpad + m) * g.Npad + n0 + b * 8);
#pragma unroll
                    for (int j = 0; j < 4; ++j) row[j] = make_longlong2(Z[jb][2 * j], Z[jb][2 * j + 1]);
                }
            }
        }  // tiles
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    }
}

// Products of a single exact chunk (K <= 256: every product of an enlarged
// corner), emulated FP64 only.  Their epilogue -- ~70 instructions per entry,
// half of them on the 16-lane integer pipe -- outweighs the 30 MMAs per
// 32 of K, and with three warps per SM quarter and one set of accumulators
// it was bound by latency (38% of issue slots) and waited for the MMAs in
// between.  Here two teams of twelve warps take turns on two sets of
// accumulators (BN <= 80: 6 BN <= 480 of 512 TMEM columns): the MMAs of one
// tile run under the epilogues of the two before it, and a warp holds eight
// columns at a time, so that 26 warps fit the register file.
// 262144 x 192 x 64 in its sweep layout: 340 -> 176 us; 8192 x 8192 x 128: 527 -> 278.
constexpr int TEAM_WARPS = 12;
constexpr int SHORT_THREADS = (2 * TEAM_WARPS + 2) * 32;
template <int NB16>
__global__ void __launch_bounds__(SHORT_THREADS, 1)
    k_oz_gemm_short(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const GemmArgs g) {
    constexpr int BN = 16 * NB16;
    constexpr uint32_t TMEM_COLS = 6 * BN <= 128 ? 128 : 6 * BN <= 256 ? 256 : 512;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t* sbase = smem_raw + (base - raw);
    uint64_t* full = (uint64_t*)(sbase + (size_t)g.stages * g.stage_bytes);
    uint64_t* empty = full + g.stages;
    uint64_t* acc_full = empty + g.stages;   // [2]
    uint64_t* acc_empty = acc_full + 2;      // [2]
    uint64_t* drain = acc_empty + 2;
    uint32_t* tmem_slot = (uint32_t*)(drain + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ntiles = g.m_tiles * g.n_tiles, nkb = g.nkb;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 32) {
        for (int st = 0; st < g.stages; ++st) {
            mbar_init(&full[st], 1);
            mbar_init(&empty[st], 1);
        }
        for (int u = 0; u < 2; ++u) {
            mbar_init(&acc_full[u], 1);
            mbar_init(&acc_empty[u], TEAM_WARPS);
        }
        mbar_init(drain, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    dep_wait();  // the operands and the outputs are touched from here on only

    if (warp == 2 * TEAM_WARPS) {
        // ---------------- TMA producer ----------------
        if (lane == 0) {
            int issued = 0;
            bool ok = true;
            for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
                const int m0 = t / g.n_tiles * BM, n0 = t % g.n_tiles * BN;
                for (int i = 0; i < nkb; ++i) {
                    const int st = issued % g.stages;
                    if (!mbar_wait(&empty[st], ((uint32_t)(issued / g.stages) & 1u) ^ 1u, g.err, g.wait_limit)) {
                        ok = false;
                        break;
                    }
                    uint8_t* sa = sbase + (size_t)st * g.stage_bytes;
                    mbar_expect_tx(&full[st], g.stage_bytes);
                    tma_load_3d(sa, &tmA, i * BK, m0, 0, &full[st]);
                    tma_load_3d(sa + g.a_bytes, &tmB, i * BK, n0, 0, &full[st]);
                    ++issued;
                }
            }
            if (*(volatile int*)g.err) {
                // let the copies still in flight land before the CTA exits
                for (int i = max(0, issued - g.stages); i < issued; ++i) {
                    const long long t0 = clock64();
                    while (!mbar_try_wait(&full[i % g.stages], (uint32_t)(i / g.stages) & 1u) &&
                           clock64() - t0 < g.wait_limit) {
                    }
                }
            }
        }
    } else if (warp == 2 * TEAM_WARPS + 1) {
        // ---------------- MMA issuer (converged warp, one elected thread) ----------------
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
        int it = 0, ti = 0;
        bool ok = true;
        for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x, ++ti) {
            const int buf = ti & 1;
            bool go = ti < 2 || mbar_wait(&acc_empty[buf], (uint32_t)((ti >> 1) - 1) & 1u, g.err, g.wait_limit);
            for (int i = 0; i < nkb; ++i, ++it) {
                const int st = it % g.stages;
                go = go && mbar_wait(&full[st], (uint32_t)(it / g.stages) & 1u, g.err, g.wait_limit);
                if (!__all_sync(0xffffffffu, go)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t sa = base + (uint32_t)st * g.stage_bytes, sb = sa + g.a_bytes;
                const uint32_t acc = tmem + (uint32_t)buf * (3 * BN), keep = i == 0 ? 0u : 1u;
                if (elect_one()) {
                    switch (g.s) {
                        case 2: issue_levels<2, BN>(acc, sa, sb, idesc, keep); break;
                        case 3: issue_levels<3, BN>(acc, sa, sb, idesc, keep); break;
                        case 4: issue_levels<4, BN>(acc, sa, sb, idesc, keep); break;
                        case 5: issue_levels<5, BN>(acc, sa, sb, idesc, keep); break;
                        default: issue_levels<6, BN>(acc, sa, sb, idesc, keep); break;
                    }
                    tc_commit(&empty[st]);
                    if (i == nkb - 1) tc_commit(&acc_full[buf]);
                }
                __syncwarp();
            }
        }
        // every MMA issued by this warp completes before TMEM is freed
        if (elect_one()) {
            tc_commit(drain);
            const long long t0 = clock64();
            while (!mbar_try_wait(drain, 0u) && clock64() - t0 < g.wait_limit) {
            }
        }
        __syncwarp();
    } else {
        // ---------------- epilogue: two teams of 3 warps per TMEM lane quarter ----------------
        const int team = warp >= TEAM_WARPS ? 1 : 0, q = warp & 3, grp = (warp - team * TEAM_WARPS) >> 2;
        constexpr int NB8 = 2 * NB16;
        const uint32_t lane_addr = tmem + (uint32_t)team * (3 * BN) + ((uint32_t)(q * 32) << 16);
        int ti = team;
        for (int t = blockIdx.x + team * gridDim.x; t < ntiles; t += 2 * gridDim.x, ti += 2) {
            const int m0 = t / g.n_tiles * BM, n0 = t % g.n_tiles * BN;
            const int m = m0 + q * 32 + lane;
            const int ea = m < g.M ? safe_exp(g.eA[m]) - 44 : 0;
            double* crow = g.C + (m < g.M ? view_offset32(g.out_r, (unsigned)m) : 0);
            if (!mbar_wait(&acc_full[team], (uint32_t)(ti >> 1) & 1u, g.err, g.wait_limit)) break;
            tc_fence_after();
            for (int b = grp; b < NB8; b += 3) {
                uint32_t r0[8], r1[8], r2[8];
                tc_ld8(lane_addr + b * 8, r0);
                tc_ld8(lane_addr + BN + b * 8, r1);
                if (g.s > 2) tc_ld8(lane_addr + 2 * BN + b * 8, r2);
                tc_wait_ld();
                if (b + 3 >= NB8) {  // the warp's last read of this tile
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&acc_empty[team]);
                }
                long long Z[8];
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    Z[j] = fixed_add_w(g.w, 0, __uint_as_float(r0[j]), __uint_as_float(r1[j]),
                                     g.s > 2 ? __uint_as_float(r2[j]) : 0.0f);
                emit8<true>(g, Z, ea, m, n0 + b * 8, crow, lane);
            }
            if (grp >= NB8) {  // fewer blocks than warps: this one read nothing
                __syncwarp();
                if (lane == 0) mbar_arrive(&acc_empty[team]);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    }
}

// split-K partials -> C: an exact int64 sum (|Z| < 2^59 at 16384 of K, so up to
// K = 2^17 in all), in FP64 beyond
constexpr int COMBINE_INT64_K = 1 << 17;
__global__ void k_oz_combine(const long long* __restrict__ PZ, int splits, int wide, int Mpad, int Npad, int M, int N,
                             const int* __restrict__ eA, const int* __restrict__ eB, double alpha, double beta,
                             double* __restrict__ C, View out_r, View out_c) {
    dep_wait(PZ, eA, eB, C);
    const size_t total = (size_t)M * N, zs = (size_t)Mpad * Npad;
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < total; t += (size_t)gridDim.x * blockDim.x) {
        const int m = (int)(t / N), n = (int)(t % N);
        const long long* p = PZ + (size_t)m * Npad + n;
        const int e = safe_exp(eA[m]) + safe_exp(eB[n]) - 44;
        double v;
        if (!wide) {
            long long z = 0;
#pragma unroll 4
            for (int q = 0; q < splits; ++q) z += p[q * zs];
            v = z_scaled(z, e);
        } else {
            v = 0.0;
            for (int q = 0; q < splits; ++q) v += (double)p[q * zs];
            v = e > BAD_EXP / 2 ? __longlong_as_double(0x7ff8000000000000ll) : scale_pow2(v, e);
        }
        if (alpha != 1.0) v *= alpha;
        double* cp = C + view_offset32(out_r, (unsigned)m) + view_offset32(out_c, (unsigned)n);
        *cp = (beta == 0.0) ? v : fma(beta, *cp, v);
    }
}

}  // namespace oz
}  // namespace ctm

// ===========================================================================
// host side
// ===========================================================================
namespace ctm {
namespace {

inline size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }
inline int k8_of(int K) { return (K + 7) & ~7; }
inline int k4_of(int K) { return (K + 3) & ~3; }

PFN_cuTensorMapEncodeTiled_v12000 tmap_encoder() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
    });
    return fn;
}

// slices [s][R][Kp], 64-byte-swizzled boxes of {64 bytes of k, rows, s}:
// BF16 (Kp = K8, 32 k per box row) or TF32 as FP32 (Kp = K4, 16 k)
bool make_map(CUtensorMap* map, const void* slices, int R, int Kp, int s, int box_rows, bool tf32 = false) {
    auto enc = tmap_encoder();
    if (!enc) return false;
    const int esz = tf32 ? 4 : 2;
    const cuuint64_t dims[3] = {(cuuint64_t)Kp, (cuuint64_t)R, (cuuint64_t)s};
    const cuuint64_t strides[2] = {(cuuint64_t)Kp * esz, (cuuint64_t)R * Kp * esz};
    const cuuint32_t box[3] = {(cuuint32_t)(64 / esz), (cuuint32_t)box_rows, (cuuint32_t)s};
    const cuuint32_t estr[3] = {1, 1, 1};
    return enc(map, tf32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3,
               const_cast<void*>(slices), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

struct Plan {
    int nb16, bn, m_tiles, n_tiles, ksplit, kb_per_split, nkb, stages;
    bool one;  // a single exact chunk: k_oz_gemm_short
    uint32_t a_bytes, stage_bytes;
    size_t smem, ws_bytes;
};

// An MMA of BN columns takes about 55 + BN/3 cycles here (measured at 64, 96
// and 144; 128-row operands from shared memory).
double mma_cycles(int bn) { return 55.0 + bn / 3.0; }

// mode 2 (3xTF32) holds 16 k per 64-byte stage row instead of 32; modes 1 and
// 2 never split K
Plan plan_of(int M, int N, int K, int s, int mode = 0) {
    Plan p{};
    p.m_tiles = (M + oz::BM - 1) / oz::BM;
    p.nkb = mode == 2 ? (k4_of(K) + 15) / 16 : (k8_of(K) + oz::BK - 1) / oz::BK;
    if (p.nkb < 1) p.nkb = 1;
    p.one = mode == 0 && p.nkb <= oz::CHUNK_KB;
    if (p.one) {
        // the width with the least work on the fullest SM: a tile costs the longer
        // of its MMAs and its epilogue (~0.55 cycles per entry and SM, measured)
        double best = -1.0;
        for (int nb = 1; nb <= 5; ++nb) {
            const double nt = std::ceil(N / (16.0 * nb));
            const double tile = std::max(2.0 * p.nkb * (s * (s + 1) / 2) * mma_cycles(16 * nb), 0.55 * 128 * 16 * nb) + 600.0;
            const double cost = std::ceil(nt * p.m_tiles / 152.0) * tile;
            if (best < 0.0 || cost < best) {
                best = cost;
                p.nb16 = nb;
            }
        }
    } else {
        // fewest 144-wide tiles, then the narrowest 16-multiple width that covers N
        const int nt = (N + 143) / 144;
        p.nb16 = std::max(1, ((N + nt - 1) / nt + 15) / 16);
    }
    p.bn = 16 * p.nb16;
    p.n_tiles = (N + p.bn - 1) / p.bn;
    const int nchunks = (p.nkb + oz::CHUNK_KB - 1) / oz::CHUNK_KB;
    const int tiles = p.m_tiles * p.n_tiles;
    // Split K when the tiles leave SMs idle, at whole chunks (the FP32 levels are
    // summed per chunk: splits inside one changed their rounding, and observables
    // of small emulated runs by 1e-9): the split whose fullest SM has the least
    // work, 2 s(s+1)/2 MMAs per k-block, a drain per chunk, and the partials'
    // pass.  64 tiles x 32 chunks in 3 splits put 22 chunks on some SMs, in 2
    // splits 16 on all.
    int ks = 1;
    if (mode == 0 && tiles < 120 && nchunks >= 2) {
        const double kb = (double)s * (s + 1) * mma_cycles(p.bn);
        double best = -1.0;
        for (int k = 2; k <= nchunks; ++k) {
            const int per = (nchunks + k - 1) / k * oz::CHUNK_KB;
            if ((nchunks * oz::CHUNK_KB + per - 1) / per != k) continue;
            const double cta = per * kb + 2500.0 * ((per + oz::CHUNK_KB - 1) / oz::CHUNK_KB) + 5000.0;
            const double cost = ((tiles * k + 151) / 152) * cta + 8.0 * k * p.m_tiles * oz::BM * p.n_tiles * p.bn / 1500.0;
            if (best < 0.0 || cost < best) {
                best = cost;
                ks = k;
            }
        }
    }
    // int64 sums of a split stay below 2^59 for K <= 16384
    const int max_kb_per_split = 16384 / oz::BK;
    if (mode == 0) ks = std::max(ks, (p.nkb + max_kb_per_split - 1) / max_kb_per_split);
    p.kb_per_split = mode == 0 ? (nchunks + ks - 1) / ks * oz::CHUNK_KB : p.nkb;
    p.ksplit = (p.nkb + p.kb_per_split - 1) / p.kb_per_split;
    p.a_bytes = (uint32_t)(s * oz::BM * oz::BK * 2);
    p.stage_bytes = p.a_bytes + (uint32_t)(s * p.bn * oz::BK * 2);
    p.stages = std::min<int>(6, (int)((220u * 1024u) / p.stage_bytes));
    p.smem = (size_t)p.stages * p.stage_bytes + 1024 + 256;
    p.ws_bytes = p.ksplit > 1 ? align256((size_t)p.ksplit * p.m_tiles * oz::BM * p.n_tiles * p.bn * 8) : 0;
    return p;
}

using GemmKernel = void (*)(const CUtensorMap, const CUtensorMap, const oz::GemmArgs);
// `done`: a bit per device on which this kernel's 227 KB shared-memory opt-in
// (a per-device function attribute) is set
cudaError_t launch_gemm(GemmKernel kern, int threads, unsigned long long* done, const Plan& p, const CUtensorMap& ta,
                        const CUtensorMap& tb, const oz::GemmArgs& g, cudaStream_t st) {
    static std::mutex mu;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    {
        std::lock_guard<std::mutex> lock(mu);
        if (!(*done >> dev & 1ull)) {
            e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
            if (e != cudaSuccess) return e;
            *done |= 1ull << dev;
        }
    }
    dim3 grid(p.m_tiles, p.n_tiles, p.ksplit);
    if (g.direct) {
        // persistent: one CTA per SM (the stage ring fills shared memory)
        int nsm = 0;
        e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        const long long tiles = (long long)p.m_tiles * p.n_tiles;
        grid = dim3((unsigned)std::min<long long>(tiles, nsm > 0 ? nsm : 1), 1, 1);
    }
    return launch_dep(kern, grid, threads, p.smem, st, ta, tb, g);
}
template <int NB16>
cudaError_t launch_mode(int mode, const Plan& p, const CUtensorMap& ta, const CUtensorMap& tb, const oz::GemmArgs& g,
                        cudaStream_t st) {
    static unsigned long long done[4] = {};
    if constexpr (NB16 <= 5)
        if (p.one) return launch_gemm(oz::k_oz_gemm_short<NB16>, oz::SHORT_THREADS, done + 3, p, ta, tb, g, st);
    if (mode == 0) return launch_gemm(oz::k_oz_gemm<NB16, 0>, oz::THREADS, done, p, ta, tb, g, st);
    if (mode == 1) return launch_gemm(oz::k_oz_gemm<NB16, 1>, oz::THREADS, done + 1, p, ta, tb, g, st);
    return launch_gemm(oz::k_oz_gemm<NB16, 2>, oz::THREADS, done + 2, p, ta, tb, g, st);
}

}  // namespace

// split buffer: slices [s][R][K8] | row max bits [R] (u64) | exponents [R] (int)
size_t oz_split_bytes(int R, int K, int s) {
    return align256((size_t)s * R * k8_of(K) * 2) + align256((size_t)R * 8) + align256((size_t)R * 4);
}
inline const int* split_exponents(const void* buf, int R, int K8, int s) {
    return (const int*)((const char*)buf + align256((size_t)s * R * K8 * 2) + align256((size_t)R * 8));
}
// TF32 split buffer: slices [2][R][K4] (FP32) | row max bits [R] | exponents [R]
size_t oz_split_tf32_bytes(int R, int K) {
    return align256((size_t)2 * R * k4_of(K) * 4) + align256((size_t)R * 8) + align256((size_t)R * 4);
}
inline const int* split_tf32_exponents(const void* buf, int R, int K4) {
    return (const int*)((const char*)buf + align256((size_t)2 * R * K4 * 4) + align256((size_t)R * 8));
}

// Whether the device runs clusters of 16 CTAs of the one-launch slicer (a
// property of the device: asked once for each).
static bool cols_cluster_of_16() {
    static std::mutex mu;
    static unsigned long long asked = 0, yes = 0;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
    std::lock_guard<std::mutex> lock(mu);
    if (asked >> dev & 1ull) return yes >> dev & 1ull;
    bool ok = true;
    for (auto k : {oz::k_split_cols_one<true>, oz::k_split_cols_one<false>}) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(16, 1, 1);
        cfg.blockDim = dim3(32 * oz::COLS_ONE_WARPS, 1, 1);
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 16;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int n = 0;
        ok = ok && cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
             cudaOccupancyMaxActiveClusters(&n, k, &cfg) == cudaSuccess && n > 0;
    }
    if (!ok) cudaGetLastError();
    asked |= 1ull << dev;
    yes |= (unsigned long long)ok << dev;
    return ok;
}

// K range of one warp in the lane = row kernels: 256, halved down to 32 until
// the operand gives every SM sixteen warps
static int cols_krange(int R, int K) {
    const long long rg = (R + 31) / 32;
    int range = 256;
    while (range > 32 && rg * ((K + range - 1) / range) < 152 * 16) range /= 2;
    return range;
}

// CTAs of the cluster that slices 32 rows in one launch, 0 where the operand
// goes the long way (maxima, then slices).  Whole products of 5 slices with
// such an A, in us, without clusters (K <= 1536: one CTA; above: the long way)
// and with them, M x N x K:
//   48x48x1200 57.0, 40.6   1200x48x1200 61.1, 54.9   1024x40x1024 52.9, 42.8
//   144x144x8192 76.4, 67.2   2048x64x2048 72.3, 63.1   20000x64x2048 430, 407
//   8192x144x1536 153, 168   30000x16x1200 302, 346   8192x144x5000 530, 557
// so clusters of 16 and those of short rows (K <= 1536) are for operands of one
// wave or two, clusters of up to 8 for K in between whatever R.
static int cols_cluster(int R, int K8) {
    const long long rg = (R + 31) / 32;
    const int warps = (K8 + 31) / 32;
    const bool small = rg * warps <= 152 * 2 * oz::COLS_ONE_WARPS;
    if (!small && K8 <= oz::COLS_ONE_MAX) return 1;
    int nc = 1;
    while (nc < 16 && nc * oz::COLS_ONE_WARPS < warps) nc *= 2;
    if (nc * oz::COLS_ONE_WARPS < warps || rg * nc > 0x7fffffffll) return 0;
    if (nc == 16) return small && cols_cluster_of_16() ? 16 : 0;
    while (nc < 8 && rg * nc < 152 && nc * 2 < warps) nc *= 2;
    return nc;
}

static void launch_rowmax_cols(unsigned blocks, cudaStream_t st, const double* X, int R, int K, const oz::View& rv,
                               const oz::View& kv, int kranges, int krange, unsigned long long* mb) {
    launch_dep(kv.n == 1 ? oz::k_rowmax_cols<true> : oz::k_rowmax_cols<false>, blocks, 128, 0, st, X, R, K, rv, kv, kranges,
               krange, mb);
}

cudaError_t oz_split_tf32(const double* X, int R, int K, const OzView& rvh, const OzView& kvh, void* buf,
                          cudaStream_t st) {
    if (R <= 0 || K <= 0 || rvh.n < 1 || rvh.n > 4 || kvh.n < 1 || kvh.n > 4) return cudaErrorInvalidValue;
    oz::View rv, kv;
    rv.n = rvh.n;
    kv.n = kvh.n;
    for (int a = 0; a < 4; ++a) {
        rv.dim[a] = rvh.dim[a];
        rv.stride[a] = rvh.stride[a];
        kv.dim[a] = kvh.dim[a];
        kv.stride[a] = kvh.stride[a];
    }
    const int K4 = k4_of(K);
    float* sl = (float*)buf;
    unsigned long long* mb = (unsigned long long*)((char*)buf + align256((size_t)2 * R * K4 * 4));
    int* ex = const_cast<int*>(split_tf32_exponents(buf, R, K4));
    cudaError_t e = cudaMemsetAsync(mb, 0, (size_t)R * 8, st);
    if (e != cudaSuccess) return e;
    const unsigned rg = (unsigned)((R + 31) / 32);
    const int krange = cols_krange(R, K);
    const unsigned kr = (unsigned)((K + krange - 1) / krange);
    const unsigned long long warps = (unsigned long long)rg * kr;
    const unsigned long long threads = (unsigned long long)R * (K4 / 4);
    if ((warps + 3) / 4 > 0x7fffffffull || (threads + 255) / 256 > 0x7fffffffull) return cudaErrorInvalidValue;
    launch_rowmax_cols((unsigned)((warps + 3) / 4), st, X, R, K, rv, kv, (int)kr, krange, mb);
    launch_dep(oz::k_split_tf32, (unsigned)((threads + 255) / 256), 256, 0, st, X, R, K, K4, rv, kv, mb, sl, ex);
    return cudaGetLastError();
}

template <int TPR>
void launch_rows_reg_t(bool vec, unsigned blocks, cudaStream_t st, const double* X, int R, int K, int K8,
                       long long rs, int s, __nv_bfloat16* sl, int* ex) {
    launch_dep(vec ? oz::k_split_rows_reg<TPR, true> : oz::k_split_rows_reg<TPR, false>, blocks, 256, 0, st, X, R, K, K8, rs,
               s, sl, ex);
}
void launch_split_rows_reg(int tpr, bool vec, unsigned blocks, cudaStream_t st, const double* X, int R, int K,
                           int K8, long long rs, int s, __nv_bfloat16* sl, int* ex) {
    switch (tpr) {
        case 1: launch_rows_reg_t<1>(vec, blocks, st, X, R, K, K8, rs, s, sl, ex); break;
        case 2: launch_rows_reg_t<2>(vec, blocks, st, X, R, K, K8, rs, s, sl, ex); break;
        case 4: launch_rows_reg_t<4>(vec, blocks, st, X, R, K, K8, rs, s, sl, ex); break;
        case 8: launch_rows_reg_t<8>(vec, blocks, st, X, R, K, K8, rs, s, sl, ex); break;
        case 16: launch_rows_reg_t<16>(vec, blocks, st, X, R, K, K8, rs, s, sl, ex); break;
        case 32: launch_rows_reg_t<32>(vec, blocks, st, X, R, K, K8, rs, s, sl, ex); break;
        case 64: launch_rows_reg_t<64>(vec, blocks, st, X, R, K, K8, rs, s, sl, ex); break;
        case 128: launch_rows_reg_t<128>(vec, blocks, st, X, R, K, K8, rs, s, sl, ex); break;
        default: launch_rows_reg_t<256>(vec, blocks, st, X, R, K, K8, rs, s, sl, ex); break;
    }
}

cudaError_t oz_split(const double* X, int R, int K, long long rs, long long cs, int s, void* buf, cudaStream_t st) {
    OzView rv{1, {R, 1, 1, 1}, {rs, 0, 0, 0}}, kv{1, {K, 1, 1, 1}, {cs, 0, 0, 0}};
    return oz_split_view(X, R, K, rv, kv, s, buf, st);
}

cudaError_t oz_split_view(const double* X, int R, int K, const OzView& rvh, const OzView& kvh, int s, void* buf,
                          cudaStream_t st) {
    if (R <= 0 || K <= 0 || s < 2 || s > oz::MAX_S || rvh.n < 1 || rvh.n > 4 || kvh.n < 1 || kvh.n > 4)
        return cudaErrorInvalidValue;
    oz::View rv, kv;
    rv.n = rvh.n;
    kv.n = kvh.n;
    for (int a = 0; a < 4; ++a) {
        rv.dim[a] = rvh.dim[a];
        rv.stride[a] = rvh.stride[a];
        kv.dim[a] = kvh.dim[a];
        kv.stride[a] = kvh.stride[a];
    }
    const long long cs = kv.stride[kv.n - 1];
    const int K8 = k8_of(K);
    __nv_bfloat16* sl = (__nv_bfloat16*)buf;
    unsigned long long* mb = (unsigned long long*)((char*)buf + align256((size_t)s * R * K8 * 2));
    int* ex = const_cast<int*>(split_exponents(buf, R, K8, s));
    const int nch = K8 / 8;
    if (cs == 1 && rv.n == 1 && kv.n == 1 && nch <= 4 * 256) {
        int tpr = 1;
        while (tpr * 4 < nch) tpr *= 2;
        const bool vec = ((uintptr_t)X % 16 == 0) && (rv.stride[0] % 2 == 0);
        const unsigned blocks = (unsigned)(((size_t)R * tpr + 255) / 256);
        launch_split_rows_reg(tpr, vec, blocks, st, X, R, K, K8, rv.stride[0], s, sl, ex);
    } else if (cs == 1) {
        cudaError_t e = cudaMemsetAsync(mb, 0, (size_t)R * 8, st);
        if (e != cudaSuccess) return e;
        const int kr = (K + oz::ROWS_KRANGE - 1) / oz::ROWS_KRANGE;
        const unsigned long long b1 = ((unsigned long long)R * kr + 7) / 8, b2 = ((unsigned long long)R * nch + 255) / 256;
        if (b1 > 0x7fffffffull || b2 > 0x7fffffffull) return cudaErrorInvalidValue;
        launch_dep(oz::k_rowmax_rows, (unsigned)b1, 256, 0, st, X, R, K, rv, kv, kr, mb);
        launch_dep(oz::k_split_rows_long, (unsigned)b2, 256, 0, st, X, R, K, K8, rv, kv, s, mb, sl, ex);
    } else if (const int nc = cols_cluster(R, K8)) {
        const int warps = std::min(oz::COLS_ONE_WARPS, ((K8 + 31) / 32 + nc - 1) / nc);
        return launch_dep_cluster(kv.n == 1 ? oz::k_split_cols_one<true> : oz::k_split_cols_one<false>, nc,
                                  (unsigned)((R + 31) / 32 * nc), 32 * warps, 0, st, X, R, K, K8, rv, kv, s, sl, ex);
    } else {
        cudaError_t e = cudaMemsetAsync(mb, 0, (size_t)R * 8, st);
        if (e != cudaSuccess) return e;
        const unsigned rg = (unsigned)((R + 31) / 32);
        const int krange = cols_krange(R, K);
        const unsigned kr = (unsigned)((K + krange - 1) / krange);
        const unsigned long long warps = (unsigned long long)rg * kr;
        const int kspan = std::min(oz::COLS_SPAN, cols_krange(R, K8)), kgroups = (K8 + kspan - 1) / kspan;
        const unsigned long long warps2 = (unsigned long long)rg * kgroups;
        if ((warps + 3) / 4 > 0x7fffffffull || (warps2 + 1) / 2 > 0x7fffffffull) return cudaErrorInvalidValue;
        launch_rowmax_cols((unsigned)((warps + 3) / 4), st, X, R, K, rv, kv, (int)kr, krange, mb);
        const unsigned blocks = (unsigned)((warps2 + 1) / 2);
        launch_dep(kv.n == 1 ? oz::k_split_cols<true> : oz::k_split_cols<false>, blocks, 64, 0, st, X, R, K, K8, rv, kv, s, mb,
                   sl, ex, kspan, kgroups);
    }
    return cudaGetLastError();
}

cudaError_t wait_probe(long long limit_cycles, int arrive, int* err, cudaStream_t st) {
    ++g_launches;
    oz::k_wait_probe<<<1, 64, 0, st>>>(limit_cycles, arrive, err);
    return cudaGetLastError();
}

size_t oz_gemm_ws_bytes(int M, int N, int K, int s, int mode) { return plan_of(M, N, K, s, mode).ws_bytes; }

cudaError_t oz_gemm(int M, int N, int K, int s, const void* Asplit, const void* Bsplit, double alpha, double beta,
                    double* C, int ldc, void* ws, size_t ws_bytes, int* err, cudaStream_t st, int mode) {
    OzView r{1, {M, 1, 1, 1}, {ldc, 0, 0, 0}}, c{1, {N, 1, 1, 1}, {1, 0, 0, 0}};
    return oz_gemm_view(M, N, K, s, Asplit, Bsplit, alpha, beta, C, r, c, ws, ws_bytes, err, st, mode);
}

cudaError_t oz_gemm_view(int M, int N, int K, int s, const void* Asplit, const void* Bsplit, double alpha,
                         double beta, double* C, const OzView& orv, const OzView& ocv, void* ws, size_t ws_bytes,
                         int* err, cudaStream_t st, int mode) {
    if (M <= 0 || N <= 0) return cudaSuccess;
    if (K <= 0 || s < 2 || s > oz::MAX_S || mode < 0 || mode > 2 || (mode == 2 && s != 2))
        return cudaErrorInvalidValue;
    const Plan p = plan_of(M, N, K, s, mode);
    if (p.stages < 2 || p.ws_bytes > ws_bytes) return cudaErrorInvalidValue;
    const int Kp = mode == 2 ? k4_of(K) : k8_of(K);
    CUtensorMap ta, tb;
    if (!make_map(&ta, Asplit, M, Kp, s, oz::BM, mode == 2) || !make_map(&tb, Bsplit, N, Kp, s, p.bn, mode == 2))
        return cudaErrorInvalidValue;
    oz::GemmArgs g{};
    g.M = M;
    g.N = N;
    g.nkb = p.nkb;
    g.kb_per_split = p.kb_per_split;
    g.s = s;
    g.stages = p.stages;
    g.a_bytes = p.a_bytes;
    g.stage_bytes = p.stage_bytes;
    g.eA = mode == 2 ? split_tf32_exponents(Asplit, M, Kp) : split_exponents(Asplit, M, Kp, s);
    g.eB = mode == 2 ? split_tf32_exponents(Bsplit, N, Kp) : split_exponents(Bsplit, N, Kp, s);
    g.direct = p.ksplit == 1;
    g.alpha = alpha;
    g.beta = beta;
    g.C = C;
    g.out_r.n = orv.n;
    g.out_c.n = ocv.n;
    for (int a = 0; a < 4; ++a) {
        g.out_r.dim[a] = orv.dim[a];
        g.out_r.stride[a] = orv.stride[a];
        g.out_c.dim[a] = ocv.dim[a];
        g.out_c.stride[a] = ocv.stride[a];
    }
    // Output columns that lie together are stored 32 or 16 bytes at a time: a
    // lane holds a row, and 8-byte stores to 32 rows left every sector written
    // in four parts (262144 x 192 x 64, row-major: 415 us).  Groups of `vec`
    // columns must be contiguous and aligned for every row.
    g.w = oz::Weights{1 << 20, 1 << 22, 1 << 28, 1};
    g.plain = alpha == 1.0 && beta == 0.0;
    // The exact-level epilogue holds a column's offset in 32 bits (in 64 it spilled:
    // 262144 x 192 x 64 227 -> 241 us): views with a negative or longer one are
    // refused, unless the product goes by the split partials.  No caller has one:
    // the outputs of a handle that fits the device end far below 2^32 elements.
    if (mode == 0 && g.direct) {
        unsigned long long last = 0;
        for (int a = 0; a < ocv.n; ++a) {
            if (ocv.dim[a] < 2) continue;
            if (ocv.stride[a] < 0 || ocv.stride[a] >= (1ll << 32)) return cudaErrorInvalidValue;
            last += (unsigned long long)(ocv.dim[a] - 1) * (unsigned long long)ocv.stride[a];
            if (last >= (1ull << 32)) return cudaErrorInvalidValue;
        }
    }
    g.vec = 1;
    if (g.plain)
        for (int v : {4, 2}) {
            bool ok = (uintptr_t)C % (8 * v) == 0 && ocv.stride[ocv.n - 1] == 1 && (ocv.n == 1 || ocv.dim[ocv.n - 1] % v == 0);
            for (int a = 0; a < ocv.n - 1; ++a) ok = ok && ocv.stride[a] % v == 0;
            for (int a = 0; a < orv.n; ++a) ok = ok && (orv.dim[a] == 1 || orv.stride[a] % v == 0);
            if (ok) {
                g.vec = v;
                break;
            }
        }
    g.Mpad = p.m_tiles * oz::BM;
    g.m_tiles = p.m_tiles;
    g.n_tiles = p.n_tiles;
    g.Npad = p.n_tiles * p.bn;
    if (!g.direct) g.PZ = (long long*)ws;
    g.err = err;
    g.wait_limit = oz::WAIT_LIMIT_CYCLES;
    cudaError_t e;
    switch (p.nb16) {
        case 1: e = launch_mode<1>(mode, p, ta, tb, g, st); break;
        case 2: e = launch_mode<2>(mode, p, ta, tb, g, st); break;
        case 3: e = launch_mode<3>(mode, p, ta, tb, g, st); break;
        case 4: e = launch_mode<4>(mode, p, ta, tb, g, st); break;
        case 5: e = launch_mode<5>(mode, p, ta, tb, g, st); break;
        case 6: e = launch_mode<6>(mode, p, ta, tb, g, st); break;
        case 7: e = launch_mode<7>(mode, p, ta, tb, g, st); break;
        case 8: e = launch_mode<8>(mode, p, ta, tb, g, st); break;
        default: e = launch_mode<9>(mode, p, ta, tb, g, st); break;
    }
    if (e != cudaSuccess || g.direct) return e;
    size_t blocks = ((size_t)M * N + 255) / 256;
    if (blocks > 152 * 16) blocks = 152 * 16;
    launch_dep(oz::k_oz_combine, (unsigned)blocks, 256, 0, st, g.PZ, p.ksplit, K > oz::COMBINE_INT64_K ? 1 : 0, g.Mpad, g.Npad,
                                                        M, N, g.eA, g.eB, alpha, beta, C, g.out_r, g.out_c);
    return cudaGetLastError();
}

}  // namespace ctm
