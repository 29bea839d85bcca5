// oz.cuh -- helpers of the exact-splitting (Ozaki) products: balanced digits
// of a scaled FP64 value in base 2^beta, their exact BF16 encoding, powers of
// two, and the canonical K-major layout of one 16-column operand chunk.
#pragma once

#include <cstdint>
#include <cstring>

#include <cuda_runtime.h>

// Element offset of (row, k) inside a 16-column chunk in the canonical K-major
// layout: 8 x 8 core matrices of 16-byte rows, the two core matrices of a row
// group 64 elements apart, row groups 128 elements apart.
static __host__ __device__ __forceinline__ int oz_kofs(int row, int k)
{
    return (row >> 3) * 128 + (k >> 3) * 64 + (row & 7) * 8 + (k & 7);
}

// Balanced base-2^beta digits of I, most significant first: I = sum_s d[s] 2^(beta (S-1-s)).
static __host__ __device__ __forceinline__ int oz_digit_step(long long &I, int beta)
{
    const long long mask = (1ll << beta) - 1, half = 1ll << (beta - 1);
    long long r = I & mask;
    I >>= beta;
    if (r > half) {
        r -= (1ll << beta);
        I += 1;
    }
    return (int)r;
}

// The same digits without the carry chain: with 2^(beta-1) - 1 added in every
// place but the first, place q of I + bias holds digit + 2^(beta-1) - 1, between 0
// and 2^beta - 1, and the first place the first digit.
static __host__ __device__ constexpr long long oz_digit_bias(int S, int beta)
{
    long long c = 0;
    for (int q = 0; q < S - 1; ++q) c += ((1ll << (beta - 1)) - 1) << (beta * q);
    return c;
}
// Digit sd as a float, without a conversion: the place's bits are put into the
// mantissa of 2^23 (the first digit, signed, into that of 1.5 2^23) and one
// subtraction leaves the digit.  Its upper 16 bits are the digit's BF16.
static __host__ __device__ __forceinline__ float oz_digit_f32(long long J, int S, int beta, int sd)
{
    const uint32_t r = (uint32_t)(J >> (beta * (S - 1 - sd)));
    const uint32_t u = sd == 0 ? 0x4B400000u + r : 0x4B000000u | (r & ((1u << beta) - 1));
#ifdef __CUDA_ARCH__
    const float f = __uint_as_float(u);
#else
    float f;
    std::memcpy(&f, &u, 4);
#endif
    return f - (sd == 0 ? 12582912.f : 8388608.f + (float)((1 << (beta - 1)) - 1));
}
static __host__ __device__ __forceinline__ int oz_digit_at(long long J, int S, int beta, int sd)
{
    return (int)oz_digit_f32(J, S, beta, sd);
}

// BF16 bits of a small integer (|d| <= 256): exact.
static __host__ __device__ __forceinline__ uint16_t oz_bf16_int(int d)
{
    const float f = (float)d;
#ifdef __CUDA_ARCH__
    const uint32_t u = __float_as_uint(f);
#else
    uint32_t u;
    std::memcpy(&u, &f, 4);
#endif
    return (uint16_t)(u >> 16);
}

// 2^e as a double (normal range).
static __host__ __device__ __forceinline__ double oz_pow2(int e)
{
    const long long b = (long long)(e + 1023) << 52;
#ifdef __CUDA_ARCH__
    return __longlong_as_double(b);
#else
    double d;
    std::memcpy(&d, &b, 8);
    return d;
#endif
}


// ---------------------------------------------------------------------------
// Integer-pipe versions of the two conversions around the digit products, so
// that they leave the FP64 pipe free (results bit for bit those of the FP64
// instructions they replace).

// round-half-even(v 2^k) for finite v with |v 2^k| < 2^62: the value of
// __double2ll_rn(v * 2^k) (the product being exact), from v's bit pattern.
static __host__ __device__ __forceinline__ long long oz_rint_pow2(double v, int k)
{
#ifdef __CUDA_ARCH__
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
#else
    unsigned long long b;
    std::memcpy(&b, &v, 8);
#endif
    const int e = (int)((b >> 52) & 0x7ffull);
    if (e == 0) return 0;  // zero or subnormal: far below 1/2 after any scale used here
    const long long m = (long long)((b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull);  // v = m 2^(e - 1075)
    const int s = e - 1075 + k;
    long long r;
    if (s >= 0) {
        r = m << s;
    } else if (s < -53) {
        r = 0;  // m 2^s < 1/2
    } else {
        const int sh = -s;
        r = m >> sh;
        const long long rem = m & ((1ll << sh) - 1), half = 1ll << (sh - 1);
        if (rem > half || (rem == half && (r & 1))) r += 1;
    }
    return (b >> 63) ? -r : r;
}

// The double nearest (ties to even) to (hi 2^w + lo) 2^p, for |hi| < 2^62,
// |lo| < 2^62, w <= 32 and a result in the normal range: the value of
// fma((double)hi, 2^w, (double)lo) * 2^p (one rounding, an exact power-of-two
// scale), built from the integer bits.
static __host__ __device__ __forceinline__ double oz_i64x2_scaled_w(long long hi, long long lo, int w, int p)
{
    // X = hi 2^w + lo, |X| < 2^95, as a sign and a magnitude of at most 95 bits
    const __int128 X = (__int128)hi * ((__int128)1 << w) + (__int128)lo;
    if (X == 0) return 0.0;
    const bool neg = X < 0;
    const unsigned __int128 u = neg ? (unsigned __int128)(-X) : (unsigned __int128)X;
    const unsigned long long uh = (unsigned long long)(u >> 64), ul = (unsigned long long)u;
#ifdef __CUDA_ARCH__
    const int lz = uh ? __clzll((long long)uh) : 64 + __clzll((long long)ul);
#else
    const int lz = uh ? __builtin_clzll(uh) : 64 + __builtin_clzll(ul);
#endif
    const int nb = 128 - lz;  // bits of |X|
    unsigned long long m;
    int e2;  // |X| rounded = m 2^e2, 2^52 <= m < 2^53
    if (nb <= 53) {
        m = ul << (53 - nb);
        e2 = nb - 53;
    } else {
        int sh = nb - 53;
        const unsigned __int128 one = 1;
        m = (unsigned long long)(u >> sh);
        const unsigned __int128 rem = u & ((one << sh) - 1), half = one << (sh - 1);
        if (rem > half || (rem == half && (m & 1ull))) m += 1;
        if (m == (1ull << 53)) {
            m >>= 1;
            sh += 1;
        }
        e2 = sh;
    }
    unsigned long long bits = ((unsigned long long)(e2 + p + 52 + 1023) << 52) | (m & 0xFFFFFFFFFFFFFull);
    if (neg) bits |= 1ull << 63;
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)bits);
#else
    double d;
    std::memcpy(&d, &bits, 8);
    return d;
#endif
}

// The same with w = 32 (the embedding layers' groups).
static __host__ __device__ __forceinline__ double oz_i64x2_scaled(long long hi, long long lo, int p)
{
    return oz_i64x2_scaled_w(hi, lo, 32, p);
}

// oz_i64x2_scaled_w for |hi| < 2^61, |lo| < 2^60, 1 <= w <= 32 and a result in the
// normal range, in 64-bit arithmetic: hi is shifted up by k <= w as far as 62 bits
// allow, lo's bits below 2^(w - k) are kept as a sticky bit (they matter only when
// the sum has 62 bits, of which 53 are kept), and one rounding to nearest even
// leaves the value of fma((double)hi, 2^w, (double)lo) * 2^p bit for bit.
static __host__ __device__ __forceinline__ double oz_i64x2_round(long long hi, long long lo, int w, int p)
{
    const unsigned long long ah = (unsigned long long)(hi < 0 ? -hi : hi);
#ifdef __CUDA_ARCH__
    const int lzh = __clzll((long long)ah);
#else
    const int lzh = ah ? __builtin_clzll(ah) : 64;
#endif
    const int k = lzh - 2 < w ? lzh - 2 : w, d = w - k;  // |hi 2^k| < 2^62
    const long long kept = lo >> d;
    const long long m = (hi << k) + kept;
    const unsigned long long sticky = (unsigned long long)(lo - (kept << d)) != 0ull ? 1ull : 0ull;
    const unsigned long long u0 = (unsigned long long)m | sticky;
    const bool neg = (long long)u0 < 0;
    const unsigned long long u = neg ? 0ull - u0 : u0;
    if (u == 0) return 0.0;
#ifdef __CUDA_ARCH__
    const int lz = __clzll((long long)u);
#else
    const int lz = __builtin_clzll(u);
#endif
    const int sh = 11 - lz;  // u has 64 - lz bits
    unsigned long long r;    // 53 bits (or 2^53 after rounding up)
    if (sh <= 0) r = u << -sh;
    else r = (u + ((1ull << (sh - 1)) - 1ull) + ((u >> sh) & 1ull)) >> sh;
    // r 2^sh 2^d 2^p; the hidden bit of r adds one to the exponent field
    const unsigned long long bits =
        ((unsigned long long)(sh + d + p + 1074) << 52) + r + (neg ? 0x8000000000000000ull : 0ull);
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)bits);
#else
    double v;
    std::memcpy(&v, &bits, 8);
    return v;
#endif
}
