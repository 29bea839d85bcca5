// fit_oz.cu -- the fitting net N_a (Eqs. fitting, fitting-detail; one net per
// centre type, Remark 1), forward and backward to the descriptor, with FP64
// accuracy and every GEMM on the 5th-generation tensor cores.
//
// Exact splitting (Ozaki's scheme).  A GEMM Y = X W with FP64 operands is
// written with a power-of-two scale per row of X (2^e_r >= max_k |X_rk|) and
// per column of W (2^f_n), and the scaled values as S signed digits in base
// 2^beta:
//   X_rk = 2^e_r sum_s a_s,rk 2^(-beta s),   W_kn = 2^f_n sum_t b_t,kn 2^(-beta t),
// with |a_1|, |b_1| <= 2^beta and |a_s|, |b_t| <= 2^(beta-1) for s, t >= 2
// (balanced digits of the integers round(X_rk 2^(beta S - e_r))).  Then
//   Y_rn = 2^(e_r + f_n) sum_g 2^(-beta g) C_g,   C_g = sum_{s+t=g} A_s B_t,
// summed over g = 2 .. S+1 (the terms beyond are below the expansions' own
// precision: FP64 rounding for the 55-bit plans of the FP64 mode, 2^-28
// relative for the 28-bit plans of the split mixed mode).  A digit
// is an integer of at most 8 bits, exact in BF16; every product is exact in
// FP32, and while
//   K 4^(beta-1) (S + 2) < 2^24
// every partial sum of every C_g is below 2^24: the FP32 tensor-core
// accumulators hold C_g exactly, in any summation order.  A longer contraction
// is cut into segments that satisfy this, added up in int64 (FP64 mode: 8 digits
// of 7 bits throughout, 36 products per 16 columns and 8 planes to read; 66 and
// 11 for the 1,600-long first layer when one segment had to hold it, with 5-bit
// digits).  The result is the exact product of the digit expansions, rounded
// once into FP64, and is reproducible bit for bit.
//
// Kernels.  k_oz_split: digits of the activations of a 128-atom tile of one
// type, S BF16 matrices in the canonical K-major layout of the MMA A operand
// (16-column chunks); k_oz_wsplit: the weights', once per set of parameters.
// k_oz_gemm: persistent over (tile, 32-column chunk of Y); a copy warp streams
// the digit chunks of A and W (cp.async.bulk, a 4-stage ring on mbarriers), an
// MMA warp issues the S(S+1)/2 digit products of 128 x 32 x 16 of a chunk as S
// MMAs into S group accumulators in tensor memory, and 8 warps combine the groups exactly, round
// once and apply the layer's bias, tanh and skip (forward) or the skip gradient
// (backward).  Every wait is bounded; on a timeout the kernel sets
// DPF_MMA_TIMEOUT, waits for its copies and MMAs, frees tensor memory and
// returns.
//
// Measured per evaluation (12,288 water atoms): the six GEMMs 2.8 -> 1.0 ms, the
// six splits 0.74 -> 0.30 ms; 192 atoms: the whole fitting net 0.96 -> 0.24 ms.
// One elected lane of a whole warp issues: behind `threadIdx.x == 0` the same MMAs
// took 139 cycles each instead of 97 in the former kernel.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <vector>

#include "dp_internal.cuh"
#include "tc.cuh"
#include "oz.cuh"

namespace {

constexpr int OZ_NST = 4;                   // pipeline stages (40 KB each at 8 digits)
constexpr int OZ_THREADS = 320;             // 8 epilogue warps, the MMA warp, the copy warp
// chunks whose sums stay exact at 8 digits of 7 bits: 400 columns, 400 4^6 10 < 2^24
constexpr int OZ_SEG = 16777215 / (4096 * 10) / DP_OZ_KC;
constexpr uint32_t OZ_TAB_BYTES = DP_TANH_NINT * DP_TANH_STRIDE * 8;
static_assert(OZ_TAB_BYTES % 16 == 0, "bulk copy of the tanh table");
constexpr int OZ_A_BLK = DP_OZ_TILE * DP_OZ_KC;  // elements of one A digit chunk (128 x 16)
constexpr int OZ_B_BLK = DP_OZ_NC * DP_OZ_KC;    // elements of one W digit chunk (32 x 16)
constexpr int OZ_WSEG = 16;                      // chunks of a weight gradient's segment (256 atoms)
constexpr int OZ_KEEP = 256;                     // columns of a row that k_oz_split may keep between its passes

struct TileRef {
    int a, first, cnt;
};

// Tile index -> (type, first row of the type-sorted rows, rows); a = -1 past the
// end.  Every centre has rpa rows.
__device__ __forceinline__ TileRef oz_tile(int tl, const int32_t *__restrict__ type_start, int ntypes, int rpa)
{
    TileRef t{-1, 0, 0};
    for (int a = 0; a < ntypes; ++a) {
        const int n_a = (type_start[a + 1] - type_start[a]) * rpa;
        const int tiles = (n_a + DP_OZ_TILE - 1) / DP_OZ_TILE;
        if (tl < tiles) {
            t.a = a;
            t.first = type_start[a] * rpa + tl * DP_OZ_TILE;
            t.cnt = min(DP_OZ_TILE, n_a - tl * DP_OZ_TILE);
            return t;
        }
        tl -= tiles;
    }
    return t;
}

// Row of a matrix [N rpa][.] that a row of the type-sorted rows stands for.
__device__ __forceinline__ int oz_row(const int32_t *__restrict__ type_perm, int q, int rpa)
{
    return rpa == 1 ? type_perm[q] : type_perm[q / rpa] * rpa + q % rpa;
}

// Exponent of a row or column from the bits of its largest |x|: 2^e > |x|.  zero: its
// digits are 0 (nothing there, or below 2^-960).  An infinity or NaN gives OZ_NAN,
// for which k_oz_gemm writes NaN.
constexpr int OZ_NAN = 30000;
__device__ __forceinline__ int oz_exponent(unsigned long long mx, int bS, bool &zero)
{
    zero = true;
    if (mx == 0) return 0;
    if (mx >= 0x7ff0000000000000ull) return OZ_NAN;
    int e;
    frexp(__longlong_as_double((long long)mx), &e);
    if (e < bS - 1020) return 0;
    zero = false;
    return e;
}

// ------------------------------------------------------------------ split --

struct OzSplitArgs {
    int mode;  // 0: x = src; 1: x = src (1 - t^2); 2: x = w_out (1 - t^2) and E_i = src . w_out + b_out
    const double *src;
    int lds;
    const double *tv;
    int ldt;
    const double *wout[DP_MAX_TYPES];
    const double *bout[DP_MAX_TYPES];
    double *Ei;
    int K, nK, beta, S;
    const int32_t *type_perm, *type_start;
    int ntypes, rpa;
    uint16_t *a;
    int32_t *aexp;
    int64_t a_stride;
    int32_t *cnt;  // part counters of the GEMM that follows (zeroed here)
    int ncnt;
    int vec;       // rows start on 16 bytes
    int keep;      // columns of a row kept in shared memory (0: none)
};

// Digits sd of 8 values (with their bias, oz_digit_bias) as 8 BF16.
template <int S, int B>
__device__ __forceinline__ uint4 oz_pack_digits(const long long (&J)[8], int sd)
{
    uint32_t f[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) f[q] = __float_as_uint(oz_digit_f32(J[q], S, B, sd));
    return make_uint4(__byte_perm(f[0], f[1], 0x7632), __byte_perm(f[2], f[3], 0x7632),
                      __byte_perm(f[4], f[5], 0x7632), __byte_perm(f[6], f[7], 0x7632));
}

// One CTA per group of 8 rows of a tile (a row group of the canonical layout):
// warp w takes the exponent (and output-layer energy) of row w, then every
// digit plane of a 16-column chunk is written as one contiguous 256-byte block:
// lane = row (0..7) + 8 * (column half) + 16 * (chunk parity), the warps
// striding over the chunk pairs.  (One warp per row group, rows one after the
// other, took 277 us for the descriptors of 12,288 water atoms and 181 us for
// 192: a chain of dependent loads on few warps.)  When the row groups are few,
// gridDim.y CTAs share one: each finds the exponents, and writes its share of the
// chunks.  Bound by instruction issue: the value's bits are rounded to an integer
// on the integer pipe, its digits read from their places without a carry chain
// and converted by one FP32 subtraction.  Products (1 - t^2) x of up to 256
// columns stay in shared memory between the passes (formed twice, 240 columns of
// 12,288 atoms took 52 us, now 43; plain values are read again: keeping them took
// 28 instead of 26 us).  With a chain, a conversion instruction
// per digit and 8-byte loads the descriptors of 12,288 atoms took 175 us and
// those of 192 atoms 32 us; now 113 and 15 us.
template <int S, int B>
__global__ void __launch_bounds__(256) k_oz_split(OzSplitArgs p)
{
    __shared__ int e_s[8];
    __shared__ int nz_s[8];
    extern __shared__ __align__(16) double v_s[];  // kept rows
    const bool keep = p.keep != 0;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tl = blockIdx.x / (DP_OZ_TILE / 8), r0 = (blockIdx.x % (DP_OZ_TILE / 8)) * 8;
    if (blockIdx.x + blockIdx.y == 0)
        for (int q = tid; q < p.ncnt; q += 256) p.cnt[q] = 0;
    const TileRef T = oz_tile(tl, p.type_start, p.ntypes, p.rpa);
    if (T.a < 0) return;
    const double *wo = p.mode == 2 ? p.wout[T.a] : nullptr;
    constexpr int bS = B * S;

    // value of column k of atom i (0 past the row's end or the tile's atoms)
    auto value = [&](int i, int k) -> double {
        if (i < 0 || k >= p.K) return 0.0;
        double v = p.mode == 2 ? wo[k] : p.src[(size_t)i * p.lds + k];
        if (p.mode != 0) {
            const double t = p.tv[(size_t)i * p.ldt + k];
            v *= fma(-t, t, 1.0);
        }
        return v;
    };

    {
        const int r = r0 + warp;
        const int i = r < T.cnt ? oz_row(p.type_perm, T.first + r, p.rpa) : -1;
        if (p.mode == 2) {
            double e = 0.0;
            if (i >= 0)
                for (int k = lane; k < p.K; k += 32) e = fma(p.src[(size_t)i * p.lds + k], wo[k], e);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
            if (i >= 0 && lane == 0 && blockIdx.y == 0) p.Ei[i] = *p.bout[T.a] + e;
        }
        // largest |x| by its bits; a row with an infinity or NaN gives NaN
        unsigned long long mx = 0;
        auto larger = [&](double v) {
            const unsigned long long b = (unsigned long long)__double_as_longlong(fabs(v));
            mx = b > mx ? b : mx;
        };
        int k0 = 0;  // columns taken two at a time
        if (keep) {
#pragma unroll 4
            for (int k = lane; k < p.nK * DP_OZ_KC; k += 32) {
                const double v = value(i, k);
                v_s[warp * p.keep + k] = v;
                larger(v);
            }
            k0 = p.K;
        } else if (p.mode == 0 && p.vec && i >= 0) {
            const double *x = p.src + (size_t)i * p.lds;
            k0 = p.K & ~1;
#pragma unroll 8
            for (int k = 2 * lane; k < k0; k += 64) {
                const double2 v = *reinterpret_cast<const double2 *>(x + k);
                larger(v.x);
                larger(v.y);
            }
        }
#pragma unroll 4
        for (int k = k0 + lane; k < p.K; k += 32) larger(value(i, k));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long q = __shfl_xor_sync(0xffffffffu, mx, o);
            mx = q > mx ? q : mx;
        }
        if (lane == 0) {
            bool zero;
            const int e = oz_exponent(mx, bS, zero);
            e_s[warp] = e;
            nz_s[warp] = !zero;
            if (blockIdx.y == 0) p.aexp[(size_t)tl * DP_OZ_TILE + r] = e;
        }
    }
    __syncthreads();

    // digits: lane handles row r0 + (lane & 7), columns kh*8 .. kh*8+7 of chunk kc
    const int jr = lane & 7, kh = (lane >> 3) & 1;
    const int r = r0 + jr;
    const int i = r < T.cnt && nz_s[jr] ? oz_row(p.type_perm, T.first + r, p.rpa) : -1;
    const int sh = bS - e_s[jr];
    uint16_t *out = p.a + (size_t)tl * p.a_stride;
    const int ofs = oz_kofs(r, kh * 8);
    for (int kc = 2 * (warp + 8 * blockIdx.y) + (lane >> 4); kc < p.nK; kc += 16 * gridDim.y) {
        const int k8 = kc * DP_OZ_KC + kh * 8;
        long long J[8];
        double v[8];
        if (keep) {
#pragma unroll
            for (int q = 0; q < 8; q += 2) {
                const double2 u = *reinterpret_cast<const double2 *>(v_s + jr * p.keep + k8 + q);
                v[q] = i < 0 ? 0.0 : u.x;
                v[q + 1] = i < 0 ? 0.0 : u.y;
            }
        } else if (p.vec && i >= 0 && k8 + 8 <= p.K) {
            const double *x = p.mode == 2 ? wo + k8 : p.src + (size_t)i * p.lds + k8;
            if (p.mode == 2) {
#pragma unroll
                for (int q = 0; q < 8; ++q) v[q] = x[q];
            } else {
#pragma unroll
                for (int q = 0; q < 8; q += 2) {
                    const double2 u = *reinterpret_cast<const double2 *>(x + q);
                    v[q] = u.x;
                    v[q + 1] = u.y;
                }
            }
            if (p.mode != 0) {
                const double *tv = p.tv + (size_t)i * p.ldt + k8;
#pragma unroll
                for (int q = 0; q < 8; q += 2) {
                    const double2 t = *reinterpret_cast<const double2 *>(tv + q);
                    v[q] *= fma(-t.x, t.x, 1.0);
                    v[q + 1] *= fma(-t.y, t.y, 1.0);
                }
            }
        } else {
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = value(i, k8 + q);
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) J[q] = oz_rint_pow2(v[q], sh) + oz_digit_bias(S, B);
#pragma unroll
        for (int sd = 0; sd < S; ++sd)
            *reinterpret_cast<uint4 *>(out + ((size_t)kc * S + sd) * OZ_A_BLK + ofs) = oz_pack_digits<S, B>(J, sd);
    }
}

cudaError_t launch_split(cudaStream_t st, OzSplitArgs &a, int tiles, int num_sms)
{
    const auto odd = [](const void *p, int ld) { return ((uintptr_t)p & 15) != 0 || (ld & 1) != 0; };
    a.vec = !((a.mode != 2 && odd(a.src, a.lds)) || (a.mode != 0 && odd(a.tv, a.ldt)));
    // rows 16 bytes apart in the banks
    a.keep = a.mode != 0 && a.K <= OZ_KEEP ? a.nK * DP_OZ_KC + 2 : 0;
    const size_t smem = (size_t)a.keep * 8 * sizeof(double);
    const int groups = tiles * (DP_OZ_TILE / 8);
    // up to 4 CTAs per SM; 16 chunks are one pass of a CTA
    const dim3 grid(groups, std::max(1, std::min(4 * num_sms / groups, (a.nK + 15) / 16)));
    if (a.S == 8 && a.beta == 7) k_oz_split<8, 7><<<grid, 256, smem, st>>>(a);
    else if (a.S == 4 && a.beta == 7) k_oz_split<4, 7><<<grid, 256, smem, st>>>(a);
    else if (a.S == 5 && a.beta == 6) k_oz_split<5, 6><<<grid, 256, smem, st>>>(a);
    else return cudaErrorInvalidValue;
    return cudaGetLastError();
}

// ------------------------------------------------------------------- gemm --

struct OzGemmArgs {
    const uint16_t *a;
    const int32_t *aexp;
    int64_t a_stride;
    const uint16_t *w;
    const int32_t *wexp;
    OzGemm g;
    const int32_t *type_perm, *type_start;
    int ntypes, rpa;
    int skip;     // skip kind of the layer
    int skip_in;  // input width of the layer
    const double *bias[DP_MAX_TYPES];
    const double *hin;  // forward: layer input (skip); backward: dL/dh_l per atom
    int ldh;
    const double *gbc[DP_MAX_TYPES];  // backward: dL/dh_l broadcast per type (last layer), else null
    double *tout;
    double *hout;
    int ldo;
    const double *tanh_tab;
    int32_t *status;
    int units;  // (tile, column chunk) pairs, tiles past the last atom included
    const double *tin;  // epi 2: tanh values of the value pass
    // weight gradients Y = X^T Z, contracted over the atoms of each type (epi 3)
    int wg, rows, nq;                 // 1; rows of Y and their tiles
    int64_t out_off[DP_MAX_TYPES];    // of a type's Y in hout
    const double *x, *z;              // X and Z
    int ldx, ldz, one;                // one: the last row of Y is the sum of Z's rows (else 0)
    // contraction shared by `parts` CTAs: their chain sums [unit][32][256 threads], arrivals per (pair, warp)
    int parts;
    long long *part;
    int32_t *cnt;
};

// One unit of k_oz_gemm: a 128-row tile of the A operand and a 32-column chunk of Y.
struct OzUnit {
    int a, tl, nchunk, nK, nseg, seg;
    int first, cnt;             // atoms of the tile; wg: first atom, atoms (of the type's, in type order)
    int sg0;                    // wg: first segment, counted over the types
    const uint16_t *as, *bs;    // digits of the first K-chunk
    size_t astep, bstep;        // ... to the next
};

__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *mbar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
            tc::smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(tc::smem_u32(mbar))
        : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t *mbar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(tc::smem_u32(mbar)), "r"(bytes)
                 : "memory");
}

// y 2^e: one multiplication while 2^e is a normal number (exact, or rounded
// once when the product is subnormal, as ldexp rounds it), ldexp otherwise
__device__ __forceinline__ double scale2(double y, int e)
{
    return (e >= -1022 && e <= 1023) ? y * oz_pow2(e) : ldexp(y, e);
}

template <int S, bool WG>
__device__ __forceinline__ bool oz_unit(const OzGemmArgs &p, int u, OzUnit &U)
{
    const OzGemm &g = p.g;
    const int ks = u % p.parts;
    u /= p.parts;
    if constexpr (!WG) {
        U.tl = u / g.nN;
        U.nchunk = u - U.tl * g.nN;
        const TileRef T = oz_tile(U.tl, p.type_start, p.ntypes, p.rpa);
        U.a = T.a;
        U.first = T.first;
        U.cnt = T.cnt;
        U.nK = g.nK;
        U.seg = g.seg;
        U.astep = (size_t)S * OZ_A_BLK;
        U.bstep = (size_t)S * OZ_B_BLK;
        U.as = p.a + (size_t)U.tl * p.a_stride;
        U.bs = p.w + g.w_off[T.a < 0 ? 0 : T.a] + (size_t)U.nchunk * g.nK * U.bstep;
    } else {
        // chunks of 16 atoms, type after type; [chunk][tile or column chunk][S][block]
        const int per = p.nq * g.nN;
        U.a = u / per;
        U.tl = (u - U.a * per) / g.nN;
        U.nchunk = u - U.a * per - U.tl * g.nN;
        int kb = 0;
        U.sg0 = 0;
        for (int a = 0; a < U.a; ++a) {
            const int nk = (p.type_start[a + 1] - p.type_start[a] + DP_OZ_KC - 1) / DP_OZ_KC;
            kb += nk;
            U.sg0 += (nk + OZ_WSEG - 1) / OZ_WSEG;
        }
        U.nK = (p.type_start[U.a + 1] - p.type_start[U.a] + DP_OZ_KC - 1) / DP_OZ_KC;
        U.seg = OZ_WSEG;
        U.first = p.type_start[U.a];
        U.cnt = p.type_start[U.a + 1] - U.first;
        U.astep = (size_t)p.nq * S * OZ_A_BLK;
        U.bstep = (size_t)g.nN * S * OZ_B_BLK;
        U.as = p.a + kb * U.astep + (size_t)U.tl * S * OZ_A_BLK;
        U.bs = p.w + kb * U.bstep + (size_t)U.nchunk * S * OZ_B_BLK;
    }
    if (p.parts > 1) {
        int per = (U.nK + p.parts - 1) / p.parts;
        if constexpr (WG) per = (per + OZ_WSEG - 1) / OZ_WSEG * OZ_WSEG;  // whole segments
        const int k0 = ks * per;
        if constexpr (WG) {
            U.sg0 += k0 / OZ_WSEG;
            U.first += k0 * DP_OZ_KC;
            U.cnt -= k0 * DP_OZ_KC;
        }
        U.as += k0 * U.astep;
        U.bs += k0 * U.bstep;
        U.nK = max(0, min(U.nK - k0, per));
    }
    U.nseg = (U.nK + U.seg - 1) / U.seg;
    return U.a >= 0;
}

// Entries of a weight gradient that the digits of a segment may not carry.  The
// digit product of n atoms errs by about 2^-58 sqrt(n) of the two columns' powers
// of two 2^e, 2^f (the groups left out); a chain of FP64 FMAs by 2^-54 or more of the
// products' size, which is far below 2^(e+f) when the columns have their outliers
// at different atoms.  A column's level l says that three quarters of its values
// are at least 2^(e-l).  The digits stand where X's column is even (OZ_EVEN; normal
// deviates have 4, a few per cent 5 or 6): Z's outliers then meet values of 2^(e-l);
// where the two levels are small together; or where the result itself is at least
// an eighth of 2^(e+f).  The others are summed from the FP64 values.  An even Z
// alone is not enough: an atom with an outlier in X has saturated units, whose Z is 0.
constexpr int OZ_EVEN = 5;
constexpr int OZ_LVL_BITS = 5;  // exponent and level in one word; level -16: zeros, NaN
__device__ __forceinline__ bool oz_digits_stand(double y, int vx, int vz)
{
    constexpr int sh = 32 - OZ_LVL_BITS;
    const int lx = (vx << sh) >> sh, lz = (vz << sh) >> sh;
    if (lx <= OZ_EVEN || lx + lz <= 2 * OZ_EVEN) return true;
    const int ey = (int)((__double_as_longlong(y) >> 52) & 0x7ff) - 1023;  // |y| >= 2^ey
    return ey >= (vx >> OZ_LVL_BITS) + (vz >> OZ_LVL_BITS) - 3;
}
// Row k, columns f .. f + 15, over na atoms of a segment by the whole warp: lanes on
// the atoms, then a transposing tree that leaves column f + n on lanes 2n, 2n + 1.
// (An entry at a time on its own lane held the warp up for 70 k cycles of dependent
// loads, and a few entries in 10,000 took the GEMM from 290 to 640 us.)
__device__ __noinline__ double oz_wdot(const OzGemmArgs &p, int at0, int na, int k, int f)
{
    const int lane = threadIdx.x & 31;
    double v[16];
#pragma unroll
    for (int n = 0; n < 16; ++n) v[n] = 0.0;
#pragma unroll 2
    for (int q = lane; q < na; q += 32) {
        const size_t i = p.type_perm[at0 + q];
        const double x = k < p.rows - 1 ? p.x[i * p.ldx + k] : p.one ? 1.0 : 0.0;
        const double *z = p.z + i * p.ldz + f;
#pragma unroll
        for (int n = 0; n < 16; ++n)
            if (f + n < p.g.N) v[n] = fma(x, z[n], v[n]);
    }
#pragma unroll
    for (int w = 16, m = 8; w >= 2; w >>= 1, m >>= 1) {
        const bool up = (lane & w) != 0;
#pragma unroll
        for (int n = 0; n < m; ++n) {
            const double send = up ? v[n] : v[m + n], keep = up ? v[m + n] : v[n];
            v[n] = keep + __shfl_xor_sync(0xffffffffu, send, w);
        }
    }
    return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

// Persistent, one CTA per SM over the units (tile, 32-column chunk of Y) in
// order, so that the CTAs at work share a tile's digits in L2.  Warps 0-7: the
// epilogue (two warps per quarter of the tensor memory's lanes, 16 columns
// each); warp 8 issues the MMAs, warp 9 the copies.  The group accumulators are
// doubled (2 x 256 columns): the epilogue of one segment runs beside the MMAs
// of the next.  A contraction longer than the accumulators hold exactly is cut
// into segments of g.seg chunks, which the epilogue adds up in int64.
//
// Bounds, per unit of a 240-long contraction at S = 8: 15 chunks of 1,152
// accumulator columns at half a cycle = 8.6 k cycles of MMAs; 40 KB of copies per
// chunk, 10.3 k at the 60 B/clk that large bulk copies reach alone; with the FP64
// tanh 20 k cycles of FP64 pipe.  As 36 MMAs of N = 32 per chunk (20 cycles each
// with A in the collector, 40 without) the chunk took a fifth longer: the first
// layer of 12,288 atoms 392 us, now 324, the gradient to the descriptor 332 and
// 274.  What is left there is the copies: every SM reads a tile's digits again
// for each of its column chunks, 3 GB in 274 us out of L2.  The tanh table sits
// in shared memory: its lookups by 32 lanes cost 32 wavefronts each through L1,
// and were 53 k cycles per unit.
template <int S, int EPI, bool SEG>
__global__ void __launch_bounds__(OZ_THREADS, 1) k_oz_gemm(OzGemmArgs p)
{
    extern __shared__ __align__(1024) unsigned char smraw[];
    __shared__ __align__(8) uint64_t full[OZ_NST], empty[OZ_NST], tfull[2], tempty[2], tabbar, drain;
    __shared__ uint32_t tslot;
    __shared__ volatile int fail;
    const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const OzGemm &g = p.g;
    constexpr bool WG = EPI == 3, OUT2 = EPI == 0 || EPI == 2;  // OUT2: tout beside hout
    constexpr uint32_t a_bytes = (uint32_t)S * OZ_A_BLK * 2, b_bytes = (uint32_t)S * OZ_B_BLK * 2;
    constexpr uint32_t stage_bytes = a_bytes + b_bytes;
    constexpr int NST = OZ_NST;
    constexpr uint32_t TBUF = 256, TCOLS = 512;
    static_assert(S * DP_OZ_NC <= TBUF, "group accumulators of one buffer");
    const double *tab = reinterpret_cast<const double *>(smraw + NST * stage_bytes);

    if (warp == 0) tc::tmem_alloc(&tslot, TCOLS);
    if (tid == 0) {
        for (int s = 0; s < NST; ++s) {
            tc::mbar_init(&full[s], 1);
            tc::mbar_init(&empty[s], 1);
        }
        for (int s = 0; s < 2; ++s) {
            tc::mbar_init(&tfull[s], 1);
            tc::mbar_init(&tempty[s], 8);
        }
        tc::mbar_init(&tabbar, 1);
        tc::mbar_init(&drain, 1);
        fail = 0;
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tbase = __shfl_sync(0xffffffffu, tslot, 0);

    if (warp == 9) {
        // copies: the tanh table, then the digit chunks of every unit
        int c = 0;
        bool ok = true;
        if (EPI == 0 && tc::elect_one()) {
            mbar_expect_tx(&tabbar, OZ_TAB_BYTES);
            bulk_g2s(smraw + NST * stage_bytes, p.tanh_tab, OZ_TAB_BYTES, &tabbar);
        }
        for (int u = blockIdx.x; u < p.units && ok; u += gridDim.x) {
            OzUnit U;
            if (!oz_unit<S, WG>(p, u, U)) break;
            for (int kc = 0; kc < U.nK; ++kc, ++c) {
                const int st = c % NST;
                if (c >= NST) ok = tc::mbar_wait(&empty[st], (c / NST - 1) & 1) && !fail;
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                if (tc::elect_one()) {
                    unsigned char *dst = smraw + (size_t)st * stage_bytes;
                    mbar_expect_tx(&full[st], stage_bytes);
                    bulk_g2s(dst, U.as + kc * U.astep, a_bytes, &full[st]);
                    bulk_g2s(dst + a_bytes, U.bs + kc * U.bstep, b_bytes, &full[st]);
                }
                __syncwarp();
            }
        }
        if (!ok) fail = 1;
        // no copy is in flight when the CTA leaves
        for (int q = c > NST ? c - NST : 0; q < c; ++q) tc::mbar_wait(&full[q % NST], (q / NST) & 1);
        if (EPI == 0) tc::mbar_wait(&tabbar, 0);
    } else if (warp == 8) {
        // the MMAs of one chunk, then the commit that frees its stage; one copy of
        // the code per stage, so that every descriptor is a constant.  Digit s of A
        // meets the digits t = 1 .. S + 1 - s of W in one MMA of N = 32 (S + 1 - s):
        // W's digit planes lie one after the other, 32 rows each, and so do the
        // accumulators of the groups s + t
        auto issue = [&](auto stage, uint32_t dbase, bool acc0) {
            constexpr int st = decltype(stage)::value;
            // descriptors of digit plane 1; plane s is (s - 1) blocks further (the
            // address field holds bytes / 16 and stays below 2^14 inside shared memory)
            const uint32_t abase = tc::smem_u32(smraw) + st * stage_bytes;
            const uint64_t ad0 = tc::make_desc(abase, 128, 256);
            const uint64_t bd = tc::make_desc(abase + a_bytes, 128, 256);
#pragma unroll
            for (int s = 1; s <= S; ++s)
                tc::mma_bf16(dbase + (uint32_t)(s - 1) * DP_OZ_NC, ad0 + (uint64_t)((s - 1) * OZ_A_BLK * 2 / 16), bd,
                             tc::make_idesc_bf16(DP_OZ_TILE, DP_OZ_NC * (S + 1 - s)), acc0 || s > 1);
            tc::mma_commit(&empty[st]);
        };
        int c = 0, sc = 0;
        bool ok = true;
        for (int u = blockIdx.x; u < p.units && ok; u += gridDim.x) {
            OzUnit U;
            if (!oz_unit<S, WG>(p, u, U)) break;
            for (int sg = 0; sg < U.nseg && ok; ++sg, ++sc) {
                const int buf = sc & 1;
                if (sc >= 2) ok = tc::mbar_wait(&tempty[buf], ((sc >> 1) - 1) & 1) && !fail;
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                tc::fence_after_sync();
                const uint32_t dbase = tbase + buf * TBUF;
                const int k0 = sg * U.seg, k1 = min(U.nK, k0 + U.seg);
                for (int kc = k0; kc < k1; ++kc, ++c) {
                    const int st = c % NST;
                    ok = tc::mbar_wait(&full[st], (c / NST) & 1) && !fail;
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                    if (tc::elect_one()) {
                        const bool acc0 = kc > k0;
                        if (st == 0) issue(std::integral_constant<int, 0>{}, dbase, acc0);
                        else if (st == 1) issue(std::integral_constant<int, 1>{}, dbase, acc0);
                        else if (st == 2) issue(std::integral_constant<int, 2>{}, dbase, acc0);
                        else issue(std::integral_constant<int, 3>{}, dbase, acc0);
                    }
                    __syncwarp();
                }
                if (ok && tc::elect_one()) tc::mma_commit(&tfull[buf]);
                __syncwarp();
            }
        }
        if (!ok) fail = 1;
        if (tc::elect_one()) tc::mma_commit(&drain);
        __syncwarp();
        tc::mbar_wait(&drain, 0);
    } else {
        // y = sum_{g=2}^{S+1} C_g 2^(beta (S + 1 - g)): the group sums are integers
        // below 2^24, combined exactly in two int64 Horner chains (the H groups of
        // largest scale, then the rest; each chain, summed over the segments of a
        // plan of oz_plan_gemm, below 2^53; a weight gradient rounds every segment)
        // and rounded once to FP64 with its scale, on the integer pipe:
        // y 2^escale = sum_g C_g 2^(-beta g).
        constexpr int H = (S + 1) / 2;
        const int w = g.beta * (S - H);
        const int half = warp >> 2, row = 32 * (warp & 3) + lane;
        const uint32_t tl_lane = tbase + ((uint32_t)(32 * (warp & 3)) << 16) + 16 * half;
        const bool vec = !WG && (p.ldo & 1) == 0 && (p.ldh & 1) == 0;  // rows start on 16 bytes
        int sc = 0;
        bool ok = true;
        if (EPI == 0) ok = __all_sync(0xffffffffu, tc::mbar_wait(&tabbar, 0));
        for (int u = blockIdx.x; u < p.units && ok; u += gridDim.x) {
            OzUnit U;
            if (!oz_unit<S, WG>(p, u, U)) break;
            const int n0 = U.nchunk * DP_OZ_NC + 16 * half;   // first of this thread's 16 columns of Y
            const int erow = U.tl * DP_OZ_TILE + row;
            int i, esc = 0;
            const int4 *fe4 = nullptr;
            if constexpr (!WG) {
                i = row < U.cnt ? oz_row(p.type_perm, U.first + row, p.rpa) : -1;
                fe4 = reinterpret_cast<const int4 *>(p.wexp + g.e_off[U.a] + n0);
                esc = (i >= 0 ? p.aexp[erow] : 0) - g.beta * (S + 1);
            } else {
                i = erow < p.rows ? erow : -1;
            }
            double *hout = p.hout + (WG ? p.out_off[U.a] : 0);
            // the skip's operands, asked for before the MMAs are waited for
            const bool bcast = EPI == 1 && p.gbc[U.a] != nullptr;
            const double *hin = bcast ? p.gbc[U.a] : (WG ? hout : p.hin) + (size_t)(i < 0 ? 0 : i) * p.ldh;
            double sk[2][8];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int q0 = n0 + 8 * h;
#pragma unroll
                for (int n = 0; n < 8; ++n) sk[h][n] = 0.0;
                if (i >= 0 && p.skip != 0) {
                    if (p.skip == 1 && vec && !bcast && q0 + 8 <= g.N) {
#pragma unroll
                        for (int n = 0; n < 8; n += 2) {
                            const double2 v = *reinterpret_cast<const double2 *>(hin + q0 + n);
                            sk[h][n] = v.x;
                            sk[h][n + 1] = v.y;
                        }
                    } else {
#pragma unroll
                        for (int n = 0; n < 8; ++n) {
                            const int q = q0 + n;
                            if (q < g.N)
                                sk[h][n] = p.skip == 1 ? hin[q]
                                           : EPI != 1  ? hin[q % p.skip_in]
                                                       : hin[q] + hin[q + p.skip_in];
                        }
                    }
                }
            }
            // group sums of 8 columns (half h of the 16) in buffer buf
            auto groups = [&](int buf, int h, long long (&a)[8], long long (&b)[8]) {
#pragma unroll
                for (int gg = 2; gg <= S + 1; ++gg) {
                    float v[8];
                    tc::tmem_ld8(tl_lane + buf * TBUF + (uint32_t)(gg - 2) * DP_OZ_NC + 8 * h, v);
#pragma unroll
                    for (int n = 0; n < 8; ++n) {
                        const long long iv = (long long)__float2int_rn(v[n]);
                        if (gg == 2) a[n] = iv;
                        else if (gg <= H + 1) a[n] = (a[n] << g.beta) + iv;
                        else if (gg == H + 2) b[n] = iv;
                        else b[n] = (b[n] << g.beta) + iv;
                    }
                }
            };
            // the value of the group sums (hi, lo) of an entry whose exponents add up to e
            auto scaled = [&](long long hi, long long lo, int e) -> double {
                if (e > -900 && e < 900) return oz_i64x2_round(hi, lo, w, e);
                if (e > 5000) return __longlong_as_double(0x7ff8000000000000ll);
                return scale2(fma((double)hi, oz_pow2(w), (double)lo), e);
            };
            auto finish = [&](int h, const long long (&hi)[8], const long long (&lo)[8], const double (&skh)[8]) {
                if (i < 0) return;
                const int q0 = n0 + 8 * h;
                double *ho = hout + (size_t)i * p.ldo + q0;
                double *to = OUT2 ? p.tout + (size_t)i * p.ldo + q0 : nullptr;
                const double *ti = EPI == 2 ? p.tin + (size_t)i * p.ldo + q0 : nullptr;
                const int4 f0 = fe4[2 * h], f1 = fe4[2 * h + 1];
                const int fe[8] = {f0.x, f0.y, f0.z, f0.w, f1.x, f1.y, f1.z, f1.w};
#pragma unroll
                for (int n2 = 0; n2 < 8; n2 += 2) {
                    double y[2], t[2];
#pragma unroll
                    for (int v = 0; v < 2; ++v) {
                        const int n = n2 + v;
                        const bool in = q0 + n < g.N;
                        y[v] = scaled(hi[n], lo[n], esc + fe[n]);
                        if constexpr (EPI == 0) {
                            t[v] = dp_tanh64(y[v] + (in ? p.bias[U.a][q0 + n] : 0.0), tab);
                            y[v] = t[v];
                        } else if constexpr (EPI == 2) {
                            const double tv = in ? ti[n] : 0.0;
                            t[v] = y[v];
                            y[v] *= fma(-tv, tv, 1.0);
                        }
                        y[v] += skh[n];
                    }
                    if (vec && q0 + n2 + 2 <= g.N) {
                        *reinterpret_cast<double2 *>(ho + n2) = make_double2(y[0], y[1]);
                        if constexpr (OUT2) *reinterpret_cast<double2 *>(to + n2) = make_double2(t[0], t[1]);
                    } else {
#pragma unroll
                        for (int v = 0; v < 2; ++v)
                            if (q0 + n2 + v < g.N) {
                                ho[n2 + v] = y[v];
                                if constexpr (OUT2) to[n2 + v] = t[v];
                            }
                    }
                }
            };
            auto wait = [&](int buf) {
                ok = tc::mbar_wait(&tfull[buf], (sc >> 1) & 1) && !fail;
                ok = __all_sync(0xffffffffu, ok);
                tc::fence_after_sync();
                return ok;
            };
            auto release = [&](int buf) {
                tc::fence_before_sync();
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&tempty[buf]);
                ++sc;
            };
            if constexpr (WG) {
                // every segment has its own exponents; its sum is rounded once and added in order
                double acc[2][8];
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int n = 0; n < 8; ++n) acc[h][n] = 0.0;
                for (int sg = 0; sg < U.nseg; ++sg) {
                    const int buf = sc & 1;
                    if (!wait(buf)) break;
                    long long a[2][8], b[2][8];
                    groups(buf, 0, a[0], b[0]);
                    groups(buf, 1, a[1], b[1]);
                    release(buf);
                    const size_t wi = (size_t)(U.sg0 + sg) * g.nN * DP_OZ_NC + n0;
                    const int va = i < 0 ? -16 & ((1 << OZ_LVL_BITS) - 1)
                                         : p.aexp[(size_t)(U.sg0 + sg) * p.nq * DP_OZ_TILE + erow];
                    unsigned bad = 0;  // entries the digits may not carry
#pragma unroll
                    for (int n4 = 0; n4 < 4; ++n4) {
                        const int4 f = *reinterpret_cast<const int4 *>(p.wexp + wi + 4 * n4);
                        const int vw[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
                        for (int v = 0; v < 4; ++v) {
                            const int q = 4 * n4 + v, h = q >> 3, n = q & 7;
                            const double y = scaled(a[h][n], b[h][n],
                                                    (va >> OZ_LVL_BITS) + (vw[v] >> OZ_LVL_BITS) - g.beta * (S + 1));
                            if (oz_digits_stand(y, va, vw[v])) acc[h][n] += y;
                            else bad |= 1u << q;
                        }
                    }
                    for (unsigned who = __ballot_sync(0xffffffffu, bad != 0); who != 0; who &= who - 1) {
                        const int src = __ffs(who) - 1, k = __shfl_sync(0xffffffffu, i, src);
                        const double y = oz_wdot(p, U.first + sg * OZ_WSEG * DP_OZ_KC,
                                                 min(U.cnt - sg * OZ_WSEG * DP_OZ_KC, OZ_WSEG * DP_OZ_KC), k, n0);
#pragma unroll
                        for (int n = 0; n < 16; ++n) {
                            const double yn = __shfl_sync(0xffffffffu, y, 2 * n);
                            if (lane == src && (bad >> n & 1u)) acc[n >> 3][n & 7] += yn;
                        }
                    }
                    __syncwarp();
                }
                if (!ok) break;
                if (p.parts > 1) {
                    // the last of the parts to arrive adds all of them up in order
                    const int ks = u % p.parts, ub = u - ks;
                    auto slot = [&](int q, int v) { return p.part + ((size_t)(ub + q) * 32 + v) * 256 + tid; };
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int n = 0; n < 8; ++n) *slot(ks, 8 * h + n) = __double_as_longlong(acc[h][n]);
                    __threadfence();
                    __syncwarp();
                    int old = 0;
                    if (lane == 0) old = atomicAdd(&p.cnt[(u / p.parts) * 8 + warp], 1);
                    old = __shfl_sync(0xffffffffu, old, 0);
                    if (old != p.parts - 1) continue;
                    __threadfence();
                    double own[16];
#pragma unroll
                    for (int n = 0; n < 16; ++n) {
                        own[n] = acc[n >> 3][n & 7];
                        acc[n >> 3][n & 7] = 0.0;
                    }
#pragma unroll 2
                    for (int q = 0; q < p.parts; ++q)
#pragma unroll
                        for (int n = 0; n < 16; ++n)
                            acc[n >> 3][n & 7] += q == ks ? own[n] : __longlong_as_double(__ldcg(slot(q, n)));
                }
                if (i >= 0) {
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int n = 0; n < 8; ++n)
                            if (n0 + 8 * h + n < g.N)
                                hout[(size_t)i * p.ldo + n0 + 8 * h + n] = acc[h][n] + sk[h][n];
                }
                __syncwarp();
            } else if constexpr (SEG) {
                long long hi[2][8], lo[2][8];
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int n = 0; n < 8; ++n) hi[h][n] = lo[h][n] = 0;
                for (int sg = 0; sg < U.nseg; ++sg) {
                    const int buf = sc & 1;
                    if (!wait(buf)) break;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        long long a[8], b[8];
                        groups(buf, h, a, b);
#pragma unroll
                        for (int n = 0; n < 8; ++n) {
                            hi[h][n] += a[n];
                            lo[h][n] += b[n];
                        }
                    }
                    release(buf);
                }
                if (!ok) break;
                if (p.parts > 1) {
                    // the last of the parts to arrive adds the others' sums (integers: in any order)
                    const int ks = u % p.parts, ub = u - ks;
                    auto slot = [&](int q, int v) { return p.part + ((size_t)(ub + q) * 32 + v) * 256 + tid; };
#pragma unroll
                    for (int h = 0; h < 2; ++h)
#pragma unroll
                        for (int n = 0; n < 8; ++n) {
                            *slot(ks, 16 * h + n) = hi[h][n];
                            *slot(ks, 16 * h + 8 + n) = lo[h][n];
                        }
                    __threadfence();
                    __syncwarp();
                    int old = 0;
                    if (lane == 0) old = atomicAdd(&p.cnt[(u / p.parts) * 8 + warp], 1);
                    old = __shfl_sync(0xffffffffu, old, 0);
                    if (old != p.parts - 1) continue;
                    __threadfence();
                    for (int q = 0; q < p.parts; ++q) {
                        if (q == ks) continue;
#pragma unroll
                        for (int h = 0; h < 2; ++h)
#pragma unroll
                            for (int n = 0; n < 8; ++n) {
                                hi[h][n] += __ldcg(slot(q, 16 * h + n));
                                lo[h][n] += __ldcg(slot(q, 16 * h + 8 + n));
                            }
                    }
                }
                finish(0, hi[0], lo[0], sk[0]);
                finish(1, hi[1], lo[1], sk[1]);
            } else {
                // one segment: 8 columns at a time, half the code
                const int buf = sc & 1;
                if (!wait(buf)) break;
#pragma unroll 1
                for (int h = 0; h < 2; ++h) {
                    long long a[8], b[8];
                    double skh[8];
#pragma unroll
                    for (int n = 0; n < 8; ++n) skh[n] = h == 0 ? sk[0][n] : sk[1][n];
                    __syncwarp();
                    groups(buf, h, a, b);
                    finish(h, a, b, skh);
                }
                release(buf);
            }
        }
        if (!ok) fail = 1;
    }
    tc::fence_before_sync();
    __syncthreads();
    if (tid == 0 && fail) atomicOr(p.status, DPF_MMA_TIMEOUT);
    if (warp == 0) tc::tmem_dealloc(tbase, TCOLS);
}

// Digits of 32 rows (chunk u) of type a's B operand, element (this thread's row, k)
// = elem(k): lane = row, the 8 warps stride over k.
template <class ELEM>
__device__ __forceinline__ void oz_write_b(const OzGemm &g, int a, int u, ELEM elem, uint16_t *__restrict__ w,
                                           int32_t *__restrict__ e, unsigned long long (&mx_s)[8][DP_OZ_NC])
{
    const int rl = threadIdx.x & 31, sl = threadIdx.x >> 5, row = u * DP_OZ_NC + rl;
    unsigned long long mx = 0;  // parameters are finite
#pragma unroll 4
    for (int k = sl; k < g.K; k += 8) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(fabs(elem(k)));
        mx = b > mx ? b : mx;
    }
    mx_s[sl][rl] = mx;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 8; ++q) mx = mx_s[q][rl] > mx ? mx_s[q][rl] : mx;
    const int bS = g.beta * g.S;
    bool zero;
    const int ex = oz_exponent(mx, bS, zero);
    if (sl == 0) e[g.e_off[a] + row] = ex;
    uint16_t *out = w + g.w_off[a] + (size_t)u * g.nK * g.S * OZ_B_BLK;
    for (int kb = sl; kb < 2 * g.nK; kb += 8) {
        const int kc = kb >> 1, kh = kb & 1;
        long long I[8];
#pragma unroll
        for (int q = 0; q < 8; ++q)
            I[q] = zero ? 0 : oz_rint_pow2(elem(kc * DP_OZ_KC + kh * 8 + q), bS - ex);
        for (int sd = g.S - 1; sd >= 0; --sd) {
            int dg[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) dg[q] = sd > 0 ? oz_digit_step(I[q], g.beta) : (int)I[q];
            uint4 v;
            v.x = (uint32_t)oz_bf16_int(dg[0]) | ((uint32_t)oz_bf16_int(dg[1]) << 16);
            v.y = (uint32_t)oz_bf16_int(dg[2]) | ((uint32_t)oz_bf16_int(dg[3]) << 16);
            v.z = (uint32_t)oz_bf16_int(dg[4]) | ((uint32_t)oz_bf16_int(dg[5]) << 16);
            v.w = (uint32_t)oz_bf16_int(dg[6]) | ((uint32_t)oz_bf16_int(dg[7]) << 16);
            *reinterpret_cast<uint4 *>(out + ((size_t)kc * g.S + sd) * OZ_B_BLK + oz_kofs(rl, kh * 8)) = v;
        }
    }
}

// Weight digits of every type, layer and direction, one CTA per 32 rows of a B
// operand: row n of the forward operand is column n of W_l, row q of the
// backward operand is row q of W_l.  (On the host this took most of a training
// step on a small frame; the parameters change every step.)
__global__ void __launch_bounds__(256) k_oz_wsplit(DevModel m, OzModel oz, uint16_t *__restrict__ w,
                                                   int32_t *__restrict__ e)
{
    __shared__ unsigned long long mx_s[8][DP_OZ_NC];
    int u = blockIdx.x, a = 0, l = 0, d = 0;
    int kin = m.m2 * m.M;
    int64_t off = 0;
    for (;;) {
        const OzGemm &t = d == 0 ? oz.fwd[l] : oz.bwd[l];
        if (u < t.nN) break;
        u -= t.nN;
        if (++d == 2) {
            d = 0;
            off += (int64_t)kin * m.fit[l] + m.fit[l];
            kin = m.fit[l];
            if (++l == m.n_fit) {
                l = 0;
                ++a;
                off = 0;
                kin = m.m2 * m.M;
            }
        }
    }
    const OzGemm &g = d == 0 ? oz.fwd[l] : oz.bwd[l];
    const double *W = m.params + m.fit_base[a] + off;
    const int F = m.fit[l], row = u * DP_OZ_NC + (threadIdx.x & 31);
    auto elem = [&](int k) -> double {
        if (k >= g.K || row >= g.N) return 0.0;
        return d == 0 ? W[(size_t)k * F + row] : W[(size_t)row * F + k];
    };
    oz_write_b(g, a, u, elem, w, e, mx_s);
}

// The same for the series of the embedding nets (embed_cheb.cu), C [T T][nn][M],
// nc terms: forward rows f, k = (neighbour type, term); backward rows k, columns f.
__global__ void __launch_bounds__(256) k_oz_series(OzGemm gf, OzGemm gb, int T, int nn, int nc, int M,
                                                   const double *__restrict__ C, uint16_t *__restrict__ w,
                                                   int32_t *__restrict__ e)
{
    __shared__ unsigned long long mx_s[8][DP_OZ_NC];
    const int a = blockIdx.x / (gf.nN + gb.nN), v = blockIdx.x - a * (gf.nN + gb.nN);
    const bool fwd = v < gf.nN;
    const OzGemm &g = fwd ? gf : gb;
    const int u = fwd ? v : v - gf.nN, row = u * DP_OZ_NC + (threadIdx.x & 31);
    auto elem = [&](int k) -> double {
        if (k >= g.K || row >= g.N) return 0.0;
        const int kk = fwd ? k : row, f = fwd ? row : k;
        return C[((size_t)(a * T + kk / nc) * nn + kk % nc) * M + f];
    };
    oz_write_b(g, a, u, elem, w, e, mx_s);
}

// --------------------------------------------- weight gradients' operands ---
//
// dPhi/dW_l = X^T Zb + dX^T dZb over the atoms of a type (the parameter gradient
// of pgrad.cu: forward with tangent and reverse mode run on the same GEMMs):
// digits of the columns of X (rows of the A operand) and of Zb (rows of the B
// operand), scaled per column and segment of 256 atoms by its largest magnitude
// there, so that an outlier takes bits from its own segment only; where it takes
// them from a result, that is summed in FP64 (oz_digits_stand).  With one scale per
// column and type, a descriptor outlier at one atom and an adjoint outlier at
// another left errors of 5e-12 to 1e-10 of the first layer's largest entry where
// FP64 sums, and these, leave 1e-15; the first layer of 12,288 atoms took 257 us,
// now 293 (the two kernels before it 169 us, now 127 in one).
// The whole fitting part on the FP64 units, with per-CTA gradient slices, took 63
// ms for 12,288 water atoms with the student's widths, now 3.8 ms; 648 atoms at
// full width: 23 -> 0.8 ms (24 GEMMs and 14 splits, bound as k_oz_gemm).

struct OzCols {
    const double *src;   // [N][ld], columns 0 .. K-1
    int ld, K, one;      // column `one` is 1 for every atom (-1: none)
    int rb, nb;          // rows per block of the operand (128 or 32), blocks
    uint16_t *out;       // [chunk of 16 atoms][nb][S][rb x 16]
    int32_t *exp;        // [segment][nb rb] exponent and level (oz_digits_stand)
};
struct OzColsPair {
    OzCols c[2];
};

// Exponents, levels and digits of one segment x 32 columns per CTA
// (thread: one column, 32 atoms, read once).
__global__ void __launch_bounds__(256) k_oz_cols(OzColsPair pr, const int32_t *__restrict__ type_perm,
                                                 const int32_t *__restrict__ type_start, int ntypes,
                                                 int32_t *__restrict__ cnt, int ncnt)
{
    constexpr int S = 8, beta = 7, W = OZ_WSEG * DP_OZ_KC, H = W / 8;
    __shared__ int perm[W];
    __shared__ unsigned long long mx_s[8][32], lv_s[2][8][32];
    const OzCols o = blockIdx.z == 0 ? pr.c[0] : pr.c[1];
    const int tid = threadIdx.x, c = tid & 31, h = tid >> 5, q = blockIdx.y * 32 + c, ncol = o.nb * o.rb;
    if (blockIdx.x + blockIdx.y + blockIdx.z == 0)  // part counters of the GEMM that follows
        for (int u = tid; u < ncnt; u += 256) cnt[u] = 0;
    int sg = blockIdx.x, a = 0, kb = 0;
    for (;; ++a) {
        if (a == ntypes) return;
        const int n = type_start[a + 1] - type_start[a], ns = (n + W - 1) / W;
        if (sg < ns) break;
        sg -= ns;
        kb += (n + DP_OZ_KC - 1) / DP_OZ_KC;
    }
    if (q >= ncol) return;  // whole CTAs: blocks are multiples of 32 columns
    const int first = type_start[a] + sg * W, n = min(W, type_start[a + 1] - first);
    static_assert(W == 256, "one atom per thread");
    perm[tid] = tid < n ? type_perm[first + tid] : -1;
    __syncthreads();
    double v[H];
    unsigned long long mx = 0;
#pragma unroll
    for (int u = 0; u < H; ++u) {
        const int i = perm[h * H + u];
        v[u] = i < 0 ? 0.0 : q < o.K ? o.src[(size_t)i * o.ld + q] : q == o.one ? 1.0 : 0.0;
        const unsigned long long b = (unsigned long long)__double_as_longlong(fabs(v[u]));
        mx = b > mx ? b : mx;
    }
    mx_s[h][c] = mx;
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 8; ++u) mx = mx_s[u][c] > mx ? mx_s[u][c] : mx;
    bool zero;
    const int ex = oz_exponent(mx, beta * S, zero);
    uint16_t *out = o.out + ((size_t)(kb + sg * OZ_WSEG) * o.nb + q / o.rb) * S * o.rb * DP_OZ_KC + oz_kofs(q % o.rb, 0);
    // values of level l or less, l = 0 .. 15, a byte each
    unsigned long long lo = 0, hi = 0;
    constexpr unsigned long long ONES = 0x0101010101010101ull;
#pragma unroll
    for (int k = 0; k < H / 8; ++k) {
        const int at = h * H + 8 * k, kc = at / DP_OZ_KC;
        long long J[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const long long I = zero ? 0 : oz_rint_pow2(v[8 * k + u], beta * S - ex);
            const int l = __clzll(I < 0 ? -I : I) - (63 - beta * S);  // |I| <= 2^56
            if (l < 8) lo += ONES << (8 * l);
            if (l < 16) hi += l < 8 ? ONES : ONES << (8 * (l - 8));
            J[u] = I + oz_digit_bias(S, beta);
        }
        if (kc * DP_OZ_KC < n) {
            uint16_t *ok = out + (size_t)kc * o.nb * S * o.rb * DP_OZ_KC + (at % DP_OZ_KC) / 8 * 64;
#pragma unroll
            for (int sd = 0; sd < S; ++sd)
                *reinterpret_cast<uint4 *>(ok + (size_t)sd * o.rb * DP_OZ_KC) = oz_pack_digits<S, beta>(J, sd);
        }
    }
    lv_s[0][h][c] = lo;
    lv_s[1][h][c] = hi;
    __syncthreads();
    if (h == 0) {
        auto count = [&](int l) {  // values of level l or less
            int v = 0;
            for (int u = 0; u < 8; ++u) v += (int)(lv_s[l >> 3][u][c] >> (8 * (l & 7)) & 0xff);
            return v;
        };
        int l = zero ? -16 : 0;  // zeros: every product with them is exact; NaN: the digits do not count
        while (l >= 0 && l < 15 && 4 * count(l) < 3 * n) ++l;
        o.exp[(size_t)blockIdx.x * ncol + q] = ex * (1 << OZ_LVL_BITS) + (l & ((1 << OZ_LVL_BITS) - 1));
    }
}

// Adjoints of the output layer: hb = cE w_out, dhb = -w_out of the atom's type,
// and its z adjoints zb = cE, dzb = -1 (column 0).
__global__ void k_oz_pg_out(DevModel m, const int32_t *__restrict__ types, int N, double cE, int F, int ld,
                            int64_t wo_off, double *__restrict__ hb, double *__restrict__ dhb,
                            double *__restrict__ zb, double *__restrict__ dzb)
{
    for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < (size_t)N * F;
         q += (size_t)gridDim.x * blockDim.x) {
        const size_t i = q / F;
        const int n = (int)(q - i * F);
        const int a = min(max(types[i], 0), m.ntypes - 1);  // as the type partition
        const double w = m.params[m.fit_base[a] + wo_off + n];
        hb[i * ld + n] = cE * w;
        dhb[i * ld + n] = -w;
        if (n == 0) {
            zb[i * ld] = cE;
            dzb[i * ld] = -1.0;
        }
    }
}

// z adjoints of a hidden layer: dzb = (1 - t^2) dhb, zb = (1 - t^2) (hb - 2 t dz dhb)
__global__ void k_oz_pg_z(int N, int F, int ld, const double *__restrict__ t, const double *__restrict__ dz,
                          const double *__restrict__ hb, const double *__restrict__ dhb, double *__restrict__ zb,
                          double *__restrict__ dzb)
{
    for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < (size_t)N * F;
         q += (size_t)gridDim.x * blockDim.x) {
        const size_t i = q / F, e = i * ld + (q - i * F);
        const double tv = t[e], one = fma(-tv, tv, 1.0), g = dhb[e];
        dzb[e] = one * g;
        zb[e] = one * fma(-2.0 * tv * dz[e], g, hb[e]);
    }
}

// Digit width, digit count and segment length of a GEMM of contraction length
// K (nK chunks) at `bits` bits per operand.  From 55 bits on: 8 digits of 7
// bits, the widest for which one 16-column chunk is exact, and as many chunks
// per segment as stay exact, spread evenly (400 columns: 400 4^6 10 < 2^24); a
// segment adds less than 2^45.1 to an int64 chain, and the widest descriptor (128 x
// 128) has 41.  Below: one segment and the widest digits
// that the whole contraction allows.
void oz_plan_gemm(OzGemm &g, int bits)
{
    g.seg = g.nK;
    if (bits >= 55) {
        g.beta = 7;
        g.S = 8;
        const int nseg = (g.nK + OZ_SEG - 1) / OZ_SEG;
        g.seg = (g.nK + nseg - 1) / nseg;
        return;
    }
    for (g.beta = 7; g.beta >= 4; --g.beta) {
        g.S = (bits + g.beta - 1) / g.beta;
        const double bound = (double)g.K * std::pow(4.0, g.beta - 1) * (g.S + 2);
        if (bound < 16777216.0) return;
    }
    g.beta = 0;
    g.S = 0;
}

// CTAs that share one long contraction (more than one segment) when the (tile,
// column chunk) pairs would leave half of the SMs idle or more: exact integer
// sums, so the result does not depend on the split; a weight gradient's parts hold
// whole segments and their FP64 sums are added in order, the same on the same GPU.
// A part keeps 8 chunks or more, below which its fixed costs (sums written and
// read, 64 KB) outweigh the MMAs (1 k cycles a chunk).  One CTA per pair took 88 us
// for the first layer of 192 water atoms and 321 us for a weight gradient over
// 12,288; now 44 and 60 us (85 us for the 240 x 240 weights, 321 before).
int oz_parts(int pairs, int nK, int num_sms)
{
    return std::max(1, std::min(num_sms / std::max(pairs, 1), nK / 8));
}

size_t gemm_smem(int S) { return (size_t)OZ_NST * S * (OZ_A_BLK + OZ_B_BLK) * 2 + OZ_TAB_BYTES; }

}  // namespace

bool dp_oz_plan(const DevModel &m, OzModel &oz, int64_t &w_elems, int64_t &e_elems, int bits)
{
    std::memset(&oz, 0, sizeof(oz));
    const int nf = m.n_fit;
    if (nf < 1 || nf > DP_MAX_LAYERS) return false;
    int kin = m.m2 * m.M;
    int fmax = 0, in_w = 0;
    w_elems = 0;
    e_elems = 0;
    for (int l = 0; l < nf; ++l) {
        const int F = m.fit[l];
        if (F > DP_MAX_FIT_W) return false;
        fmax = std::max(fmax, F);
        OzGemm *gs[2] = {&oz.fwd[l], &oz.bwd[l]};
        const int Ks[2] = {kin, F}, Ns[2] = {F, kin};
        for (int d = 0; d < 2; ++d) {
            OzGemm &g = *gs[d];
            g.K = Ks[d];
            g.N = Ns[d];
            g.nK = (g.K + DP_OZ_KC - 1) / DP_OZ_KC;
            g.nN = (g.N + DP_OZ_NC - 1) / DP_OZ_NC;
            oz_plan_gemm(g, bits);
            if (!(g.S == 4 || g.S == 5 || g.S == 8)) return false;
            in_w = std::max(in_w, g.nK * g.S * OZ_A_BLK);
            for (int a = 0; a < m.ntypes; ++a) {
                g.w_off[a] = w_elems;
                w_elems += (int64_t)g.nN * g.nK * g.S * OZ_B_BLK;
                g.e_off[a] = e_elems;
                e_elems += (int64_t)g.nN * DP_OZ_NC;
            }
        }
        kin = F;
    }
    oz.in_w = in_w;
    oz.fmax = fmax;
    oz.ok = 1;
    return true;
}

cudaError_t dp_launch_oz_weights(cudaStream_t st, const DevModel &m, const OzModel &oz, uint16_t *w, int32_t *e,
                                 int64_t *launches)
{
    int grid = 0;
    for (int l = 0; l < m.n_fit; ++l) grid += oz.fwd[l].nN + oz.bwd[l].nN;
    k_oz_wsplit<<<grid * m.ntypes, 256, 0, st>>>(m, oz, w, e);
    *launches += 1;
    return cudaGetLastError();
}

namespace {

// The launches of one pass of the fitting net over N centres.
struct OzRun {
    cudaStream_t st;
    const DevModel &m;
    const OzModel &oz;
    const OzBuffers &ob;
    int N;
    const NlistBuffers &nb;
    double *Ei;
    int num_sms;
    int32_t *status;
    int64_t *launches;
    int T, nf, tiles, K1;
    size_t plane;
    // parameter offsets of layer l (W_l, b_l) and of the output layer inside a type's block
    int64_t woff[DP_MAX_LAYERS], boff[DP_MAX_LAYERS], wo_off;

    OzRun(cudaStream_t st_, const DevModel &m_, const OzModel &oz_, const OzBuffers &ob_, int N_,
          const NlistBuffers &nb_, double *Ei_, int num_sms_, int32_t *status_, int64_t *launches_)
        : st(st_), m(m_), oz(oz_), ob(ob_), N(N_), nb(nb_), Ei(Ei_), num_sms(num_sms_), status(status_),
          launches(launches_), T(m_.ntypes), nf(m_.n_fit), tiles((N_ + DP_OZ_TILE - 1) / DP_OZ_TILE + m_.ntypes),
          K1(m_.m2 * m_.M), plane((size_t)ob_.nmax * oz_.fmax)
    {
        int64_t off = 0;
        int kin = K1;
        for (int l = 0; l < nf; ++l) {
            woff[l] = off;
            off += (int64_t)kin * m.fit[l];
            boff[l] = off;
            off += m.fit[l];
            kin = m.fit[l];
        }
        wo_off = off;
    }

    cudaError_t init() const
    {
        return tiles > ob.tiles ? cudaErrorInvalidValue : cudaSuccess;
    }

    cudaError_t split(int mode, const double *src, int lds, const double *tv, const OzGemm &g) const
    {
        OzSplitArgs a;
        std::memset(&a, 0, sizeof(a));
        a.mode = mode;
        a.src = src;
        a.lds = lds;
        a.tv = tv;
        a.ldt = oz.fmax;
        for (int t = 0; t < T; ++t) {
            a.wout[t] = m.params + m.fit_base[t] + wo_off;
            a.bout[t] = m.params + m.fit_base[t] + wo_off + m.fit[nf - 1];
        }
        a.Ei = Ei;
        a.K = g.K;
        a.nK = g.nK;
        a.beta = g.beta;
        a.S = g.S;
        a.type_perm = nb.type_perm;
        a.type_start = nb.type_start;
        a.ntypes = T;
        a.rpa = 1;
        a.a = ob.a;
        a.aexp = ob.aexp;
        a.a_stride = ob.a_stride;
        a.cnt = ob.cnt;
        a.ncnt = g.seg < g.nK ? ob.slots * 8 : 0;
        *launches += 1;
        return launch_split(st, a, tiles, num_sms);
    }

    template <int S, int EPI, bool SEG>
    cudaError_t launch_as(const OzGemmArgs &a) const
    {
        const size_t smem = gemm_smem(S);
        cudaError_t e = cudaFuncSetAttribute(k_oz_gemm<S, EPI, SEG>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem);
        if (e != cudaSuccess) return e;
        k_oz_gemm<S, EPI, SEG><<<std::min(a.units, num_sms), OZ_THREADS, smem, st>>>(a);
        *launches += 1;
        return cudaGetLastError();
    }

    // epi 0: forward (bias, tanh, skip); 1: backward (skip gradient); 2: tangent forward; 3: weight gradient
    template <int S>
    cudaError_t launch_epi(const OzGemmArgs &a, int epi) const
    {
        const bool seg = a.g.seg < a.g.nK;
        if (epi == 3) return launch_as<S, 3, true>(a);
        if (epi == 0) return seg ? launch_as<S, 0, true>(a) : launch_as<S, 0, false>(a);
        if (epi == 1) return seg ? launch_as<S, 1, true>(a) : launch_as<S, 1, false>(a);
        return seg ? launch_as<S, 2, true>(a) : launch_as<S, 2, false>(a);
    }

    cudaError_t launch(OzGemmArgs &a, int epi) const
    {
        a.type_perm = nb.type_perm;
        a.type_start = nb.type_start;
        a.ntypes = T;
        a.rpa = 1;
        a.tanh_tab = m.tanh_tab;
        a.status = status;
        // the type partition makes at most T - 1 tiles more than the atoms fill
        const int nK = a.wg ? N / (DP_OZ_KC * T) : a.g.nK;
        const int pairs = a.wg ? a.units : (N + DP_OZ_TILE - 1) / DP_OZ_TILE * a.g.nN;
        a.parts = 1;
        if (a.wg || a.g.seg < a.g.nK) a.parts = std::max(1, std::min(oz_parts(pairs, nK, num_sms), ob.slots / a.units));
        a.units *= a.parts;
        a.part = ob.part;
        a.cnt = ob.cnt;
        // plans of 4 and 5 digits have one segment and no tangent
        if (a.g.S == 8) return launch_epi<8>(a, epi);
        if (a.g.S == 5) return epi == 0 ? launch_as<5, 0, false>(a) : launch_as<5, 1, false>(a);
        return epi == 0 ? launch_as<4, 0, false>(a) : launch_as<4, 1, false>(a);
    }

    // hin: the skip's operand (with bcast_wout the output weights)
    cudaError_t gemm(const OzGemm &g, int epi, int skip, int skip_in, int l, const double *hin, int ldh,
                     bool bcast_wout, const double *tin, double *tout, double *hout, int ldo) const
    {
        OzGemmArgs a;
        std::memset(&a, 0, sizeof(a));
        a.a = ob.a;
        a.aexp = ob.aexp;
        a.a_stride = ob.a_stride;
        a.w = oz.w;
        a.wexp = oz.wexp;
        a.g = g;
        a.skip = skip;
        a.skip_in = skip_in;
        for (int t = 0; t < T; ++t) {
            a.bias[t] = m.params + m.fit_base[t] + boff[l];
            a.gbc[t] = bcast_wout ? m.params + m.fit_base[t] + wo_off : nullptr;
        }
        a.hin = hin;
        a.ldh = ldh;
        a.tin = tin;
        a.tout = tout;
        a.hout = hout;
        a.ldo = ldo;
        a.units = tiles * g.nN;
        return launch(a, epi);
    }
};

}  // namespace

cudaError_t dp_launch_fit_oz(cudaStream_t st, const DevModel &m, const OzModel &oz, const OzBuffers &ob, int N,
                             const NlistBuffers &nb, EvalBuffers eb, int num_sms, int32_t *status,
                             int64_t *launches)
{
    const OzRun r(st, m, oz, ob, N, nb, eb.Ei, num_sms, status, launches);
    const int nf = r.nf, K1 = r.K1;
    const size_t plane = r.plane;
    double *H[2] = {ob.h, ob.h + plane};
    double *G[2] = {ob.g, ob.g + plane};
    cudaError_t e = r.init();
    if (e != cudaSuccess) return e;
    // forward: h_l = skip(h_{l-1}) + tanh(h_{l-1} W_l + b_l), h_{-1} = D
    int kin = K1;
    for (int l = 0; l < nf; ++l) {
        const double *x = l == 0 ? eb.D : H[(l - 1) & 1];
        const int ldx = l == 0 ? K1 : oz.fmax;
        if ((e = r.split(0, x, ldx, nullptr, oz.fwd[l])) != cudaSuccess) return e;
        if ((e = r.gemm(oz.fwd[l], 0, dp_skip_kind(kin, m.fit[l]), kin, l, x, ldx, false, nullptr,
                        ob.t + (size_t)l * plane, H[l & 1], oz.fmax)) != cudaSuccess)
            return e;
        kin = m.fit[l];
    }
    // output layer (E_i) and dL/dz of the last layer (dL/dh = w_out)
    if ((e = r.split(2, H[(nf - 1) & 1], oz.fmax, ob.t + (size_t)(nf - 1) * plane, oz.bwd[nf - 1])) != cudaSuccess)
        return e;
    // backward: dL/dh_{l-1} = (dL/dz_l) W_l^T + skip'(dL/dh_l)
    for (int l = nf - 1; l >= 0; --l) {
        const int kin_l = l == 0 ? K1 : m.fit[l - 1];
        const bool last = l == nf - 1;
        double *out = l == 0 ? eb.gD : G[(l - 1) & 1];
        const int ldo = l == 0 ? K1 : oz.fmax;
        if ((e = r.gemm(oz.bwd[l], 1, dp_skip_kind(kin_l, m.fit[l]), kin_l, l, last ? nullptr : G[l & 1], oz.fmax,
                        last, nullptr, nullptr, out, ldo)) != cudaSuccess)
            return e;
        if (l > 0)
            if ((e = r.split(1, G[(l - 1) & 1], oz.fmax, ob.t + (size_t)(l - 1) * plane, oz.bwd[l - 1])) != cudaSuccess)
                return e;
    }
    return cudaSuccess;
}

size_t dp_oz_grad_elems(const DevModel &m, const OzModel &oz, int64_t natoms, int which)
{
    const size_t K = (size_t)m.m2 * m.M > (size_t)oz.fmax ? (size_t)m.m2 * m.M : (size_t)oz.fmax;
    const size_t nq = K / DP_OZ_TILE + 1, nn = (oz.fmax + DP_OZ_NC - 1) / DP_OZ_NC;
    const size_t chunks = (size_t)natoms / DP_OZ_KC + m.ntypes;
    const size_t segs = (size_t)natoms / (OZ_WSEG * DP_OZ_KC) + m.ntypes;
    switch (which) {
    case 0: return chunks * nq * 8 * OZ_A_BLK;
    case 1: return chunks * nn * 8 * OZ_B_BLK;
    case 2: return segs * (nq * DP_OZ_TILE + nn * DP_OZ_NC);
    default: return 6 * (size_t)natoms * oz.fmax;
    }
}

cudaError_t dp_launch_pgrad_fit_oz(cudaStream_t st, const DevModel &m, const OzModel &oz, const OzBuffers &ob,
                                   const OzGradBuffers &og, const int32_t *types, int N, double cE,
                                   const NlistBuffers &nb, EvalBuffers eb, PGradBuffers pb, int num_sms,
                                   int32_t *status, double *grad, int64_t *launches)
{
    const OzRun r(st, m, oz, ob, N, nb, eb.Ei, num_sms, status, launches);
    const int nf = r.nf, K1 = r.K1, T = r.T, ld = oz.fmax;
    const size_t plane = r.plane;
    cudaError_t e = r.init();
    if (e != cudaSuccess) return e;
    // per layer: tanh values, tangent pre-activations, outputs, their tangents
    auto keep = [&](int kind, int l) { return pb.fit_scr + (size_t)(kind * nf + l) * plane; };
    double *hb[2] = {og.x, og.x + plane}, *dhb[2] = {og.x + 2 * plane, og.x + 3 * plane};
    double *zb = og.x + 4 * plane, *dzb = og.x + 5 * plane;

    // forward, value and tangent
    int kin = K1;
    for (int l = 0; l < nf; ++l) {
        const double *x = l == 0 ? eb.D : keep(2, l - 1), *dx = l == 0 ? pb.dD : keep(3, l - 1);
        const int ldx = l == 0 ? K1 : ld, sk = dp_skip_kind(kin, m.fit[l]);
        if ((e = r.split(0, x, ldx, nullptr, oz.fwd[l])) != cudaSuccess) return e;
        if ((e = r.gemm(oz.fwd[l], 0, sk, kin, l, x, ldx, false, nullptr, keep(0, l), keep(2, l), ld)) != cudaSuccess)
            return e;
        if ((e = r.split(0, dx, ldx, nullptr, oz.fwd[l])) != cudaSuccess) return e;
        if ((e = r.gemm(oz.fwd[l], 2, sk, kin, l, dx, ldx, false, keep(0, l), keep(1, l), keep(3, l), ld)) !=
            cudaSuccess)
            return e;
        kin = m.fit[l];
    }

    // gradient of a layer's weights and, as the row after them, its bias
    auto weights = [&](const double *x, const double *dx, int ldx, int K, int F, int64_t off) -> cudaError_t {
        const int nq = K / DP_OZ_TILE + 1, nN = (F + DP_OZ_NC - 1) / DP_OZ_NC;  // K + 1 rows
        for (int pass = 0; pass < 2; ++pass) {
            const int segs = N / (OZ_WSEG * DP_OZ_KC) + T;
            OzColsPair c;
            int32_t *expb = og.exp + (size_t)segs * nq * DP_OZ_TILE;
            c.c[0] = OzCols{pass == 0 ? x : dx, ldx, K, pass == 0 ? K : -1, DP_OZ_TILE, nq, og.a, og.exp};
            c.c[1] = OzCols{pass == 0 ? zb : dzb, ld, F, -1, DP_OZ_NC, nN, og.b, expb};
            k_oz_cols<<<dim3(segs, std::max(nq * DP_OZ_TILE, nN * DP_OZ_NC) / 32, 2), 256, 0, st>>>(
                c, nb.type_perm, nb.type_start, T, ob.cnt, ob.slots * 8);
            *launches += 1;
            OzGemmArgs a;
            std::memset(&a, 0, sizeof(a));
            a.a = og.a;
            a.aexp = og.exp;
            a.w = og.b;
            a.wexp = expb;
            a.x = c.c[0].src;
            a.z = c.c[1].src;
            a.ldx = ldx;
            a.ldz = ld;
            a.one = pass == 0;
            a.g.N = F;
            a.g.nN = nN;
            a.g.beta = 7;
            a.g.S = 8;
            a.skip = pass;  // the second product is added to the first
            a.wg = 1;
            a.rows = K + 1;
            a.nq = nq;
            a.hout = grad;
            a.ldo = a.ldh = F;
            for (int t = 0; t < T; ++t) a.out_off[t] = m.fit_base[t] + off;
            a.units = T * nq * nN;
            const cudaError_t e2 = r.launch(a, 3);
            if (e2 != cudaSuccess) return e2;
        }
        return cudaSuccess;
    };

    // reverse mode of cE E - dE
    const int Fl = m.fit[nf - 1];
    auto blocks = [&](int F) { return (int)std::min<size_t>(((size_t)N * F + 255) / 256, 8192); };
    k_oz_pg_out<<<blocks(Fl), 256, 0, st>>>(m, types, N, cE, Fl, ld, r.wo_off, hb[(nf - 1) & 1], dhb[(nf - 1) & 1], zb,
                                            dzb);
    *launches += 1;
    if ((e = weights(keep(2, nf - 1), keep(3, nf - 1), ld, Fl, 1, r.wo_off)) != cudaSuccess) return e;
    for (int l = nf - 1; l >= 0; --l) {
        const int F = m.fit[l], kl = l == 0 ? K1 : m.fit[l - 1], sk = dp_skip_kind(kl, F);
        double *h = hb[l & 1], *dh = dhb[l & 1];
        k_oz_pg_z<<<blocks(F), 256, 0, st>>>(N, F, ld, keep(0, l), keep(1, l), h, dh, zb, dzb);
        *launches += 1;
        if ((e = weights(l == 0 ? eb.D : keep(2, l - 1), l == 0 ? pb.dD : keep(3, l - 1), l == 0 ? K1 : ld, kl, F,
                         r.woff[l])) != cudaSuccess)
            return e;
        double *out = l == 0 ? pb.Db : hb[(l - 1) & 1], *dout = l == 0 ? pb.dDb : dhb[(l - 1) & 1];
        const int ldo = l == 0 ? K1 : ld;
        if ((e = r.split(0, zb, ld, nullptr, oz.bwd[l])) != cudaSuccess) return e;
        if ((e = r.gemm(oz.bwd[l], 1, sk, kl, l, h, ld, false, nullptr, nullptr, out, ldo)) != cudaSuccess) return e;
        if ((e = r.split(0, dzb, ld, nullptr, oz.bwd[l])) != cudaSuccess) return e;
        if ((e = r.gemm(oz.bwd[l], 1, sk, kl, l, dh, ld, false, nullptr, nullptr, dout, ldo)) != cudaSuccess) return e;
    }
    return cudaGetLastError();
}

bool dp_oz_series_plan(const DevModel &m, int n, OzSeries &os)
{
    const int Kt = m.ntypes * n;
    os.gf.K = os.gb.N = Kt;
    os.gf.N = os.gb.K = m.M;
    int64_t w = 0, e = 0;
    for (OzGemm *g : {&os.gf, &os.gb}) {
        g->nK = (g->K + DP_OZ_KC - 1) / DP_OZ_KC;
        g->nN = (g->N + DP_OZ_NC - 1) / DP_OZ_NC;
        g->beta = 7;
        g->S = 8;
        g->seg = g->nK;
        if (g->nK > OZ_SEG) return false;
        for (int a = 0; a < m.ntypes; ++a) {
            g->w_off[a] = w;
            w += (int64_t)g->nN * g->nK * g->S * OZ_B_BLK;
            g->e_off[a] = e;
            e += (int64_t)g->nN * DP_OZ_NC;
        }
    }
    os.w_elems = w;
    os.e_elems = e;
    return true;
}

cudaError_t dp_launch_oz_series(cudaStream_t st, const DevModel &m, const OzSeries &os, int nn, int n, const double *C,
                                int64_t *launches)
{
    k_oz_series<<<m.ntypes * (os.gf.nN + os.gb.nN), 256, 0, st>>>(os.gf, os.gb, m.ntypes, nn, n, m.M, C, os.w, os.e);
    *launches += 1;
    return cudaGetLastError();
}

// Digits needed for four rows per centre, and their capacity in the fitting net's buffer.
bool dp_oz_series_fits(const DevModel &m, const OzSeries &os, const OzBuffers &ob, int N)
{
    const int64_t tiles = (4 * (int64_t)N + DP_OZ_TILE - 1) / DP_OZ_TILE + m.ntypes;
    return tiles * std::max(os.gf.nK, os.gb.nK) * 8 * OZ_A_BLK <= (int64_t)ob.tiles * ob.a_stride;
}

cudaError_t dp_launch_oz_rows(cudaStream_t st, const DevModel &m, const OzSeries &os, const OzGemm &g, uint16_t *a_dig,
                              int N, const double *x, int ldx, double *y, int ldy, const NlistBuffers &nb, int num_sms,
                              int32_t *status, int64_t *launches)
{
    const int tiles = (4 * N + DP_OZ_TILE - 1) / DP_OZ_TILE + m.ntypes;
    const int64_t stride = (int64_t)g.nK * 8 * OZ_A_BLK;
    OzSplitArgs sp;
    std::memset(&sp, 0, sizeof(sp));
    sp.src = x;
    sp.lds = ldx;
    sp.K = g.K;
    sp.nK = g.nK;
    sp.beta = g.beta;
    sp.S = g.S;
    sp.type_perm = nb.type_perm;
    sp.type_start = nb.type_start;
    sp.ntypes = m.ntypes;
    sp.rpa = 4;
    sp.a = a_dig;
    sp.aexp = os.aexp;
    sp.a_stride = stride;
    cudaError_t e = launch_split(st, sp, tiles, num_sms);
    if (e != cudaSuccess) return e;
    OzGemmArgs a;
    std::memset(&a, 0, sizeof(a));
    a.a = a_dig;
    a.aexp = os.aexp;
    a.a_stride = stride;
    a.parts = 1;
    a.w = os.w;
    a.wexp = os.e;
    a.g = g;
    a.type_perm = nb.type_perm;
    a.type_start = nb.type_start;
    a.ntypes = m.ntypes;
    a.rpa = 4;
    a.hin = y;
    a.hout = y;
    a.ldh = a.ldo = ldy;
    a.status = status;
    a.units = tiles * g.nN;
    const size_t smem = gemm_smem(8);
    e = cudaFuncSetAttribute(k_oz_gemm<8, 1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_oz_gemm<8, 1, false><<<std::min(a.units, num_sms), OZ_THREADS, smem, st>>>(a);
    *launches += 2;
    return cudaGetLastError();
}
