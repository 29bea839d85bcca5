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
// of 7 bits throughout, 36 MMAs per 16 columns and 8 planes to read; 66 and 11
// for the 1,600-long first layer when one segment had to hold it, with 5-bit
// digits).  The result is the exact product of the digit expansions, rounded
// once into FP64, and is reproducible bit for bit.
//
// Kernels.  k_oz_split: digits of the activations of a 128-atom tile of one
// type, S BF16 matrices in the canonical K-major layout of the MMA A operand
// (16-column chunks).  The weights' digits are made once on the host.
// k_oz_gemm: persistent over (tile, 32-column chunk of Y); a copy warp streams
// the digit chunks of A and W (cp.async.bulk, a 4-stage ring on mbarriers), an
// MMA warp issues S(S+1)/2 MMAs of 128 x 32 x 16 per chunk into S group
// accumulators in tensor memory, and 8 warps combine the groups exactly, round
// once and apply the layer's bias, tanh and skip (forward) or the skip gradient
// (backward).  Every wait is bounded; on a timeout the kernel sets
// DPF_MMA_TIMEOUT, waits for its copies and MMAs, frees tensor memory and
// returns.
//
// Measured per evaluation (12,288 water atoms): the six GEMMs 2.8 -> 1.22 ms,
// the six splits 0.74 -> 0.43 ms; 192 atoms: the whole fitting net 0.96 -> 0.33
// ms.  One elected lane of a whole warp issues: behind `threadIdx.x == 0` the
// same MMAs took 139 cycles each instead of 97 in the former kernel.
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
constexpr uint32_t OZ_TAB_BYTES = DP_TANH_NINT * DP_TANH_STRIDE * 8;
static_assert(OZ_TAB_BYTES % 16 == 0, "bulk copy of the tanh table");
constexpr int OZ_A_BLK = DP_OZ_TILE * DP_OZ_KC;  // elements of one A digit chunk (128 x 16)
constexpr int OZ_B_BLK = DP_OZ_NC * DP_OZ_KC;    // elements of one W digit chunk (32 x 16)

struct TileRef {
    int a, first, cnt;
};

// Tile index -> (type, first position in type_perm, atoms); a = -1 past the end.
__device__ __forceinline__ TileRef oz_tile(int tl, const int32_t *__restrict__ type_start, int ntypes)
{
    TileRef t{-1, 0, 0};
    for (int a = 0; a < ntypes; ++a) {
        const int n_a = type_start[a + 1] - type_start[a];
        const int tiles = (n_a + DP_OZ_TILE - 1) / DP_OZ_TILE;
        if (tl < tiles) {
            t.a = a;
            t.first = type_start[a] + tl * DP_OZ_TILE;
            t.cnt = min(DP_OZ_TILE, n_a - tl * DP_OZ_TILE);
            return t;
        }
        tl -= tiles;
    }
    return t;
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
    int ntypes;
    uint16_t *a;
    int32_t *aexp;
    int64_t a_stride;
};

// One CTA per group of 8 rows of a tile (a row group of the canonical layout):
// warp w takes the exponent (and output-layer energy) of row w, then every
// digit plane of a 16-column chunk is written as one contiguous 256-byte block:
// lane = row (0..7) + 8 * (column half) + 16 * (chunk parity), the warps
// striding over the chunk pairs.  (One warp per row group, rows one after the
// other, took 277 us for the descriptors of 12,288 water atoms and 181 us for
// 192: a chain of dependent loads on few warps.)  The conversions run on the
// integer pipe.
__global__ void __launch_bounds__(256) k_oz_split(OzSplitArgs p)
{
    __shared__ int e_s[8];
    __shared__ int nz_s[8];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tl = blockIdx.x / (DP_OZ_TILE / 8), r0 = (blockIdx.x % (DP_OZ_TILE / 8)) * 8;
    const TileRef T = oz_tile(tl, p.type_start, p.ntypes);
    if (T.a < 0) return;
    const double *wo = p.mode == 2 ? p.wout[T.a] : nullptr;
    const int bS = p.beta * p.S;

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
        const int i = r < T.cnt ? p.type_perm[T.first + r] : -1;
        if (p.mode == 2) {
            double e = 0.0;
            if (i >= 0)
                for (int k = lane; k < p.K; k += 32) e = fma(p.src[(size_t)i * p.lds + k], wo[k], e);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
            if (i >= 0 && lane == 0) p.Ei[i] = *p.bout[T.a] + e;
        }
        // largest |x| by its bits (NaN left out)
        unsigned long long mx = 0;
#pragma unroll 4
        for (int k = lane; k < p.K; k += 32) {
            const unsigned long long b = (unsigned long long)__double_as_longlong(fabs(value(i, k)));
            if (b > mx && b <= 0x7ff0000000000000ull) mx = b;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long q = __shfl_xor_sync(0xffffffffu, mx, o);
            mx = q > mx ? q : mx;
        }
        if (lane == 0) {
            int e = 0;
            const double m = __longlong_as_double((long long)mx);
            bool zero = !(m > 0.0);
            if (!zero) {
                frexp(m, &e);
                if (e < bS - 1020) zero = true;  // below 2^-960: a zero row
            }
            e_s[warp] = zero ? 0 : e;
            nz_s[warp] = !zero;
            p.aexp[(size_t)tl * DP_OZ_TILE + r] = zero ? 0 : e;
        }
    }
    __syncthreads();

    // digits: lane handles row r0 + (lane & 7), columns kh*8 .. kh*8+7 of chunk kc
    const int jr = lane & 7, kh = (lane >> 3) & 1;
    const int r = r0 + jr;
    const int i = r < T.cnt && nz_s[jr] ? p.type_perm[T.first + r] : -1;
    const int sh = bS - e_s[jr];
    uint16_t *out = p.a + (size_t)tl * p.a_stride;
    const int ofs = oz_kofs(r, kh * 8);
    for (int kc = 2 * warp + (lane >> 4); kc < p.nK; kc += 16) {
        const int k8 = kc * DP_OZ_KC + kh * 8;
        long long I[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) I[q] = oz_rint_pow2(value(i, k8 + q), sh);
        for (int sd = p.S - 1; sd >= 0; --sd) {
            int d[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) d[q] = sd > 0 ? oz_digit_step(I[q], p.beta) : (int)I[q];
            uint4 u;
            u.x = (uint32_t)oz_bf16_int(d[0]) | ((uint32_t)oz_bf16_int(d[1]) << 16);
            u.y = (uint32_t)oz_bf16_int(d[2]) | ((uint32_t)oz_bf16_int(d[3]) << 16);
            u.z = (uint32_t)oz_bf16_int(d[4]) | ((uint32_t)oz_bf16_int(d[5]) << 16);
            u.w = (uint32_t)oz_bf16_int(d[6]) | ((uint32_t)oz_bf16_int(d[7]) << 16);
            *reinterpret_cast<uint4 *>(out + ((size_t)kc * p.S + sd) * OZ_A_BLK + ofs) = u;
        }
    }
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
    int ntypes;
    int epi;      // 0: forward (bias, tanh, skip); 1: backward (skip gradient)
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

// Persistent, one CTA per SM over the units (tile, 32-column chunk of Y) in
// order, so that the CTAs at work share a tile's digits in L2.  Warps 0-7: the
// epilogue (two warps per quarter of the tensor memory's lanes, 16 columns
// each); warp 8 issues the MMAs, warp 9 the copies.  The group accumulators are
// doubled (2 x 256 columns): the epilogue of one segment runs beside the MMAs
// of the next.  A contraction longer than the accumulators hold exactly is cut
// into segments of g.seg chunks, which the epilogue adds up in int64.
//
// Bounds, per unit of a 240-long contraction at S = 8: 15 chunks x 36 MMAs of
// 20 cycles with A held in the collector (40 without, and 40 when two CTAs of
// one SM alternate: measured) = 10.8 k cycles, 40 KB of copies per chunk at the
// 60 B/clk that large bulk copies reach = 10.3 k; with the FP64 tanh 20 k
// cycles of FP64 pipe.  The tanh table sits in shared memory: its lookups by 32
// lanes cost 32 wavefronts each through L1, and were 53 k cycles per unit.
template <int S>
__global__ void __launch_bounds__(OZ_THREADS, 1) k_oz_gemm(OzGemmArgs p)
{
    extern __shared__ __align__(1024) unsigned char smraw[];
    __shared__ __align__(8) uint64_t full[OZ_NST], empty[OZ_NST], tfull[2], tempty[2], tabbar, drain;
    __shared__ uint32_t tslot;
    __shared__ volatile int fail;
    const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const OzGemm &g = p.g;
    const int nK = g.nK, nseg = (nK + g.seg - 1) / g.seg;
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
        if (p.epi == 0 && tc::elect_one()) {
            mbar_expect_tx(&tabbar, OZ_TAB_BYTES);
            bulk_g2s(smraw + NST * stage_bytes, p.tanh_tab, OZ_TAB_BYTES, &tabbar);
        }
        for (int u = blockIdx.x; u < p.units && ok; u += gridDim.x) {
            const int tl = u / g.nN, nchunk = u - tl * g.nN;
            const TileRef T = oz_tile(tl, p.type_start, p.ntypes);
            if (T.a < 0) break;
            const uint16_t *asrc = p.a + (size_t)tl * p.a_stride;
            const uint16_t *bsrc = p.w + g.w_off[T.a] + (size_t)nchunk * nK * S * OZ_B_BLK;
            for (int kc = 0; kc < nK; ++kc, ++c) {
                const int st = c % NST;
                if (c >= NST) ok = tc::mbar_wait(&empty[st], (c / NST - 1) & 1) && !fail;
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                if (tc::elect_one()) {
                    unsigned char *dst = smraw + (size_t)st * stage_bytes;
                    mbar_expect_tx(&full[st], stage_bytes);
                    bulk_g2s(dst, asrc + (size_t)kc * S * OZ_A_BLK, a_bytes, &full[st]);
                    bulk_g2s(dst + a_bytes, bsrc + (size_t)kc * S * OZ_B_BLK, b_bytes, &full[st]);
                }
                __syncwarp();
            }
        }
        if (!ok) fail = 1;
        // no copy is in flight when the CTA leaves
        for (int q = c > NST ? c - NST : 0; q < c; ++q) tc::mbar_wait(&full[q % NST], (q / NST) & 1);
        if (p.epi == 0) tc::mbar_wait(&tabbar, 0);
    } else if (warp == 8) {
        const uint32_t idesc = tc::make_idesc_bf16(DP_OZ_TILE, DP_OZ_NC);
        // the MMAs of one chunk, then the commit that frees its stage; one copy of
        // the code per stage, so that every descriptor is a constant
        auto issue = [&](auto stage, uint32_t dbase, bool acc0) {
            constexpr int st = decltype(stage)::value;
            // descriptors of digit plane 1; plane s is (s - 1) blocks further (the
            // address field holds bytes / 16 and stays below 2^14 inside shared memory)
            const uint32_t abase = tc::smem_u32(smraw) + st * stage_bytes;
            const uint64_t ad0 = tc::make_desc(abase, 128, 256);
            const uint64_t bd0 = tc::make_desc(abase + a_bytes, 128, 256);
#pragma unroll
            for (int s = 1; s <= S; ++s) {
                const uint64_t ad = ad0 + (uint64_t)((s - 1) * OZ_A_BLK * 2 / 16);
#pragma unroll
                for (int t = 1; t + s <= S + 1; ++t) {
                    const uint32_t dc = dbase + (uint32_t)(s + t - 2) * DP_OZ_NC;
                    const uint64_t bd = bd0 + (uint64_t)((t - 1) * OZ_B_BLK * 2 / 16);
                    const bool acc = acc0 || s > 1;
                    if (s == S) tc::mma_bf16(dc, ad, bd, idesc, acc);
                    else if (t == 1) tc::mma_bf16_a<0>(dc, ad, bd, idesc, acc);
                    else if (t + s <= S) tc::mma_bf16_a<1>(dc, ad, bd, idesc, acc);
                    else tc::mma_bf16_a<2>(dc, ad, bd, idesc, acc);
                }
            }
            tc::mma_commit(&empty[st]);
        };
        int c = 0, sc = 0;
        bool ok = true;
        for (int u = blockIdx.x; u < p.units && ok; u += gridDim.x) {
            if (oz_tile(u / g.nN, p.type_start, p.ntypes).a < 0) break;
            for (int sg = 0; sg < nseg && ok; ++sg, ++sc) {
                const int buf = sc & 1;
                if (sc >= 2) ok = tc::mbar_wait(&tempty[buf], ((sc >> 1) - 1) & 1) && !fail;
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                tc::fence_after_sync();
                const uint32_t dbase = tbase + buf * TBUF;
                const int k1 = min(nK, (sg + 1) * g.seg);
                for (int kc = sg * g.seg; kc < k1; ++kc, ++c) {
                    const int st = c % NST;
                    ok = tc::mbar_wait(&full[st], (c / NST) & 1) && !fail;
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                    if (tc::elect_one()) {
                        const bool acc0 = kc > sg * g.seg;
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
        // largest scale, then the rest; each chain, summed over the segments, below
        // 2^53 for every plan of oz_plan_gemm) and rounded once to FP64 with its
        // scale, on the integer pipe: y 2^escale = sum_g C_g 2^(-beta g).
        constexpr int H = (S + 1) / 2;
        const int w = g.beta * (S - H);
        const int half = warp >> 2, row = 32 * (warp & 3) + lane;
        const uint32_t tl_lane = tbase + ((uint32_t)(32 * (warp & 3)) << 16) + 16 * half;
        const bool vec = (p.ldo & 1) == 0 && (p.ldh & 1) == 0;  // rows start on 16 bytes
        int sc = 0;
        bool ok = true;
        if (p.epi == 0) ok = __all_sync(0xffffffffu, tc::mbar_wait(&tabbar, 0));
        for (int u = blockIdx.x; u < p.units && ok; u += gridDim.x) {
            const int tl = u / g.nN, nchunk = u - tl * g.nN;
            const TileRef T = oz_tile(tl, p.type_start, p.ntypes);
            if (T.a < 0) break;
            const int i = row < T.cnt ? p.type_perm[T.first + row] : -1;
            const int n0 = nchunk * DP_OZ_NC + 16 * half;   // first of this thread's 16 columns of Y
            const int esc = (i >= 0 ? p.aexp[(size_t)tl * DP_OZ_TILE + row] : 0) - g.beta * (S + 1);
            const int4 *fe4 = reinterpret_cast<const int4 *>(p.wexp + g.e_off[T.a] + n0);
            // the skip's operands, asked for before the MMAs are waited for
            const bool bcast = p.epi != 0 && p.gbc[T.a] != nullptr;
            const double *hin = bcast ? p.gbc[T.a] : p.hin + (size_t)(i < 0 ? 0 : i) * p.ldh;
            double sk[16];
#pragma unroll
            for (int n = 0; n < 16; ++n) sk[n] = 0.0;
            if (i >= 0) {
                if (p.skip == 1 && vec && !bcast && n0 + 16 <= g.N) {
#pragma unroll
                    for (int n = 0; n < 16; n += 2) {
                        const double2 v = *reinterpret_cast<const double2 *>(hin + n0 + n);
                        sk[n] = v.x;
                        sk[n + 1] = v.y;
                    }
                } else if (p.skip != 0) {
#pragma unroll
                    for (int n = 0; n < 16; ++n)
                        if (n0 + n < g.N) {
                            const int q = n0 + n;
                            sk[n] = p.skip == 1 ? hin[q]
                                    : p.epi == 0 ? hin[q % p.skip_in]
                                                 : hin[q] + hin[q + p.skip_in];
                        }
                }
            }
            long long hi[16], lo[16];
#pragma unroll
            for (int n = 0; n < 16; ++n) hi[n] = lo[n] = 0;
            for (int sg = 0; sg < nseg; ++sg, ++sc) {
                const int buf = sc & 1;
                ok = tc::mbar_wait(&tfull[buf], (sc >> 1) & 1) && !fail;
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                tc::fence_after_sync();
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    long long a[8], b[8];
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
#pragma unroll
                    for (int n = 0; n < 8; ++n) {
                        hi[8 * h + n] += a[n];
                        lo[8 * h + n] += b[n];
                    }
                }
                tc::fence_before_sync();
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&tempty[buf]);
            }
            if (!ok) break;
            if (i < 0) continue;
            double *ho = p.hout + (size_t)i * p.ldo + n0;
            double *to = p.epi == 0 ? p.tout + (size_t)i * p.ldo + n0 : nullptr;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int4 f4 = fe4[q];
                const int fe[4] = {f4.x, f4.y, f4.z, f4.w};
#pragma unroll
                for (int n2 = 0; n2 < 4; n2 += 2) {
                    double y[2], t[2];
#pragma unroll
                    for (int v = 0; v < 2; ++v) {
                        const int n = 4 * q + n2 + v, e = esc + fe[n2 + v];
                        y[v] = e > -900 && e < 900 ? oz_i64x2_scaled_w(hi[n], lo[n], w, e)
                                                   : scale2(fma((double)hi[n], oz_pow2(w), (double)lo[n]), e);
                        if (p.epi == 0) {
                            const int col = n0 + n;
                            t[v] = dp_tanh64(y[v] + (col < g.N ? p.bias[T.a][col] : 0.0), tab);
                            y[v] = t[v];
                        }
                        y[v] += sk[n];
                    }
                    const int n = 4 * q + n2;
                    if (vec && n0 + n + 2 <= g.N) {
                        *reinterpret_cast<double2 *>(ho + n) = make_double2(y[0], y[1]);
                        if (p.epi == 0) *reinterpret_cast<double2 *>(to + n) = make_double2(t[0], t[1]);
                    } else {
#pragma unroll
                        for (int v = 0; v < 2; ++v)
                            if (n0 + n + v < g.N) {
                                ho[n + v] = y[v];
                                if (p.epi == 0) to[n + v] = t[v];
                            }
                    }
                }
            }
        }
        if (!ok) fail = 1;
    }
    tc::fence_before_sync();
    __syncthreads();
    if (tid == 0 && fail) atomicOr(p.status, DPF_MMA_TIMEOUT);
    if (warp == 0) tc::tmem_dealloc(tbase, TCOLS);
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
    const int F = m.fit[l], rl = threadIdx.x & 31, sl = threadIdx.x >> 5, row = u * DP_OZ_NC + rl;
    auto elem = [&](int k) -> double {
        if (k >= g.K || row >= g.N) return 0.0;
        return d == 0 ? W[(size_t)k * F + row] : W[(size_t)row * F + k];
    };
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
    const double big = __longlong_as_double((long long)mx);
    const int bS = g.beta * g.S;
    int ex = 0;
    bool zero = !(big > 0.0);
    if (!zero) {
        frexp(big, &ex);
        if (ex < bS - 1020) zero = true;
    }
    if (zero) ex = 0;
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

// Digit width, digit count and segment length of a GEMM of contraction length
// K (nK chunks) at `bits` bits per operand.  From 55 bits on: 8 digits of 7
// bits, the widest for which one 16-column chunk is exact, and as many chunks
// per segment as stay exact, spread evenly (400 columns: 400 4^6 10 < 2^24); the
// int64 chains hold 2^8 segments.  Below: one segment and the widest digits
// that the whole contraction allows.
void oz_plan_gemm(OzGemm &g, int bits)
{
    g.seg = g.nK;
    if (bits >= 55) {
        g.beta = 7;
        g.S = 8;
        const int most = 16777215 / (4096 * (g.S + 2)) / DP_OZ_KC;  // 25 chunks
        const int nseg = (g.nK + most - 1) / most;
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

cudaError_t dp_launch_fit_oz(cudaStream_t st, const DevModel &m, const OzModel &oz, const OzBuffers &ob, int N,
                             const NlistBuffers &nb, EvalBuffers eb, int num_sms, int32_t *status,
                             int64_t *launches)
{
    const int nf = m.n_fit, T = m.ntypes;
    const int tiles = (N + DP_OZ_TILE - 1) / DP_OZ_TILE + T;
    if (tiles > ob.tiles) return cudaErrorInvalidValue;
    {
        cudaError_t e = cudaFuncSetAttribute(k_oz_gemm<8>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)gemm_smem(8));
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k_oz_gemm<5>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gemm_smem(5));
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k_oz_gemm<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gemm_smem(4));
        if (e != cudaSuccess) return e;
    }
    const int K1 = m.m2 * m.M;
    const size_t plane = (size_t)ob.nmax * oz.fmax;
    double *H[2] = {ob.h, ob.h + plane};
    double *G[2] = {ob.g, ob.g + plane};
    // parameter offsets of layer l (W_l, b_l) and of the output layer inside a type's block
    int64_t boff[DP_MAX_LAYERS], wo_off = 0;
    {
        int64_t off = 0;
        int kin = K1;
        for (int l = 0; l < nf; ++l) {
            off += (int64_t)kin * m.fit[l];
            boff[l] = off;
            off += m.fit[l];
            kin = m.fit[l];
        }
        wo_off = off;
    }
    const int split_blocks = tiles * (DP_OZ_TILE / 8);

    auto split = [&](int mode, const double *src, int lds, const double *tv, const OzGemm &g) -> cudaError_t {
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
        a.Ei = eb.Ei;
        a.K = g.K;
        a.nK = g.nK;
        a.beta = g.beta;
        a.S = g.S;
        a.type_perm = nb.type_perm;
        a.type_start = nb.type_start;
        a.ntypes = T;
        a.a = ob.a;
        a.aexp = ob.aexp;
        a.a_stride = ob.a_stride;
        k_oz_split<<<split_blocks, 256, 0, st>>>(a);
        *launches += 1;
        return cudaGetLastError();
    };
    auto gemm = [&](const OzGemm &g, int epi, int skip, int skip_in, int l, const double *hin, int ldh,
                    bool bcast_wout, double *tout, double *hout, int ldo) -> cudaError_t {
        OzGemmArgs a;
        std::memset(&a, 0, sizeof(a));
        a.a = ob.a;
        a.aexp = ob.aexp;
        a.a_stride = ob.a_stride;
        a.w = oz.w;
        a.wexp = oz.wexp;
        a.g = g;
        a.type_perm = nb.type_perm;
        a.type_start = nb.type_start;
        a.ntypes = T;
        a.epi = epi;
        a.skip = skip;
        a.skip_in = skip_in;
        for (int t = 0; t < T; ++t) {
            a.bias[t] = m.params + m.fit_base[t] + boff[l];
            a.gbc[t] = bcast_wout ? m.params + m.fit_base[t] + wo_off : nullptr;
        }
        a.hin = hin;
        a.ldh = ldh;
        a.tout = tout;
        a.hout = hout;
        a.ldo = ldo;
        a.tanh_tab = m.tanh_tab;
        a.status = status;
        a.units = tiles * g.nN;
        const int grid = std::min(a.units, num_sms);
        const size_t smem = gemm_smem(g.S);
        if (g.S == 4) k_oz_gemm<4><<<grid, OZ_THREADS, smem, st>>>(a);
        else if (g.S == 5) k_oz_gemm<5><<<grid, OZ_THREADS, smem, st>>>(a);
        else k_oz_gemm<8><<<grid, OZ_THREADS, smem, st>>>(a);
        *launches += 1;
        return cudaGetLastError();
    };

    cudaError_t e;
    // forward: h_l = skip(h_{l-1}) + tanh(h_{l-1} W_l + b_l), h_{-1} = D
    int kin = K1;
    for (int l = 0; l < nf; ++l) {
        const double *x = l == 0 ? eb.D : H[(l - 1) & 1];
        const int ldx = l == 0 ? K1 : oz.fmax;
        if ((e = split(0, x, ldx, nullptr, oz.fwd[l])) != cudaSuccess) return e;
        if ((e = gemm(oz.fwd[l], 0, dp_skip_kind(kin, m.fit[l]), kin, l, x, ldx, false,
                      ob.t + (size_t)l * plane, H[l & 1], oz.fmax)) != cudaSuccess)
            return e;
        kin = m.fit[l];
    }
    // output layer (E_i) and dL/dz of the last layer (dL/dh = w_out)
    if ((e = split(2, H[(nf - 1) & 1], oz.fmax, ob.t + (size_t)(nf - 1) * plane, oz.bwd[nf - 1])) != cudaSuccess)
        return e;
    // backward: dL/dh_{l-1} = (dL/dz_l) W_l^T + skip'(dL/dh_l)
    for (int l = nf - 1; l >= 0; --l) {
        const int kin_l = l == 0 ? K1 : m.fit[l - 1];
        const bool last = l == nf - 1;
        double *out = l == 0 ? eb.gD : G[(l - 1) & 1];
        const int ldo = l == 0 ? K1 : oz.fmax;
        if ((e = gemm(oz.bwd[l], 1, dp_skip_kind(kin_l, m.fit[l]), kin_l, l, last ? nullptr : G[l & 1], oz.fmax,
                      last, nullptr, out, ldo)) != cudaSuccess)
            return e;
        if (l > 0)
            if ((e = split(1, G[(l - 1) & 1], oz.fmax, ob.t + (size_t)(l - 1) * plane, oz.bwd[l - 1])) != cudaSuccess)
                return e;
    }
    return cudaSuccess;
}
