// embed_cheb.cu -- FP64 environment matrix, embedding net and descriptor
// (Algorithm 2; Eqs. embedding, embedding-first, embedding-rest, descrpt) and
// their backward, with every embedding net as a Chebyshev series in its one
// input s(r).
//
// An embedding net is M functions of the single number s.  They are analytic
// (tanh of affine maps), so their Chebyshev series on s in [0, S] converge
// geometrically: the water, copper and student nets reach 1e-17 of their size
// with 17 to 20 terms.  The series turn the two contractions of the path inside
// out:
//   T_cf  = scale sum_b sum_n P^b_nc C^b_nf,   P^b_nc = sum_rows R~_c T_n(t),
//   dE/dR~_c + ... per row from  U^b_nc = sum_f C^b_nf gT_cf:
//   sum_f G_f gT_cf = sum_n U_nc T_n(t),  sum_f (dG_f/ds) gT_cf = sum_n V_nc T_n(t),
// V the coefficients of the derivative (Mason and Handscomb, Chebyshev
// Polynomials, 2003, sec. 2.4).  A row costs 4 n (forward) and 8 n (backward)
// FMAs instead of a net with its s-derivative and 12 M FMAs; what depends on M
// is done once per atom.  G is never formed.
//
// The coefficients are made on the device when a context first evaluates a set
// of parameters: k_cheb_nodes evaluates the nets at the NN Chebyshev nodes in
// double-double arithmetic (Dekker 1971, Knuth's two-sum), k_cheb_coef the discrete
// transform, also in double-double, so the stored coefficients are the series'
// rounded to FP64.  dp_cheb_terms keeps the terms until the derivative of what
// is left is below 2^-55 of the net's size; a net that 44 terms do not resolve,
// or that the series misses between its nodes (k_cheb_check), makes the context use the kernels of embed_x.cu / embed.cu instead.  Rows
// with s > S (r < 0.75 A, dp_cheb_domain) evaluate the net itself, one row at a time.
//
// What bounds the kernels: the FP64 pipe (16 cycles per warp instruction and SM).
// One 128-thread CTA per atom, several per SM, so that the phases of different
// atoms overlap; rows one per thread, then the per-atom products over (term,
// component) and (component, feature) items, which large boxes take to the tensor
// cores (dp_cheb_gemm).  Measured per evaluation of 139,968 water atoms (20
// terms): forward 159 -> 6.9 ms, backward 25.0 -> 13.5 ms against the kernels of
// embed_x.cu that evaluate the nets and keep G and dG/ds; 32,000 copper atoms: 79
// -> 2.3 and 12.8 -> 4.2 ms; 192 water atoms: 0.37 -> 0.04 and
// 0.17 -> 0.05 ms.  Errors against extended precision are the same (forces
// 1e-15 of their norm on water, 2e-14 on copper, both ways).
#include <cmath>

#include "atom_cta.cuh"
#include "cheb.cuh"

namespace {

constexpr int NN = DP_CHEB_NN;
constexpr int CT = DP_ATOM_CT;  // threads of a CTA = rows of a chunk (128)
constexpr int LDT = CT + 1;   // row pitch of the T_n(t) table (odd: lanes on n hit different banks)
constexpr unsigned FULL = 0xffffffffu;

// ------------------------------------------------------- double-double ------

struct dd {
    double h, l;
};

__device__ __forceinline__ dd two_sum(double a, double b)
{
    const double s = __dadd_rn(a, b), v = __dsub_rn(s, a);
    return {s, __dadd_rn(__dsub_rn(a, __dsub_rn(s, v)), __dsub_rn(b, v))};
}
__device__ __forceinline__ dd quick_sum(double a, double b)
{
    const double s = __dadd_rn(a, b);
    return {s, __dsub_rn(b, __dsub_rn(s, a))};
}
__device__ __forceinline__ dd dd_add(dd a, dd b)
{
    dd s = two_sum(a.h, b.h);
    const dd t = two_sum(a.l, b.l);
    s = quick_sum(s.h, __dadd_rn(s.l, t.h));
    return quick_sum(s.h, __dadd_rn(s.l, t.l));
}
__device__ __forceinline__ dd dd_mul(dd a, dd b)
{
    const double p = __dmul_rn(a.h, b.h);
    double e = __fma_rn(a.h, b.h, -p);
    e = __fma_rn(a.h, b.l, e);
    e = __fma_rn(a.l, b.h, e);
    return quick_sum(p, e);
}
__device__ __forceinline__ dd dd_neg(dd a) { return {-a.h, -a.l}; }
__device__ __forceinline__ dd dd_div(dd a, dd b)
{
    const double q = __ddiv_rn(a.h, b.h);
    dd r = dd_add(a, dd_neg(dd_mul(b, {q, 0.0})));
    const double q2 = __ddiv_rn(r.h, b.h);
    r = dd_add(r, dd_neg(dd_mul(b, {q2, 0.0})));
    return dd_add(quick_sum(q, q2), {__ddiv_rn(r.h, b.h), 0.0});
}

// sin (odd = 1) or cos (odd = 0) of |x| <= pi / 4 by Taylor's series
__device__ dd dd_trig(dd x, int odd)
{
    const dd x2 = dd_neg(dd_mul(x, x));
    dd term = odd ? x : dd{1.0, 0.0}, sum = term;
    for (int k = odd + 1; k < 32; k += 2) {
        term = dd_div(dd_mul(term, x2), {(double)k * (double)(k + 1), 0.0});
        sum = dd_add(sum, term);
    }
    return sum;
}

// tanh of |x| <= 1/64: the odd Taylor series (remainder below 1e-25)
__device__ __forceinline__ dd dd_tanh_small(dd x)
{
    const double u = x.h * x.h;
    double p = 21844.0 / 6081075.0;
    p = fma(p, u, -1382.0 / 155925.0);
    p = fma(p, u, 62.0 / 2835.0);
    p = fma(p, u, -17.0 / 315.0);
    p = fma(p, u, 2.0 / 15.0);
    p = fma(p, u, -1.0 / 3.0);
    return dd_add(x, {x.h * (u * p), 0.0});
}

__global__ void k_cheb_setup(double *__restrict__ trig)
{
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    const dd pi = {3.141592653589793116, 1.2246467991473532e-16};
    if (q < 4 * NN) {
        // cos(pi q / (2 NN)) through the symmetries of the cosine
        int j = q > 2 * NN ? 4 * NN - q : q;
        const bool neg = j > NN;
        if (neg) j = 2 * NN - j;
        const bool s = 2 * j > NN;
        const dd th = dd_div(dd_mul(pi, {(double)(s ? NN - j : j), 0.0}), {2.0 * NN, 0.0});
        dd v = dd_trig(th, s ? 1 : 0);
        if (neg) v = dd_neg(v);
        trig[2 * q] = v.h;
        trig[2 * q + 1] = v.l;
    } else if (q < 4 * NN + DP_CHEB_NTANH) {
        // tanh(k / 32): the series at k / 32 / 2^m <= 1/2048 (remainder 1e-38), doubled m times
        const int k = q - 4 * NN;
        double v = k / 32.0;
        int m = 0;
        for (; v > 1.0 / 2048.0; ++m) v *= 0.5;
        const dd z = {v, 0.0}, u = dd_mul(z, z);
        const double c[7] = {1.0, -1.0, 2.0, -17.0, 62.0, -1382.0, 21844.0};
        const double d[7] = {1.0, 3.0, 15.0, 315.0, 2835.0, 155925.0, 6081075.0};
        dd p = dd_div({c[6], 0.0}, {d[6], 0.0});
        for (int i = 5; i >= 0; --i) p = dd_add(dd_mul(p, u), dd_div({c[i], 0.0}, {d[i], 0.0}));
        dd t = dd_mul(z, p);
        for (; m > 0; --m) t = dd_div(dd_add(t, t), dd_add({1.0, 0.0}, dd_mul(t, t)));
        trig[2 * q] = t.h;
        trig[2 * q + 1] = t.l;
    }
}

// tanh(x) to about 1e-21: tanh(k/32 + t) = (A + B) / (1 + A B); 1 beyond 22
// (1 - tanh(22) = 1.6e-19)
__device__ dd dd_tanh(dd x, const double *__restrict__ tab)
{
    if (!(fabs(x.h) < 22.0)) return x.h != x.h ? x : dd{copysign(1.0, x.h), 0.0};
    const bool neg = x.h < 0.0;
    if (neg) x = dd_neg(x);
    const int k = (int)rint(x.h * 32.0);
    const dd A = {tab[2 * k], tab[2 * k + 1]};
    const dd B = dd_tanh_small(dd_add(x, {-k / 32.0, 0.0}));
    const dd t = dd_div(dd_add(A, B), dd_add({1.0, 0.0}, dd_mul(A, B)));
    return neg ? dd_neg(t) : t;
}

// One CTA per (net, node): the net at s_k = S/2 (1 + cos(pi (2k+1) / (2 NN))),
// thread o on output o of each layer.
__global__ void __launch_bounds__(CT) k_cheb_nodes(DevModel m, double scale, const double *__restrict__ trig,
                                                   double *__restrict__ y)
{
    __shared__ dd h[2][DP_MAX_EMB_W];
    const int net = blockIdx.x / NN, k = blockIdx.x % NN, o = threadIdx.x;
    const double *W = m.params + m.emb_base[net];
    const int q = 2 * k + 1;
    dd s = dd_add({1.0, 0.0}, {trig[2 * q], trig[2 * q + 1]});
    s = dd_div(s, {scale, 0.0});
    const double *tab = trig + 2 * 4 * NN;
    int win = m.emb[0], cur = 0;
    if (o < win) h[0][o] = dd_tanh(dd_add(dd_mul(s, {W[o], 0.0}), {W[win + o], 0.0}), tab);
    W += 2 * win;
    for (int l = 1; l < m.n_emb; ++l) {
        __syncthreads();
        const int wout = m.emb[l], sk = dp_skip_kind(win, wout);
        if (o < wout) {
            dd z = {W[win * wout + o], 0.0};
            for (int p = 0; p < win; ++p) z = dd_add(z, dd_mul(h[cur][p], {W[p * wout + o], 0.0}));
            z = dd_tanh(z, tab);
            if (sk) z = dd_add(z, h[cur][o < win ? o : o - win]);
            h[cur ^ 1][o] = z;
        }
        W += win * wout + wout;
        win = wout;
        cur ^= 1;
    }
    if (o < m.M) {
        double *out = y + ((size_t)blockIdx.x * m.M + o) * 2;
        out[0] = h[cur][o].h;   // each thread reads what it wrote
        out[1] = h[cur][o].l;
    }
}

// One CTA per (net, n): C_n = (2 - [n = 0]) / NN sum_k cos(pi n (2k+1) / (2 NN)) y_k
__global__ void __launch_bounds__(CT) k_cheb_coef(DevModel m, const double *__restrict__ trig,
                                                  const double *__restrict__ y, double *__restrict__ C,
                                                  double *__restrict__ Ct, double *__restrict__ mx)
{
    __shared__ double wm[CT / 32];
    const int net = blockIdx.x / NN, n = blockIdx.x % NN, f = threadIdx.x, M = m.M, T = m.ntypes;
    double v = 0.0;
    if (f < M) {
        dd acc = {0.0, 0.0};
        for (int k = 0; k < NN; ++k) {
            const int j = (n * (2 * k + 1)) % (4 * NN);
            const double *yk = y + ((size_t)(net * NN + k) * M + f) * 2;
            acc = dd_add(acc, dd_mul({trig[2 * j], trig[2 * j + 1]}, {yk[0], yk[1]}));
        }
        acc = dd_div(acc, {n == 0 ? (double)NN : 0.5 * NN, 0.0});
        v = acc.h;
        C[(size_t)blockIdx.x * M + f] = v;
        Ct[((size_t)(net / T) * M + f) * (T * NN) + (net % T) * NN + n] = v;
    }
    v = fabs(v);
    bool bad = !(v <= 1e300);
    for (int s = 16; s > 0; s >>= 1) v = fmax(v, __shfl_xor_sync(FULL, v, s));
    if ((f & 31) == 0) wm[f >> 5] = v;
    bad = __syncthreads_or(bad);
    if (f == 0) {
        for (int w = 1; w < CT / 32; ++w) v = fmax(v, wm[w]);
        mx[blockIdx.x] = bad ? 1e301 : v;
    }
}

// Coefficients of the derivative, V_n = (2 / S) (2 - [n = 0]) sum_{m = n+1, n+3, ..} m C_m
// (the terms decrease geometrically: smallest first).
__global__ void __launch_bounds__(CT) k_cheb_deriv(DevModel m, double scale, const double *__restrict__ C,
                                                   double *__restrict__ V)
{
    const int net = blockIdx.x / NN, n = blockIdx.x % NN, f = threadIdx.x;
    if (f >= m.M) return;
    double v = 0.0;
    for (int q = NN - 1 - (NN - n) % 2; q > n; q -= 2) v = fma((double)q, C[(size_t)(net * NN + q) * m.M + f], v);
    V[(size_t)blockIdx.x * m.M + f] = v * ((n == 0 ? 1.0 : 2.0) * scale);
}

// ---------------------------------------------------------- rows beyond S ---

// The net with its s-derivative at s, by the whole CTA (rows with s > S only):
// G in ga[0..M), dG/ds in da.  ga, da, gb, db: DP_MAX_EMB_W doubles each.
__device__ void net_direct(const DevModel &m, int net, double s, double *&ga, double *&da, double *&gb, double *&db)
{
    const int o = threadIdx.x;
    const double *W = m.params + m.emb_base[net];
    int win = m.emb[0];
    __syncthreads();
    if (o < win) {
        const double w0 = W[o], t = dp_tanh64(fma(s, w0, W[win + o]), m.tanh_tab);
        ga[o] = t;
        da[o] = fma(-t, t, 1.0) * w0;
    }
    W += 2 * win;
    for (int l = 1; l < m.n_emb; ++l) {
        __syncthreads();
        const int wout = m.emb[l], sk = dp_skip_kind(win, wout);
        if (o < wout) {
            double z = W[win * wout + o], dz = 0.0;
            for (int p = 0; p < win; ++p) {
                const double w = W[p * wout + o];
                z = fma(ga[p], w, z);
                dz = fma(da[p], w, dz);
            }
            const double t = dp_tanh64(z, m.tanh_tab);
            const int os = o < win ? o : o - win;
            gb[o] = t + (sk ? ga[os] : 0.0);
            db[o] = fma(fma(-t, t, 1.0), dz, sk ? da[os] : 0.0);
        }
        double *u = ga;
        ga = gb;
        gb = u;
        u = da;
        da = db;
        db = u;
        W += win * wout + wout;
        win = wout;
    }
    __syncthreads();
}

// Type block of row q of the atom (rows of all blocks one after the other);
// start[b] is the first row of block b, start[T] the number of rows.
__device__ __forceinline__ int row_block(const int *start, int T, int q)
{
    int b = 0;
    while (b + 1 < T && q >= start[b + 1]) ++b;
    return b;
}

// The series (all NN terms) against the net in FP64 at the points between the nodes
// and the ends of the domain, s = S/2 (1 + cos(pi j / NN)): a unit that turns between
// two nodes (at s = 0 the first node is at S / 3734) leaves coefficients that look
// resolved.  Where they differ by more than 2^-40 of the net's size, mx marks the net
// as not resolved.  One CTA per (net, point).
__global__ void __launch_bounds__(CT) k_cheb_check(DevModel m, double scale, const double *__restrict__ trig,
                                                   const double *__restrict__ C, double *__restrict__ mx)
{
    __shared__ double fbuf[4][DP_MAX_EMB_W];
    __shared__ double wm[CT / 32];
    const int net = blockIdx.x / (NN + 1), j = blockIdx.x % (NN + 1), f = threadIdx.x, M = m.M;
    const double t = trig[4 * j], t2 = t + t;
    double *ga = fbuf[0], *da = fbuf[1], *gb = fbuf[2], *db = fbuf[3];
    net_direct(m, net, (1.0 + t) / scale, ga, da, gb, db);
    double diff = 0.0, size = 0.0;
    if (f < M) {
        double v = 0.0, p0 = 1.0, p1 = t;
#pragma unroll 8
        for (int n = 0; n < NN; ++n) {
            const double c = C[(size_t)(net * NN + n) * M + f], p2 = fma(t2, p1, -p0);
            v = fma(c, p0, v);
            size = fmax(size, fabs(c));
            p0 = p1;
            p1 = p2;
        }
        diff = fabs(v - ga[f]);
    }
    for (int s = 16; s > 0; s >>= 1) size = fmax(size, __shfl_xor_sync(FULL, size, s));
    if ((f & 31) == 0) wm[f >> 5] = size;
    __syncthreads();
    for (int w = 0; w < CT / 32; ++w) size = fmax(size, wm[w]);
    if (__syncthreads_or(!(diff <= 0x1p-40 * size)) && f == 0) mx[net * NN] = 1e301;
}

// Adds the rows beyond S to T (Ts [4][M], scaled), in row order, by the whole CTA.
__device__ __forceinline__ void far_rows_T(const DevModel &m, double S, int a, int i, const int *start,
                                           double (&fbuf)[4][DP_MAX_EMB_W], const double *pair_d, double *Ts)
{
    const int T = m.ntypes, M = m.M, tid = threadIdx.x;
    const double irc = 1.0 / (m.rcut - m.rcut_smth);
    double *ga = fbuf[0], *da = fbuf[1], *gb = fbuf[2], *db = fbuf[3];
    for (int q = 0; q < start[T]; ++q) {
        const int b = row_block(start, T, q);
        const double *d = pair_d + ((size_t)i * m.nm + m.sel_off[b] + (q - start[b])) * 3;
        const double dv[3] = {d[0], d[1], d[2]};
        const double r = __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(dv[0], dv[0]), __dmul_rn(dv[1], dv[1])),
                                              __dmul_rn(dv[2], dv[2])));
        double s, ds, inv;
        dp_switch_inv(r, m.rcut_smth, m.rcut, irc, s, ds, inv);
        if (s <= S) continue;  // uniform: every thread has the same row
        net_direct(m, a * T + b, s, ga, da, gb, db);
        const double sr = s * inv;
        for (int p = tid; p < 4 * M; p += CT) {
            const int c = p / M;
            Ts[p] += (c == 0 ? s : sr * dv[c - 1]) * ga[p - c * M] * m.desc_scale;
        }
        __syncthreads();
    }
}

// D = T_<^T T of one atom by the whole CTA.
__device__ __forceinline__ void descriptor(const DevModel &m, int i, const double *Ts, double *__restrict__ Dout)
{
    const int M = m.M, nd = m.m2 * M;
    for (int q = threadIdx.x; q < nd; q += CT) {
        const int a2 = q / M, b2 = q - a2 * M;
        double acc = Ts[a2] * Ts[b2];
        acc = fma(Ts[M + a2], Ts[M + b2], acc);
        acc = fma(Ts[2 * M + a2], Ts[2 * M + b2], acc);
        acc = fma(Ts[3 * M + a2], Ts[3 * M + b2], acc);
        Dout[(size_t)i * nd + q] = acc;
    }
}

// ---------------------------------------------------------------- forward ---

// MOM: the CTA stops at the scaled moments, written to Tout as [4][T nc] rows of
// the atom, with a flag in Dout[i] when it has rows beyond S; T and D follow in
// other kernels (dp_launch_cheb_fwd).
template <bool MOM>
__global__ void __launch_bounds__(CT) k_cheb_fwd(DevModel m, ChebModel cm, const double *__restrict__ x,
                                                 const int32_t *__restrict__ types, Box3 box,
                                                 const int32_t *__restrict__ type_perm,
                                                 const int32_t *__restrict__ nlist, const int32_t *__restrict__ nreal,
                                                 double *__restrict__ pair_d, double *__restrict__ Tout,
                                                 double *__restrict__ Dout)
{
    extern __shared__ __align__(16) double sm[];
    const int nc = cm.n, M = m.M, T = m.ntypes, nm = m.nm, tid = threadIdx.x;
    double *R4 = sm;                       // [CT][4] rows of R~
    double *part = R4 + CT * 4;            // [2][CT][4] moment partials of the row slices
    double *Mom = part + 2 * CT * 4;       // [T nc][4]
    double *Ts = Mom + T * nc * 4;         // [4][M]
    double *Tch = Ts + 4 * M;              // [nc][LDT] T_n(t) of the chunk's rows
    __shared__ int start[DP_MAX_TYPES + 1];
    __shared__ double fbuf[4][DP_MAX_EMB_W];  // rows beyond S
    const int i = type_perm[blockIdx.x];
    const int a = types[i];
    const bool a_ok = (unsigned)a < (unsigned)T;
    if (tid == 0) {
        int r = 0;
        for (int b = 0; b < T; ++b) {
            start[b] = r;
            r += a_ok ? nreal[(size_t)i * T + b] : 0;
        }
        start[T] = r;
    }
    for (int p = tid; p < T * nc * 4; p += CT) Mom[p] = 0.0;
    __syncthreads();
    const int R = start[T];
    const double xi[3] = {x[3 * i], x[3 * i + 1], x[3 * i + 2]};
    const double irc = 1.0 / (m.rcut - m.rcut_smth);
    const int ns = CT / nc;                    // row slices of the moment sums
    const int mn = tid % nc, msl = tid / nc;   // this thread's term and slice
    bool any_far = false;
    int seg = 0;
    for (int c0 = 0; c0 < R; c0 += CT) {
        const int q = c0 + tid;
        bool far = false;
        if (q < R) {
            const int b = row_block(start, T, q);
            const size_t slot = (size_t)i * nm + m.sel_off[b] + (q - start[b]);
            const int j = nlist[slot];
            const double xj[3] = {x[3 * j], x[3 * j + 1], x[3 * j + 2]};
            double d[3], s, ds, inv;
            dp_switch_inv(dp_pinned_dist(xi, xj, box, d), m.rcut_smth, m.rcut, irc, s, ds, inv);
            pair_d[slot * 3] = d[0];
            pair_d[slot * 3 + 1] = d[1];
            pair_d[slot * 3 + 2] = d[2];
            const double sr = s * inv;
            far = !(s <= cm.S);
            double *Rq = R4 + tid * 4;
            Rq[0] = far ? 0.0 : s;
            Rq[1] = far ? 0.0 : sr * d[0];
            Rq[2] = far ? 0.0 : sr * d[1];
            Rq[3] = far ? 0.0 : sr * d[2];
            const double t = far ? 0.0 : fma(s, cm.scale, -1.0), t2 = t + t;
            double p0 = 1.0, p1 = t;
            Tch[tid] = 1.0;
            for (int n = 1; n < nc; ++n) {
                Tch[n * LDT + tid] = p1;
                const double p2 = fma(t2, p1, -p0);
                p0 = p1;
                p1 = p2;
            }
        }
        any_far = __syncthreads_or(far) || any_far;
        for (int b = 0; b < T; ++b) {
            const int lo = max(start[b] - c0, 0), hi = min(start[b + 1] - c0, CT);
            if (lo >= hi) continue;
            double *pt = part + (seg & 1) * CT * 4;
            if (msl < ns) {
                double acc[4] = {0.0, 0.0, 0.0, 0.0};
                const double *tn = Tch + mn * LDT;
                for (int r = lo + msl; r < hi; r += ns) {
                    const double tv = tn[r];
                    const double2 u = *reinterpret_cast<const double2 *>(R4 + r * 4);
                    const double2 w = *reinterpret_cast<const double2 *>(R4 + r * 4 + 2);
                    acc[0] = fma(tv, u.x, acc[0]);
                    acc[1] = fma(tv, u.y, acc[1]);
                    acc[2] = fma(tv, w.x, acc[2]);
                    acc[3] = fma(tv, w.y, acc[3]);
                }
#pragma unroll
                for (int c = 0; c < 4; ++c) pt[tid * 4 + c] = acc[c];
            }
            __syncthreads();
            for (int p = tid; p < nc * 4; p += CT) {
                double v = Mom[b * nc * 4 + p];
                for (int u = 0; u < ns; ++u) v += pt[u * nc * 4 + p];
                Mom[b * nc * 4 + p] = v;
            }
            ++seg;
        }
        __syncthreads();
    }
    if constexpr (MOM) {
        for (int p = tid; p < T * nc * 4; p += CT)
            Tout[((size_t)i * 4 + (p & 3)) * (T * nc) + (p >> 2)] = Mom[p] * m.desc_scale;
        if (tid == 0) Dout[i] = any_far ? 1.0 : 0.0;
        return;
    }
    // T = scale sum_k P_k C_k, items (c, f)
    {
        const double *C = cm.C + (size_t)(a_ok ? a : 0) * T * NN * M;
        for (int p0 = tid; p0 < 4 * M; p0 += 4 * CT) {
            double acc[4] = {0.0, 0.0, 0.0, 0.0};
            int c[4], f[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int p = p0 + u * CT;
                c[u] = p / M;
                f[u] = p - c[u] * M;
            }
            for (int b = 0; b < T; ++b) {
                if (start[b] == start[b + 1]) continue;
                const double *Cb = C + (size_t)b * NN * M, *mo = Mom + b * nc * 4;
#pragma unroll 4
                for (int n = 0; n < nc; ++n)
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (p0 + u * CT < 4 * M) acc[u] = fma(mo[n * 4 + c[u]], Cb[n * M + f[u]], acc[u]);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (p0 + u * CT < 4 * M) Ts[p0 + u * CT] = acc[u] * m.desc_scale;
        }
    }
    __syncthreads();
    if (any_far) far_rows_T(m, cm.S, a, i, start, fbuf, pair_d, Ts);
    for (int p = tid; p < 4 * M; p += CT) Tout[(size_t)i * 4 * M + p] = Ts[p];
    descriptor(m, i, Ts, Dout);
}

// T of one atom finished (rows beyond S added) and D = T_<^T T, one CTA per atom.
__global__ void __launch_bounds__(CT) k_cheb_desc(DevModel m, double S, const int32_t *__restrict__ types,
                                                  const int32_t *__restrict__ type_perm,
                                                  const int32_t *__restrict__ nreal, const double *__restrict__ flag,
                                                  const double *__restrict__ pair_d, double *__restrict__ Tio,
                                                  double *__restrict__ Dout)
{
    __shared__ double Ts[4 * DP_MAX_EMB_W];
    __shared__ int start[DP_MAX_TYPES + 1];
    __shared__ double fbuf[4][DP_MAX_EMB_W];
    const int M = m.M, T = m.ntypes, tid = threadIdx.x;
    const int i = type_perm[blockIdx.x];
    for (int p = tid; p < 4 * M; p += CT) Ts[p] = Tio[(size_t)i * 4 * M + p];
    const bool far = flag[i] != 0.0;
    if (far && tid == 0) {
        int r = 0;
        for (int b = 0; b < T; ++b) {
            start[b] = r;
            r += nreal[(size_t)i * T + b];
        }
        start[T] = r;
    }
    __syncthreads();
    if (far) {
        far_rows_T(m, S, types[i], i, start, fbuf, pair_d, Ts);
        for (int p = tid; p < 4 * M; p += CT) Tio[(size_t)i * 4 * M + p] = Ts[p];
    }
    descriptor(m, i, Ts, Dout);
}

// dE/dT of one atom per CTA, as [4][M].
__global__ void __launch_bounds__(CT) k_cheb_gT(DevModel m, const int32_t *__restrict__ type_perm,
                                                const double *__restrict__ Tin, const double *__restrict__ gD,
                                                double *__restrict__ gT)
{
    extern __shared__ __align__(16) double sm[];
    const int M = m.M, m2 = m.m2, tid = threadIdx.x, LDG = M | 1;
    double *Ts = sm, *lp = Ts + 4 * M, *gs = lp + 8 * m2;
    const size_t i = type_perm[blockIdx.x];
    for (int p = tid; p < 4 * M; p += CT) Ts[p] = Tin[i * 4 * M + p];
    for (int p = tid; p < m2 * M; p += CT) gs[(p / M) * LDG + p % M] = gD[i * m2 * M + p];
    __syncthreads();
    dp_atom_gT(gs, LDG, Ts, lp, m2, M, m.desc_scale, [&](int c, int xx, double v) { gT[(i * 4 + c) * M + xx] = v; });
}

// --------------------------------------------------------------- backward ---

// PRE: dE/dT (gD, as [4][M]) and U (Tin, as [4][T nc]) of the atom are there already.
template <bool PRE>
__global__ void __launch_bounds__(CT) k_cheb_bwd(DevModel m, ChebModel cm, const int32_t *__restrict__ types,
                                                 const int32_t *__restrict__ type_perm,
                                                 const int32_t *__restrict__ nreal, const double *__restrict__ Tin,
                                                 const double *__restrict__ gD, double *__restrict__ pair_g,
                                                 double *__restrict__ f_own, double *__restrict__ vir_part)
{
    extern __shared__ __align__(16) double sm[];
    const int nc = cm.n, M = m.M, m2 = m.m2, T = m.ntypes, nm = m.nm, tid = threadIdx.x;
    const int Kt = T * nc, LDG = M | 1;
    double *UV = sm;                        // [Kt][8]: U_nc, V_nc
    double *g4 = UV + Kt * 8;               // [M][4]: gT_cf
    double *Ts = g4 + M * 4;                // [4][M]
    double *lp = Ts + 4 * M;                // [2][4][m2] partial long sums
    double *gs = lp + 8 * m2;               // [m2][LDG] dE/dD, then [slices][Kt][4] partials of U
    __shared__ int start[DP_MAX_TYPES + 1];
    __shared__ double fbuf[4][DP_MAX_EMB_W];
    __shared__ double fsum[CT / 32][8], wsum[CT / 32][16];
    __shared__ unsigned farbits[(DP_MAX_NM + CT) / 32];
    const int i = type_perm[blockIdx.x];
    const int a = types[i];
    const bool a_ok = (unsigned)a < (unsigned)T;
    if (tid == 0) {
        int r = 0;
        for (int b = 0; b < T; ++b) {
            start[b] = r;
            r += a_ok ? nreal[(size_t)i * T + b] : 0;
        }
        start[T] = r;
    }
    if constexpr (PRE) {
        for (int p = tid; p < Kt * 4; p += CT) UV[(p % Kt) * 8 + p / Kt] = Tin[(size_t)i * 4 * Kt + p];
    } else {
        for (int p = tid; p < 4 * M; p += CT) Ts[p] = Tin[(size_t)i * 4 * M + p];
        {
            const double *g = gD + (size_t)i * m2 * M;
            for (int p = tid; p < m2 * M; p += CT) gs[(p / M) * LDG + p % M] = g[p];
        }
        __syncthreads();
        dp_atom_gT(gs, LDG, Ts, lp, m2, M, m.desc_scale, [&](int c, int xx, double v) { g4[xx * 4 + c] = v; });
        __syncthreads();
        // U_kc = sum_f C_kf gT_cf: thread = (term k of the centre's nets, feature slice)
        {
            const double *Ct = cm.Ct + (size_t)(a_ok ? a : 0) * M * T * NN;
            const int nsl = Kt < CT ? CT / Kt : 1;
            for (int p = tid; p < Kt * nsl; p += CT) {
                const int fs = p / Kt, k = p - fs * Kt, b = k / nc;
                const double *ck = Ct + b * NN + (k - b * nc);
                double acc[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
                for (int f = fs; f < M; f += nsl) {
                    const double cv = ck[(size_t)f * T * NN];
                    const double2 u = *reinterpret_cast<const double2 *>(g4 + f * 4);
                    const double2 w = *reinterpret_cast<const double2 *>(g4 + f * 4 + 2);
                    acc[0] = fma(cv, u.x, acc[0]);
                    acc[1] = fma(cv, u.y, acc[1]);
                    acc[2] = fma(cv, w.x, acc[2]);
                    acc[3] = fma(cv, w.y, acc[3]);
                }
#pragma unroll
                for (int c = 0; c < 4; ++c) gs[p * 4 + c] = acc[c];
            }
            __syncthreads();
            for (int p = tid; p < Kt * 4; p += CT) {
                double v = gs[p];
                for (int u = 1; u < nsl; ++u) v += gs[u * Kt * 4 + p];
                UV[(p >> 2) * 8 + (p & 3)] = v;
            }
        }
        __syncthreads();
    }
    __syncthreads();
    const int R = start[T];
    // V: the derivative's coefficients, d/ds = (2 / S) d/dt, v_n = (2 - [n = 0]) sum_{m = n+1, n+3, ..} m u_m
    for (int p = tid; p < Kt * 4; p += CT) {
        const int k = p >> 2, c = p & 3, b = k / nc, n = k - b * nc;
        const double *u = UV + b * nc * 8 + c;
        double v = 0.0;
        for (int q = n + 1; q < nc; q += 2) v = fma((double)q, u[q * 8], v);
        UV[k * 8 + 4 + c] = v * ((n == 0 ? 1.0 : 2.0) * cm.scale);
    }
    __syncthreads();

    const double irc = 1.0 / (m.rcut - m.rcut_smth);
    double fo[3] = {0.0, 0.0, 0.0}, vir[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) vir[q] = 0.0;
    // pair gradient of a row from its sums P_c = sum_f G_f gT_cf and Q = sum_c R~_c sum_f (dG_f/ds) gT_cf
    auto chain = [&](double *pg, const double *d, double inv, double s, double ds, const double *P, double Q) {
        const double u[3] = {d[0] * inv, d[1] * inv, d[2] * inv};
        const double dot = P[1] * u[0] + P[2] * u[1] + P[3] * u[2];
        const double sr = s * inv;
        const double coef = (P[0] + Q) * ds + ds * dot - sr * dot;
#pragma unroll
        for (int e = 0; e < 3; ++e) {
            const double gv = fma(u[e], coef, sr * P[1 + e]);
            pg[e] = gv;
            fo[e] += gv;
#pragma unroll
            for (int f = 0; f < 3; ++f) vir[f * 3 + e] -= d[f] * gv;
        }
    };
    auto radius = [](const double *d) {
        return __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(d[0], d[0]), __dmul_rn(d[1], d[1])), __dmul_rn(d[2], d[2])));
    };
    bool any_far = false;
    for (int c0 = 0; c0 < R; c0 += CT) {
        const int q = c0 + tid;
        bool far = false;
        if (q < R) {
            const int b = row_block(start, T, q);
            double *pg = pair_g + ((size_t)i * nm + m.sel_off[b] + (q - start[b])) * 3;
            const double d[3] = {pg[0], pg[1], pg[2]};
            double s, ds, inv;
            dp_switch_inv(radius(d), m.rcut_smth, m.rcut, irc, s, ds, inv);
            far = !(s <= cm.S);
            if (!far) {
                const double sr = s * inv;
                const double t = fma(s, cm.scale, -1.0), t2 = t + t;
                const double2 *uv = reinterpret_cast<const double2 *>(UV + b * nc * 8);
                double P[4] = {uv[0].x, uv[0].y, uv[1].x, uv[1].y};
                double Qc[4] = {uv[2].x, uv[2].y, uv[3].x, uv[3].y};
                double p0 = 1.0, p1 = t;
#pragma unroll 2
                for (int n = 1; n < nc; ++n) {
                    const double2 a0 = uv[n * 4], a1 = uv[n * 4 + 1], a2 = uv[n * 4 + 2], a3 = uv[n * 4 + 3];
                    P[0] = fma(a0.x, p1, P[0]);
                    P[1] = fma(a0.y, p1, P[1]);
                    P[2] = fma(a1.x, p1, P[2]);
                    P[3] = fma(a1.y, p1, P[3]);
                    Qc[0] = fma(a2.x, p1, Qc[0]);
                    Qc[1] = fma(a2.y, p1, Qc[1]);
                    Qc[2] = fma(a3.x, p1, Qc[2]);
                    Qc[3] = fma(a3.y, p1, Qc[3]);
                    const double p2 = fma(t2, p1, -p0);
                    p0 = p1;
                    p1 = p2;
                }
                chain(pg, d, inv, s, ds, P, s * Qc[0] + sr * (d[0] * Qc[1] + d[1] * Qc[2] + d[2] * Qc[3]));
            }
        }
        const unsigned bal = __ballot_sync(FULL, far);
        if ((tid & 31) == 0) farbits[(c0 + tid) >> 5] = bal;
        any_far |= far;
    }
    if (__syncthreads_or(any_far)) {
        // rows beyond S in row order; their d is still in place
        double *ga = fbuf[0], *da = fbuf[1], *gb = fbuf[2], *db = fbuf[3];
        if constexpr (PRE) {
            for (int p = tid; p < 4 * M; p += CT) g4[(p % M) * 4 + p / M] = gD[(size_t)i * 4 * M + p];
            __syncthreads();
        }
        for (int q = 0; q < R; ++q) {
            if (!((farbits[q >> 5] >> (q & 31)) & 1u)) continue;
            const int b = row_block(start, T, q);
            double *pg = pair_g + ((size_t)i * nm + m.sel_off[b] + (q - start[b])) * 3;
            const double d[3] = {pg[0], pg[1], pg[2]};
            double s, ds, inv;
            dp_switch_inv(radius(d), m.rcut_smth, m.rcut, irc, s, ds, inv);
            net_direct(m, a * T + b, s, ga, da, gb, db);
            double p[8];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                p[c] = tid < M ? ga[tid] * g4[tid * 4 + c] : 0.0;
                p[4 + c] = tid < M ? da[tid] * g4[tid * 4 + c] : 0.0;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int c = 0; c < 8; ++c) p[c] += __shfl_xor_sync(FULL, p[c], o);
            if ((tid & 31) == 0)
#pragma unroll
                for (int c = 0; c < 8; ++c) fsum[tid >> 5][c] = p[c];
            __syncthreads();
            if (tid == 0) {
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    for (int w = 1; w < CT / 32; ++w) p[c] += fsum[w][c];
                const double sr = s * inv;
                chain(pg, d, inv, s, ds, p, s * p[4] + sr * (d[0] * p[5] + d[1] * p[6] + d[2] * p[7]));
            }
            __syncthreads();
        }
    }
    dp_atom_sum12(fo, vir, wsum, f_own, vir_part, i);
}

// ------------------------------------------------- parameter gradient ------
//
// Phi = sum_i (cE E_i - dE_i) with dE_i the tangent of E_i along
// delta r_ij = lambda_j - lambda_i (csrc/pgrad.cu).  With the moments
//   P_n = sum_rows R~ T_n,  dP_n = sum_rows dR~ T_n,  Q_n = sum_rows R~ ds T_n,
// T = scale P C and dT = scale (dP C + Q V).  The adjoints of C and V are sums
// over the atoms, sum (P Tb + dP dTb) and sum Q dTb; both go back through the
// discrete transform to the net's values and derivatives at the NN nodes, and
// reverse mode runs through the net with its s-tangent at NN points instead of
// at every row.  (Folding V's adjoint into C's would multiply it by n^2 and
// lose two digits to the cancellation over the nodes.)  12,288 water atoms,
// student widths: 70 -> 4.2 ms (the net, its tangent and its reverse mode at
// every row before); 648 atoms, full width: 13.8 -> 0.6 ms.

constexpr int PM = 12;  // moments per term: P, dP, Q (4 components each)

// T, dT, D, dD and the moments of one atom per CTA, as k_cheb_fwd with the tangent.
__global__ void __launch_bounds__(CT) k_chebpg_fwd(DevModel m, ChebModel cm, const double *__restrict__ x,
                                                   const int32_t *__restrict__ types, Box3 box,
                                                   const double *__restrict__ lam,
                                                   const int32_t *__restrict__ type_perm,
                                                   const int32_t *__restrict__ nlist,
                                                   const int32_t *__restrict__ nreal, double *__restrict__ Tout,
                                                   double *__restrict__ dTout, double *__restrict__ Dout,
                                                   double *__restrict__ dDout, double *__restrict__ momout,
                                                   int32_t *far_flag)
{
    extern __shared__ __align__(16) double sm[];
    const int nc = cm.n, M = m.M, T = m.ntypes, nm = m.nm, tid = threadIdx.x;
    double *RM = sm;                       // [CT][PM] R~, dR~, R~ ds
    double *part = RM + CT * PM;           // [CT][PM]
    double *Mom = part + CT * PM;          // [T nc][PM]
    double *Ts = Mom + T * nc * PM;        // [8][M] T, dT
    double *Tch = Ts + 8 * M;              // [nc][LDT] T_n(t)
    __shared__ int start[DP_MAX_TYPES + 1];
    const int i = type_perm[blockIdx.x];
    const int a = types[i];
    const bool a_ok = (unsigned)a < (unsigned)T;
    if (tid == 0) {
        int r = 0;
        for (int b = 0; b < T; ++b) {
            start[b] = r;
            r += a_ok ? nreal[(size_t)i * T + b] : 0;
        }
        start[T] = r;
    }
    for (int p = tid; p < T * nc * PM; p += CT) Mom[p] = 0.0;
    __syncthreads();
    const int R = start[T];
    const double xi[3] = {x[3 * i], x[3 * i + 1], x[3 * i + 2]};
    const double li[3] = {lam[3 * i], lam[3 * i + 1], lam[3 * i + 2]};
    const double irc = 1.0 / (m.rcut - m.rcut_smth);
    const int ns = CT / nc, mn = tid % nc, msl = tid / nc;
    bool any_far = false;
    for (int c0 = 0; c0 < R; c0 += CT) {
        const int q = c0 + tid;
        if (q < R) {
            const int b = row_block(start, T, q);
            const int j = nlist[(size_t)i * nm + m.sel_off[b] + (q - start[b])];
            const double xj[3] = {x[3 * j], x[3 * j + 1], x[3 * j + 2]};
            double d[3], s, ds, inv;
            dp_switch_inv(dp_pinned_dist(xi, xj, box, d), m.rcut_smth, m.rcut, irc, s, ds, inv);
            const double u[3] = {d[0] * inv, d[1] * inv, d[2] * inv};
            const double dr[3] = {lam[3 * j] - li[0], lam[3 * j + 1] - li[1], lam[3 * j + 2] - li[2]};
            const double udr = u[0] * dr[0] + u[1] * dr[1] + u[2] * dr[2];
            double *Rq = RM + tid * PM;
            const double dst = ds * udr;  // the tangent of s
            Rq[0] = s;
            Rq[4] = dst;
            Rq[8] = s * dst;
#pragma unroll
            for (int e = 0; e < 3; ++e) {
                Rq[1 + e] = s * u[e];
                Rq[5 + e] = dst * u[e] + s * inv * (dr[e] - u[e] * udr);
                Rq[9 + e] = s * u[e] * dst;
            }
            any_far |= !(s <= cm.S);
            const double t = fma(s, cm.scale, -1.0), t2 = t + t;
            double p0 = 1.0, p1 = t;
            Tch[tid] = 1.0;
            for (int n = 1; n < nc; ++n) {
                Tch[n * LDT + tid] = p1;
                const double p2 = fma(t2, p1, -p0);
                p0 = p1;
                p1 = p2;
            }
        }
        __syncthreads();
        for (int b = 0; b < T; ++b) {
            const int lo = max(start[b] - c0, 0), hi = min(start[b + 1] - c0, CT);
            if (lo >= hi) continue;
            if (msl < ns) {
                double acc[PM];
#pragma unroll
                for (int c = 0; c < PM; ++c) acc[c] = 0.0;
                for (int r = lo + msl; r < hi; r += ns) {
                    const double tv = Tch[mn * LDT + r];
                    const double *Rq = RM + r * PM;
#pragma unroll
                    for (int c = 0; c < PM; ++c) acc[c] = fma(tv, Rq[c], acc[c]);
                }
#pragma unroll
                for (int c = 0; c < PM; ++c) part[tid * PM + c] = acc[c];
            }
            __syncthreads();
            for (int p = tid; p < nc * PM; p += CT) {
                double v = Mom[b * nc * PM + p];
                for (int u = 0; u < ns; ++u) v += part[u * nc * PM + p];
                Mom[b * nc * PM + p] = v;
            }
            __syncthreads();
        }
    }
    if (any_far) atomicOr(far_flag, 1);
    for (int p = tid; p < T * nc * PM; p += CT) momout[(size_t)i * T * nc * PM + p] = Mom[p];
    {
        const size_t net0 = (size_t)(a_ok ? a : 0) * T * NN * M;
        for (int p = tid; p < 8 * M; p += CT) {
            const int c = p / M, f = p - c * M;
            double acc = 0.0;
            for (int b = 0; b < T; ++b) {
                if (start[b] == start[b + 1]) continue;
                const double *Cb = cm.C + net0 + (size_t)b * NN * M + f, *Vb = cm.V + net0 + (size_t)b * NN * M + f;
                const double *mo = Mom + b * nc * PM + c;
                if (c < 4) {
#pragma unroll 4
                    for (int n = 0; n < nc; ++n) acc = fma(mo[n * PM], Cb[n * M], acc);
                } else {
#pragma unroll 4
                    for (int n = 0; n < nc; ++n)
                        acc = fma(mo[n * PM], Cb[n * M], fma(mo[n * PM + 4], Vb[n * M], acc));
                }
            }
            Ts[p] = acc * m.desc_scale;
        }
    }
    __syncthreads();
    for (int p = tid; p < 4 * M; p += CT) {
        Tout[(size_t)i * 4 * M + p] = Ts[p];
        dTout[(size_t)i * 4 * M + p] = Ts[4 * M + p];
    }
    const int nd = m.m2 * M;
    for (int q = tid; q < nd; q += CT) {
        const int a2 = q / M, b2 = q - a2 * M;
        double acc = 0.0, dacc = 0.0;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const double ta = Ts[c * M + a2], tb = Ts[c * M + b2];
            acc = fma(ta, tb, acc);
            dacc = fma(Ts[(4 + c) * M + a2], tb, dacc);
            dacc = fma(ta, Ts[(4 + c) * M + b2], dacc);
        }
        Dout[(size_t)i * nd + q] = acc;
        dDout[(size_t)i * nd + q] = dacc;
    }
}

// Tb and dTb of one atom per CTA from dPhi/dD (Db) and dPhi/d(dD) (dDb), over T
// and dT: D = T_<^T T, dD = dT_<^T T + T_<^T dT; the scale of T folded in.
__global__ void __launch_bounds__(CT) k_chebpg_tb(DevModel m, double *__restrict__ Tio, double *__restrict__ dTio,
                                                  const double *__restrict__ Db, const double *__restrict__ dDb,
                                                  const int32_t *far_flag)
{
    if (*far_flag) return;
    extern __shared__ __align__(16) double sm[];
    const int M = m.M, m2 = m.m2, tid = threadIdx.x, LDG = M | 1;
    const size_t i = blockIdx.x;
    double *Ts = sm, *dTs = Ts + 4 * M;  // [4][M] each
    double *lp = dTs + 4 * M;            // [2][4][m2] long sums of Tb, dTb
    double *g = lp + 8 * m2;             // [m2][LDG] one of the two adjoints
    for (int p = tid; p < 4 * M; p += CT) {
        Ts[p] = Tio[i * 4 * M + p];
        dTs[p] = dTio[i * 4 * M + p];
    }
    constexpr int OWN = (4 * DP_MAX_EMB_W + CT - 1) / CT;
    double tb[OWN], dtb[OWN];
#pragma unroll
    for (int u = 0; u < OWN; ++u) tb[u] = dtb[u] = 0.0;
    for (int pass = 0; pass < 2; ++pass) {  // dDb with (dT -> Tb, T -> dTb), then Db with (T -> Tb)
        const double *src = (pass == 0 ? dDb : Db) + i * m2 * M;
        const double *A = pass == 0 ? dTs : Ts;
        __syncthreads();
        for (int p = tid; p < m2 * M; p += CT) g[(p / M) * LDG + p % M] = src[p];
        __syncthreads();
        for (int p = tid; p < 4 * m2; p += CT) {
            const int c = p / m2, xx = p - c * m2;
            double v = 0.0, dv = 0.0;
            for (int b = 0; b < M; ++b) {
                const double gv = g[xx * LDG + b];
                v = fma(gv, A[c * M + b], v);
                if (pass == 0) dv = fma(gv, Ts[c * M + b], dv);
            }
            lp[p] = v;
            lp[4 * m2 + p] = dv;
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < OWN; ++u) {
            const int p = tid + u * CT;
            if (p < 4 * M) {
                const int c = p / M, xx = p - c * M;
                double v = xx < m2 ? lp[c * m2 + xx] : 0.0, dv = xx < m2 && pass == 0 ? lp[4 * m2 + c * m2 + xx] : 0.0;
                for (int a2 = 0; a2 < m2; ++a2) {
                    const double gv = g[a2 * LDG + xx];
                    v = fma(gv, A[c * M + a2], v);
                    if (pass == 0) dv = fma(gv, Ts[c * M + a2], dv);
                }
                tb[u] += v;
                dtb[u] += dv;
            }
        }
    }
#pragma unroll
    for (int u = 0; u < OWN; ++u) {
        const int p = tid + u * CT;
        if (p < 4 * M) {
            Tio[i * 4 * M + p] = tb[u] * m.desc_scale;
            dTio[i * 4 * M + p] = dtb[u] * m.desc_scale;
        }
    }
}

// Partial adjoints of C and V: CTA (split, centre type, 16 terms of the type's
// nets side by side) sums P Tb + dP dTb and Q dTb over its share of the type's
// atoms; thread = (4 terms, features u, u + 32, ...).
constexpr int CBK = 16;
constexpr int CBA = 4;  // atoms staged at once
__global__ void __launch_bounds__(CT) k_chebpg_cb(DevModel m, int nc, const int32_t *__restrict__ type_perm,
                                                  const int32_t *__restrict__ type_start,
                                                  const double *__restrict__ mom, const double *__restrict__ Tb,
                                                  const double *__restrict__ dTb, double *__restrict__ part,
                                                  const int32_t *far_flag)
{
    if (*far_flag) return;
    extern __shared__ __align__(16) double sm[];
    const int M = m.M, T = m.ntypes, Kt = T * nc, tid = threadIdx.x;
    const int a = blockIdx.y, k0 = blockIdx.z * CBK;
    double *ms = sm;                   // [CBA][PM][CBK]
    double *ts = ms + CBA * PM * CBK;  // [CBA][8][M]: Tb, dTb
    const int s0 = type_start[a], cnt = type_start[a + 1] - s0;
    const int lo = (int)((long long)blockIdx.x * cnt / gridDim.x), hi = (int)((long long)(blockIdx.x + 1) * cnt / gridDim.x);
    const int kq = (tid >> 5) * 4, fl = tid & 31;
    double acc[4][4], accv[4][4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] = accv[u][v] = 0.0;
    for (int b0 = lo; b0 < hi; b0 += CBA) {
        const int n = min(CBA, hi - b0);
        __syncthreads();
        for (int p = tid; p < n * PM * CBK; p += CT) {
            const int at = p / (PM * CBK), k = (p / PM) % CBK, c = p % PM;
            const size_t i = type_perm[s0 + b0 + at];
            ms[(at * PM + c) * CBK + k] = k0 + k < Kt ? mom[(i * Kt + k0 + k) * PM + c] : 0.0;
        }
        for (int p = tid; p < n * 8 * M; p += CT) {
            const int at = p / (8 * M), r = p - at * 8 * M;
            const size_t i = type_perm[s0 + b0 + at];
            ts[p] = r < 4 * M ? Tb[i * 4 * M + r] : dTb[i * 4 * M + r - 4 * M];
        }
        __syncthreads();
        for (int at = 0; at < n; ++at)
#pragma unroll 2
            for (int c = 0; c < 4; ++c) {
                const double *mp = ms + (at * PM + c) * CBK + kq;
                double mv[3][4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    mv[0][u] = mp[u];
                    mv[1][u] = mp[4 * CBK + u];
                    mv[2][u] = mp[8 * CBK + u];
                }
#pragma unroll
                for (int v = 0; v < 4; ++v)
                    if (fl + 32 * v < M) {
                        const double tv = ts[(at * 8 + c) * M + fl + 32 * v], dv = ts[(at * 8 + 4 + c) * M + fl + 32 * v];
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            acc[u][v] = fma(mv[0][u], tv, fma(mv[1][u], dv, acc[u][v]));
                            accv[u][v] = fma(mv[2][u], dv, accv[u][v]);
                        }
                    }
            }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int k = k0 + kq + u;
        if (k >= Kt) continue;
        const int b = k / nc, n = k - b * nc;
        const size_t nets = (size_t)T * T;
        double *pc = part + ((2 * (size_t)blockIdx.x * nets + a * T + b) * NN + n) * M, *pv = pc + nets * NN * M;
#pragma unroll
        for (int v = 0; v < 4; ++v)
            if (fl + 32 * v < M) {
                pc[fl + 32 * v] = acc[u][v];
                pv[fl + 32 * v] = accv[u][v];
            }
    }
}

// Sum of the partial adjoints in a fixed order, into the first one.
__global__ void k_chebpg_sum(double *__restrict__ part, size_t elems, int splits, const int32_t *far_flag)
{
    if (*far_flag) return;
    for (size_t p = blockIdx.x * (size_t)blockDim.x + threadIdx.x; p < elems; p += (size_t)gridDim.x * blockDim.x) {
        double v = part[p];
#pragma unroll 8
        for (int q = 1; q < splits; ++q) v += part[q * elems + p];
        part[p] = v;
    }
}

// One CTA per (net, node): the adjoints of the net's value and derivative there,
// Gb_f = sum_n w_nk Cb_nf and G'b_f = sum_n w_nk Vb_nf with w_nk = (2 - [n = 0]) / NN
// cos(pi n (2k+1) / (2 NN)), and reverse mode through the layers with their
// s-tangents; h, dh, zb and dzb of every layer go to node[net][k][0 .. 3][.].
__global__ void __launch_bounds__(CT) k_chebpg_node(DevModel m, int nc, double scale, const double *__restrict__ trig,
                                                    const double *__restrict__ Cb, const double *__restrict__ Vb,
                                                    double *__restrict__ node, int se, const int32_t *far_flag)
{
    if (*far_flag) return;
    __shared__ double h[DP_MAX_LAYERS][DP_MAX_EMB_W], dh[DP_MAX_LAYERS][DP_MAX_EMB_W], t[DP_MAX_LAYERS][DP_MAX_EMB_W],
        dz[DP_MAX_LAYERS][DP_MAX_EMB_W];
    __shared__ double g[DP_MAX_EMB_W], dg[DP_MAX_EMB_W], zb[DP_MAX_EMB_W], dzb[DP_MAX_EMB_W];
    const int net = blockIdx.x / NN, k = blockIdx.x % NN, o = threadIdx.x, M = m.M;
    const double *P = m.params + m.emb_base[net];
    const double s = (1.0 + trig[2 * (2 * k + 1)]) / scale;
    if (o < m.emb[0]) {
        const double tv = dp_tanh64(fma(s, P[o], P[m.emb[0] + o]), m.tanh_tab);
        h[0][o] = t[0][o] = tv;
        dz[0][o] = P[o];
        dh[0][o] = fma(-tv, tv, 1.0) * P[o];
    }
    int off = 2 * m.emb[0];
    for (int l = 1; l < m.n_emb; ++l) {
        __syncthreads();
        const int win = m.emb[l - 1], wout = m.emb[l], sk = dp_skip_kind(win, wout);
        if (o < wout) {
            double z = P[off + win * wout + o], d = 0.0;
            for (int p = 0; p < win; ++p) {
                const double w = P[off + p * wout + o];
                z = fma(h[l - 1][p], w, z);
                d = fma(dh[l - 1][p], w, d);
            }
            const double tv = dp_tanh64(z, m.tanh_tab);
            const int os = o < win ? o : o - win;
            t[l][o] = tv;
            dz[l][o] = d;
            h[l][o] = tv + (sk ? h[l - 1][os] : 0.0);
            dh[l][o] = fma(fma(-tv, tv, 1.0), d, sk ? dh[l - 1][os] : 0.0);
        }
        off += win * wout + wout;
    }
    if (o < M) {
        double v = 0.0, dv = 0.0;
        for (int n = nc - 1; n >= 0; --n) {
            const double w = trig[2 * ((n * (2 * k + 1)) % (4 * NN))] * (n == 0 ? 1.0 / NN : 2.0 / NN);
            v = fma(w, Cb[((size_t)net * NN + n) * M + o], v);
            dv = fma(w, Vb[((size_t)net * NN + n) * M + o], dv);
        }
        g[o] = v;
        dg[o] = dv;
    }
    double *nd = node + (size_t)blockIdx.x * 4 * se;
    int lo = se;
    for (int l = m.n_emb - 1; l >= 0; --l) {
        __syncthreads();
        const int out = m.emb[l], in = l > 0 ? m.emb[l - 1] : 0;
        lo -= out;
        if (o < out) {
            const double one = fma(-t[l][o], t[l][o], 1.0), d = dg[o];
            dzb[o] = one * d;
            zb[o] = one * fma(-2.0 * t[l][o] * dz[l][o], d, g[o]);
            nd[lo + o] = h[l][o];
            nd[se + lo + o] = dh[l][o];
            nd[2 * se + lo + o] = zb[o];
            nd[3 * se + lo + o] = dzb[o];
        }
        __syncthreads();
        if (l > 0) {
            off -= in * out + out;
            const int sk = dp_skip_kind(in, out);
            double v = 0.0, d = 0.0;
            if (o < in) {
                for (int p = 0; p < out; ++p) {
                    const double w = P[off + o * out + p];
                    v = fma(w, zb[p], v);
                    d = fma(w, dzb[p], d);
                }
                if (sk) {
                    v += g[o];
                    d += dg[o];
                }
                if (sk == 2) {
                    v += g[o + in];
                    d += dg[o + in];
                }
            }
            __syncthreads();
            if (o < in) {
                g[o] = v;
                dg[o] = d;
            }
        }
    }
}

// Gradient of every embedding parameter from the nodes: dW[q][o] = sum_k h_k[q]
// zb_k[o] + dh_k[q] dzb_k[o] (layer 0: h = s, dh = 1), db[o] = sum_k zb_k[o].
__global__ void k_chebpg_grad(DevModel m, double scale, const double *__restrict__ trig, const double *__restrict__ node, int se,
                              double *__restrict__ grad, const int32_t *far_flag)
{
    if (*far_flag) return;
    const int net = blockIdx.y;
    const double *nd = node + (size_t)net * NN * 4 * se;
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < m.emb_net_size; p += gridDim.x * blockDim.x) {
        int l = 0, lo = 0, r = p, in = 1;  // layer, its offset in the node arrays, index in the layer
        while (r >= (in + 1) * m.emb[l]) {
            r -= (in + 1) * m.emb[l];
            lo += m.emb[l];
            in = m.emb[l];
            ++l;
        }
        const int out = m.emb[l], q = r / out, o = r - q * out;
        double v = 0.0, w = 0.0;
        for (int k = 0; k < NN; ++k) {
            const double *n = nd + (size_t)k * 4 * se;
            double hv = 1.0, dv = 0.0;
            if (q < in) {
                hv = l == 0 ? (1.0 + trig[2 * (2 * k + 1)]) / scale : n[lo - in + q];
                dv = l == 0 ? 1.0 : n[se + lo - in + q];
            }
            v = fma(hv, n[2 * se + lo + o], v);
            w = fma(dv, n[3 * se + lo + o], w);
        }
        grad[m.emb_base[net] + p] = v + w;
    }
}

size_t pg_fwd_smem(const DevModel &m, int nc)
{
    return sizeof(double) * (2 * CT * PM + (size_t)m.ntypes * nc * PM + 8 * m.M + (size_t)nc * LDT);
}

size_t pg_tb_smem(const DevModel &m) { return sizeof(double) * (8 * (size_t)m.M + 8 * m.m2 + (size_t)m.m2 * (m.M | 1)); }

size_t fwd_smem(const DevModel &m, int nc)
{
    return sizeof(double) * (CT * 4 + 2 * CT * 4 + (size_t)m.ntypes * nc * 4 + 4 * m.M + (size_t)nc * LDT);
}

size_t pre_smem(const DevModel &m, int nc) { return sizeof(double) * ((size_t)m.ntypes * nc * 8 + 4 * (size_t)m.M); }

size_t bwd_smem(const DevModel &m, int nc)
{
    const size_t Kt = (size_t)m.ntypes * nc, nsl = Kt < CT ? CT / Kt : 1;
    const size_t g = (size_t)m.m2 * (m.M | 1), u = Kt * nsl * 4;
    return sizeof(double) * (Kt * 8 + 8 * (size_t)m.M + 8 * (size_t)m.m2 + (g > u ? g : u));
}

constexpr size_t SMEM_MAX = 220 * 1024;  // dynamic, next to ~7 KB of static shared memory

}  // namespace

bool dp_cheb_supported(const DevModel &m) { return bwd_smem(m, NN) <= SMEM_MAX && fwd_smem(m, NN) <= SMEM_MAX; }

size_t dp_cheb_elems(const DevModel &m, int which)
{
    const size_t nets = (size_t)m.ntypes * m.ntypes;
    switch (which) {
    case 0:
    case 1:
    case 2: return nets * NN * m.M;
    case 3: return nets * NN * m.M * 2;
    case 4: return nets * NN;
    default: return 2 * (4 * NN + DP_CHEB_NTANH);
    }
}

cudaError_t dp_launch_cheb_setup(cudaStream_t st, ChebBuffers cb, int64_t *launches)
{
    k_cheb_setup<<<(4 * NN + DP_CHEB_NTANH + 127) / 128, 128, 0, st>>>(cb.trig);
    *launches += 1;
    return cudaGetLastError();
}

cudaError_t dp_launch_cheb_build(cudaStream_t st, const DevModel &m, double scale, ChebBuffers cb, int64_t *launches)
{
    const int grid = m.ntypes * m.ntypes * NN;
    k_cheb_nodes<<<grid, CT, 0, st>>>(m, scale, cb.trig, cb.y);
    k_cheb_coef<<<grid, CT, 0, st>>>(m, cb.trig, cb.y, cb.C, cb.Ct, cb.mx);
    k_cheb_deriv<<<grid, CT, 0, st>>>(m, scale, cb.C, cb.V);
    k_cheb_check<<<m.ntypes * m.ntypes * (NN + 1), CT, 0, st>>>(m, scale, cb.trig, cb.C, cb.mx);
    *launches += 4;
    return cudaGetLastError();
}

int dp_cheb_terms(const DevModel &m, const double *mx)
{
    int need = 4;
    for (int net = 0; net < m.ntypes * m.ntypes; ++net) {
        const double *c = mx + net * NN;
        double size = 0.0, tail = 0.0;
        for (int n = 0; n < NN; ++n) size = c[n] > size ? c[n] : size;
        if (!(size <= 1e300)) return 0;
        // the derivative of the terms n .., by s / S, is 2 sum n^2 |C_n| or less (3/4 of
        // it are asked for: as by s at S = 4/3)
        int n = NN;
        for (; n > 0; --n) {
            tail += 1.5 * (double)(n - 1) * (n - 1) * c[n - 1];
            if (tail > 0x1p-55 * size) break;
        }
        need = n > need ? n : need;
    }
    need = (need + 3) / 4 * 4;
    return need <= NN - 4 ? need : 0;
}

// The products with the series, T = scale P C and U = C dE/dT, as exact digit
// products on the tensor cores (fit_oz.cu), four rows per atom: their 8 M T n FMAs
// per atom leave the FP64 units (40% of the forward's there) for two splits, two
// GEMMs, one kernel that forms D and one that forms dE/dT.  The rows use buffers
// that are free at that point, hence M2 >= 4 and Kt <= M: the moments dE/dD's,
// dE/dT D's, U T's, the flag of rows beyond S E_i's.  Per evaluation, fused ->
// apart: 139,968 water atoms forward 13.0 -> 6.9 ms, backward 16.7 -> 13.5 ms;
// 32,000 copper 2.9 -> 2.3 and 4.6 -> 4.2; 2,187 water (whole step) 1.17 ->
// 1.13; 192 water 0.51 -> 0.53.  The line is the work that
// pays for the four more launches: equal at 1,029 water atoms (40 terms) and
// 2,048 copper atoms (20 terms), 100 features each.
bool dp_cheb_gemm(const DevModel &m, int n, int N)
{
    const int Kt = m.ntypes * n;
    return m.m2 >= 4 && Kt <= m.M && (int64_t)N * Kt * m.M >= (1 << 22);
}

cudaError_t dp_launch_cheb_fwd(cudaStream_t st, const DevModel &m, const ChebModel &cm, const double *x,
                               const int32_t *types, Box3 box, int N, const FormatBuffers &fb,
                               const NlistBuffers &nb, EvalBuffers eb, const OzSeries *os, uint16_t *a_dig, int num_sms,
                               int32_t *status, int64_t *launches)
{
    const size_t smem = fwd_smem(m, cm.n);
    cudaError_t e = cudaFuncSetAttribute(k_cheb_fwd<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_MAX);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_cheb_fwd<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_MAX);
    if (e != cudaSuccess) return e;
    *launches += 1;
    if (!os) {
        k_cheb_fwd<false><<<N, CT, smem, st>>>(m, cm, x, types, box, nb.type_perm, fb.nlist, fb.nreal, eb.pair_g, eb.T,
                                               eb.D);
        return cudaGetLastError();
    }
    const int Kt = m.ntypes * cm.n;
    k_cheb_fwd<true><<<N, CT, smem, st>>>(m, cm, x, types, box, nb.type_perm, fb.nlist, fb.nreal, eb.pair_g, eb.gD,
                                          eb.Ei);
    if ((e = dp_launch_oz_rows(st, m, *os, os->gf, a_dig, N, eb.gD, Kt, eb.T, m.M, nb, num_sms, status, launches)) !=
        cudaSuccess)
        return e;
    k_cheb_desc<<<N, CT, 0, st>>>(m, cm.S, types, nb.type_perm, fb.nreal, eb.Ei, eb.pair_g, eb.T, eb.D);
    *launches += 1;
    return cudaGetLastError();
}

cudaError_t dp_launch_cheb_bwd(cudaStream_t st, const DevModel &m, const ChebModel &cm, const int32_t *types, int N,
                               const FormatBuffers &fb, const NlistBuffers &nb, EvalBuffers eb, const OzSeries *os,
                               uint16_t *a_dig, int num_sms, int32_t *status, int64_t *launches)
{
    cudaError_t e = cudaFuncSetAttribute(k_cheb_bwd<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_MAX);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_cheb_bwd<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_MAX);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_cheb_gT, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_MAX);
    if (e != cudaSuccess) return e;
    *launches += 1;
    if (!os) {
        k_cheb_bwd<false><<<N, CT, bwd_smem(m, cm.n), st>>>(m, cm, types, nb.type_perm, fb.nreal, eb.T, eb.gD, eb.pair_g,
                                                            eb.f_own, eb.vir_part);
        return cudaGetLastError();
    }
    const int Kt = m.ntypes * cm.n;
    const size_t gsm = sizeof(double) * (4 * (size_t)m.M + 8 * (size_t)m.m2 + (size_t)m.m2 * (m.M | 1));
    k_cheb_gT<<<N, CT, gsm, st>>>(m, nb.type_perm, eb.T, eb.gD, eb.D);
    if ((e = dp_launch_oz_rows(st, m, *os, os->gb, a_dig, N, eb.D, m.M, eb.T, Kt, nb, num_sms, status, launches)) !=
        cudaSuccess)
        return e;
    k_cheb_bwd<true><<<N, CT, pre_smem(m, cm.n), st>>>(m, cm, types, nb.type_perm, fb.nreal, eb.T, eb.D, eb.pair_g,
                                                      eb.f_own, eb.vir_part);
    *launches += 1;
    return cudaGetLastError();
}

bool dp_cheb_grad_supported(const DevModel &m, int n)
{
    return n > 0 && pg_fwd_smem(m, n) <= SMEM_MAX && pg_tb_smem(m) <= SMEM_MAX;
}

size_t dp_cheb_grad_elems(const DevModel &m, int n, int64_t natoms, int which)
{
    const size_t nets = (size_t)m.ntypes * m.ntypes;
    size_t se = 0;
    for (int l = 0; l < m.n_emb; ++l) se += m.emb[l];
    switch (which) {
    case 0: return (size_t)natoms * m.ntypes * n * PM;
    case 1: return (size_t)dp_cheb_splits(m.ntypes, natoms) * 2 * nets * NN * m.M;
    default: return nets * NN * 4 * se;
    }
}

cudaError_t dp_launch_chebpg_fwd(cudaStream_t st, const DevModel &m, const ChebModel &cm, const double *x,
                                 const int32_t *types, Box3 box, int N, const double *lam, const FormatBuffers &fb,
                                 const NlistBuffers &nb, EvalBuffers eb, PGradBuffers pb, ChebGradBuffers gb,
                                 int64_t *launches)
{
    cudaError_t e = cudaMemsetAsync(gb.far, 0, sizeof(int32_t), st);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_chebpg_fwd, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_MAX);
    if (e != cudaSuccess) return e;
    k_chebpg_fwd<<<N, CT, pg_fwd_smem(m, cm.n), st>>>(m, cm, x, types, box, lam, nb.type_perm, fb.nlist, fb.nreal,
                                                     eb.T, pb.dT, eb.D, pb.dD, gb.mom, gb.far);
    *launches += 1;
    return cudaGetLastError();
}

cudaError_t dp_launch_chebpg_bwd(cudaStream_t st, const DevModel &m, const ChebModel &cm, int N,
                                 const NlistBuffers &nb, EvalBuffers eb, PGradBuffers pb, ChebGradBuffers gb,
                                 const double *trig, double *grad, int64_t *launches)
{
    const int T = m.ntypes, Kt = T * cm.n;
    int se = 0;
    for (int l = 0; l < m.n_emb; ++l) se += m.emb[l];
    cudaError_t e = cudaFuncSetAttribute(k_chebpg_tb, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_MAX);
    const size_t csm = sizeof(double) * CBA * (PM * CBK + 8 * (size_t)m.M);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_chebpg_cb, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)csm);
    if (e != cudaSuccess) return e;
    k_chebpg_tb<<<N, CT, pg_tb_smem(m), st>>>(m, eb.T, pb.dT, pb.Db, pb.dDb, gb.far);
    const int splits = dp_cheb_splits(T, N);
    k_chebpg_cb<<<dim3(splits, T, (Kt + CBK - 1) / CBK), CT, csm, st>>>(
        m, cm.n, nb.type_perm, nb.type_start, gb.mom, eb.T, pb.dT, gb.part, gb.far);
    const size_t elems = 2 * (size_t)T * T * NN * m.M;
    k_chebpg_sum<<<(int)((elems + 255) / 256), 256, 0, st>>>(gb.part, elems, splits, gb.far);
    k_chebpg_node<<<T * T * NN, CT, 0, st>>>(m, cm.n, cm.scale, trig, gb.part, gb.part + elems / 2, gb.node, se, gb.far);
    k_chebpg_grad<<<dim3((m.emb_net_size + 255) / 256, T * T), 256, 0, st>>>(m, cm.scale, trig, gb.node, se, grad, gb.far);
    *launches += 5;
    return cudaGetLastError();
}
