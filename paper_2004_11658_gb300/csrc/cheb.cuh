// cheb.cuh -- the embedding nets of an FP64 context as Chebyshev series in s
// (csrc/embed_cheb.cu): shapes, buffers and launchers.
#pragma once

#include "cheb_domain.h"
#include "dp_internal.cuh"

// Nodes (and stored terms) per net.  The domain s in [0, S] (dp_cheb_domain) is
// mapped to t = (2 / S) s - 1.
constexpr int DP_CHEB_NN = 48;

struct ChebModel {
    int n;             // terms used by every net (0: not resolved, the series is not used)
    double S, scale;   // domain and 2 / S
    const double *C;   // [T T][NN][M]: G_f(s) = sum_n C[net][n][f] T_n(t)
    const double *Ct;  // [T][M][T NN]: the same values, the nets of centre type a side by side
    const double *V;   // [T T][NN][M]: dG_f/ds = sum_n V[net][n][f] T_n(t)
};

// Device scratch of the construction; bytes of one context's buffers.
struct ChebBuffers {
    double *C, *Ct, *V;
    double *y;      // node values, [T T][NN][M][2] (high and low part)
    double *mx;     // [T T][NN] max_f |C|
    double *trig;   // [4 NN][2] cos(pi j / (2 NN)), then [DP_CHEB_NTANH][2] tanh(k / 32)
};
constexpr int DP_CHEB_NTANH = 705;

bool dp_cheb_supported(const DevModel &m);
size_t dp_cheb_elems(const DevModel &m, int which);  // doubles of C, Ct, V, y, mx, trig (which = 0..5)
cudaError_t dp_launch_cheb_setup(cudaStream_t st, ChebBuffers cb, int64_t *launches);
// Coefficients of every net from the device parameters.
cudaError_t dp_launch_cheb_build(cudaStream_t st, const DevModel &m, double scale, ChebBuffers cb, int64_t *launches);
// Terms needed for the nets of the host copy of mx, 0 if not resolved.
int dp_cheb_terms(const DevModel &m, const double *mx);

// os: the products with the series on the tensor cores (dp_cheb_gemm), a_dig
// their digit scratch; null: on the FP64 units, fused.
bool dp_cheb_gemm(const DevModel &m, int n, int N);
cudaError_t dp_launch_cheb_fwd(cudaStream_t st, const DevModel &m, const ChebModel &cm, const double *x,
                               const int32_t *types, Box3 box, int N, const FormatBuffers &fb,
                               const NlistBuffers &nb, EvalBuffers eb, const OzSeries *os, uint16_t *a_dig, int num_sms,
                               int32_t *status, int64_t *launches);
cudaError_t dp_launch_cheb_bwd(cudaStream_t st, const DevModel &m, const ChebModel &cm, const int32_t *types, int N,
                               const FormatBuffers &fb, const NlistBuffers &nb, EvalBuffers eb, const OzSeries *os,
                               uint16_t *a_dig, int num_sms, int32_t *status, int64_t *launches);

// Parameter gradient through the series (csrc/embed_cheb.cu): T, dT, D, dD of
// every atom with the moments kept, then, from dPhi/dD and dPhi/d(dD), the
// gradient of the embedding nets' parameters by way of the coefficients.
struct ChebGradBuffers {
    double *mom;    // [N][T n][12] moments (k_chebpg_fwd)
    double *part;   // [dp_cheb_splits][2][T T][NN][M] partial adjoints of C and V
    double *node;   // [T T][NN][4][sum of widths] layer outputs and z adjoints at the nodes, with tangents
    int32_t *far;   // set when a row lies beyond S: the caller's other kernels run instead
};
// Atom shares of a centre type: 24 atoms each, so that several CTAs share an SM
// (64 shares in all took 2.0 ms for 12,288 water atoms with the student's widths,
// 1.25 as now), between 64 and 256 in all (the buffer's size).
inline int dp_cheb_splits(int ntypes, int64_t natoms)
{
    const int64_t s = natoms / (24 * ntypes), lo = ntypes > 8 ? 8 : 64 / ntypes, hi = 4 * lo;
    return (int)(s < lo ? lo : s > hi ? hi : s);
}
// Terms the gradient keeps: the parameter derivatives' series converge as the
// nets' with a polynomial factor, which 8 more terms cover (nets of 29 to 46 terms
// needed at most 2 more, in 40-digit arithmetic), and the last 4 for nets of 44.
inline int dp_cheb_grad_terms(int n) { return n + 8 < DP_CHEB_NN ? n + 8 : DP_CHEB_NN; }
size_t dp_cheb_grad_elems(const DevModel &m, int n, int64_t natoms, int which);  // doubles of mom, part, node
bool dp_cheb_grad_supported(const DevModel &m, int n);
cudaError_t dp_launch_chebpg_fwd(cudaStream_t st, const DevModel &m, const ChebModel &cm, const double *x,
                                 const int32_t *types, Box3 box, int N, const double *lam, const FormatBuffers &fb,
                                 const NlistBuffers &nb, EvalBuffers eb, PGradBuffers pb, ChebGradBuffers gb,
                                 int64_t *launches);
// Overwrites eb.T and pb.dT; writes grad[0 .. T T emb_net_size).
cudaError_t dp_launch_chebpg_bwd(cudaStream_t st, const DevModel &m, const ChebModel &cm, int N,
                                 const NlistBuffers &nb, EvalBuffers eb, PGradBuffers pb, ChebGradBuffers gb,
                                 const double *trig, double *grad, int64_t *launches);
