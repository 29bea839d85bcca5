// cheb.cuh -- the embedding nets of an FP64 context as Chebyshev series in s
// (csrc/embed_cheb.cu): shapes, buffers and launchers.
#pragma once

#include "dp_internal.cuh"

// Nodes (and stored terms) per net, and the resolved domain s in [0, S], mapped
// to t = (2 / S) s - 1.  S = 4/3 is r = 0.75 A, below the O-H bond; nearer rows
// evaluate the net itself.  (S = 2 needs 24 terms instead of 20.)
constexpr int DP_CHEB_NN = 48;
constexpr double DP_CHEB_SCALE = 1.5;               // 2 / S
constexpr double DP_CHEB_S = 2.0 / DP_CHEB_SCALE;

struct ChebModel {
    int n;             // terms used by every net (0: not resolved, the series is not used)
    const double *C;   // [T T][NN][M]: G_f(s) = sum_n C[net][n][f] T_n(t)
    const double *Ct;  // [T][M][T NN]: the same values, the nets of centre type a side by side
};

// Device scratch of the construction; bytes of one context's buffers.
struct ChebBuffers {
    double *C, *Ct;
    double *y;      // node values, [T T][NN][M][2] (high and low part)
    double *mx;     // [T T][NN] max_f |C|
    double *trig;   // [4 NN][2] cos(pi j / (2 NN)), then [DP_CHEB_NTANH][2] tanh(k / 32)
};
constexpr int DP_CHEB_NTANH = 705;

bool dp_cheb_supported(const DevModel &m);
size_t dp_cheb_elems(const DevModel &m, int which);  // doubles of C, Ct, y, mx, trig (which = 0..4)
cudaError_t dp_launch_cheb_setup(cudaStream_t st, ChebBuffers cb, int64_t *launches);
// Coefficients of every net from the device parameters.
cudaError_t dp_launch_cheb_build(cudaStream_t st, const DevModel &m, ChebBuffers cb, int64_t *launches);
// Terms needed for the nets of the host copy of mx, 0 if not resolved.
int dp_cheb_terms(const DevModel &m, const double *mx);

cudaError_t dp_launch_cheb_fwd(cudaStream_t st, const DevModel &m, const ChebModel &cm, const double *x,
                               const int32_t *types, Box3 box, int N, const FormatBuffers &fb,
                               const NlistBuffers &nb, EvalBuffers eb, int64_t *launches);
cudaError_t dp_launch_cheb_bwd(cudaStream_t st, const DevModel &m, const ChebModel &cm, const int32_t *types, int N,
                               const FormatBuffers &fb, const NlistBuffers &nb, EvalBuffers eb, int64_t *launches);
