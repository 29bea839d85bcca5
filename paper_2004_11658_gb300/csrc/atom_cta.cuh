// atom_cta.cuh -- pieces of the backward kernels that take one atom per
// 128-thread CTA (embed_cheb.cu, mixed.cu).
#pragma once

#include "dp_internal.cuh"

constexpr int DP_ATOM_CT = 128;

// dE/dT of one atom, gT[c][x] = scale ([x < m2] sum_b gD[x][b] T[c][b] + sum_{a < m2} gD[a][x] T[c][a]),
// handed to out(c, x, value).  gs: dE/dD [m2][LDG] and Ts: T [4][M] in shared
// memory; lp: 8 m2 doubles of it.  The 4 m2 long sums two threads each first.
template <class OUT>
__device__ __forceinline__ void dp_atom_gT(const double *gs, int LDG, const double *Ts, double *lp, int m2, int M,
                                           double scale, OUT out)
{
    const int tid = threadIdx.x;
    for (int p = tid; p < 8 * m2; p += DP_ATOM_CT) {
        const int h = p / (4 * m2), e = p - h * 4 * m2, c = e / m2, xx = e - c * m2;
        const double *gr = gs + xx * LDG, *tr = Ts + c * M;
        double v0 = 0.0, v1 = 0.0;
        int b = h;
        for (; b + 2 < M; b += 4) {
            v0 = fma(gr[b], tr[b], v0);
            v1 = fma(gr[b + 2], tr[b + 2], v1);
        }
        for (; b < M; b += 2) v0 = fma(gr[b], tr[b], v0);
        lp[p] = v0 + v1;
    }
    __syncthreads();
    for (int p = tid; p < 4 * M; p += DP_ATOM_CT) {
        const int c = p / M, xx = p - c * M;
        double v0 = 0.0, v1 = 0.0;
        int a2 = 0;
        for (; a2 + 1 < m2; a2 += 2) {
            v0 = fma(gs[a2 * LDG + xx], Ts[c * M + a2], v0);
            v1 = fma(gs[(a2 + 1) * LDG + xx], Ts[c * M + a2 + 1], v1);
        }
        if (a2 < m2) v0 = fma(gs[a2 * LDG + xx], Ts[c * M + a2], v0);
        v0 += v1;
        if (xx < m2) v0 += lp[c * m2 + xx] + lp[4 * m2 + c * m2 + xx];
        out(c, xx, v0 * scale);
    }
}

// Own force fo[3] and virial vir[9] summed over the CTA and written for atom i:
// a transposing shuffle tree (16 adds instead of 60), then the warps in order.
__device__ __forceinline__ void dp_atom_sum12(const double (&fo)[3], const double (&vir)[9],
                                              double (&wsum)[DP_ATOM_CT / 32][16], double *__restrict__ f_own,
                                              double *__restrict__ vir_part, size_t i)
{
    const int tid = threadIdx.x, lane = tid & 31;
    double p[16];
#pragma unroll
    for (int q = 0; q < 3; ++q) p[q] = fo[q];
#pragma unroll
    for (int q = 0; q < 9; ++q) p[3 + q] = vir[q];
#pragma unroll
    for (int q = 12; q < 16; ++q) p[q] = 0.0;
#pragma unroll
    for (int w = 16, n = 8; w >= 2; w >>= 1, n >>= 1) {
        const bool up = (lane & w) != 0;
#pragma unroll
        for (int k = 0; k < n; ++k) {
            const double send = up ? p[k] : p[n + k];
            const double keep = up ? p[n + k] : p[k];
            p[k] = keep + __shfl_xor_sync(0xffffffffu, send, w);
        }
    }
    p[0] += __shfl_xor_sync(0xffffffffu, p[0], 1);
    if ((lane & 1) == 0) wsum[tid >> 5][lane >> 1] = p[0];
    __syncthreads();
    if (tid < 12) {
        double v = wsum[0][tid];
        for (int w = 1; w < DP_ATOM_CT / 32; ++w) v += wsum[w][tid];
        if (tid < 3) f_own[i * 3 + tid] = v;
        else vir_part[i * 9 + tid - 3] = v;
    }
}
