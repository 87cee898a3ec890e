// In-CTA Householder QR in shared memory, the fallback of the orthogonalisation kernels (tt_qr.cu,
// tt_solve.cu).
#pragma once

#include "tt_internal.cuh"

// Householder QR of an m x q column-major matrix held in shared memory (q small).
// On exit: A holds Q (m x p, p = min(m, q)) in its first p columns, R (p x q) in Rm (q x q,
// row-major, rows >= p zero), with diag(R) >= 0.

__device__ inline float warp_sum(float v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ inline void block_householder_qr(float* A, int m, int q, float* Rm, float* tau, float* colsc) {
  const int p = min(m, q);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int j = 0; j < p; ++j) {
    float* x = A + (int64_t)j * m;
    // norm of x[j+1 : m]
    if (warp == 0) {
      float ss = 0.f;
      for (int i = j + 1 + lane; i < m; i += 32) ss = fmaf(x[i], x[i], ss);
      ss = warp_sum(ss);
      if (lane == 0) {
        float alpha = x[j];
        float xn = sqrtf(ss);
        if (xn == 0.f) {
          tau[j] = 0.f;
          colsc[0] = 0.f;
        } else {
          float beta = -copysignf(hypotf(alpha, xn), alpha);
          tau[j] = (beta - alpha) / beta;
          colsc[0] = 1.f / (alpha - beta);
          x[j] = beta;
        }
      }
    }
    __syncthreads();
    const float sc = colsc[0];
    const float tj = tau[j];
    if (tj != 0.f)
      for (int i = j + 1 + threadIdx.x; i < m; i += blockDim.x) x[i] *= sc;
    __syncthreads();
    if (tj != 0.f) {
      // apply H_j = I - tau v v^T (v_j = 1) to columns j+1..q-1, one warp per column
      for (int cc = j + 1 + warp; cc < q; cc += nw) {
        float* y = A + (int64_t)cc * m;
        float w = 0.f;
        for (int i = j + 1 + lane; i < m; i += 32) w = fmaf(x[i], y[i], w);
        w = warp_sum(w) + y[j];
        w *= tj;
        if (lane == 0) y[j] -= w;
        for (int i = j + 1 + lane; i < m; i += 32) y[i] = fmaf(-w, x[i], y[i]);
      }
    }
    __syncthreads();
  }
  // R (upper trapezoid) out, zero below
  for (int idx = threadIdx.x; idx < q * q; idx += blockDim.x) {
    int i = idx / q, jj = idx - i * q;
    Rm[idx] = (i < p && jj >= i) ? A[(int64_t)jj * m + i] : 0.f;
  }
  __syncthreads();
  // form Q in place (backward accumulation of the reflectors), columns 0..p-1
  for (int j = p - 1; j >= 0; --j) {
    float* x = A + (int64_t)j * m;
    const float tj = tau[j];
    for (int cc = j + 1 + warp; cc < p; cc += nw) {
      float* y = A + (int64_t)cc * m;
      float w = 0.f;
      for (int i = j + 1 + lane; i < m; i += 32) w = fmaf(x[i], y[i], w);
      w = (warp_sum(w) + y[j]) * tj;
      if (lane == 0) y[j] -= w;
      for (int i = j + 1 + lane; i < m; i += 32) y[i] = fmaf(-w, x[i], y[i]);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
      if (i < j)
        x[i] = 0.f;
      else if (i == j)
        x[i] = 1.f - tj;
      else
        x[i] = -tj * x[i];
    }
    __syncthreads();
  }
  // non-negative diagonal of R
  for (int j = 0; j < p; ++j) {
    if (Rm[j * q + j] < 0.f) {
      for (int t = threadIdx.x; t < q; t += blockDim.x) Rm[j * q + t] = -Rm[j * q + t];
      for (int i = threadIdx.x; i < m; i += blockDim.x) A[(int64_t)j * m + i] = -A[(int64_t)j * m + i];
    }
    __syncthreads();
  }
}
