// Orthogonalisation steps of Algorithm 1 for ranks up to 32, one CTA of 512 threads each:
//   k_qr_left_tiles : [Q, R] = qr(G_k^L), G_k <- Q, G_{k+1} <- R G_{k+1}^R            (k < d - 1)
//   k_lq_tiles      : the right-to-left steps k = k1 .. k0: (G_k^R)^T = Q R, G_k^R <- Q^T,
//                     G_{k-1}^L <- G_{k-1}^L R^T
// Both are CholeskyQR2 on the unfolding A (m rows, q <= Q columns, Q a multiple of 4) in shared
// memory, rows Q (+ 4) floats apart, columns q .. Q-1 zero: twice W = A^T A, W = L L^T, A <- A L^{-T};
// then R = L_2^T L_1^T. With a positive diagonal the factorisation is unique. A pivot at or below 1e-6
// of W's largest diagonal entry (condition number above about 1e3, rank deficiency) and unfoldings
// with fewer rows than columns take Householder reflections instead (zero-padded factors). Every sum
// has a fixed order.
// Bound: latency of one CTA (m = 1000, q = 10: about 28,000 cycles, of which 3,700 the first loads,
// 2 x 3,000 the Gram, 2 x 4,400 the factorisation by one warp, 2 x 1,700 the row solves, 2,700 R on the
// neighbour). The Gram as 4 x 4 tiles over row groups takes any q with 16 accumulators per thread; the
// former kernels held whole rows and their q (q + 1) / 2 products in registers, up to q = 16, and went
// through one generic kernel above. Warm, m = 1000, q = 10: QR step 17.8 -> 13.7 us, LQ sweep of the
// 100^4 cores 50 -> 38 us; 256 x 256 x 3 x 128 at rank 20: LQ sweep 120 -> 39 us, first QR step 81 -> 23.
#include <algorithm>

#include "tt_householder.cuh"

namespace {

constexpr int QT = 512;

template <int Q>
struct QrTiles {
  static constexpr int QP = Q % 8 == 0 ? Q + 4 : Q;  // row pitch: 16-byte row reads hit all banks
  static constexpr int B = Q / 4;
  static constexpr int NT = B * (B + 1) / 2;  // 4 x 4 tiles of the lower triangle of W
  static constexpr int NG = 480 / NT;  // row groups: thread t sums tile t % NT over group t / NT
  static constexpr int NS = 16 * NT >= QT ? 1 : QT / (16 * NT);  // slices of the sum over the groups
  // floats of scratch: partial tiles, slice sums, L_1^T, L_2^T, 1 / diagonals
  static constexpr int PART = NG * NT * 16;
  static constexpr int SCRATCH = PART + NS * NT * 16 + 2 * Q * Q + 2 * Q;
};

// One step of CholeskyQR: W = A^T A, L^T of W = L L^T into LT (Q x Q, row j = column j of L) and the
// reciprocals of its diagonal into dinv, A <- A L^{-T}; false (A unchanged) on a small pivot.
template <int Q>
__device__ bool cholqr_pass(float* As, int m, int q, float* part, float* slice, float* LT, float* dinv, int* flag) {
  using S = QrTiles<Q>;
  constexpr int QP = S::QP, NT = S::NT, NG = S::NG, NS = S::NS;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  {
    const int tile = t % NT, g = t / NT;
    int ti = 0;
    while ((ti + 1) * (ti + 2) / 2 <= tile) ++ti;
    const int tj = tile - ti * (ti + 1) / 2;
    if (g < NG) {
      float acc[4][4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
      const float* pi = As + 4 * ti;
      const float* pj = As + 4 * tj;
#pragma unroll 4
      for (int r = g; r < m; r += NG) {
        const float4 x = *reinterpret_cast<const float4*>(pi + r * QP);
        const float4 y = *reinterpret_cast<const float4*>(pj + r * QP);
        const float xa[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float2 xx = make_float2(xa[i], xa[i]);
          const float2 lo = tt_ffma2(xx, make_float2(y.x, y.y), make_float2(acc[i][0], acc[i][1]));
          const float2 hi = tt_ffma2(xx, make_float2(y.z, y.w), make_float2(acc[i][2], acc[i][3]));
          acc[i][0] = lo.x, acc[i][1] = lo.y, acc[i][2] = hi.x, acc[i][3] = hi.y;
        }
      }
      float4* out = reinterpret_cast<float4*>(part + (size_t)(g * NT + tile) * 16);
#pragma unroll
      for (int i = 0; i < 4; ++i) out[i] = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
    }
  }
  __syncthreads();
  for (int e = t; e < NS * NT * 16; e += QT) {  // groups of a slice, in order
    const int s = e / (NT * 16), k = e - s * (NT * 16);
    float sum = 0.f;
#pragma unroll 8
    for (int g = s; g < NG; g += NS) sum += part[(size_t)g * NT * 16 + k];
    slice[e] = sum;
  }
  __syncthreads();
  for (int e = t; e < Q * Q; e += QT) {  // W's lower triangle, row-major, unit pivots in the padding
    const int i = e / Q, k = e - i * Q;
    float v = i == k ? 1.f : 0.f;
    if (i < q && k <= i) {
      const int bi = i >> 2, at = (bi * (bi + 1) / 2 + (k >> 2)) * 16 + (i & 3) * 4 + (k & 3);
      v = 0.f;
#pragma unroll
      for (int s = 0; s < NS; ++s) v += slice[s * NT * 16 + at];
    }
    part[e] = v;
  }
  __syncthreads();
  if (warp == 0) {
    // One warp factors W, right-looking, lane i holding row i with the pivot column always in w[0]: the
    // loop over the columns stays rolled, because this code runs from a cold instruction cache
    // (unrolled it took 23,700 of 47,000 cycles at q = 10, and 3,600 where the second pass found it
    // cached). Columns go to LT unscaled and are scaled at the end.
    const int i = min(lane, Q - 1);
    float w[Q];
#pragma unroll
    for (int u = 0; u < Q / 4; ++u) {
      const float4 x = *reinterpret_cast<const float4*>(part + i * Q + 4 * u);
      w[4 * u] = x.x, w[4 * u + 1] = x.y, w[4 * u + 2] = x.z, w[4 * u + 3] = x.w;
    }
    float dmax = i < q ? part[i * Q + i] : 0.f;
    for (int o = 16; o > 0; o >>= 1) dmax = fmaxf(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
    bool ok = dmax > 0.f && isfinite(dmax);
    const float thr = 1e-6f * dmax;
    __syncwarp();
#pragma unroll 1
    for (int j = 0; j < Q; ++j) {
      const float c = w[0], p = __shfl_sync(0xffffffffu, c, j);
      if (!(p > thr) || !isfinite(p)) ok = ok && j >= q;
      const float f = -c * (1.f / fmaxf(p, 1e-30f));
      if (lane < Q) LT[j * Q + lane] = lane >= j ? c : 0.f;
#pragma unroll
      for (int k = 1; k < Q; ++k) w[k - 1] = fmaf(f, __shfl_sync(0xffffffffu, c, j + k), w[k]);
    }
    __syncwarp();
    if (lane < Q) {
      const float l = sqrtf(fmaxf(LT[lane * Q + lane], 1e-30f));
      dinv[lane] = 1.f / l;
      part[lane] = l;
    }
    __syncwarp();
    for (int e = lane; e < Q * Q; e += 32) {
      const int j = e / Q, k = e - j * Q;
      LT[e] = k == j ? part[j] : LT[e] * dinv[j];
    }
    if (lane == 0) *flag = ok;
  }
  __syncthreads();
  if (!*flag) return false;
  // rows: x L^T = a, two at a time so that both read the same L
  for (int r0 = t; r0 < m; r0 += 2 * QT) {
    const int r1 = r0 + QT;
    float a[Q], b[Q];
    const float4* p0 = reinterpret_cast<const float4*>(As + (size_t)r0 * QP);
    const float4* p1 = reinterpret_cast<const float4*>(As + (size_t)(r1 < m ? r1 : r0) * QP);
#pragma unroll
    for (int u = 0; u < Q / 4; ++u) {
      const float4 x = p0[u], y = p1[u];
      a[4 * u] = x.x, a[4 * u + 1] = x.y, a[4 * u + 2] = x.z, a[4 * u + 3] = x.w;
      b[4 * u] = y.x, b[4 * u + 1] = y.y, b[4 * u + 2] = y.z, b[4 * u + 3] = y.w;
    }
#pragma unroll
    for (int j = 0; j < Q; ++j) {
      const float d = dinv[j];
      a[j] *= d;
      b[j] *= d;
#pragma unroll
      for (int u = j / 4; u < Q / 4; ++u) {
        const float4 l = *reinterpret_cast<const float4*>(LT + j * Q + 4 * u);
        const float la[4] = {l.x, l.y, l.z, l.w};
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (4 * u + e > j) {
            a[4 * u + e] = fmaf(-a[j], la[e], a[4 * u + e]);
            b[4 * u + e] = fmaf(-b[j], la[e], b[4 * u + e]);
          }
      }
    }
    float4* o0 = reinterpret_cast<float4*>(As + (size_t)r0 * QP);
    float4* o1 = reinterpret_cast<float4*>(As + (size_t)r1 * QP);
#pragma unroll
    for (int u = 0; u < Q / 4; ++u) {
      o0[u] = make_float4(a[4 * u], a[4 * u + 1], a[4 * u + 2], a[4 * u + 3]);
      if (r1 < m) o1[u] = make_float4(b[4 * u], b[4 * u + 1], b[4 * u + 2], b[4 * u + 3]);
    }
  }
  __syncthreads();
  return true;
}

// CholeskyQR2 of As (destroyed when it returns false); R (Q x Q row-major, upper triangular) into Rm
template <int Q>
__device__ bool cholqr2(float* As, int m, int q, float* scratch, float* Rm, int* flag) {
  using S = QrTiles<Q>;
  float* slice = scratch + S::PART;
  float* L1 = slice + S::NS * S::NT * 16;
  float* L2 = L1 + Q * Q;
  float* dinv = L2 + Q * Q;
  if (!cholqr_pass<Q>(As, m, q, scratch, slice, L1, dinv, flag)) return false;
  if (!cholqr_pass<Q>(As, m, q, scratch, slice, L2, dinv + Q, flag)) return false;
  for (int e = threadIdx.x; e < Q * Q; e += QT) {  // R = L_2^T L_1^T (zero outside l = i .. j)
    const int i = e / Q, j = e - i * Q;
    float acc = 0.f;
#pragma unroll 4
    for (int l = 0; l < Q; ++l) acc = fmaf(L2[i * Q + l], L1[l * Q + j], acc);
    Rm[e] = acc;
  }
  __syncthreads();
  return true;
}

// y = R x for `n` vectors of q floats, component b of vector c at X[c * cs + b * bs], in place
template <int Q>
__device__ void apply_r(const float* Rm, float* X, int n, int q, int cs, int bs) {
  for (int c0 = threadIdx.x; c0 < n; c0 += 2 * QT) {
    const bool two = c0 + QT < n;
    float* p0 = X + (size_t)c0 * cs;
    float* p1 = two ? p0 + (size_t)QT * cs : p0;
    float x[Q], y[Q];
#pragma unroll
    for (int b = 0; b < Q; ++b) {
      x[b] = b < q ? p0[(size_t)b * bs] : 0.f;
      y[b] = b < q ? p1[(size_t)b * bs] : 0.f;
    }
#pragma unroll
    for (int a = 0; a < Q; ++a) {
      float sx = 0.f, sy = 0.f;
#pragma unroll
      for (int u = a / 4; u < Q / 4; ++u) {  // entries of R left of the diagonal are zero
        const float4 r = *reinterpret_cast<const float4*>(Rm + a * Q + 4 * u);
        sx = fmaf(r.x, x[4 * u], fmaf(r.y, x[4 * u + 1], fmaf(r.z, x[4 * u + 2], fmaf(r.w, x[4 * u + 3], sx))));
        sy = fmaf(r.x, y[4 * u], fmaf(r.y, y[4 * u + 1], fmaf(r.z, y[4 * u + 2], fmaf(r.w, y[4 * u + 3], sy))));
      }
      if (a < q) {
        p0[(size_t)a * bs] = sx;
        if (two) p1[(size_t)a * bs] = sy;
      }
    }
  }
}

// Position idx = t, t + QT, t + 2 QT, ... as (idx / n, idx mod n) without a division per step
struct Walk {
  int hi, lo;
  const int n, dh, dl;
  __device__ explicit Walk(int n_) : hi((int)threadIdx.x / n_), lo((int)threadIdx.x % n_), n(n_), dh(QT / n_), dl(QT % n_) {}
  __device__ void next() {
    hi += dh;
    lo += dl;
    if (lo >= n) {
      lo -= n;
      ++hi;
    }
  }
};

__device__ __forceinline__ void cp_async4(float* dst, const float* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async16(float* dst, const float* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_done() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// asynchronous copy of n floats into 16-byte-aligned shared memory
__device__ __forceinline__ void fetch_flat(float* dst, const float* src, int n) {
  if ((reinterpret_cast<uintptr_t>(src) & 15) == 0) {
    for (int i = 4 * threadIdx.x; i + 3 < n; i += 4 * QT) cp_async16(dst + i, src + i);
    for (int i = (n & ~3) + threadIdx.x; i < n; i += QT) cp_async4(dst + i, src + i);
  } else {
    for (int i = threadIdx.x; i < n; i += QT) cp_async4(dst + i, src + i);
  }
}

// Shared memory (floats): As (m x QP, rounded up to the dense m x q of the fallback) | NX (the
// neighbour core, 16-byte aligned) | scratch | Rm (Q x Q) | tau (Q) | colsc (4)
template <int Q>
size_t qr_smem(int64_t m, int64_t nx) {
  return sizeof(float) * ((size_t)m * QrTiles<Q>::QP + (size_t)((nx + 3) & ~3) + QrTiles<Q>::SCRATCH + Q * Q + Q + 4);
}

template <int Q>
__global__ void __launch_bounds__(QT, 1) k_qr_left_tiles(float* core, float* next, int r0, int n, int q, int ncols, int prefetch,
                                                           const int* status) {
  extern __shared__ __align__(16) float sm[];
  __shared__ int flag;
  constexpr int QP = QrTiles<Q>::QP;
  if (*status != 0) return;
  const int m = r0 * n, t = threadIdx.x, nx = prefetch ? q * ncols : 0;
  float* As = sm;
  float* NX = As + (size_t)m * QP;
  float* scratch = NX + ((nx + 3) & ~3);
  float* Rm = scratch + QrTiles<Q>::SCRATCH;
  float* tau = Rm + Q * Q;
  fetch_flat(NX, next, nx);
  bool ok = m >= q;
  if (ok) {  // columns m floats apart -> rows; four columns per 16-byte store
    constexpr int U = 4;
    Walk ld(m), st(m);
    for (int k0 = t; k0 < m * (Q / 4); k0 += U * QT) {
      float v[U][4];
#pragma unroll
      for (int u = 0; u < U; ++u, ld.next())
#pragma unroll
        for (int e = 0; e < 4; ++e)
          v[u][e] = 4 * ld.hi + e < q ? core[(size_t)(4 * ld.hi + e) * m + ld.lo] : 0.f;
#pragma unroll
      for (int u = 0; u < U; ++u, st.next())
        if (st.hi < Q / 4) *reinterpret_cast<float4*>(As + st.lo * QP + 4 * st.hi) = make_float4(v[u][0], v[u][1], v[u][2], v[u][3]);
    }
    __syncthreads();
    ok = cholqr2<Q>(As, m, q, scratch, Rm, &flag);
    if (ok)
      for (Walk w(m); w.hi < Q / 4; w.next()) {
        const float4 x = *reinterpret_cast<const float4*>(As + w.lo * QP + 4 * w.hi);
        const float xa[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (4 * w.hi + e < q) core[(size_t)(4 * w.hi + e) * m + w.lo] = xa[e];
      }
  }
  if (!ok) {  // Householder on a dense column-major copy (pitch m)
    __syncthreads();
    for (int idx = t; idx < m * q; idx += QT) As[idx] = core[idx];
    __syncthreads();
    block_householder_qr(As, m, q, scratch, tau, tau + Q);
    const int p = min(m, q);
    for (int idx = t; idx < m * q; idx += QT) core[idx] = (idx / m < p) ? As[idx] : 0.f;
    for (int e = t; e < Q * Q; e += QT) {  // R from pitch q
      const int i = e / Q, j = e - i * Q;
      Rm[e] = i < q && j < q ? scratch[i * q + j] : 0.f;
    }
  }
  cp_async_done();
  __syncthreads();
  // G_{k+1}^R <- R G_{k+1}^R, a column is q consecutive floats; without room beside A in pieces
  // through A's place
  const int per = prefetch ? ncols : m * QP / q;
  float* X = prefetch ? NX : As;
  for (int c0 = 0; c0 < ncols; c0 += per) {
    const int nc = min(per, ncols - c0);
    if (!prefetch) {
      __syncthreads();
      for (int i = t; i < nc * q; i += QT) X[i] = next[(size_t)c0 * q + i];
      __syncthreads();
    }
    apply_r<Q>(Rm, X, nc, q, q, 1);
    __syncthreads();
    for (int i = t; i < nc * q; i += QT) next[(size_t)c0 * q + i] = X[i];
  }
}

struct LqArgs {
  float* core[TT_MAX_D];
  int r[TT_MAX_D + 1];
  int n[TT_MAX_D];
  int k1, k0;
  int mmax;   // rows of As
  int nxmax;  // floats of NX (a multiple of 4); 0: no room, the neighbours pass through As
};

// The cores pass through shared memory once: core k-1 is fetched while core k is factored, takes R^T
// there and is repacked as the next unfolding.
template <int Q>
__global__ void __launch_bounds__(QT, 1) k_lq_tiles(LqArgs a, const int* status) {
  extern __shared__ __align__(16) float sm[];
  __shared__ int flag;
  constexpr int QP = QrTiles<Q>::QP;
  if (*status != 0) return;
  const int t = threadIdx.x;
  float* As = sm;
  float* NX = As + (size_t)a.mmax * QP;
  float* scratch = NX + a.nxmax;
  float* Rm = scratch + QrTiles<Q>::SCRATCH;
  float* tau = Rm + Q * Q;
  // rows i of (G_k^R)^T: q consecutive floats each
  auto pack = [&](const float* src, int m, int q) {
    Walk w(q);
#pragma unroll 8
    for (int idx = t; idx < m * q; idx += QT, w.next()) As[w.hi * QP + w.lo] = src[idx];
    for (int r = t; r < m; r += QT)
      for (int a2 = q; a2 < Q; ++a2) As[r * QP + a2] = 0.f;
  };
  auto unpack = [&](float* dst, int m, int q) {
    Walk w(q);
    for (int idx = t; idx < m * q; idx += QT, w.next()) dst[idx] = As[w.hi * QP + w.lo];
  };
  pack(a.core[a.k1], a.n[a.k1] * a.r[a.k1 + 1], a.r[a.k1]);
  for (int k = a.k1; k >= a.k0; --k) {
    const int m = a.n[k] * a.r[k + 1], q = a.r[k], rows = a.r[k - 1] * a.n[k - 1];
    float *core = a.core[k], *prev = a.core[k - 1];
    __syncthreads();  // As is packed, NX is free
    if (a.nxmax) {
      fetch_flat(NX, prev, rows * q);
      if (k != a.k1) unpack(core, m, q);  // core k so far lies in As alone; the fallback reads it from memory
    }
    bool ok = m >= q;
    if (ok) ok = cholqr2<Q>(As, m, q, scratch, Rm, &flag);
    if (ok) {
      unpack(core, m, q);
    } else {
      __syncthreads();
      for (int idx = t; idx < m * q; idx += QT) {  // dense, column a2 of pitch m
        const int a2 = idx / m, i = idx - a2 * m;
        As[idx] = core[a2 + (size_t)q * i];
      }
      __syncthreads();
      block_householder_qr(As, m, q, scratch, tau, tau + Q);
      const int p = min(m, q);
      for (int idx = t; idx < m * q; idx += QT) {
        const int a2 = idx / m, i = idx - a2 * m;
        core[a2 + (size_t)q * i] = a2 < p ? As[idx] : 0.f;
      }
      for (int e = t; e < Q * Q; e += QT) {
        const int i = e / Q, j = e - i * Q;
        Rm[e] = i < q && j < q ? scratch[i * q + j] : 0.f;
      }
    }
    cp_async_done();
    __syncthreads();
    // G_{k-1}^L <- G_{k-1}^L R^T: row t is R applied to row t
    if (a.nxmax) {
      apply_r<Q>(Rm, NX, rows, q, 1, rows);
      __syncthreads();
      if (k > a.k0)
        pack(NX, a.n[k - 1] * q, a.r[k - 1]);
      else
        for (int i = t; i < rows * q; i += QT) prev[i] = NX[i];
    } else {
      const int per = a.mmax * QP / q;
      for (int t0 = 0; t0 < rows; t0 += per) {
        const int nr = min(per, rows - t0);
        for (int idx = t; idx < nr * q; idx += QT) {
          const int b = idx / nr, i = idx - b * nr;
          As[idx] = prev[t0 + i + (size_t)rows * b];
        }
        __syncthreads();
        apply_r<Q>(Rm, As, nr, q, 1, nr);
        __syncthreads();
        for (int idx = t; idx < nr * q; idx += QT) {
          const int b = idx / nr, i = idx - b * nr;
          prev[t0 + i + (size_t)rows * b] = As[idx];
        }
        __syncthreads();
      }
      if (k > a.k0) pack(prev, a.n[k - 1] * q, a.r[k - 1]);
    }
  }
}

template <int Q>
bool launch_left(tt_ctx* c, float* core, float* next, int r0, int n, int q, int ncols, cudaError_t* err) {
  const int64_t m = (int64_t)r0 * n, nx = (int64_t)q * ncols;
  const int prefetch = qr_smem<Q>(m, nx) <= TT_SMEM_MAX;
  const size_t smem = qr_smem<Q>(m, prefetch ? nx : 0);
  if (smem > TT_SMEM_MAX) return false;
  *err = tt_allow_smem(k_qr_left_tiles<Q>);
  if (*err != cudaSuccess) return true;
  k_qr_left_tiles<Q><<<1, QT, smem, c->stream>>>(core, next, r0, n, q, ncols, prefetch, c->d_status);
  *err = cudaGetLastError();
  return true;
}

template <int Q>
bool launch_lq(tt_ctx* c, LqArgs a, cudaError_t* err) {
  if (qr_smem<Q>(a.mmax, a.nxmax) > TT_SMEM_MAX) a.nxmax = 0;
  const size_t smem = qr_smem<Q>(a.mmax, a.nxmax);
  if (smem > TT_SMEM_MAX) return false;
  *err = tt_allow_smem(k_lq_tiles<Q>);
  if (*err != cudaSuccess) return true;
  k_lq_tiles<Q><<<1, QT, smem, c->stream>>>(a, c->d_status);
  *err = cudaGetLastError();
  return true;
}

// f<Q> for the smallest instance that holds q columns; false above 32
#define TT_QR_DISPATCH(q, call)            \
  ((q) <= 4    ? call(4)                   \
   : (q) <= 8  ? call(8)                   \
   : (q) <= 12 ? call(12)                  \
   : (q) <= 16 ? call(16)                  \
   : (q) <= 20 ? call(20)                  \
   : (q) <= 24 ? call(24)                  \
   : (q) <= 32 ? call(32)                  \
               : false)

}  // namespace

bool tt_qr_left_tiles(tt_ctx* c, float* core, float* next, int k, cudaError_t* err) {
  const int q = c->r[k + 1], ncols = (int)(c->n[k + 1] * c->r[k + 2]);
#define TT_CALL(QQ) launch_left<QQ>(c, core, next, c->r[k], (int)c->n[k], q, ncols, err)
  return TT_QR_DISPATCH(q, TT_CALL);
#undef TT_CALL
}

bool tt_lq_tiles(tt_ctx* c, float* const* cores, int k1, int k0, cudaError_t* err) {
  LqArgs a;
  a.k1 = k1;
  a.k0 = k0;
  a.mmax = a.nxmax = 0;
  int q = 1;
  for (int k = k0 - 1; k <= k1; ++k) {
    a.core[k] = cores[k];
    a.n[k] = (int)c->n[k];
    if (k >= k0) {
      q = std::max(q, c->r[k]);
      a.mmax = std::max(a.mmax, (int)c->n[k] * c->r[k + 1]);
      a.nxmax = std::max(a.nxmax, (int)((c->r[k - 1] * c->n[k - 1] * c->r[k] + 3) & ~3));
    }
  }
  for (int k = 0; k <= c->d; ++k) a.r[k] = c->r[k];
#define TT_CALL(QQ) launch_lq<QQ>(c, a, err)
  return TT_QR_DISPATCH(q, TT_CALL);
#undef TT_CALL
}
