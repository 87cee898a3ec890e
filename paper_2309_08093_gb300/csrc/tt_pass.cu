// Part (a) for several modes from one read of A (Alg. 1, Eqs. (eqn_h), (eqn_v)). With the modes cut
// into a head (the first ones) and a tail (the others), A is a list of contiguous slabs, one per
// tail index t, and the definition of Y_k regroups in two ways:
//
// k_head_pass, modes 0 and 1 (head = modes 0, 1; slab n_0 x n_1). With c_t the hash of the tail
// modes, Z_c = sum over the slabs with c_t = c of sign_t * slab, and
//     Y_0[(c + h_1(i_1)) mod J, i_0] += v_1(i_1) Z_c[i_0, i_1],
//     Y_1[(c + h_0(i_0)) mod J, i_1] += v_0(i_0) Z_c[i_0, i_1].
// A CTA walks slabs in the order of c (the plan of mode 1), sums a run of equal c in registers and
// adds each finished run to both sketches: one read of A where one launch per mode took two.
//
// k_tail_pass, the last one or two modes (head = the modes before them). With q_t the CountSketch of
// slab t under the head's hashes (J buckets, the same pattern for every slab) the tail modes s, l give
//     Y_l[(c + h_s(i_s)) mod J, i_l] += v_s(i_s) q_t[c],   Y_s[(c + h_l(i_l)) mod J, i_s] += v_l(i_l) q_t[c],
// again one read of A for both. The modes between (d >= 5) keep one launch each (tt_unfold.cu).
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "tt_unfold.cuh"

namespace {

__device__ __forceinline__ void red4(float* p, float4 v) { atomicAdd(reinterpret_cast<float4*>(p), v); }

// Sum of the n values p[0], p[stride], ..., which are left zero: an unevaluated pair of floats (two-sums),
// so that only its rounding to one float counts
__device__ __forceinline__ float take_copies(float* p, int64_t stride, int n) {
  float s = 0.f, e = 0.f;
  for (int c = 0; c < n; c += 8) {
    float v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = c + u < n ? p[(c + u) * stride] : 0.f;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      if (c + u < n) p[(c + u) * stride] = 0.f;
      const float t = s + v[u], b = t - s;
      e += (s - (t - b)) + (v[u] - b);
      s = t;
    }
  }
  return isfinite(e) ? s + e : s;  // (an infinite sum has no error term)
}

// Copies of an accumulator whose entries take `adds` FP32 adds one after the other: about 0.8 sqrt(adds), a
// power of two, which leaves an entry no more rounding than the sums of one launch per mode (register runs,
// a column copy per work item, Y_k). FP8, whose runs are exact there, asks for more by larger `adds`.
int copies_of(double adds) {
  int c = 1;
  while (3.0 * c * c < adds && c < 64) c *= 2;
  return c;
}

// ---------------------------------------------------------------------------------------------
// head pass

struct HeadArgs {
  const char* A;
  const float* scales;
  const uint32_t* plan;  // slabs grouped by c: fibre index of the slab | sign in bit 31
  const int32_t* key;    // c of each plan entry
  const int32_t *h0, *h1;
  const int8_t *v0, *v1;
  float* Y0r;  // c0 copies of J x p0, row b = bucket b of Y_0 (FP8: before the finite scales)
  float* Y1r;  // c1 copies of J x p1, row b = bucket b of Y_1
  int c0, c1;  // powers of two
  int64_t R;   // slabs
  int J, n0, n1, p0, p1;
  int G1, nch;  // columns i_1 per chunk of a slab, chunks
  int nseg;     // segments of the plan
  int pitch;    // floats per column of the transposition tile (a multiple of 32)
  uint32_t inv_n0;  // 2^32 / n_0 rounded up
  float* zero[2];   // sketches of the tail pass (which follows): zeroed on the side
  int64_t nzero[2];
};
constexpr int HEAD_BATCH = 256;  // plan entries staged at a time
constexpr int HEAD_TMAX = 320;   // two CTAs per SM at 102 registers
// entries of a slab's chunk per thread
template <int DT>
constexpr int head_acc() { return DT == TT_F64 ? 16 : 32; }

// 16-byte words [v ^ (i_1 / 4 mod 8)] of column i_1: with a pitch of 32 floats the 16-byte stores of
// a column and the reads below (8 column groups x 4 consecutive rows) both touch every bank once
__device__ __forceinline__ int tile_at(int i1, int i0, int pitch) {
  return i1 * pitch + ((((i0 >> 2) ^ ((i1 >> 2) & 7)) << 2) | (i0 & 3));
}

// VB bytes of A as 32-bit words. A is read with the streaming hint here and in the tail pass, so that the
// accumulators' copies stay in L2 beside it (100^4 FP32, all modes: 308 -> 297 us).
template <int VB>
__device__ __forceinline__ void head_load(const char* p, uint32_t* r) {
  if constexpr (VB == 16) {
    const uint4 u = __ldcs(reinterpret_cast<const uint4*>(p));
    r[0] = u.x, r[1] = u.y, r[2] = u.z, r[3] = u.w;
  } else if constexpr (VB == 8) {
    const uint2 u = __ldcs(reinterpret_cast<const uint2*>(p));
    r[0] = u.x, r[1] = u.y;
  } else if constexpr (VB == 4) {
    r[0] = __ldcs(reinterpret_cast<const uint32_t*>(p));
  } else if constexpr (VB == 2) {
    r[0] = __ldcs(reinterpret_cast<const unsigned short*>(p));
  } else {
    r[0] = __ldcs(reinterpret_cast<const unsigned char*>(p));
  }
}

// acc[e] += s * entry e of the loaded words (s = +-1)
template <int DT, int EPV>
__device__ __forceinline__ void head_add(const uint32_t* w, float s, float* acc) {
  if constexpr (DT == TT_F32 && EPV > 1) {
#pragma unroll
    for (int e = 0; e < EPV; e += 2) {
      const float2 d = tt_ffma2(make_float2(s, s), make_float2(__uint_as_float(w[e]), __uint_as_float(w[e + 1])),
                                make_float2(acc[e], acc[e + 1]));
      acc[e] = d.x, acc[e + 1] = d.y;
    }
  } else if constexpr (DT == TT_F32) {
    acc[0] = fmaf(s, __uint_as_float(w[0]), acc[0]);
  } else if constexpr (DT == TT_F64) {
#pragma unroll
    for (int e = 0; e < EPV; ++e) {
      const unsigned long long b = ((unsigned long long)w[2 * e + 1] << 32) | w[2 * e];
      acc[e] = fmaf(s, (float)__longlong_as_double((long long)b), acc[e]);
    }
  } else if constexpr (DT == TT_BF16) {
    const unsigned short sb = tt_bf16_sign(s);
    if constexpr (EPV == 1) {
      acc[0] = tt_fma_bf16((unsigned short)w[0], sb, acc[0]);
    } else {
#pragma unroll
      for (int e = 0; e < EPV; e += 2) tt_fma_bf16x2(w[e >> 1], sb, acc[e], acc[e + 1]);
    }
  } else {
    const unsigned short sh = tt_f16_sign(s);
    if constexpr (EPV == 1) {
      acc[0] = tt_fma_e4m3((unsigned short)w[0], sh, acc[0]);
    } else {
#pragma unroll
      for (int e = 0; e < EPV; e += 4) tt_fma_e4m3x4(w[e >> 2], sh, acc[e], acc[e + 1], acc[e + 2], acc[e + 3]);
    }
  }
}

// Bound: DRAM while runs are long (100^4 FP32, J = 1024, 9.8 slabs per run: 80 us with k_head_out, 170 us
// with one launch per mode), the flushes' L2 atomics and tile traffic beside it when they are short
// (J = 4096, 2.4 slabs per run: 128 and 206 us). The flushes go to L2 as 16-byte atomic adds
// along rows (5.9 TB/s of sums, measured alone) because shared-memory float atomics at random
// buckets sustain half of that (0.75 T adds/s) and need a copy of the columns per CTA. Two CTAs per
// SM: one flushes while the other loads.
// A slab's chunk is read as a run of VB-byte vectors, whatever columns they lie in: thread t holds
// the vectors t + T j. U slabs are loaded ahead of the sums.
// Accuracy: a bucket of Y_0 (Y_1) takes about runs * n_1 / J (runs * n_0 / J) of these adds one after the
// other, and the rounding error of FP32 sums grows with their square root; so segments add to one of c0
// (c1) copies of the rows in turn, and k_head_out adds the copies up. FP8 rows of Y_0 are summed before
// their scales, exactly while |sums| < 2^15. (One sum per row: 83 and 126 us.) Relative error, one sum / copies / one launch per mode:
// Y_1 of 100^4 FP32 1.8e-7 / 8.2e-8 / 9.5e-8, Y_0 of 256 x 256 x 3 x 128 FP32 1.3e-7 / 5.8e-8 / 8.9e-8,
// of 40^5 FP8 1.3e-7 / 2.5e-8 / 4.6e-8.
template <int DT, int VB>
__global__ void __launch_bounds__(HEAD_TMAX, 2) k_head_pass(HeadArgs a) {
  constexpr int EB = TtElem<DT>::bytes;
  constexpr int EPV = VB / EB;                // entries per vector
  constexpr int NV = head_acc<DT>() / EPV;    // vectors per thread
  constexpr int W = VB < 4 ? 1 : VB / 4;      // registers per vector
  constexpr int U = NV * W >= 32 ? 1 : 32 / (NV * W);
  extern __shared__ __align__(16) float hsm[];
  const int T = blockDim.x, t = threadIdx.x;
  for (int z = 0; z < 2; ++z)
    for (int64_t i = (int64_t)blockIdx.x * T + t; i < a.nzero[z]; i += (int64_t)gridDim.x * T) a.zero[z][i] = 0.f;
  const int n0 = a.n0, J = a.J, pitch = a.pitch;
  const int ch = blockIdx.x % a.nch, seg = blockIdx.x / a.nch;
  const int c0 = ch * a.G1, g1 = min(a.G1, a.n1 - c0), g1p = (g1 + 3) & ~3;
  const int rows_tile = (a.G1 + 3) & ~3, n0p = (n0 + 3) & ~3;
  float* tile = hsm;                                        // rows_tile x pitch
  float* cf0 = tile + (size_t)rows_tile * pitch;            // n0p: v_0 (times the FP8 scale)
  float* sc0 = cf0 + n0p;                                   // n0p: what of the FP8 scale k_head_out leaves
  int* hh0 = reinterpret_cast<int*>(sc0 + n0p);             // n0p
  int* hh1 = hh0 + n0p;                                     // rows_tile: h_1, sign in bit 31
  uint32_t* sw = reinterpret_cast<uint32_t*>(hh1 + rows_tile);  // HEAD_BATCH
  int* sk = reinterpret_cast<int*>(sw + HEAD_BATCH);        // HEAD_BATCH
  for (int i = t; i < n0p; i += T) {
    const float s = a.scales && i < n0 ? __ldg(a.scales + i) : 1.f;
    sc0[i] = isfinite(s) ? 1.f : s;
    cf0[i] = i < n0 && __ldg(a.v0 + i) < 0 ? -s : s;
    hh0[i] = i < n0 ? __ldg(a.h0 + i) : 0;
  }
  for (int i = t; i < g1; i += T) hh1[i] = __ldg(a.h1 + c0 + i) | (__ldg(a.v1 + c0 + i) < 0 ? (int)0x80000000 : 0);
  for (int i = t; i < rows_tile * pitch; i += T) tile[i] = 0.f;  // the padding stays zero
  const int64_t eb = a.R * seg / a.nseg, ee = a.R * (seg + 1) / a.nseg;
  const int ne = n0 * g1;  // entries of a slab's chunk
  const char* base = a.A + (int64_t)c0 * n0 * EB + (int64_t)t * VB;
  const int64_t fb = (int64_t)n0 * EB;
  float* const y0r = a.Y0r + (int64_t)(seg & (a.c0 - 1)) * J * a.p0;
  float* const y1r = a.Y1r + (int64_t)(seg & (a.c1 - 1)) * J * a.p1;
  const bool quads = EPV >= 4 && (n0 & 3) == 0;  // every four entries lie in one column
  float acc[NV][EPV];
#pragma unroll
  for (int j = 0; j < NV; ++j)
#pragma unroll
    for (int e = 0; e < EPV; ++e) acc[j][e] = 0.f;

  // the finished run of group c: rows of Y_0 and Y_1 (16-byte atomic adds), through the tile where a
  // thread's entries are not a row's
  auto flush = [&](int c) {
    __syncthreads();  // the tile's last readers are done
    if (quads) {
#pragma unroll
      for (int j = 0; j < NV; ++j)
#pragma unroll
        for (int e = 0; e + 3 < EPV; e += 4) {
            const int en = (t + T * j) * EPV + e;
            if (en < ne) {
              const int i1 = (int)__umulhi((uint32_t)en, a.inv_n0), i0 = en - i1 * n0;
              const int hw = hh1[i1];
              const float s1 = hw < 0 ? -1.f : 1.f;
              const float4 z = make_float4(acc[j][e], acc[j][e + 1], acc[j][e + 2], acc[j][e + 3]);
              *reinterpret_cast<float4*>(tile + tile_at(i1, i0, pitch)) = z;
              float4 m = make_float4(s1 * z.x, s1 * z.y, s1 * z.z, s1 * z.w);
              if (DT == TT_FP8E4M3) m.x *= sc0[i0], m.y *= sc0[i0 + 1], m.z *= sc0[i0 + 2], m.w *= sc0[i0 + 3];
              red4(y0r + (int64_t)tt_modj(c + (hw & 0x7FFFFFFF), J) * a.p0 + i0, m);
            }
          }
    } else {
#pragma unroll
      for (int j = 0; j < NV; ++j)
#pragma unroll
        for (int e = 0; e < EPV; ++e) {
          const int en = (t + T * j) * EPV + e;
          if (en < ne) {
            const int i1 = (int)__umulhi((uint32_t)en, a.inv_n0), i0 = en - i1 * n0;
            tile[tile_at(i1, i0, pitch)] = acc[j][e];
          }
        }
    }
#pragma unroll
    for (int j = 0; j < NV; ++j)
#pragma unroll
      for (int e = 0; e < EPV; ++e) acc[j][e] = 0.f;
    __syncthreads();
    // the columns of the tile as rows of Y_1: 4 rows i_0 x 32 columns i_1 per warp step
    const int g = t & 7, q = (t >> 3) & 3;
    const int nq = n0p >> 2, ng = (g1p + 31) >> 5;
    for (int task = t >> 5; task < nq * ng; task += T >> 5) {
      const int ig = task / nq, i0 = 4 * (task - ig * nq) + q, i1 = 32 * ig + 4 * g;
      if (i0 < n0 && i1 < g1p) {
        const float* src = tile + tile_at(i1, i0, pitch);  // columns i1 .. i1 + 3 share the swizzle
        const float s = cf0[i0];
        red4(y1r + (int64_t)tt_modj(c + hh0[i0], J) * a.p1 + c0 + i1,
             make_float4(s * src[0], s * src[pitch], s * src[2 * pitch], s * src[3 * pitch]));
      }
    }
    if (!quads)  // and the rows of Y_0
      for (int i = t; i < nq * g1; i += T) {
        const int i1 = i / nq, i0 = 4 * (i - i1 * nq);
        const int hw = hh1[i1];
        const float s1 = hw < 0 ? -1.f : 1.f;
        const float4 z = *reinterpret_cast<const float4*>(tile + tile_at(i1, i0, pitch));
        float4 m = make_float4(s1 * z.x, s1 * z.y, s1 * z.z, s1 * z.w);
        if (DT == TT_FP8E4M3) m.x *= sc0[i0], m.y *= sc0[i0 + 1], m.z *= sc0[i0 + 2], m.w *= sc0[i0 + 3];
        red4(y0r + (int64_t)tt_modj(c + (hw & 0x7FFFFFFF), J) * a.p0 + i0, m);
      }
  };

  int cur = -1;
  for (int64_t b0 = eb; b0 < ee; b0 += HEAD_BATCH) {
    const int nb = (int)min((int64_t)HEAD_BATCH, ee - b0);
    __syncthreads();
    for (int i = t; i < nb; i += T) {
      sw[i] = __ldg(a.plan + b0 + i);
      sk[i] = __ldg(a.key + b0 + i);
    }
    __syncthreads();
    for (int i = 0; i < nb; i += U) {
      uint32_t r[U][NV][W];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (U == 1 || i + u < nb) {
          const char* p = base + (int64_t)(sw[i + u] & 0x7FFFFFFFu) * fb;
#pragma unroll
          for (int j = 0; j < NV; ++j)
            if ((t + T * j) * EPV < ne) head_load<VB>(p + T * j * VB, r[u][j]);
        }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (U == 1 || i + u < nb) {
          const int c = sk[i + u];
          if (c != cur) {
            if (cur >= 0) flush(cur);
            cur = c;
          }
          const float s = (sw[i + u] >> 31) ? -1.f : 1.f;
#pragma unroll
          for (int j = 0; j < NV; ++j)
            if ((t + T * j) * EPV < ne) head_add<DT, EPV>(r[u][j], s, acc[j]);
        }
    }
  }
  if (cur >= 0) flush(cur);
}

// Y_0 and Y_1 (column-major, J x n) from the copies of the row-major J x p accumulators, 32 x 32 tiles;
// the accumulators are left zero for the next head pass
struct HeadOutArgs {
  float *Y0r, *Y1r, *Y0, *Y1;
  const float* scales;  // of Y_0's columns (null: none)
  int J, n0, n1, p0, p1, c0, c1, tiles0;
};
__global__ void __launch_bounds__(1024) k_head_out(HeadOutArgs a) {
  __shared__ float tl[32][33];
  const bool first = (int)blockIdx.y < a.tiles0;
  const int n = first ? a.n0 : a.n1, p = first ? a.p0 : a.p1, J = a.J;
  const int i0 = 32 * ((int)blockIdx.y - (first ? 0 : a.tiles0)), b0 = 32 * blockIdx.x;
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
  if (b0 + y < J && i0 + x < n) {
    float s = first && a.scales ? __ldg(a.scales + i0 + x) : 1.f;
    if (!isfinite(s)) s = 1.f;  // (k_head_pass applied it)
    tl[y][x] = s * take_copies((first ? a.Y0r : a.Y1r) + (int64_t)(b0 + y) * p + i0 + x, (int64_t)J * p, first ? a.c0 : a.c1);
  }
  __syncthreads();
  if (b0 + x < J && i0 + y < n) (first ? a.Y0 : a.Y1)[(int64_t)(i0 + y) * J + b0 + x] = tl[x][y];
}

// ---------------------------------------------------------------------------------------------
// tail pass

// The plans of both passes for one draw, one CTA each.
// CTA b < nchunk: the head's pattern of the tail pass, the same for every slab. The entries of a
// slab, cut into chunks of `chunk` entries, are listed by bucket (sum of the head modes' hashes mod
// J) within each chunk, in blocks of four 16-bit entry numbers; a bucket's last block is filled up
// with a number from `chunk` on, an entry that is staged as zero (FP8: there are n_0 of them, one of each
// row, and the one of a row that the bucket holds is taken). Bucket word: first block | blocks << 16.
// Sign word: the signs (product of the head modes' v) of 32 entries.
// CTA nchunk (when R > 0): the slabs of the head pass sorted by c, the hash of the modes 2 .. d-1
// (plan word: fibre index of the slab | sign << 31). One CTA sorts up to 2^15 slabs; with more the
// grid-wide plan of mode 1 (tt_context.cu) is used.
// Both are counting sorts: counts in shared memory, a scan over the J buckets, placement in shared
// memory and coalesced stores. Bound by the latency of one CTA: with the tables' draw 14 us of a
// fresh-draw call at 101 x 84 x 93 x 100 (22 us when every entry was hashed twice and stored where it
// belongs), 15 us at 100^4 (30).
struct PassPlanArgs {
  const int32_t* h;
  const int8_t* v;
  int64_t n[TT_MAX_D], noff[TT_MAX_D];
  int d, nh, J, chunk, nchunk, blocks;
  int64_t E;
  uint16_t* list;    // 4 * blocks numbers per chunk
  uint32_t* bucket;  // J words per chunk
  uint32_t* sign;    // (chunk + 31) / 32 words per chunk
  int nkeys;         // entries or slabs that a CTA sorts, at most
  int zeros;         // zero entries behind a staged chunk: a row each (FP8) or one
  int64_t R;         // slabs of the head pass (0: not planned here)
  uint32_t* plan;
  int32_t* key;
};
constexpr int64_t HEAD_PLAN_MAX = 1 << 15;
// floats of a pass's accumulators, 48 MB: they are to stay in L2 beside A (300 x 300 x 33 x 33 at J = 8192
// with 79 MB: head pass 359 us, one launch per mode 312)
constexpr int64_t PASS_COPIES_MAX = 12 << 20;

__global__ void __launch_bounds__(1024) k_pass_plans(PassPlanArgs a) {
  extern __shared__ int psm[];  // J counts, then cursors
  uint16_t* keys = reinterpret_cast<uint16_t*>(psm + ((a.J + 1) & ~1));  // buckets (J <= 8192), sign in bit 15
  uint16_t* ord = keys + a.nkeys;  // the sorted numbers, on their way to coalesced stores
  __shared__ int wsum[32];
  const int t = threadIdx.x, T = blockDim.x, lane = t & 31, warp = t >> 5;
  const bool slabs = (int)blockIdx.x == a.nchunk;
  const int m0 = slabs ? 2 : 0, m1 = slabs ? a.d : a.nh;  // modes that are hashed
  const int64_t e0 = slabs ? 0 : (int64_t)blockIdx.x * a.chunk;
  const int ne = slabs ? (int)a.R : (int)min((int64_t)a.chunk, a.E - e0);
  for (int b = t; b < a.J; b += T) psm[b] = 0;
  __syncthreads();
  uint32_t* sign = a.sign + (int64_t)blockIdx.x * ((a.chunk + 31) / 32);
  constexpr int U = 4;  // entries whose table lookups are in flight together
  for (int i0 = t; i0 - t < ne; i0 += U * T) {
    uint32_t rem[U];
    int key[U], neg[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      rem[u] = (uint32_t)(e0 + min(i0 + u * T, ne - 1));
      key[u] = neg[u] = 0;
    }
    for (int s = m0; s < m1; ++s) {
      const uint32_t n = (uint32_t)a.n[s];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint32_t q = rem[u] / n, x = rem[u] - q * n;
        rem[u] = q;
        key[u] = tt_modj(key[u] + __ldg(a.h + a.noff[s] + x), a.J);
        neg[u] ^= __ldg(a.v + a.noff[s] + x) < 0;
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = i0 + u * T;
      const uint32_t w = __ballot_sync(0xffffffffu, neg[u] && i < ne);
      if (i < ne) {
        atomicAdd(psm + key[u], 1);
        keys[i] = (uint16_t)(key[u] | neg[u] << 15);
        if (!slabs && lane == 0) sign[i >> 5] = w;
      }
    }
  }
  __syncthreads();
  // exclusive scan of the J counts (block counts for a pattern): each thread a run of buckets
  const int per = (a.J + T - 1) / T, lo = min(a.J, t * per), hi = min(a.J, lo + per);
  int sum = 0;
  for (int b = lo; b < hi; ++b) sum += slabs ? psm[b] : (psm[b] + 3) >> 2;
  int inc = sum;
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) wsum[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    int x = wsum[lane];
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    wsum[lane] = x;
  }
  __syncthreads();
  int at = (warp ? wsum[warp - 1] : 0) + inc - sum;
  uint32_t* bucket = a.bucket + (int64_t)blockIdx.x * a.J;
  for (int b = lo; b < hi; ++b) {
    const int cnt = psm[b];
    if (slabs) {
      psm[b] = at;
      at += cnt;
    } else {
      const int nb = (cnt + 3) >> 2;
      bucket[b] = (uint32_t)at | (uint32_t)nb << 16;
      psm[b] = 4 * at;
      at += nb;
    }
  }
  __syncthreads();
  for (int i = t; i < ne; i += T) ord[atomicAdd(psm + (keys[i] & 0x7FFF), 1)] = (uint16_t)i;
  __syncthreads();
  if (!slabs) {  // fill up last blocks (they start at multiples of 4)
    for (int b = lo; b < hi; ++b) {
      int p = psm[b];
      if (p & 3)
        for (const int e = ord[p - 1], m = a.zeros, z = a.chunk + ((e - a.chunk) % m + m) % m; p & 3; ++p) ord[p] = (uint16_t)z;
    }
    __syncthreads();
  }
  if (slabs) {
    for (int p = t; p < ne; p += T) {
      const int i = ord[p], key = keys[i];
      a.plan[p] = (uint32_t)((int64_t)i * a.n[1]) | (uint32_t)(key >> 15) << 31;
      a.key[p] = key & 0x7FFF;
    }
  } else {  // (wsum[31]: blocks of all buckets)
    uint2* list = reinterpret_cast<uint2*>(a.list) + (int64_t)blockIdx.x * a.blocks;
    for (int p = t; p < wsum[31]; p += T) list[p] = reinterpret_cast<const uint2*>(ord)[p];
  }
}

struct TailArgs {
  const char* A;
  const float* scales;
  const uint16_t* list;
  const uint32_t *bucket, *sign;
  const int32_t *hs, *hl;  // hashes and signs of the tail modes s (null: one tail mode) and l
  const int8_t *vs, *vl;
  float *Ys, *Yl;  // cs copies of J x n_s, cl copies of J x n_l, column-major, zeroed
  int cs, cl;      // powers of two
  int64_t E;       // entries of a slab
  int J, n0, chunk, nchunk, blocks, ns, nl, ngl;  // ngl: groups of V indices i_l
  int parts;       // lanes that share a bucket's list (a power of two)
  uint32_t inv_n0;  // 2^32 / n_0 rounded up (FP8: entry number -> i_0)
  int64_t units;   // nchunk * ngl * ns
};

constexpr int TAIL_T = 1024;
// Slabs that Y_l's registers sum before they are added to a copy. FP8 launches of one mode add a row's
// entries exactly before its scale rounds them, so their sums are the shortest to match.
__host__ __device__ constexpr int tail_run(int dtype) { return dtype == TT_FP8E4M3 ? 4 : 8; }

// What a thread stages per slab group: JJ loads of EPW entries from each of V slabs. An entry of the
// staged chunk holds its V slabs' signed values side by side (V * SB bytes), so that one
// shared-memory load per list number serves V slabs. FP64 is staged as FP32.
template <int DT, int V, int EPW>
struct TailShape {
  static constexpr int EB = TtElem<DT>::bytes;
  static constexpr int SB = EB == 8 ? 4 : EB;
  static constexpr int JJ = EB == 8 ? 5 : 20 / V;
  static constexpr int ENT = V * SB;  // bytes of a staged entry
};

// q += x for the two FP32 values of 64-bit words (add.rn.f32x2): kept in 64-bit registers, so that the
// shared-memory load feeds the add without moves
__device__ __forceinline__ void add2(unsigned long long& q, unsigned long long x) {
  asm("add.rn.f32x2 %0, %0, %1;" : "+l"(q) : "l"(x));
}

// One CTA of 1024 threads per SM; unit = (chunk, group of V indices i_l, i_s), consecutive units in one
// CTA. Thread t owns bucket b of Y_l and so, per i_s, the head's bucket b - h_s(i_s): it sums that
// bucket's list from the staged slabs (random 8-byte shared-memory loads), keeps Y_l's column sums in
// registers while i_s advances (tail_run slabs at most), and adds its q to Y_s with atomics that are
// contiguous across a warp. The next unit's slabs are loaded into registers meanwhile. The signs go on
// when a slab is staged.
// Accuracy: FP32 sums of n terms one after the other carry a rounding error that grows with sqrt(n), and
// a bucket of Y_s takes up to n_l * nchunk of these adds, one of Y_l n_s * nchunk. They are cut in two
// levels: units go to one of cs (cl) copies of Y_s (Y_l) in turn, and k_tail_out adds the copies up; the
// lists are summed block by block where a bucket has several. Relative error of Y_s, one sum / in levels /
// one launch per mode: 256 x 256 x 3 x 128 FP32 5.4e-7 / 1.1e-7 / 2.0e-7, 40^5 FP8 2.2e-7 / 7.3e-8 /
// 7.8e-8, 100^4 FP32 1.8e-7 / 7.9e-8 / 9.5e-8.
// Bound: instruction issue (64% active; 123 M warp instructions) and the random shared-memory loads
// (141 k of 333 k cycles). 100^4 FP32: 176 us for both modes at J = 4096 (161 us without the copies, one
// launch per mode 206 us).
// FP8 scales that are infinite or NaN: the lists' padding, a zero times such a scale, must stay out of the
// sums. Such tensors take the WILD instance, which skips it entry by entry; both are launched and the CTAs of
// the one that does not apply return once they have read the scales (3 us; a test in the sums: 13 us of
// 234 at 40^5).
template <int DT, int V, int EPW, int RPT, bool WILD = false>
__global__ void __launch_bounds__(TAIL_T, 1) k_tail_pass(TailArgs a) {
  using Sh = TailShape<DT, V, EPW>;
  constexpr int EB = Sh::EB, JJ = Sh::JJ, ENT = Sh::ENT, T = TAIL_T;
  using Word = typename std::conditional<EB == 8, double, uint32_t>::type;
  extern __shared__ __align__(16) unsigned char tsm[];
  const int zeros = DT == TT_FP8E4M3 ? a.n0 : 1;
  unsigned char* buf = tsm;  // chunk + zeros entries
  uint2* sl = reinterpret_cast<uint2*>(buf + (((size_t)(a.chunk + zeros) * ENT + 15) & ~(size_t)15));  // blocks
  uint32_t* sb = reinterpret_cast<uint32_t*>(sl + a.blocks);                                 // J
  float* ssc = reinterpret_cast<float*>(sb + a.J);                                           // n0 FP8 scales
  const int t = threadIdx.x, J = a.J, parts = a.parts;
  const int part = t & (parts - 1), row0 = t / parts, rstep = T / parts;
  if (DT == TT_FP8E4M3) {
    bool wild = false;
    for (int i = t; i < a.n0; i += T) {
      ssc[i] = __ldg(a.scales + i);
      wild = wild || !isfinite(ssc[i]);
    }
    if ((__syncthreads_or(wild) != 0) != WILD) return;
  }
  for (int i = t; i < zeros * ENT; i += T) buf[(size_t)a.chunk * ENT + i] = 0;
  const int64_t u0 = a.units * blockIdx.x / gridDim.x, u1 = a.units * (blockIdx.x + 1) / gridDim.x;
  if (u0 >= u1) return;
  int is = (int)(u0 % a.ns), gl = (int)((u0 / a.ns) % a.ngl), ch = (int)(u0 / a.ns / a.ngl);

  Word pw[JJ][V];
  int nj = 0;  // loads of this thread in the chunk last fetched
  // slabs past the last index l read the last one's values, which are not added to any column
  auto fetch = [&](int ch_, int gl_, int is_) {
    const int ne = (int)min((int64_t)a.chunk, a.E - (int64_t)ch_ * a.chunk);
    nj = (ne / EPW - t + T - 1) / T;
#pragma unroll
    for (int v = 0; v < V; ++v) {
      const int il = min(V * gl_ + v, a.nl - 1);
      const char* p = a.A + (((int64_t)il * a.ns + is_) * a.E + (int64_t)ch_ * a.chunk) * EB + t * (EPW * EB);
#pragma unroll
      for (int jj = 0; jj < JJ; ++jj) {
        if (jj < nj) {
          const char* q = p + T * jj * (EPW * EB);
          if constexpr (EPW * EB == 8) pw[jj][v] = __ldcs(reinterpret_cast<const double*>(q));
          else if constexpr (EPW * EB == 4) pw[jj][v] = __ldcs(reinterpret_cast<const uint32_t*>(q));
          else if constexpr (EPW * EB == 2) pw[jj][v] = __ldcs(reinterpret_cast<const unsigned short*>(q));
          else pw[jj][v] = __ldcs(reinterpret_cast<const unsigned char*>(q));
        }
      }
    }
  };
  uint32_t smask = 0;  // signs of this thread's entries, bit EPW * jj + e
  auto stage = [&]() {
#pragma unroll
    for (int jj = 0; jj < JJ; ++jj) {
      if (jj >= nj) continue;
      unsigned char* dst = buf + (size_t)((t + T * jj) * EPW) * ENT;
      if constexpr (EB == 8) {
        const float s = __uint_as_float(0x3F800000u | (smask << (31 - jj) & 0x80000000u));
        *reinterpret_cast<float2*>(dst) = make_float2(s * (float)pw[jj][0], s * (float)pw[jj][1]);
      } else if constexpr (EB == 4) {
        const uint32_t m = smask << (31 - jj) & 0x80000000u;
        *reinterpret_cast<uint2*>(dst) = make_uint2(pw[jj][0] ^ m, pw[jj][1] ^ m);
      } else if constexpr (EB == 2 && EPW == 2) {
        const uint32_t m = (smask >> (2 * jj) & 1u) << 15 | (smask >> (2 * jj + 1) & 1u) << 31;
        uint32_t w[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) w[v] = pw[jj][v] ^ m;
        *reinterpret_cast<uint4*>(dst) = make_uint4(__byte_perm(w[0], w[1], 0x5410), __byte_perm(w[2], w[3], 0x5410),
                                                    __byte_perm(w[0], w[1], 0x7632), __byte_perm(w[2], w[3], 0x7632));
      } else if constexpr (EB == 2) {
        const uint32_t m = (smask >> jj & 1u) * 0x80008000u;
        *reinterpret_cast<uint32_t*>(dst) = (pw[jj][0] | pw[jj][1] << 16) ^ m;
      } else if constexpr (EPW == 4) {
        const uint32_t m = ((smask >> (4 * jj) & 15u) * 0x00204081u & 0x01010101u) << 7;
        uint32_t w[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) w[v] = pw[jj][v] ^ m;
        const uint32_t t0 = __byte_perm(w[0], w[1], 0x5140), t1 = __byte_perm(w[2], w[3], 0x5140);
        const uint32_t t2 = __byte_perm(w[0], w[1], 0x7362), t3 = __byte_perm(w[2], w[3], 0x7362);
        *reinterpret_cast<uint4*>(dst) = make_uint4(__byte_perm(t0, t1, 0x5410), __byte_perm(t0, t1, 0x7632),
                                                    __byte_perm(t2, t3, 0x5410), __byte_perm(t2, t3, 0x7632));
      } else {
        *reinterpret_cast<unsigned short*>(dst) =
            (unsigned short)((pw[jj][0] | pw[jj][1] << 8) ^ (smask >> jj & 1u) * 0x8080u);
      }
    }
  };
  int i0base = 0;  // i_0 of the chunk's first entry
  // q += the V values of the chunk's entry number x
  auto gather = [&](uint32_t x, float (&q)[V]) {
    const unsigned char* src = buf + x * ENT;
    if constexpr (EB == 2) {
      tt_fma_bf16x2(*reinterpret_cast<const uint32_t*>(src), 0x3F80, q[0], q[1]);
      if constexpr (V == 4) tt_fma_bf16x2(*reinterpret_cast<const uint32_t*>(src + 4), 0x3F80, q[2], q[3]);
    } else {
      const uint32_t y = x + i0base;
      const float s = ssc[y - __umulhi(y, a.inv_n0) * a.n0];
      if constexpr (V == 4) {
        float d[4] = {0.f, 0.f, 0.f, 0.f};
        tt_fma_e4m3x4(*reinterpret_cast<const uint32_t*>(src), 0x3C00, d[0], d[1], d[2], d[3]);
#pragma unroll
        for (int v = 0; v < 4; ++v) q[v] = fmaf(s, d[v], q[v]);
      } else {
        const uint32_t w = *reinterpret_cast<const unsigned short*>(src);
        q[0] = fmaf(s, tt_e4m3_to_float(w), q[0]);
        q[1] = fmaf(s, tt_e4m3_to_float(w >> 8), q[1]);
      }
    }
  };
  float acc[RPT][V];
#pragma unroll
  for (int j = 0; j < RPT; ++j)
#pragma unroll
    for (int v = 0; v < V; ++v) acc[j][v] = 0.f;
  auto flush = [&](int gl_, int at) {  // the group's columns of Y_l, into copy `at` mod cl
    if (part == 0) {
      float* yl = a.Yl + (int64_t)(at & (a.cl - 1)) * J * a.nl;
#pragma unroll
      for (int j = 0; j < RPT; ++j) {
        const int b = row0 + rstep * j;
        if (b < J) {
#pragma unroll
          for (int v = 0; v < V; ++v)
            if (V * gl_ + v < a.nl && acc[j][v] != 0.f) atomicAdd(yl + (int64_t)J * (V * gl_ + v) + b, acc[j][v]);
        }
      }
    }
#pragma unroll
    for (int j = 0; j < RPT; ++j)
#pragma unroll
      for (int v = 0; v < V; ++v) acc[j][v] = 0.f;
  };

  fetch(ch, gl, is);
  int ch_in = -1;
  for (int64_t u = u0; u < u1; ++u) {
    __syncthreads();  // the staged chunk and lists are no longer read
    if (ch != ch_in) {
      const uint2* gl2 = reinterpret_cast<const uint2*>(a.list) + (int64_t)ch * a.blocks;
      for (int i = t; i < a.blocks; i += T) sl[i] = __ldg(gl2 + i);
      for (int b = t; b < J; b += T) sb[b] = __ldg(a.bucket + (int64_t)ch * J + b);
      const uint32_t* sg = a.sign + (int64_t)ch * ((a.chunk + 31) / 32);
      smask = 0;
#pragma unroll
      for (int jj = 0; jj < JJ; ++jj) {
        const int i = (t + T * jj) * EPW;
        if (jj < nj) smask |= (__ldg(sg + (i >> 5)) >> (i & 31) & ((1u << EPW) - 1u)) << (EPW * jj);
      }
      if (DT == TT_FP8E4M3) i0base = (int)((int64_t)ch * a.chunk % a.n0);
      ch_in = ch;
    }
    stage();
    __syncthreads();
    int nis = is + 1, ngl = gl, nch = ch;
    if (nis == a.ns) {
      nis = 0;
      if (++ngl == a.ngl) ngl = 0, ++nch;
    }
    if (u + 1 < u1) fetch(nch, ngl, nis);  // in flight during the sums below
    int hs = 0;
    float vs = 1.f;
    int hl[V];
    float vl[V];
    float* ys = nullptr;
    const int nv = min(V, a.nl - V * gl);
    if (a.hs) {
      hs = __ldg(a.hs + is);
      vs = __ldg(a.vs + is) < 0 ? -1.f : 1.f;
      ys = a.Ys + (int64_t)J * (((ch * a.ngl + gl) & (a.cs - 1)) * a.ns + is);
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const int il = min(V * gl + v, a.nl - 1);
        hl[v] = __ldg(a.hl + il);
        vl[v] = __ldg(a.vl + il) < 0 ? -1.f : 1.f;
      }
    }
#pragma unroll
    for (int j = 0; j < RPT; ++j) {
      const int b = row0 + rstep * j;  // bucket of Y_l; the head's bucket c = b - h_s(i_s)
      if (RPT > 1 && rstep * j >= J) break;
      int c = b - hs;
      if (c < 0) c += J;
      const uint32_t se = b < J ? sb[c] : 0u;
      const int p0 = (int)(se & 0xFFFFu), pe = p0 + (int)(se >> 16);
      float q[V];
#pragma unroll
      for (int v = 0; v < V; ++v) q[v] = 0.f;
      if constexpr (EB >= 4) {
        const unsigned long long* src = reinterpret_cast<const unsigned long long*>(buf);
        unsigned long long qq = 0;
        for (int p = p0 + part; p < pe; p += parts) {
          const uint2 x = sl[p];
          unsigned long long lo = src[x.x & 0xFFFFu], hi = src[x.y & 0xFFFFu];  // a block in pairs
          add2(lo, src[x.x >> 16]);
          add2(hi, src[x.y >> 16]);
          add2(lo, hi);
          add2(qq, lo);
        }
        q[0] = __uint_as_float((uint32_t)qq), q[1] = __uint_as_float((uint32_t)(qq >> 32));
      } else {
        for (int p = p0 + part; p < pe; p += parts) {
          const uint2 x = sl[p];
          if constexpr (WILD) {
            for (uint32_t y : {x.x & 0xFFFFu, x.x >> 16, x.y & 0xFFFFu, x.y >> 16})
              if (y < (uint32_t)a.chunk) gather(y, q);
          } else if constexpr (RPT <= 2) {  // buckets of several blocks: each block on its own
            float qb[V] = {};
            gather(x.x & 0xFFFFu, qb);
            gather(x.x >> 16, qb);
            gather(x.y & 0xFFFFu, qb);
            gather(x.y >> 16, qb);
#pragma unroll
            for (int v = 0; v < V; ++v) q[v] += qb[v];
          } else {
            gather(x.x & 0xFFFFu, q);
            gather(x.x >> 16, q);
            gather(x.y & 0xFFFFu, q);
            gather(x.y >> 16, q);
          }
        }
      }
      if (parts > 1)
#pragma unroll
        for (int v = 0; v < V; ++v)
          for (int o = 1; o < parts; o <<= 1) q[v] += __shfl_xor_sync(0xffffffffu, q[v], o);
#pragma unroll
      for (int v = 0; v < V; ++v) acc[j][v] = fmaf(vs, q[v], acc[j][v]);
      if (a.hs && part == 0 && pe > p0) {
#pragma unroll
        for (int v = 0; v < V; ++v)
          if (v < nv) atomicAdd(ys + tt_modj(c + hl[v], J), vl[v] * q[v]);
      }
    }
    constexpr int RUN = tail_run(DT);
    if (ngl != gl || nch != ch || u + 1 == u1 || (is + 1) % RUN == 0) flush(gl, ch * ((a.ns + RUN - 1) / RUN) + is / RUN);
    is = nis, gl = ngl, ch = nch;
  }
}

// The copies of Y_s and of Y_l added up (and left zero for the next tail pass); bound by the L2 reads and
// stores of the copies.
struct TailOutArgs {
  float* src[2];
  float* dst[2];
  int64_t n[2];  // entries of a copy
  int copies[2];
};
__global__ void __launch_bounds__(256) k_tail_out(TailOutArgs a) {
  for (int z = 0; z < 2; ++z)
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < a.n[z]; i += (int64_t)gridDim.x * 256)
      a.dst[z][i] = take_copies(a.src[z] + i, a.n[z], a.copies[z]);
}

// CTAs of a pass with per_sm resident on an SM: one wave.
// - In a sweep it covers four fifths of the SMs: the passes' CTAs hold an SM's registers until they
//   end, and the chain's kernels (in a batch, also the other tensors') run on the rest. 100^4 FP32:
//   732 us per monitored sweep with a whole wave, 674, 639 and 640 us with 136, 120 and 104 tail CTAs,
//   626 with the head pass cut the same way. Batch of 4 tensors, the largest 66 M entries: 465 us
//   with a whole wave, 423 with four fifths.
// - In a batch also at most one CTA per 64 KB of A, so that small tensors' passes run side by side. 28
//   batches of 4 to 32 tensors, mean speed against one launch per mode: 1.10 with 512 KB, 1.28 (256),
//   1.32 (128), 1.33 (64 and 32); 256 tensors 1.24 from 256 KB down. Longer shares leave a tensor's
//   chain waiting for a few CTAs (6 tensors of 5.5 M entries in all: 705 us, 310 with 64 KB).
int64_t pass_ctas(const tt_ctx* c, int per_sm) {
  const int64_t sms = tt_sm_count();
  int64_t ctas = std::max<int64_t>(1, c->in_sweep ? sms * 4 / 5 : sms) * std::max(1, per_sm);
  if (c->item_bytes > 0) ctas = std::min(ctas, 16 * c->N * tt_elem_bytes(c->dtype) / c->item_bytes);
  return std::max<int64_t>(1, ctas);
}

// shared memory of k_tail_pass: a staged chunk and its zero entries, lists, buckets, row scales
size_t tail_smem(int64_t chunk, int64_t blocks, int64_t J, int64_t entry_bytes, int64_t nscales) {
  return ((size_t)((chunk + std::max<int64_t>(nscales, 1)) * entry_bytes + 15) & ~(size_t)15) + (size_t)(8 * blocks + 4 * J + 4 * nscales);
}

template <int DT, int V, int EPW>
int launch_tail_v(tt_ctx* c, TailArgs a) {
  using Sh = TailShape<DT, V, EPW>;
  a.ngl = (a.nl + V - 1) / V;
  a.units = (int64_t)a.nchunk * a.ngl * a.ns;
  a.parts = 1;
  while (a.parts < 8 && 2 * a.parts * a.J <= TAIL_T) a.parts *= 2;
  const size_t smem = tail_smem(a.chunk, a.blocks, a.J, Sh::ENT, DT == TT_FP8E4M3 ? a.n0 : 0);
  void (*kern)(TailArgs) = a.J <= 1024   ? k_tail_pass<DT, V, EPW, 1>
                           : a.J <= 2048 ? k_tail_pass<DT, V, EPW, 2>
                           : a.J <= 4096 ? k_tail_pass<DT, V, EPW, 4>
                                         : k_tail_pass<DT, V, EPW, 8>;
  TT_CUDA(c, tt_allow_smem(kern));
  const int blocks = (int)std::min<int64_t>(a.units, pass_ctas(c, 1));
  kern<<<blocks, TAIL_T, smem, c->stream>>>(a);
  TT_LAUNCH(c, "k_tail_pass");
  if constexpr (DT == TT_FP8E4M3) {  // (eight buckets per thread hold any J)
    TT_CUDA(c, tt_allow_smem(k_tail_pass<DT, V, EPW, 8, true>));
    k_tail_pass<DT, V, EPW, 8, true><<<blocks, TAIL_T, smem, c->stream>>>(a);
    TT_LAUNCH(c, "k_tail_pass");
  }
  return TT_OK;
}

template <int DT>
int launch_tail(tt_ctx* c, const TailArgs& a) {
  constexpr int EB = TtElem<DT>::bytes;
  if constexpr (EB >= 4) {
    return launch_tail_v<DT, 2, 1>(c, a);
  } else {
    // 32-bit loads where every slab starts on a 4-byte boundary
    if (reinterpret_cast<uintptr_t>(a.A) % 4 == 0 && a.E * EB % 4 == 0) return launch_tail_v<DT, 4, 4 / EB>(c, a);
    return launch_tail_v<DT, 2, 1>(c, a);
  }
}

int head_cols(const tt_ctx* c) {  // columns i_1 per chunk
  // at most what the threads hold, and 128 KB of transposition tile
  const int64_t cap = std::min<int64_t>(HEAD_TMAX * (c->dtype == TT_F64 ? head_acc<TT_F64>() : head_acc<TT_F32>()) / c->n[0],
                                        (128 * 1024 / 4) / ((c->n[0] + 31) & ~31));
  if (cap >= c->n[1]) return (int)c->n[1];
  const int64_t nch = (c->n[1] + (cap & ~3) - 1) / std::max<int64_t>(4, cap & ~3);
  return (int)(((c->n[1] + nch - 1) / nch + 3) & ~3);
}

struct HeadGeom {
  int G1, nch, threads;
  size_t smem;
  int per_sm;  // CTAs per SM, at most
};
HeadGeom head_geom(const tt_ctx* c) {
  HeadGeom g;
  g.G1 = head_cols(c);
  g.nch = (int)((c->n[1] + g.G1 - 1) / g.G1);
  const int per_warp = 32 * (c->dtype == TT_F64 ? head_acc<TT_F64>() : head_acc<TT_F32>());  // entries
  g.threads = (int)((c->n[0] * g.G1 + per_warp - 1) / per_warp) * 32;
  const size_t rows = (size_t)((g.G1 + 3) & ~3), pitch = (size_t)((c->n[0] + 31) & ~31);
  g.smem = sizeof(float) * (rows * pitch + 3 * (size_t)c->p0 + rows + 2 * HEAD_BATCH);
  g.per_sm = std::max(1, std::min({32, 2 * HEAD_TMAX / g.threads, (int)(228 * 1024 / (g.smem + 1024))}));
  return g;
}

template <int DT, int VB>
int launch_head_vb(tt_ctx* c, HeadArgs a) {
  const HeadGeom g = head_geom(c);
  auto kern = k_head_pass<DT, VB>;
  TT_CUDA(c, tt_allow_smem(kern));
  int per_sm = 1;
  TT_CUDA(c, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, g.threads, g.smem));
  a.nseg = (int)std::max<int64_t>(1, std::min<int64_t>(a.R, pass_ctas(c, std::min(per_sm, g.per_sm)) / a.nch));
  kern<<<a.nseg * a.nch, g.threads, g.smem, c->stream>>>(a);
  TT_LAUNCH(c, "k_head_pass");
  return TT_OK;
}

// the widest vectors that slabs and chunks start on (a column need not)
template <int DT>
int launch_head(tt_ctx* c, const HeadArgs& a) {
  constexpr int EB = TtElem<DT>::bytes;
  const uint64_t at = reinterpret_cast<uintptr_t>(a.A) | (uint64_t)a.n0 * a.n1 * EB | (a.nch > 1 ? (uint64_t)a.n0 * a.G1 * EB : 0);
  if (at % 16 == 0) return launch_head_vb<DT, 16>(c, a);
  if (at % 8 == 0) return launch_head_vb<DT, 8>(c, a);
  if constexpr (EB <= 4)
    if (at % 4 == 0) return launch_head_vb<DT, 4>(c, a);
  if constexpr (EB < 4) return launch_head_vb<DT, EB>(c, a);
  return tt_fail(c, TT_EINVAL, "A is not aligned to its storage type");
}

// entries per chunk: what a CTA's threads can fetch at once (JJ loads each). FP8 slabs on 4-byte
// boundaries come four entries to a load; the other narrow types keep to what entry loads reach too.
int64_t tail_chunk_max(const tt_ctx* c, int64_t E) {
  if (c->dtype == TT_F64) return TAIL_T * 5;
  return c->dtype == TT_FP8E4M3 && E % 4 == 0 ? TAIL_T * 20 : TAIL_T * 10;
}

// whether the tail pass can take this A: chunks sized for four entries to a load need its base on a
// 4-byte boundary
bool tail_takes(const tt_ctx* c, const void* A) {
  return c->pass_tail && (c->tail_chunk <= TAIL_T * 10 || reinterpret_cast<uintptr_t>(A) % 4 == 0);
}

}  // namespace

// Which modes the passes cover, from the shape alone. Workspaces of both sketch draws follow from it.
// The head pass needs slabs that fill a CTA's warps (512 entries) and columns that leave room for four
// in a chunk; its row accumulators stay in L2 (32 MB). The tail pass needs chunks of at least that
// size, and a slab that is not much sparser than the J buckets each unit adds to Y_s. With two tail modes
// every slab costs a unit of its own, so that many small slabs are slower than one launch per mode (4 x 10^6
// to 10^8 entries: 1.6 and 3 times its time below 1024 entries a slab, 0.12 to 2.3 below 2048, where fibres
// off the 16-byte grid make the launches slow, 0.7 above): those take no pass. Where the copies
// of a pass exceed 48 MB each mode takes half as many, and where those do, no pass: with fewer its
// sums would be off by more than those of one launch per mode. J up to 8192: eight buckets per thread.
// One row per slab column (n_0 = 1) goes one launch per mode: the passes divide entry numbers by n_0 with a
// multiplication by 2^32 / n_0, which has no 32-bit value then.
// The deterministic mode has its own kernels; the batch autotuner times launches per mode.
void tt_pass_plan(tt_ctx* c) {
  c->pass_head = c->pass_tail = false;
  c->tail_modes = 0;
  if (c->det || (c->flags & TT_FLAG_BATCH_AUTOTUNE) || c->J > 8192 || c->n[0] == 1) return;
  const int64_t e2 = c->n[0] * c->n[1];
  const bool fp8 = c->dtype == TT_FP8E4M3;
  c->p0 = (int)((c->n[0] + 3) & ~3);
  c->p1 = (int)((c->n[1] + 3) & ~3);
  c->pass_head = e2 >= 512 && c->n[0] <= HEAD_TMAX * head_acc<TT_F64>() / 4 && (int64_t)c->J * (c->p0 + c->p1) <= (8 << 20);
  if (c->pass_head) {
    const HeadGeom g = head_geom(c);
    const double R = (double)c->N / e2, segs = std::max(1.0, std::min(R, 152.0 * g.per_sm / g.nch));  // (152 SMs)
    const double runs = c->J * -std::expm1(-R / c->J) + segs;  // groups c that slabs have, and cut ones
    const double cap = segs * segs, adds0 = runs * c->n[1] / c->J, adds1 = (fp8 ? 1.9 : 1.0) * runs * c->n[0] / c->J;
    c->pass_head = false;
    for (double part = 1.0; part >= 0.5 && !c->pass_head; part /= 2) {
      c->head_c0 = fp8 ? 1 : copies_of(part * std::min(cap, adds0));
      c->head_c1 = copies_of(part * std::min(cap, adds1));
      c->pass_head = tt_head_copies(c) <= PASS_COPIES_MAX;
    }
  }
  const int nt = c->d >= 4 ? 2 : c->d == 3 ? 1 : 0;
  if (nt) {
    const int64_t E = c->stride[c->d - nt];
    // the longest chunk, halved until an SM's shared memory holds it (long FP8 rows bring a scale each)
    bool fits = false;
    for (int64_t cm = tail_chunk_max(c, E); !fits && cm >= 2048; cm /= 2) {
      c->tail_nchunk = (int)std::min<int64_t>((E + cm - 1) / cm, 65);
      c->tail_chunk = (int)((std::min(cm, (E + c->tail_nchunk - 1) / c->tail_nchunk) + 3) & ~3);
      // a bucket's blocks: all full but its last one
      c->tail_blocks = c->tail_chunk / 4 + std::min(c->J, c->tail_chunk);
      fits = tail_smem(c->tail_chunk, c->tail_blocks, c->J, fp8 ? 4 : 8, fp8 ? c->n[0] : 0) <= TT_SMEM_MAX;
    }
    const bool small = nt == 2 && c->N > 4000000 && (c->n[0] * tt_elem_bytes(c->dtype) % 16 ? E < 1024 : E < 2048);
    c->pass_tail = fits && E >= 512 && !small && E * 8 >= c->J && c->tail_nchunk <= 64;
    if (c->pass_tail) {
      const int run = tail_run(c->dtype);
      const double slabs = (double)c->tail_nchunk * c->n[c->d - 1];  // that a bucket of Y_s meets
      const double adds_s = (fp8 ? 3 : 1) * slabs * -std::expm1(-(double)c->tail_chunk / c->J);
      const double adds_l = (fp8 ? 4 : 1) * (double)c->tail_nchunk * (nt == 2 ? (c->n[c->d - 2] + run - 1) / run : 1);
      c->pass_tail = false;
      c->tail_modes = nt;
      for (double part = 1.0; part >= 0.5 && !c->pass_tail; part /= 2) {
        c->tail_cs = nt == 2 ? copies_of(part * adds_s) : 1;
        c->tail_cl = copies_of(part * adds_l);
        c->pass_tail = tt_tail_copies(c) <= PASS_COPIES_MAX;
      }
      if (!c->pass_tail) c->tail_modes = 0;
    }
  }
  c->head_sorted = c->pass_head && c->N / e2 <= HEAD_PLAN_MAX;
}

int64_t tt_head_copies(const tt_ctx* c) { return (int64_t)c->J * (c->head_c0 * c->p0 + c->head_c1 * c->p1); }

int64_t tt_tail_copies(const tt_ctx* c) {
  int64_t n = 0;
  if (c->tail_cs > 1) n += c->tail_cs * c->J * c->n[c->d - 2];
  if (c->tail_cl > 1) n += c->tail_cl * c->J * c->n[c->d - 1];
  return n;
}

unsigned tt_pass_mask(const tt_ctx* c, const void* A) {
  unsigned m = c->pass_head ? 3u : 0u;
  for (int s = 0; s < c->tail_modes && tail_takes(c, A); ++s) m |= 1u << (c->d - 1 - s);
  return m;
}

// modes whose fibre plan an all-modes data sketch reads: every mode without a pass, and mode 1 where
// the head pass takes its slabs from it
unsigned tt_pass_plans(const tt_ctx* c, const void* A) {
  return (((1u << c->d) - 1u) & ~tt_pass_mask(c, A)) | (c->pass_head && !c->head_sorted ? 2u : 0u);
}

int tt_launch_pass_plans(tt_ctx* c) {
  PassPlanArgs p{};
  p.h = c->d_h;
  p.v = c->d_v;
  p.d = c->d;
  p.nh = c->d - c->tail_modes;
  for (int s = 0; s < TT_MAX_D; ++s) {
    p.n[s] = s < c->d ? c->n[s] : 1;
    p.noff[s] = s < c->d ? c->noff[s] : 0;
  }
  p.J = c->J;
  p.chunk = c->tail_chunk;
  p.nchunk = c->pass_tail ? c->tail_nchunk : 0;
  p.blocks = c->tail_blocks;
  p.zeros = c->dtype == TT_FP8E4M3 ? (int)c->n[0] : 1;
  p.E = c->stride[p.nh];
  p.list = c->d_tlist;
  p.bucket = c->d_tbucket;
  p.sign = c->d_tbucket + (int64_t)c->J * c->tail_nchunk;
  p.R = c->head_sorted ? c->R[1] : 0;
  p.plan = c->d_hplan;
  p.key = c->d_rkey;
  const int ctas = p.nchunk + (c->head_sorted ? 1 : 0);
  if (ctas == 0) return TT_OK;
  // at most 4 J (J <= 8192) + 2 * 2^15 + 8 blocks (chunk / 4 + J): 202 KB
  p.nkeys = (int)((std::max<int64_t>(p.nchunk ? p.chunk : 0, p.R) + 3) & ~3);
  const size_t smem = sizeof(int) * (size_t)((c->J + 1) & ~1) +
                      sizeof(uint16_t) * (p.nkeys + std::max<size_t>(p.nchunk ? 4 * (size_t)p.blocks : 0, p.R));
  TT_CUDA(c, tt_allow_smem(k_pass_plans));
  k_pass_plans<<<ctas, 1024, smem, c->stream>>>(p);
  TT_LAUNCH(c, "k_pass_plans");
  return TT_OK;
}

int tt_launch_head_pass(tt_ctx* c, const void* A, const float* scales, float* const* Y) {
  HeadArgs a{};
  a.A = (const char*)A;
  a.scales = scales;
  a.plan = c->head_sorted ? c->d_hplan : c->d_rplan[1];
  a.key = c->d_rkey;
  a.h0 = c->d_h;
  a.v0 = c->d_v;
  a.h1 = c->d_h + c->noff[1];
  a.v1 = c->d_v + c->noff[1];
  a.R = c->R[1];
  a.J = c->J;
  a.n0 = (int)c->n[0];
  a.n1 = (int)c->n[1];
  a.p0 = c->p0;
  a.p1 = c->p1;
  a.Y0r = c->d_y01;
  a.Y1r = c->d_y01 + (int64_t)c->head_c0 * c->J * c->p0;
  a.c0 = c->head_c0;
  a.c1 = c->head_c1;
  const HeadGeom g = head_geom(c);
  a.G1 = g.G1;
  a.nch = g.nch;
  a.pitch = (a.n0 + 31) & ~31;
  a.inv_n0 = (uint32_t)((((uint64_t)1 << 32) + a.n0 - 1) / a.n0);
  for (int z = 0; z < c->tail_modes; ++z)
    if ((z == 0 ? c->tail_cl : c->tail_cs) == 1) {
      a.zero[z] = Y[c->d - 1 - z];
      a.nzero[z] = (int64_t)c->J * c->n[c->d - 1 - z];
    }
  if (!c->y01_zero) TT_CUDA(c, cudaMemsetAsync(c->d_y01, 0, sizeof(float) * (size_t)tt_head_copies(c), c->stream));
  c->y01_zero = false;
  switch (c->dtype) {
    case TT_F64: TT_TRY(launch_head<TT_F64>(c, a)); break;
    case TT_F32: TT_TRY(launch_head<TT_F32>(c, a)); break;
    case TT_BF16: TT_TRY(launch_head<TT_BF16>(c, a)); break;
    default: TT_TRY(launch_head<TT_FP8E4M3>(c, a)); break;
  }
  const HeadOutArgs o = {a.Y0r, a.Y1r, Y[0], Y[1], c->dtype == TT_FP8E4M3 ? scales : nullptr,
                         c->J,  a.n0,  a.n1, a.p0, a.p1, a.c0, a.c1, (a.n0 + 31) / 32};
  k_head_out<<<dim3((c->J + 31) / 32, o.tiles0 + (a.n1 + 31) / 32), 1024, 0, c->stream>>>(o);
  TT_LAUNCH(c, "k_head_out");
  c->y01_zero = true;
  return TT_OK;
}

int tt_launch_tail_pass(tt_ctx* c, const void* A, const float* scales, float* Ys, float* Yl) {
  const int l = c->d - 1, s = c->d - 2;
  TailArgs a{};
  a.A = (const char*)A;
  a.scales = scales;
  a.list = c->d_tlist;
  a.bucket = c->d_tbucket;
  a.sign = c->d_tbucket + (int64_t)c->J * c->tail_nchunk;
  a.blocks = c->tail_blocks;
  a.inv_n0 = (uint32_t)((((uint64_t)1 << 32) + c->n[0] - 1) / c->n[0]);
  a.hl = c->d_h + c->noff[l];
  a.vl = c->d_v + c->noff[l];
  a.cs = c->tail_cs;
  a.cl = c->tail_cl;
  if (c->tail_modes == 2) {
    a.hs = c->d_h + c->noff[s];
    a.vs = c->d_v + c->noff[s];
    a.Ys = a.cs > 1 ? c->d_ysl : Ys;
  }
  const int64_t ls = a.cs > 1 ? (int64_t)c->J * c->n[s] : 0, ll = (int64_t)c->J * c->n[l];  // a copy's entries
  a.Yl = a.cl > 1 ? c->d_ysl + a.cs * ls : Yl;
  for (int k = l; k > l - c->tail_modes && !c->pass_head; --k)  // (the head pass zeroes them)
    if ((k == l ? a.cl : a.cs) == 1)
      TT_CUDA(c, cudaMemsetAsync(k == l ? Yl : Ys, 0, sizeof(float) * (size_t)c->J * c->n[k], c->stream));
  const bool copies = a.cs > 1 || a.cl > 1;
  if (copies && !c->ysl_zero)
    TT_CUDA(c, cudaMemsetAsync(c->d_ysl, 0, sizeof(float) * (size_t)tt_tail_copies(c), c->stream));
  if (copies) c->ysl_zero = false;
  a.E = c->stride[c->d - c->tail_modes];
  a.J = c->J;
  a.n0 = (int)c->n[0];
  a.chunk = c->tail_chunk;
  a.nchunk = c->tail_nchunk;
  a.ns = c->tail_modes == 2 ? (int)c->n[s] : 1;
  a.nl = (int)c->n[l];
  switch (c->dtype) {
    case TT_F64: TT_TRY(launch_tail<TT_F64>(c, a)); break;
    case TT_F32: TT_TRY(launch_tail<TT_F32>(c, a)); break;
    case TT_BF16: TT_TRY(launch_tail<TT_BF16>(c, a)); break;
    default: TT_TRY(launch_tail<TT_FP8E4M3>(c, a)); break;
  }
  if (!copies) return TT_OK;
  TailOutArgs o{};
  if (a.cs > 1) o.src[0] = a.Ys, o.dst[0] = Ys, o.n[0] = ls, o.copies[0] = a.cs;
  if (a.cl > 1) o.src[1] = a.Yl, o.dst[1] = Yl, o.n[1] = ll, o.copies[1] = a.cl;
  k_tail_out<<<(int)std::min<int64_t>((std::max(o.n[0], o.n[1]) + 255) / 256, 8 * tt_sm_count()), 256, 0, c->stream>>>(o);
  TT_LAUNCH(c, "k_tail_out");
  c->ysl_zero = true;
  return TT_OK;
}

// The data sketches of all modes on c->stream: the passes, then one launch per remaining mode; ev[k]
// (when given) is recorded after Y_k.
int tt_launch_unfold_all(tt_ctx* c, const void* A, const float* scales, float* const* Y, cudaEvent_t* ev) {
  TT_TRY(tt_ensure_plans(c, tt_pass_plans(c, A), true));
  const unsigned mask = tt_pass_mask(c, A);
  auto mark = [&](int k) -> int {  // Y_k is done
    if (ev) TT_CUDA(c, cudaEventRecord(ev[k], c->stream));
    return TT_OK;
  };
  // a pass is timed as one read of A that its modes share
  auto timed = [&](int k0, int k1, auto&& pass) -> int {
    TT_TRY(tt_prof_begin(c, k0, k1));
    TT_TRY(pass());
    TT_TRY(tt_prof_end(c));
    for (int k = k0; k <= k1; ++k) TT_TRY(mark(k));
    return TT_OK;
  };
  if (c->pass_head) TT_TRY(timed(0, 1, [&] { return tt_launch_head_pass(c, A, scales, Y); }));
  for (int k = 0; k < c->d; ++k)
    if (!(mask & (1u << k))) {
      TT_TRY(tt_launch_unfold_planned(c, A, scales, k, Y[k]));
      TT_TRY(mark(k));
    }
  const int l = c->d - 1;
  if (tail_takes(c, A))
    TT_TRY(timed(c->d - c->tail_modes, l, [&] { return tt_launch_tail_pass(c, A, scales, Y[l - 1], Y[l]); }));
  return TT_OK;
}
