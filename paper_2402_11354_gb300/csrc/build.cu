// Index-time PEOs data (Sec. 4.2 steps (1)-(3)): per edge e = u - v the block
// norms, ||e||, w_reg, e_res and the L+1 extreme-value codes, and the edge's node
// term of the statistic (S(t(v)), from v's projection table); per node the
// projection table.  With a dimension permutation (Appendix D.1) both work on the
// permuted vectors: coordinate k of a row is read from coordinate perm[k].  Every sum
// is a plain sequential FP32 sum (compiled with --fmad=false), one thread per output,
// so the results are reproducible bit for bit.
//
// Three forms.  Up to 16 vectors per block (m <= 16, every configuration's m) the tiled
// kernels: a thread takes whole edges (or rows) and all 16 sums of each, so that a vector
// element read from shared memory serves several edges.  Where the blocks have 8..64
// coordinates, a multiple of 4, the edges take the screened form instead: estimates of the
// sums on the tensor cores settle most codes.  For larger m one CTA per node with a thread
// per sum (node_proj_kernel, build_codes_kernel).
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>

#include <string.h>

#include <algorithm>
#include <type_traits>
#include <vector>

#include "device.cuh"
#include "internal.h"

namespace peos {
namespace {

constexpr int kBuildThreads = 256;

__global__ void __launch_bounds__(kBuildThreads) build_codes_kernel(const float* __restrict__ X, long long n, int d,
                                                                    const int32_t* __restrict__ nbrs, int R, int L,
                                                                    int m, const float* __restrict__ A,
                                                                    const float* __restrict__ B,
                                                                    const int32_t* __restrict__ perm,
                                                                    const float* __restrict__ node_proj,
                                                                    int proj_stride, uint8_t* __restrict__ rec,
                                                                    size_t rec_stride, int bits, int cpw,
                                                                    int nwords) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int dp = d / L;
  float* e = reinterpret_cast<float*>(smem_raw);   // [R][d]  e, later e_res
  float* n2 = e + (size_t)R * d;                    // [R][L]  block norms squared
  float* bn = n2 + R * L;                           // [R][L]  block norms
  float* en = bn + R * L;                           // [R]
  float* wr = en + R;                               // [R]
  float* mean = wr + R;                             // [R]
  float* cr = mean + R;                             // [R]  sqrt(L) w_res
  float* proj = cr + R;                             // [R][L+1][m]
  int32_t* ids = reinterpret_cast<int32_t*>(proj + (size_t)R * (L + 1) * m);  // [R]
  int32_t* sel = ids + R;                                                      // [R][L+1] argmax j | sign << 16
  float* tvs = reinterpret_cast<float*>(sel + (size_t)R * (L + 1));           // [(L+1) m] t(v)
  const int tid = threadIdx.x;

  for (long long v = blockIdx.x; v < n; v += gridDim.x) {
    for (int s = tid; s < R; s += blockDim.x) ids[s] = nbrs[(size_t)v * R + s];
    for (int t = tid; t < (L + 1) * m; t += blockDim.x) tvs[t] = node_proj[(size_t)v * proj_stride + t];
    __syncthreads();
    for (int idx = tid; idx < R * d; idx += blockDim.x) {
      const int s = idx / d, k = idx - s * d;
      const int32_t u = ids[s];
      const int kk = perm ? __ldg(perm + k) : k;
      e[idx] = (u >= 0) ? (X[(size_t)u * d + kk] - X[(size_t)v * d + kk]) : 0.0f;
    }
    __syncthreads();
    // step (1): block norms
    for (int t = tid; t < R * L; t += blockDim.x) {
      const int s = t / L, i = t - s * L;
      const float* ei = e + (size_t)s * d + i * dp;
      float acc = 0.0f;
      for (int k = 0; k < dp; ++k) {
        const float x = ei[k];
        acc = acc + x * x;
      }
      n2[t] = acc;
      bn[t] = sqrtf(acc);
    }
    __syncthreads();
    for (int s = tid; s < R; s += blockDim.x) {
      float tot2 = 0.0f, sum = 0.0f;
      for (int i = 0; i < L; ++i) {
        tot2 = tot2 + n2[s * L + i];
        sum = sum + bn[s * L + i];
      }
      const float norm = sqrtf(tot2);
      en[s] = norm;
      if (norm == 0.0f) {
        wr[s] = 1.0f;
        cr[s] = 0.0f;
        mean[s] = 0.0f;
      } else {
        float w = sum / (sqrtf((float)L) * norm);
        if (w > 1.0f) w = 1.0f;
        wr[s] = w;
        cr[s] = sqrtf((float)L) * sqrtf(fmaxf(0.0f, 1.0f - w * w));
        mean[s] = sum / (float)L;
      }
    }
    __syncthreads();
    // step (3), i = 1..L: projections of e_i onto the a^i_j
    for (int t = tid; t < R * L * m; t += blockDim.x) {
      const int s = t / (L * m);
      const int rem = t - s * L * m;
      const int i = rem / m, j = rem - i * m;
      const float* a = A + ((size_t)i * m + j) * dp;
      const float* ei = e + (size_t)s * d + i * dp;
      float acc = 0.0f;
      for (int k = 0; k < dp; ++k) acc = acc + __ldg(a + k) * ei[k];
      proj[((size_t)s * (L + 1) + i + 1) * m + j] = acc;
    }
    __syncthreads();
    // step (1): e_res = e - e_reg, block i scaled by 1 - mean(||e_k||) / ||e_i||
    for (int idx = tid; idx < R * d; idx += blockDim.x) {
      const int s = idx / d, k = idx - s * d;
      const int i = k / dp;
      const float b = bn[s * L + i];
      const float coef = (b > 0.0f) ? (1.0f - mean[s] / b) : 0.0f;
      e[idx] = e[idx] * coef;
    }
    __syncthreads();
    // step (3), e[0]: projections of e_res onto the b_j
    for (int t = tid; t < R * m; t += blockDim.x) {
      const int s = t / m, j = t - s * m;
      const float* b = B + (size_t)j * d;
      const float* er = e + (size_t)s * d;
      float acc = 0.0f;
      for (int k = 0; k < d; ++k) acc = acc + __ldg(b + k) * er[k];
      proj[((size_t)s * (L + 1)) * m + j] = acc;
    }
    __syncthreads();
    // argmax_j |.|, lowest j on ties, sgn(0) = +1 (a degenerate edge, ||e|| = 0, gets +1)
    for (int t = tid; t < R * (L + 1); t += blockDim.x) {
      const int s = t / (L + 1);
      const float* p = proj + (size_t)t * m;
      int best = 0;
      float bv = fabsf(p[0]);
      for (int j = 1; j < m; ++j) {
        const float av = fabsf(p[j]);
        if (av > bv) {
          bv = av;
          best = j;
        }
      }
      const int neg = (en[s] != 0.0f && !(p[best] >= 0.0f)) ? 1 : 0;
      sel[t] = (en[s] == 0.0f ? 0 : best) | (neg << 16);
    }
    __syncthreads();
    // packed per edge (see code_bits)
    uint8_t* r = rec + (size_t)v * rec_stride;
    uint64_t* cwords = reinterpret_cast<uint64_t*>(r + rec_codes_offset(R));
    for (int t = tid; t < R * nwords; t += blockDim.x) {
      const int s = t / nwords, w = t - s * nwords;
      uint64_t word = 0;
      if (ids[s] >= 0) {
        for (int k = 0; k < cpw; ++k) {
          const int c = w * cpw + k;
          if (c > L) break;
          const int q = sel[s * (L + 1) + c];
          const uint64_t code = (uint64_t)(q & 0xffff) | ((uint64_t)(q >> 16) << (bits - 1));
          word |= code << (k * bits);
        }
      }
      cwords[(size_t)w * R + s] = word;
    }
    // node term S(t(v)) = w_reg sum_{c=1..L} sgn t(v)[c][j_c] + sqrt(L) w_res sgn t(v)[0][j_0]
    for (int s = tid; s < R; s += blockDim.x) {
      const bool ok = ids[s] >= 0;
      float svv = 0.0f;
      if (ok) {
        float h1 = 0.0f;
        for (int c = 1; c <= L; ++c) {
          const int q = sel[s * (L + 1) + c];
          const float val = tvs[c * m + (q & 0xffff)];
          h1 = h1 + ((q >> 16) ? -val : val);
        }
        const int q0 = sel[s * (L + 1)];
        const float v0 = tvs[q0 & 0xffff];
        const float h2 = (q0 >> 16) ? -v0 : v0;
        svv = wr[s] * h1 + cr[s] * h2;
      }
      reinterpret_cast<float4*>(r)[s] = ok ? make_float4(en[s], wr[s], cr[s], svv) : make_float4(0.f, 0.f, 0.f, 0.f);
      reinterpret_cast<int32_t*>(r + rec_ids_offset(R))[s] = ids[s];
    }
    // zero the gap before the codes and the padding after them
    for (size_t b = rec_ids_offset(R) + 4 * (size_t)R + tid; b < rec_codes_offset(R); b += blockDim.x) r[b] = 0;
    const size_t used = rec_codes_offset(R) + 8 * (size_t)nwords * R;
    for (size_t b = used + tid; b < rec_stride; b += blockDim.x) r[b] = 0;
    __syncthreads();
  }
}

// projection table of every node: out[v][c][j], one thread per entry
__global__ void node_proj_kernel(const float* __restrict__ X, long long n, int d, int L, int m,
                                 const float* __restrict__ A, const float* __restrict__ B,
                                 const int32_t* __restrict__ perm, float* __restrict__ out, int out_stride) {
  const int tw = out_stride;  // (L+1)*m entries, then zero padding
  const int dp = d / L;
  const long long total = n * (long long)tw;
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const long long v = t / tw;
    const int e = (int)(t - v * tw);
    const int c = e / m, j = e - c * m;
    const float* x = X + (size_t)v * d;
    float acc = 0.0f;
    if (c > L) {
      // padding entry
    } else if (c == 0) {
      // block by block: a sequential partial sum per block of d/L dims, then the partials
      const float* b = B + (size_t)j * d;
      for (int i = 0; i < L; ++i) {
        float part = 0.0f;
        for (int k = 0; k < dp; ++k) {
          const int t = i * dp + k;
          part = part + __ldg(b + t) * __ldg(x + (perm ? __ldg(perm + t) : t));
        }
        acc = acc + part;
      }
    } else {
      const int i = c - 1;
      const float* a = A + ((size_t)i * m + j) * dp;
      for (int k = 0; k < dp; ++k) {
        const int t = i * dp + k;
        acc = acc + __ldg(a + k) * __ldg(x + (perm ? __ldg(perm + t) : t));
      }
    }
    out[t] = acc;
  }
}

// ||v||^2 of every row, a plain sequential FP32 sum per row (one thread per row)
__global__ void row_norms_kernel(const float* __restrict__ X, long long n, int d, float* __restrict__ norms) {
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (long long)gridDim.x * blockDim.x) {
    const float* x = X + (size_t)v * d;
    float acc = 0.0f;
    for (int k = 0; k < d; ++k) acc = acc + __ldg(x + k) * __ldg(x + k);
    norms[v] = acc;
  }
}

// ---- the tiled form, m <= 16 -------------------------------------------------------
//
// What bounds it: 2 d m multiplies and as many separate adds per edge (the order of the
// sums is fixed, so no FMA), 4,096 pairs at d = 128: 3.0 ms of the FP32 pipes for the 13.6M
// edges of a 1M-node graph (R = 32, 1M x 128).  One thread per dot product (the form for
// m > 16) reads two operands per multiply and add and computes the empty slots too: 257 ms
// there.  Here a lane owns two edges and keeps the 16 sums of each in registers: per
// coordinate the warp reads 64 bytes of vectors (one broadcast) and one coordinate of each
// edge.  A warp walks its nodes' slots, keeps the valid edges in a queue and works on full
// tiles of 64, so empty slots cost nothing (13.6 of 32 slots are edges).  Measured in this
// form: index build of 1M x 128 269 -> 10.6 ms, of 50,000 x 960 (L = 24) 106 -> 5.7 ms (the
// screened form below takes both further).  Issue slots are
// then 57% busy and the rest waits on the rows' gathers: 16 warps 10.4 ms, 20 warps 9.4, 24
// warps 9.3 (and slower at d = 960); four edges per lane 12.5, coordinates of the next chunk
// kept in registers 10.8 (one build alone, before its index is freed).
constexpr int kTileWarps = 20;     // one CTA per SM
constexpr int kEdgesPerLane = 2;
constexpr int kEdgeTile = 32 * kEdgesPerLane;
constexpr int kRowsPerLane = 2;    // node tables: rows per lane, one where two leave warps without rows
constexpr int kTileDims = 16;      // coordinates staged at a time
// row pitch of the staged tile in 16-byte units: odd, so that lanes reading 16 bytes of 32
// consecutive rows meet no bank conflict
constexpr int kTilePitch = kTileDims / 4 + 1;
constexpr int kNodeChunk = 8;      // nodes a warp takes from the work counter at a time
constexpr int kVecs = 16;          // vectors per block after zero padding
// the vectors (2 d x 16 floats) sit in shared memory up to this d, else they are read
// through L1 (every lane reads the same address)
constexpr int kMaxSmemVecDim = 256;

// acc[j] += w[j] * x for the 16 vectors' element at one coordinate, two roundings each (the
// packed multiply and add would be fused into one rounding, and measured no faster)
__device__ __forceinline__ void mac16(float (&acc)[kVecs], const float4 (&w)[kVecs / 4], float x) {
#pragma unroll
  for (int q = 0; q < kVecs / 4; ++q) {
    acc[4 * q] = __fadd_rn(acc[4 * q], __fmul_rn(w[q].x, x));
    acc[4 * q + 1] = __fadd_rn(acc[4 * q + 1], __fmul_rn(w[q].y, x));
    acc[4 * q + 2] = __fadd_rn(acc[4 * q + 2], __fmul_rn(w[q].z, x));
    acc[4 * q + 3] = __fadd_rn(acc[4 * q + 3], __fmul_rn(w[q].w, x));
  }
}

// argmax_j |p_j|, lowest j on ties, as best | (sign << 16), sgn(0) = +1; the zero padding
// past m never exceeds a kept value
__device__ __forceinline__ int argmax16(const float (&p)[kVecs]) {
  int best = 0;
  float bv = fabsf(p[0]), pv = p[0];
#pragma unroll
  for (int j = 1; j < kVecs; ++j) {
    const float ax = fabsf(p[j]);
    if (ax > bv) {
      bv = ax;
      pv = p[j];
      best = j;
    }
  }
  return best | ((pv >= 0.0f) ? 0 : 1 << 16);
}

struct TileArgs {
  const float* X;
  long long n;
  int d;
  int L, m;
  const float* W;       // 2 d rows of 16 floats: the b_j, then the a^i_j, k-major
  const int32_t* perm;  // or null
  float* node_proj;     // node tables: written by the row kernel, read by the edge kernel
  int proj_stride;
  // rows
  float* norms;         // ||v||^2, or null (permuted coordinates: another order of the sum)
  // edges
  const int32_t* nbrs;
  int R;
  uint8_t* rec;
  size_t rec_stride;
  int bits, cpw, nwords;
  // edges, screened form
  const uint4* frag;    // the vectors as MMA fragments: [L][ksteps][4][32] {hi, hi, lo, lo}
  const float* amax;    // [L + 1] largest ||a^i_j|| of block i over j; last: largest ||b_j||_i over j, i
  int ksteps;           // steps of 16 coordinates per block
  float2* blocks;       // per warp: {squared block norm, code} of the tile's edges, [L][kEdgeTile]
  int* work;
};

// The vectors of the CTA in shared memory (or their global copy).
template <bool WSMEM>
__device__ __forceinline__ const float4* tile_vectors(const TileArgs& a, float4* s_w) {
  const float4* g = reinterpret_cast<const float4*>(a.W);
  if (!WSMEM) return g;
  for (int i = threadIdx.x; i < 2 * a.d * (kVecs / 4); i += blockDim.x) s_w[i] = __ldg(g + i);
  __syncthreads();
  return s_w;
}

template <bool WSMEM>
__device__ __forceinline__ void load_vec(const float4* w, int k, float4 (&out)[kVecs / 4]) {
#pragma unroll
  for (int q = 0; q < kVecs / 4; ++q) out[q] = WSMEM ? w[(size_t)k * (kVecs / 4) + q] : __ldg(w + (size_t)k * (kVecs / 4) + q);
}

// four coordinates of a row from c0 (a multiple of 4), through the permutation if there is one
template <bool PERM>
__device__ __forceinline__ float4 row4(const float* X, long long row, int d, int c0, const int32_t* perm) {
  const float* x = X + (size_t)row * d;
  if (!PERM) return __ldg(reinterpret_cast<const float4*>(x + c0));
  return make_float4(__ldg(x + __ldg(perm + c0)), __ldg(x + __ldg(perm + c0 + 1)), __ldg(x + __ldg(perm + c0 + 2)),
                     __ldg(x + __ldg(perm + c0 + 3)));
}

// One pass over the coordinates of a staged chunk: KU (4, 2 or 1, a divisor of the block
// length) coordinates of each of the lane's E rows at a time; `flush` runs at block ends.
template <int E, int KU, bool WSMEM, class X, class Flush>
__device__ __forceinline__ void tile_walk(const float4* s_e, const float4* w, int cw, int dp, int& kk, int lane,
                                          float (&acc)[E][kVecs], X&& element, Flush&& flush) {
  const float* rows = reinterpret_cast<const float*>(s_e);
#pragma unroll 1
  for (int k = 0; k < cw; k += KU) {
    float x[E][KU];
#pragma unroll
    for (int r = 0; r < E; ++r) {
      const float* p = rows + (size_t)(r * 32 + lane) * (kTilePitch * 4) + k;
      if constexpr (KU == 4) {
        const float4 v = *reinterpret_cast<const float4*>(p);
        x[r][0] = v.x;
        x[r][1] = v.y;
        x[r][2] = v.z;
        x[r][3] = v.w;
      } else if constexpr (KU == 2) {
        const float2 v = *reinterpret_cast<const float2*>(p);
        x[r][0] = v.x;
        x[r][1] = v.y;
      } else {
        x[r][0] = *p;
      }
    }
#pragma unroll
    for (int q = 0; q < KU; ++q) {
      float4 wv[kVecs / 4];
      load_vec<WSMEM>(w, k + q, wv);
#pragma unroll
      for (int r = 0; r < E; ++r) mac16(acc[r], wv, element(r, x[r][q]));
    }
    kk += KU;
    if (kk == dp) {
      flush();
      kk = 0;
    }
  }
}

template <int E>
__device__ __forceinline__ void clear(float (&acc)[E][kVecs]) {
#pragma unroll
  for (int r = 0; r < E; ++r)
#pragma unroll
    for (int j = 0; j < kVecs; ++j) acc[r][j] = 0.0f;
}

// Projection table of every row, out[v][c][j], and ||v||^2: a warp takes 32 ROWS rows, ROWS per
// lane; first the a^i (one sum per block), then the b_j (block by block: a partial sum per
// block of d/L dims, then the partials).
template <int ROWS, int KU, bool PERM, bool WSMEM>
__global__ void __launch_bounds__(kTileWarps * 32, 1) node_rows_kernel(TileArgs a) {
  constexpr int kRowTile = 32 * ROWS;
  const int warps = blockDim.x >> 5;  // kTileWarps, fewer where the rows make less than that per SM
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float4* s_w = reinterpret_cast<float4*>(smem_raw);
  const float4* w = tile_vectors<WSMEM>(a, s_w);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float4* s_e = s_w + (WSMEM ? 2 * a.d * (kVecs / 4) : 0) + (size_t)warp * kRowTile * kTilePitch;
  const int d = a.d, L = a.L, m = a.m, dp = d / L;
  const long long tiles = (a.n + kRowTile - 1) / kRowTile;
  for (long long t = (long long)blockIdx.x * warps + warp; t < tiles; t += (long long)gridDim.x * warps) {
    const long long v0 = t * kRowTile;
    auto stage = [&](int c0, int c4) {
      __syncwarp();
#pragma unroll 4
      for (int i = lane; i < kRowTile * (kTileDims / 4); i += 32) {
        const int row = i / (kTileDims / 4), col = i % (kTileDims / 4);
        if (col < c4 && v0 + row < a.n) s_e[row * kTilePitch + col] = row4<PERM>(a.X, v0 + row, d, c0 + 4 * col, a.perm);
      }
      __syncwarp();
    };
    auto store = [&](int r, int c, const float (&p)[kVecs]) {
      const long long v = v0 + r * 32 + lane;
      if (v >= a.n) return;
      float* o = a.node_proj + (size_t)v * a.proj_stride + c * m;
      if (m == kVecs) {
#pragma unroll
        for (int q = 0; q < kVecs / 4; ++q)
          reinterpret_cast<float4*>(o)[q] = make_float4(p[4 * q], p[4 * q + 1], p[4 * q + 2], p[4 * q + 3]);
      } else {
#pragma unroll
        for (int j = 0; j < kVecs; ++j)
          if (j < m) o[j] = p[j];
      }
    };
    float acc[ROWS][kVecs];
    float nrm[ROWS];
#pragma unroll
    for (int r = 0; r < ROWS; ++r) nrm[r] = 0.0f;
    clear(acc);
    int kk = 0, c = 1;
    for (int c0 = 0; c0 < d; c0 += kTileDims) {
      const int cw = min(kTileDims, d - c0);
      stage(c0, cw >> 2);
      tile_walk<ROWS, KU, WSMEM>(
          s_e, w + (size_t)(d + c0) * (kVecs / 4), cw, dp, kk, lane, acc,
          [&](int r, float x) {
            nrm[r] = nrm[r] + x * x;
            return x;
          },
          [&] {
#pragma unroll
            for (int r = 0; r < ROWS; ++r) store(r, c, acc[r]);
            clear(acc);
            ++c;
          });
    }
    if (a.norms) {
#pragma unroll
      for (int r = 0; r < ROWS; ++r)
        if (v0 + r * 32 + lane < a.n) a.norms[v0 + r * 32 + lane] = nrm[r];
    }
    float tot[ROWS][kVecs];
    clear(tot);
    for (int c0 = 0; c0 < d; c0 += kTileDims) {
      const int cw = min(kTileDims, d - c0);
      stage(c0, cw >> 2);
      tile_walk<ROWS, KU, WSMEM>(
          s_e, w + (size_t)c0 * (kVecs / 4), cw, dp, kk, lane, acc, [&](int, float x) { return x; },
          [&] {
#pragma unroll
            for (int r = 0; r < ROWS; ++r)
#pragma unroll
              for (int j = 0; j < kVecs; ++j) tot[r][j] = tot[r][j] + acc[r][j];
            clear(acc);
          });
    }
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
      store(r, 0, tot[r]);
      const long long v = v0 + r * 32 + lane;
      if (v < a.n)
        for (int e = (L + 1) * m; e < a.proj_stride; ++e) a.node_proj[(size_t)v * a.proj_stride + e] = 0.0f;
    }
  }
}

// A warp's queue of valid edges, filled in slot order from the nodes it takes: the slots'
// ids go to the records and empty slots are zeroed on the way.
template <int TILE>
struct EdgeQueue {
  static constexpr int kSlots = TILE + 32;
  int32_t *u, *v, *s;     // [kSlots] in shared memory: neighbour, node, slot
  long long v0 = 0;       // the chunk's first node
  int slots = 0, at = 0;  // its slots, and how many are queued or written
  int queued = 0;
  bool more = true;

  __device__ __forceinline__ explicit EdgeQueue(int32_t* mem) : u(mem), v(mem + kSlots), s(mem + 2 * kSlots) {}

  // at least TILE edges, or all that are left; the tile's edges (warp-wide)
  __device__ __forceinline__ int fill(const TileArgs& a, int lane) {
    const int R = a.R;
    const size_t ids_end = rec_ids_offset(R) + 4 * (size_t)R, codes_at = rec_codes_offset(R);
    const size_t used = codes_at + 8 * (size_t)a.nwords * R;
    const int gap4 = (int)(codes_at - ids_end) / 4, pad4 = (int)(a.rec_stride - used) / 4;
    while (queued < TILE && more) {
      if (at >= slots) {
        int c = 0;
        if (lane == 0) c = atomicAdd(a.work, 1);
        v0 = (long long)__shfl_sync(kFull, c, 0) * kNodeChunk;
        if (v0 >= a.n) {
          more = false;
          break;
        }
        const int nn = (int)min((long long)kNodeChunk, a.n - v0);
        slots = nn * R;
        at = 0;
        for (int t = lane; t < nn * (gap4 + pad4); t += 32) {
          const int w = t / (gap4 + pad4), b = t - w * (gap4 + pad4);
          uint8_t* r = a.rec + (size_t)(v0 + w) * a.rec_stride;
          *reinterpret_cast<uint32_t*>(b < gap4 ? r + ids_end + 4 * b : r + used + 4 * (b - gap4)) = 0u;
        }
      }
      const int t = at + lane;
      int32_t id = -1;
      int slot = 0;
      long long node = v0;
      if (t < slots) {
        id = __ldg(a.nbrs + (size_t)v0 * R + t);
        const int lv = t / R;
        node = v0 + lv;
        slot = t - lv * R;
        uint8_t* r = a.rec + (size_t)node * a.rec_stride;
        reinterpret_cast<int32_t*>(r + rec_ids_offset(R))[slot] = id;
        if (id < 0) {
          reinterpret_cast<float4*>(r)[slot] = make_float4(0.f, 0.f, 0.f, 0.f);
          for (int k = 0; k < a.nwords; ++k) reinterpret_cast<uint64_t*>(r + codes_at)[(size_t)k * R + slot] = 0;
        }
      }
      const unsigned have = __ballot_sync(kFull, id >= 0);
      if (id >= 0) {
        const int p = queued + __popc(have & ((1u << lane) - 1u));
        u[p] = id;
        v[p] = (int32_t)node;
        s[p] = slot;
      }
      queued += __popc(have);
      at += 32;
    }
    __syncwarp();
    return min(queued, TILE);
  }

  // the tile is done: the rest moves to the front
  __device__ __forceinline__ void drop(int cnt, int lane) {
    const int rest = queued - cnt;
    int32_t ru = 0, rv = 0, rs = 0;
    __syncwarp();
    if (lane < rest) {
      ru = u[cnt + lane];
      rv = v[cnt + lane];
      rs = s[cnt + lane];
    }
    __syncwarp();
    if (lane < rest) {
      u[lane] = ru;
      v[lane] = rv;
      s[lane] = rs;
    }
    queued = rest;
  }
};

// Edge records.  Per tile of 64 edges two passes over the coordinates: the a^i sums and
// the block norms (their codes and squared norms go to `blocks`), then, the block norms'
// mean being known, the b_j sums of e_res.
template <int KU, bool PERM, bool WSMEM>
__global__ void __launch_bounds__(kTileWarps * 32, 1) build_edges_kernel(TileArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float4* s_w = reinterpret_cast<float4*>(smem_raw);
  const float4* w = tile_vectors<WSMEM>(a, s_w);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  using Queue = EdgeQueue<kEdgeTile>;
  constexpr size_t kWarpBytes = (size_t)kEdgeTile * kTilePitch * 16 + (size_t)Queue::kSlots * 12;
  unsigned char* base =
      reinterpret_cast<unsigned char*>(s_w + (WSMEM ? 2 * a.d * (kVecs / 4) : 0)) + (size_t)warp * kWarpBytes;
  float4* s_e = reinterpret_cast<float4*>(base);
  Queue queue(reinterpret_cast<int32_t*>(base + (size_t)kEdgeTile * kTilePitch * 16));
  const int32_t *q_u = queue.u, *q_v = queue.v, *q_s = queue.s;
  const int d = a.d, L = a.L, m = a.m, dp = d / L, R = a.R;
  float2* blk = a.blocks + ((size_t)blockIdx.x * kTileWarps + warp) * L * kEdgeTile;
  const size_t codes_at = rec_codes_offset(R);

  for (;;) {
    const int cnt = queue.fill(a, lane);
    if (cnt == 0) break;

    auto stage = [&](int c0) {
      const int c4 = min(kTileDims, d - c0) >> 2;
      __syncwarp();
#pragma unroll 4
      for (int i = lane; i < kEdgeTile * (kTileDims / 4); i += 32) {
        const int e = i / (kTileDims / 4), col = i % (kTileDims / 4);
        if (col < c4 && e < cnt) {
          const float4 x = row4<PERM>(a.X, q_u[e], d, c0 + 4 * col, a.perm);
          const float4 y = row4<PERM>(a.X, q_v[e], d, c0 + 4 * col, a.perm);
          s_e[e * kTilePitch + col] = make_float4(x.x - y.x, x.y - y.y, x.z - y.z, x.w - y.w);
        }
      }
      __syncwarp();
    };

    // ---- pass 1: block norms and the codes e[1..L]
    float acc[kEdgesPerLane][kVecs];
    clear(acc);
    int kk = 0, c = 0;
    {
      float n2[kEdgesPerLane];
#pragma unroll
      for (int r = 0; r < kEdgesPerLane; ++r) n2[r] = 0.0f;
      for (int c0 = 0; c0 < d; c0 += kTileDims) {
        const int cw = min(kTileDims, d - c0);
        stage(c0);
        tile_walk<kEdgesPerLane, KU, WSMEM>(
            s_e, w + (size_t)(d + c0) * (kVecs / 4), cw, dp, kk, lane, acc,
            [&](int r, float x) {
              n2[r] = n2[r] + x * x;
              return x;
            },
            [&] {
#pragma unroll
              for (int r = 0; r < kEdgesPerLane; ++r) {
                blk[(size_t)c * kEdgeTile + r * 32 + lane] = make_float2(n2[r], __int_as_float(argmax16(acc[r])));
                n2[r] = 0.0f;
              }
              clear(acc);
              ++c;
            });
      }
    }
    // ---- ||e||, the weights, the packed codes and the regular part of the node term
    float mean[kEdgesPerLane];
#pragma unroll
    for (int r = 0; r < kEdgesPerLane; ++r) {
      const int e = r * 32 + lane;
      mean[r] = 0.0f;
      if (e >= cnt) continue;
      float tot2 = 0.0f, sum = 0.0f;
#pragma unroll 4
      for (int i = 0; i < L; ++i) {
        const float b2 = blk[(size_t)i * kEdgeTile + e].x;
        tot2 = tot2 + b2;
        sum = sum + sqrtf(b2);
      }
      const float norm = sqrtf(tot2);
      float wr = 1.0f, cr = 0.0f;
      if (norm != 0.0f) {
        wr = sum / (sqrtf((float)L) * norm);
        if (wr > 1.0f) wr = 1.0f;
        cr = sqrtf((float)L) * sqrtf(fmaxf(0.0f, 1.0f - wr * wr));
        mean[r] = sum / (float)L;
      }
      uint8_t* rec = a.rec + (size_t)q_v[e] * a.rec_stride;
      uint64_t* cwords = reinterpret_cast<uint64_t*>(rec + codes_at) + q_s[e];
      const float* tv = a.node_proj + (size_t)q_v[e] * a.proj_stride;
      float h1 = 0.0f;
      uint64_t word = 0;
      int k = 1, wi = 0;
      for (int i0 = 0; i0 < L; i0 += 4) {
        int sel[4];
        float val[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          // a degenerate edge gets code +1 everywhere
          sel[q] = (i0 + q < L && norm != 0.0f) ? __float_as_int(blk[(size_t)(i0 + q) * kEdgeTile + e].y) : 0;
          val[q] = i0 + q < L ? __ldg(tv + (i0 + q + 1) * m + (sel[q] & 0xffff)) : 0.0f;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (i0 + q >= L) break;
          h1 = h1 + ((sel[q] >> 16) ? -val[q] : val[q]);
          word |= ((uint64_t)(sel[q] & 0xffff) | ((uint64_t)(sel[q] >> 16) << (a.bits - 1))) << (k * a.bits);
          if (++k == a.cpw) {
            cwords[(size_t)wi * R] = word;
            word = 0;
            k = 0;
            ++wi;
          }
        }
      }
      if (k > 0) cwords[(size_t)wi * R] = word;
      reinterpret_cast<float4*>(rec)[q_s[e]] = make_float4(norm, wr, cr, h1);  // h1 becomes the node term below
    }
    // ---- pass 2: e_res = e - e_reg (block i scaled by 1 - mean(||e_k||) / ||e_i||) and e[0]
    {
      float coef[kEdgesPerLane];
      auto scale = [&](int i) {
#pragma unroll
        for (int r = 0; r < kEdgesPerLane; ++r) {
          const float b = sqrtf(blk[(size_t)i * kEdgeTile + r * 32 + lane].x);
          coef[r] = (b > 0.0f) ? (1.0f - mean[r] / b) : 0.0f;
        }
      };
      scale(0);
      c = 0;
      for (int c0 = 0; c0 < d; c0 += kTileDims) {
        const int cw = min(kTileDims, d - c0);
        stage(c0);
        tile_walk<kEdgesPerLane, KU, WSMEM>(
            s_e, w + (size_t)c0 * (kVecs / 4), cw, dp, kk, lane, acc, [&](int r, float x) { return x * coef[r]; },
            [&] {
              if (++c < L) scale(c);
            });
      }
    }
#pragma unroll
    for (int r = 0; r < kEdgesPerLane; ++r) {
      const int e = r * 32 + lane;
      if (e < cnt) {
        uint8_t* rec = a.rec + (size_t)q_v[e] * a.rec_stride;
        float4* sc = reinterpret_cast<float4*>(rec) + q_s[e];
        uint64_t* cwords = reinterpret_cast<uint64_t*>(rec + codes_at) + q_s[e];
        float4 f = *sc;
        const int sel = f.x == 0.0f ? 0 : argmax16(acc[r]);
        const float v0f = __ldg(a.node_proj + (size_t)q_v[e] * a.proj_stride + (sel & 0xffff));
        const float h2 = (sel >> 16) ? -v0f : v0f;
        f.w = f.y * f.w + f.z * h2;
        *sc = f;
        *cwords = *cwords | (uint64_t)(sel & 0xffff) | ((uint64_t)(sel >> 16) << (a.bits - 1));
      }
    }
    queue.drop(cnt, lane);
  }
}

// ---- the screened form: blocks of 8..64 coordinates, a multiple of 4 -----------------
//
// A code is an argmax over 16 sums, and only that: sums good to five digits settle nearly all
// (left: 0.13% of the block codes and 0.5% of the e[0] of 1M x 128, 0.22% and 2.6% of 50,000 x 960).  A warp takes 32 edges and forms, on the tensor cores, every e_i . a^i_j
// and e_i . b_j (two BF16 terms of each factor, three products, mma.sync on fragments built
// straight from the staged rows); per block it keeps the two largest |e_i . a^i_j|, and the
// b_j sums of e_res follow from two running sums, sum_i P_i and sum_i P_i / ||e_i||, since
// block i of e_res is e_i (1 - mean / ||e_i||).  Where the two largest are closer than the
// error bound of both the estimate and the sequential FP32 sum, the 16 sums are formed again
// in that order and decide, so the codes are those of the tiled form bit for bit.  The block
// norms are sequential FP32 sums as there (a lane per edge).
//
// What bounds it: per tile of 32 edges about 7,000 warp instructions and the rows' gathers;
// at 16 warps per SM (128 registers: 32 of them the two running sums) 51% of the issue slots
// are busy.  Rows come by asynchronous copies (1M x 128: plain loads 7.9 ms for the whole
// build, copies 7.3; 20 warps 8.6), and the sums formed in order keep 16 vector elements in
// flight (7.3 -> 7.0; 50,000 x 960: 5.1 -> 3.6 ms, where they had been a third of the time).
// Whole build, tiled form against this one: 1M x 128 10.6 -> 7.0 ms, 50,000 x 960 5.7 -> 3.6.
constexpr int kScreenWarps = 16;  // one CTA per SM
constexpr int kScreenDims = 64;   // coordinates staged at a time: whole blocks, at most this many
constexpr int kMaxCoef = 96;      // blocks per edge (L <= 95, see kMaxCodeWords)

// coordinates staged at a time and the staged row's pitch in 16-byte units: odd, so that
// neither a lane per row nor four lanes per row meet a bank conflict
__host__ __device__ inline int screen_dims(int dp) { return dp * (kScreenDims / dp); }
__host__ __device__ inline int screen_pitch(int dp) { return (screen_dims(dp) / 4) | 1; }
size_t screen_warp_bytes(int dp) {
  return (size_t)32 * screen_pitch(dp) * 16 + (size_t)EdgeQueue<32>::kSlots * 12 + (size_t)kMaxCoef * 4;
}

__device__ __forceinline__ uint32_t bf16x2(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}
// hi and lo BF16 terms of four values, as two packed pairs each
__device__ __forceinline__ void split4(const float4& x, uint32_t (&hi)[2], uint32_t (&lo)[2]) {
  hi[0] = bf16x2(x.x, x.y);
  hi[1] = bf16x2(x.z, x.w);
  lo[0] = bf16x2(x.x - __uint_as_float(hi[0] << 16), x.y - __uint_as_float(hi[0] & 0xffff0000u));
  lo[1] = bf16x2(x.z - __uint_as_float(hi[1] << 16), x.w - __uint_as_float(hi[1] & 0xffff0000u));
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// The two largest of a row's 16 values |p_j|, as keys: the value's bits with the low five
// replaced by (j, sign).  A quad of lanes holds four rows, four values of each per lane;
// lane c of the quad gets row c's result.
struct Top2 {
  uint32_t first, second;
};
__device__ __forceinline__ uint32_t top_key(float p, int j) {
  const uint32_t b = __float_as_uint(p);
  return (b & 0x7fffffe0u) | (uint32_t)(2 * j) | (b >> 31);
}
__device__ __forceinline__ Top2 top_merge(const Top2& x, const Top2& y) {
  return Top2{max(x.first, y.first), max(min(x.first, y.first), max(x.second, y.second))};
}
__device__ __forceinline__ Top2 quad_top2(const float (&row)[4][4], int t) {
  // row[q][i]: value i of row q on this lane; columns 2t, 2t + 1, 8 + 2t, 9 + 2t
  Top2 m[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const uint32_t a = top_key(row[q][0], 2 * t), b = top_key(row[q][1], 2 * t + 1), c = top_key(row[q][2], 2 * t + 8),
                   d = top_key(row[q][3], 2 * t + 9);
    m[q] = top_merge(Top2{max(a, b), min(a, b)}, Top2{max(c, d), min(c, d)});
  }
  // lanes t and t ^ 2 share rows {0, 1} / {2, 3}, then t and t ^ 1 one row each
  const bool up2 = t & 2, up1 = t & 1;
  Top2 k[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const Top2 keep = up2 ? m[q + 2] : m[q], give = up2 ? m[q] : m[q + 2];
    const Top2 got{__shfl_xor_sync(kFull, give.first, 2), __shfl_xor_sync(kFull, give.second, 2)};
    k[q] = top_merge(keep, got);
  }
  const Top2 keep = up1 ? k[1] : k[0], give = up1 ? k[0] : k[1];
  const Top2 got{__shfl_xor_sync(kFull, give.first, 1), __shfl_xor_sync(kFull, give.second, 1)};
  return top_merge(keep, got);
}
// settled: the largest is ahead of the second by more than twice the bound on a value's error
// (and the keys' own truncation), so it is the argmax and has the sign of its estimate
__device__ __forceinline__ bool top_settled(const Top2& k, float err) {
  const float v1 = __uint_as_float(k.first & 0x7fffffe0u), v2 = __uint_as_float(k.second & 0x7fffffe0u);
  return v1 - v2 > 2.0f * err + v1 * 0x1p-17f;
}
__device__ __forceinline__ int top_code(const Top2& k) { return (int)((k.first >> 1) & 15u) | (int)((k.first & 1u) << 16); }

// argmax over the sums p_j of lanes j = 0..15, as argmax16 (warp-wide; the result on every lane)
__device__ __forceinline__ int lanes_argmax(float p) {
  float pv = __shfl_sync(kFull, p, 0), bv = fabsf(pv);
  int best = 0;
  for (int j = 1; j < kVecs; ++j) {
    const float x = __shfl_sync(kFull, p, j), ax = fabsf(x);
    if (ax > bv) {
      bv = ax;
      pv = x;
      best = j;
    }
  }
  return best | ((pv >= 0.0f) ? 0 : 1 << 16);
}

// sum_k w[16 k] x[k] in order, n a multiple of 4; 16 vector elements in flight
__device__ __forceinline__ float ordered_sum(const float* w, const float* x, int n) {
  float p = 0.0f;
  int k = 0;
  for (; k + 16 <= n; k += 16) {
    float v[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) v[q] = __ldg(w + (size_t)(k + q) * kVecs);
#pragma unroll
    for (int q = 0; q < 16; ++q) p = p + v[q] * x[k + q];
  }
  for (; k < n; k += 4) {
#pragma unroll
    for (int q = 0; q < 4; ++q) p = p + __ldg(w + (size_t)(k + q) * kVecs) * x[k + q];
  }
  return p;
}

template <bool PERM, bool FSMEM>
__global__ void __launch_bounds__(kScreenWarps * 32, 1) build_edges_screened_kernel(TileArgs a, float c_a, float c_b,
                                                                                   float c_fp) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, t = lane & 3;
  const int d = a.d, L = a.L, m = a.m, dp = d / L, R = a.R, KS = a.ksteps;
  const int pitch = screen_pitch(dp), cd = screen_dims(dp);
  const uint4* frag = a.frag;
  unsigned char* mem = smem_raw;
  if (FSMEM) {
    uint4* f = reinterpret_cast<uint4*>(smem_raw);
    const int nf = L * KS * 4 * 32;
    for (int i = threadIdx.x; i < nf; i += blockDim.x) f[i] = __ldg(a.frag + i);
    __syncthreads();
    frag = f;
    mem += (size_t)nf * 16;
  }
  mem += (size_t)warp * ((size_t)32 * pitch * 16 + (size_t)EdgeQueue<32>::kSlots * 12 + (size_t)kMaxCoef * 4);
  float4* s_e = reinterpret_cast<float4*>(mem);
  EdgeQueue<32> queue(reinterpret_cast<int32_t*>(mem + (size_t)32 * pitch * 16));
  float* s_coef = reinterpret_cast<float*>(mem + (size_t)32 * pitch * 16 + (size_t)EdgeQueue<32>::kSlots * 12);
  const float* rows = reinterpret_cast<const float*>(s_e);
  const size_t codes_at = rec_codes_offset(R);
  const float bmax = __ldg(a.amax + L);

  // lane l owns edge l of the tile; in the MMA fragments edge 4 r + 2 mt + h is row 8 h + r of
  // the mt-th 16-row tile (r = 0..7), so a quad's four rows belong to its four lanes
  for (;;) {
    const int cnt = queue.fill(a, lane);
    if (cnt == 0) break;
    const bool have = lane < cnt;
    const int32_t u = have ? queue.u[lane] : 0, v = have ? queue.v[lane] : 0;
    const int slot = have ? queue.s[lane] : 0;
    if (!PERM) {  // the rows' later lines come into L2 while the first coordinates are worked on
      const int lines = (d * 4 + 127) >> 7;
      if (have)
        for (int l = 0; l < lines; ++l) {
          const char* p = reinterpret_cast<const char*>(a.X + (size_t)u * d) + ((size_t)l << 7);
          asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
        }
    }
    uint8_t* rec = a.rec + (size_t)v * a.rec_stride;
    uint64_t* cwords = reinterpret_cast<uint64_t*>(rec + codes_at) + slot;
    const float* tv = a.node_proj + (size_t)v * a.proj_stride;

    float tot2 = 0.0f, sum = 0.0f, h1 = 0.0f, pending = 0.0f;
    bool pending_neg = false;
    uint64_t word = 0, word0 = 0;
    int wk = 1, wi = 0;
    float S1[4][4], S2[4][4];  // [row of the quad][value]: sum_i P_i and sum_i P_i / ||e_i||
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int x = 0; x < 4; ++x) S1[q][x] = S2[q][x] = 0.0f;

    bool tiny = false;  // a block whose squared norm loses its precision: e[0] is settled in order
    int i = 0;          // the block
    for (int c0 = 0; c0 < d; c0 += cd) {
      const int cw4 = min(cd, d - c0) >> 2;
      __syncwarp();
      {
        // 32 rows of cw4 pieces, a piece per lane and step
        const int dr = 32 / cw4, dc = 32 - dr * cw4;
        int e = lane / cw4, col = lane - e * cw4;
        if (!PERM) {
          // the neighbours' pieces all in flight at once, straight into shared memory; v's
          // few rows are subtracted when they have arrived (each lane its own pieces)
          int e1 = e, col1 = col;
          for (int j = 0; j < cw4; ++j) {
            if (e1 < cnt)
              asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                               (uint32_t)__cvta_generic_to_shared(s_e + e1 * pitch + col1)),
                           "l"(a.X + (size_t)queue.u[e1] * d + c0 + 4 * col1)
                           : "memory");
            e1 += dr;
            col1 += dc;
            if (col1 >= cw4) {
              col1 -= cw4;
              ++e1;
            }
          }
          asm volatile("cp.async.wait_all;" ::: "memory");
        }
#pragma unroll 4
        for (int j = 0; j < cw4; ++j) {
          if (e < cnt) {
            const float4 y = row4<PERM>(a.X, queue.v[e], d, c0 + 4 * col, a.perm);
            const float4 x = PERM ? row4<PERM>(a.X, queue.u[e], d, c0 + 4 * col, a.perm) : s_e[e * pitch + col];
            s_e[e * pitch + col] = make_float4(x.x - y.x, x.y - y.y, x.z - y.z, x.w - y.w);
          }
          e += dr;
          col += dc;
          if (col >= cw4) {
            col -= cw4;
            ++e;
          }
        }
      }
      __syncwarp();
#pragma unroll 1
      for (int b0 = 0; b0 < cw4 * 4; b0 += dp, ++i) {
        // the block's bound and, from global memory, the first step's vectors, ahead of their use
        const uint4* f = frag + ((size_t)i * KS * 4) * 32 + lane;
        const float am = __ldg(a.amax + i);
        uint4 w[4];
        if (!FSMEM) {
#pragma unroll
          for (int nt = 0; nt < 4; ++nt) w[nt] = __ldg(f + nt * 32);
        }
        // block norm of the lane's own edge, in order
        float n2 = 0.0f;
        uint32_t any = 0;
        for (int k = 0; k < dp; k += 4) {
          const float4 x = s_e[lane * pitch + ((b0 + k) >> 2)];
          n2 = n2 + x.x * x.x;
          n2 = n2 + x.y * x.y;
          n2 = n2 + x.z * x.z;
          n2 = n2 + x.w * x.w;
          any |= __float_as_uint(x.x) | __float_as_uint(x.y) | __float_as_uint(x.z) | __float_as_uint(x.w);
        }
        const bool zero = (any & 0x7fffffffu) == 0u;  // every sum is 0: code +1
        const bool small = !zero && !(n2 >= 1e-30f);
        tiny = tiny || small;
        const float bn = sqrtf(n2);
        tot2 = tot2 + n2;
        sum = sum + bn;
        const float inv = bn > 0.0f ? __frcp_rn(bn) : 0.0f;
        // P = e_i . (a^i_0..15, b_0..15)
        float c[2][4][4];
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
          for (int nt = 0; nt < 4; ++nt)
#pragma unroll
            for (int x = 0; x < 4; ++x) c[mt][nt][x] = 0.0f;
        for (int ks = 0; ks < KS; ++ks) {
          uint32_t hi[2][4], lo[2][4];
          const bool in = 16 * ks + 4 * t < dp;
#pragma unroll
          for (int mt = 0; mt < 2; ++mt)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const int e = (lane & ~3) + 2 * mt + h;
              const float4 x = in ? s_e[e * pitch + ((b0 + 16 * ks) >> 2) + t] : make_float4(0.f, 0.f, 0.f, 0.f);
              uint32_t xh[2], xl[2];
              split4(x, xh, xl);
              hi[mt][h] = xh[0];
              hi[mt][2 + h] = xh[1];
              lo[mt][h] = xl[0];
              lo[mt][2 + h] = xl[1];
            }
          uint4 next[4];
          if (!FSMEM) {
#pragma unroll
            for (int nt = 0; nt < 4; ++nt)
              next[nt] = ks + 1 < KS ? __ldg(f + (4 + nt) * 32) : make_uint4(0u, 0u, 0u, 0u);
          }
#pragma unroll
          for (int nt = 0; nt < 4; ++nt) {
            if (FSMEM) w[nt] = f[nt * 32];
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) {
              mma_bf16(c[mt][nt], hi[mt], w[nt].x, w[nt].y);
              mma_bf16(c[mt][nt], lo[mt], w[nt].x, w[nt].y);
              mma_bf16(c[mt][nt], hi[mt], w[nt].z, w[nt].w);
            }
            if (!FSMEM) w[nt] = next[nt];
          }
          f += 4 * 32;
        }
        // row q = 2 mt + h of the quad: columns 2t, 2t + 1 of n-tiles 0, 1 (a) and 2, 3 (b)
        float pa[4][4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int mt = q >> 1, h = q & 1;
          const float iq = __shfl_sync(kFull, inv, (lane & ~3) + q);
#pragma unroll
          for (int x = 0; x < 4; ++x) {
            pa[q][x] = c[mt][x >> 1][2 * h + (x & 1)];
            const float pb = c[mt][2 + (x >> 1)][2 * h + (x & 1)];
            S1[q][x] = S1[q][x] + (iq != 0.0f ? pb : 0.0f);
            S2[q][x] = fmaf(pb, iq, S2[q][x]);
          }
        }
        const Top2 top = quad_top2(pa, t);
        // a lane without an edge (stale rows in s_e) reads code 0: its estimates could name a vector
        // past m, and node 0's table ends there in an index of one node
        int sel = have && !zero ? top_code(top) : 0;
        const bool open = have && !zero && (small || !top_settled(top, c_a * am * bn));
        for (unsigned todo = __ballot_sync(kFull, open); todo; todo &= todo - 1) {
          const int e = __ffs(todo) - 1;
          float p = 0.0f;
          if (lane < kVecs) {
            p = ordered_sum(a.W + (size_t)(d + i * dp) * kVecs + lane, rows + (size_t)e * pitch * 4 + b0, dp);
          }
          const int got = lanes_argmax(p);
          if (lane == e) sel = got;
        }
        // the code; its table entry is added a block later, when it has arrived
        h1 = h1 + (pending_neg ? -pending : pending);
        pending = __ldg(tv + (i + 1) * m + (sel & 0xffff));
        pending_neg = (sel >> 16) != 0;
        word |= ((uint64_t)(sel & 0xffff) | ((uint64_t)(sel >> 16) << (a.bits - 1))) << (wk * a.bits);
        if (++wk == a.cpw) {
          if (wi == 0) word0 = word;
          else if (have) cwords[(size_t)wi * R] = word;
          word = 0;
          wk = 0;
          ++wi;
        }
      }
    }
    h1 = h1 + (pending_neg ? -pending : pending);
    if (wk > 0) {
      if (wi == 0) word0 = word;
      else if (have) cwords[(size_t)wi * R] = word;
    }
    const float norm = sqrtf(tot2);
    float wr = 1.0f, cr = 0.0f, mean = 0.0f;
    if (norm != 0.0f) {
      wr = sum / (sqrtf((float)L) * norm);
      if (wr > 1.0f) wr = 1.0f;
      cr = sqrtf((float)L) * sqrtf(fmaxf(0.0f, 1.0f - wr * wr));
      mean = sum / (float)L;
    }
    // ---- e[0]: the sums of e_res with the b_j
    float pb[4][4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float mq = __shfl_sync(kFull, mean, (lane & ~3) + q);
#pragma unroll
      for (int x = 0; x < 4; ++x) pb[q][x] = S1[q][x] - mq * S2[q][x];
    }
    const Top2 top = quad_top2(pb, t);
    int sel0 = top_code(top);
    // sum_i | ||e_i|| - mean | <= sqrt(L (sum ||e_i||^2 - L mean^2)), the weight of the estimates'
    // errors; the two running sums and the sequential sum round relative to sum ||e_i||
    const float spread = sqrtf((float)L * fmaxf(tot2 - sum * mean, 0.0f) + 1e-6f * (float)L * tot2);
    const bool open = have && norm != 0.0f && (tiny || !top_settled(top, bmax * (c_b * spread + c_fp * sum)));
    for (unsigned todo = __ballot_sync(kFull, open); todo; todo &= todo - 1) {
      const int e = __ffs(todo) - 1;
      const int32_t eu = queue.u[e], ev = queue.v[e];
      const float em = __shfl_sync(kFull, mean, e);
      float* lin = reinterpret_cast<float*>(s_e);  // the edge's d coordinates, in order
      __syncwarp();
      for (int k = 4 * lane; k < d; k += 128) {
        const float4 x = row4<PERM>(a.X, eu, d, k, a.perm), y = row4<PERM>(a.X, ev, d, k, a.perm);
        *reinterpret_cast<float4*>(lin + k) = make_float4(x.x - y.x, x.y - y.y, x.z - y.z, x.w - y.w);
      }
      __syncwarp();
      for (int i = lane; i < L; i += 32) {
        float n2 = 0.0f;
        for (int k = 0; k < dp; ++k) n2 = n2 + lin[i * dp + k] * lin[i * dp + k];
        const float b = sqrtf(n2);
        s_coef[i] = (b > 0.0f) ? (1.0f - em / b) : 0.0f;
      }
      __syncwarp();
      for (int k = lane; k < d; k += 32) lin[k] = lin[k] * s_coef[k / dp];
      __syncwarp();
      const int got = lanes_argmax(lane < kVecs ? ordered_sum(a.W + lane, lin, d) : 0.0f);
      if (lane == e) sel0 = got;
    }
    if (have) {
      if (norm == 0.0f) {  // a degenerate edge gets code +1 everywhere
        sel0 = 0;
        h1 = 0.0f;
        for (int i = 0; i < L; ++i) h1 = h1 + __ldg(tv + (i + 1) * m);
        word0 = 0;
        for (int k = 1; k < a.nwords; ++k) cwords[(size_t)k * R] = 0;
      }
      const float v0f = __ldg(tv + (sel0 & 0xffff));
      const float h2 = (sel0 >> 16) ? -v0f : v0f;
      reinterpret_cast<float4*>(rec)[slot] = make_float4(norm, wr, cr, wr * h1 + cr * h2);
      cwords[0] = word0 | (uint64_t)(sel0 & 0xffff) | ((uint64_t)(sel0 >> 16) << (a.bits - 1));
    }
    queue.drop(cnt, lane);
  }
}

int num_sms() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 1;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 1;
  return sms > 0 ? sms : 1;
}

// The compact index (8- or 16-bit edge scalars; Sec. 4.3's space analysis, Sec. 6.4's
// PEOs (Compact)): one warp per node rewrites its FP32 record.  Per scalar kind (||e||,
// w_reg, sqrt(L) w_res) over the node's valid edges: s = max |x|, step = s / Qb
// (Qb = 2^(bits-1) - 1), q = rint(x / step) clamped to [-Qb, Qb] (0 when step = 0); the
// search reads x' = (float) q * step.  The node term is recomputed from the stored
// weights, sv = w_reg' sum_{c=1..L} sgn t(v)[c][j_c] + (sqrt(L) w_res)' sgn t(v)[0][j_0]
// (the same FP32 order as build_codes_kernel), and kept in FP32, so that the statistic
// the search forms, (S(t(q)) - sv) / ||x||, is the one of the stored weights.  Ids and
// codes are copied unchanged.
template <int SB>
__global__ void compact_records_kernel(const uint8_t* __restrict__ src, size_t src_stride, long long n, int R,
                                       int words, const float* __restrict__ node_proj, int proj_stride, int L, int m,
                                       uint8_t* __restrict__ dst, size_t dst_stride) {
  using Q4 = typename std::conditional<SB == 16, short4, char4>::type;
  constexpr float kQb = SB == 16 ? 32767.0f : 127.0f;
  const int lane = threadIdx.x & 31;
  const int bits = code_bits(m), cpw = codes_per_word(m);
  const unsigned long long mask = (1ull << bits) - 1ull;
  const int half = 1 << (bits - 1);
  const long long warps = (long long)gridDim.x * (blockDim.x >> 5);
  for (long long v = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); v < n; v += warps) {
    const uint8_t* r = src + (size_t)v * src_stride;
    uint8_t* o = dst + (size_t)v * dst_stride;
    const float4* sc = reinterpret_cast<const float4*>(r);
    const int32_t* ids = reinterpret_cast<const int32_t*>(r + rec_ids_offset(R));
    const uint64_t* cs = reinterpret_cast<const uint64_t*>(r + rec_codes_offset(R));
    const float* tv = node_proj + (size_t)v * proj_stride;
    float4 x[2];
    int32_t id[2];
    float mx[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int sl = h * 32 + lane;
      id[h] = sl < R ? ids[sl] : -1;
      x[h] = sl < R ? sc[sl] : make_float4(0.f, 0.f, 0.f, 0.f);
      if (id[h] >= 0) {
        mx[0] = fmaxf(mx[0], fabsf(x[h].x));
        mx[1] = fmaxf(mx[1], fabsf(x[h].y));
        mx[2] = fmaxf(mx[2], fabsf(x[h].z));
      }
    }
    float step[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) mx[k] = fmaxf(mx[k], __shfl_xor_sync(kFull, mx[k], off));
      step[k] = mx[k] / kQb;
    }
    if (lane == 0) *reinterpret_cast<float4*>(o) = make_float4(step[0], step[1], step[2], 0.0f);
    auto quant = [&](float val, float st, bool ok) -> int {
      if (!ok || !(st > 0.0f)) return 0;
      float q = rintf(val / st);
      q = fminf(fmaxf(q, -kQb), kQb);
      return (int)q;
    };
    // 16-bit form: sv[R] then q[R]; 8-bit form: {q, sv} pairs of 8 bytes
    float* svo = reinterpret_cast<float*>(o + (SB == 16 ? rec_sv_offset(R) : rec_pair_offset() + 4));
    Q4* qo = reinterpret_cast<Q4*>(o + (SB == 16 ? rec_q_offset(R) : rec_pair_offset()));
    constexpr int kStep = SB == 16 ? 1 : 2;  // elements of 4 bytes (sv) / of sizeof(Q4) (q) per edge
    int32_t* io = reinterpret_cast<int32_t*>(o + rec_ids_offset(R, SB));
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int sl = h * 32 + lane;
      if (sl < R) {
        const bool ok = id[h] >= 0;
        Q4 q;
        q.x = quant(x[h].x, step[0], ok);
        q.y = quant(x[h].y, step[1], ok);
        q.z = quant(x[h].z, step[2], ok);
        q.w = 0;
        float svv = 0.0f;
        if (ok) {
          const float wq = (float)q.y * step[1], cq = (float)q.z * step[2];
          // the edge's codes e[0..L] from its packed words: code c sits in word c / cpw
          float h1 = 0.0f, h2 = 0.0f;
          for (int c = 0; c <= L; ++c) {
            const unsigned long long word = cs[(size_t)(c / cpw) * R + sl];
            const int code = (int)((word >> ((c % cpw) * bits)) & mask);
            const float val = tv[c * m + (code & (half - 1))];
            const float sv_c = (code & half) ? -val : val;
            if (c == 0) h2 = sv_c; else h1 = h1 + sv_c;
          }
          svv = wq * h1 + cq * h2;
        }
        qo[(size_t)kStep * sl] = q;
        svo[(size_t)kStep * sl] = svv;
        io[sl] = id[h];
      }
    }
    // codes, then zero the gaps and the padding
    uint64_t* cd = reinterpret_cast<uint64_t*>(o + rec_codes_offset(R, SB));
    for (int t = lane; t < words * R; t += 32) cd[t] = cs[t];
    if (SB == 16)
      for (size_t b = rec_sv_offset(R) + 4 * (size_t)R + lane; b < rec_q_offset(R); b += 32) o[b] = 0;
    for (size_t b = rec_ids_offset(R, SB) + 4 * (size_t)R + lane; b < rec_codes_offset(R, SB); b += 32) o[b] = 0;
    for (size_t b = rec_codes_offset(R, SB) + 8 * (size_t)words * R + lane; b < dst_stride; b += 32) o[b] = 0;
  }
}

}  // namespace

cudaError_t launch_compact_records(const uint8_t* src, size_t src_stride, int64_t n, int R, int words,
                                   const float* node_proj, int proj_stride, int L, int m, int sbits, uint8_t* dst,
                                   size_t dst_stride, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  if (R > 64 || !node_proj) return cudaErrorInvalidValue;
  const int threads = 256;
  long long blocks = (n + 7) / 8;
  if (blocks > 65535LL * 16) blocks = 65535LL * 16;
  if (sbits == 16)
    compact_records_kernel<16><<<(unsigned)blocks, threads, 0, st>>>(src, src_stride, n, R, words, node_proj,
                                                                     proj_stride, L, m, dst, dst_stride);
  else if (sbits == 8)
    compact_records_kernel<8><<<(unsigned)blocks, threads, 0, st>>>(src, src_stride, n, R, words, node_proj,
                                                                    proj_stride, L, m, dst, dst_stride);
  else
    return cudaErrorInvalidValue;
  return cudaGetLastError();
}

namespace {

// The tiled kernels' variant for the block length: 4, 2 or 1 coordinates per step, rows
// read through a permutation or not, the vectors in shared memory or not.
// ROWS = 0: the edge kernel, else the row kernel with that many rows per lane.
template <int ROWS, int KU, bool PERM, bool WSMEM>
cudaError_t launch_tile(const TileArgs& a, int grid, int warps, cudaStream_t st) {
  const void* fn;
  size_t per_warp;
  if constexpr (ROWS == 0) {
    fn = (const void*)build_edges_kernel<KU, PERM, WSMEM>;
    per_warp = (size_t)kEdgeTile * kTilePitch * 16 + (size_t)(kEdgeTile + 32) * 12;
  } else {
    fn = (const void*)node_rows_kernel<ROWS, KU, PERM, WSMEM>;
    per_warp = (size_t)32 * ROWS * kTilePitch * 16;
  }
  const size_t smem = (WSMEM ? (size_t)2 * a.d * kVecs * sizeof(float) : 0) + per_warp * warps;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  TileArgs copy = a;
  void* args[] = {&copy};
  return cudaLaunchKernel(fn, dim3((unsigned)grid), dim3(warps * 32), args, smem, st);
}
template <int ROWS, int KU>
cudaError_t launch_tile_ku(const TileArgs& a, int grid, int warps, cudaStream_t st) {
  const bool ws = a.d <= kMaxSmemVecDim;
  if (a.perm) return ws ? launch_tile<ROWS, KU, true, true>(a, grid, warps, st) : launch_tile<ROWS, KU, true, false>(a, grid, warps, st);
  return ws ? launch_tile<ROWS, KU, false, true>(a, grid, warps, st) : launch_tile<ROWS, KU, false, false>(a, grid, warps, st);
}
template <int ROWS>
cudaError_t launch_tile_any(const TileArgs& a, int grid, int warps, cudaStream_t st) {
  const int dp = a.d / a.L;
  return dp % 4 == 0   ? launch_tile_ku<ROWS, 4>(a, grid, warps, st)
         : dp % 2 == 0 ? launch_tile_ku<ROWS, 2>(a, grid, warps, st)
                       : launch_tile_ku<ROWS, 1>(a, grid, warps, st);
}

int edges_grid(int64_t n) { return (int)std::min<int64_t>(num_sms(), (n + kNodeChunk - 1) / kNodeChunk); }

// The shapes of the screened form: a lane's four coordinates of a step lie in one block and
// start on 16 bytes (blocks a multiple of 4), a step of 16 is at least half full, and whole
// blocks fit the 64 staged coordinates.  Others take the tiled form.
bool screened(int d, int L, int m) {
  const int dp = d / L;
  return m <= kVecs && dp % 4 == 0 && dp >= 8 && dp <= kScreenDims && L < kMaxCoef && 32 * screen_pitch(dp) * 4 >= d;
}

// The fragment table and the norms of the screened form, from the k-major vectors W (2 d rows
// of 16: the b_j, then the a^i_j).  Coordinate 4 t + x of a step of 16 sits where the MMA's
// A fragment has lane t's x-th element.
struct ScreenTables {
  std::vector<uint32_t> frag;
  std::vector<float> amax;
};
uint16_t host_bf16(float f) {  // round to nearest even (finite values)
  uint32_t u;
  memcpy(&u, &f, 4);
  return (uint16_t)((u + 0x7fffu + ((u >> 16) & 1u)) >> 16);
}
float host_widen(uint16_t h) {
  const uint32_t u = (uint32_t)h << 16;
  float f;
  memcpy(&f, &u, 4);
  return f;
}
ScreenTables screen_tables(const float* W, int d, int L) {
  const int dp = d / L, KS = (dp + 15) / 16;
  ScreenTables T;
  T.frag.assign((size_t)L * KS * 4 * 32 * 4, 0u);
  T.amax.assign((size_t)L + 1, 0.0f);
  auto at = [&](int i, int k, int col) -> float {  // column 0..15: a^i, 16..31: b
    if (k >= dp) return 0.0f;
    return col < 16 ? W[((size_t)d + (size_t)i * dp + k) * kVecs + col] : W[((size_t)i * dp + k) * kVecs + col - 16];
  };
  for (int i = 0; i < L; ++i) {
    for (int col = 0; col < 32; ++col) {
      double n2 = 0.0;
      for (int k = 0; k < dp; ++k) n2 += (double)at(i, k, col) * at(i, k, col);
      float& most = T.amax[col < 16 ? i : L];
      most = std::max(most, (float)(sqrt(n2) * (1.0 + 1e-6)));
    }
    for (int ks = 0; ks < KS; ++ks)
      for (int nt = 0; nt < 4; ++nt)
        for (int lane = 0; lane < 32; ++lane) {
          const int g = lane >> 2, t = lane & 3;
          uint32_t* o = &T.frag[((((size_t)i * KS + ks) * 4 + nt) * 32 + lane) * 4];
          for (int r = 0; r < 2; ++r) {
            uint32_t hi = 0, lo = 0;
            for (int x = 0; x < 2; ++x) {
              const float v = at(i, 16 * ks + 4 * t + 2 * r + x, 8 * nt + g);
              const uint16_t h = host_bf16(v), l = host_bf16(v - host_widen(h));
              hi |= (uint32_t)h << (16 * x);
              lo |= (uint32_t)l << (16 * x);
            }
            o[r] = hi;
            o[2 + r] = lo;
          }
        }
  }
  return T;
}

template <bool PERM, bool FSMEM>
cudaError_t launch_screened(const TileArgs& a, int grid, size_t smem, cudaStream_t st) {
  auto fn = build_edges_screened_kernel<PERM, FSMEM>;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  // a value's error relative to ||a|| ||e_i||: three products of two-term BF16 factors (dropped
  // and rounded terms 3.05 2^-16), their FP32 accumulation (2^-23 per product), and the
  // sequential sum it stands for (2^-24 per coordinate, with the norms' own rounding); for
  // e_res the same relative to spread (d coordinates), and relative to sum ||e_i|| the
  // rounding of the two running sums and of the coefficients, (2 L + 8) 2^-24, times 1.5
  const int dp = a.d / a.L;
  const double c = 3.05 * 0x1p-16 + 48.0 * a.ksteps * 0x1p-23 + (2.0 * dp + 8.0) * 0x1p-24;
  const double c_res = c + (a.d + 4.0) * 0x1p-24, fp = 1.5 * (2.0 * a.L + 8.0) * 0x1p-24;
  fn<<<(unsigned)grid, kScreenWarps * 32, smem, st>>>(a, (float)(c * 1.01), (float)(c_res * 1.01), (float)fp);
  return cudaGetLastError();
}

}  // namespace

int codes_padded_vecs() { return kVecs; }

size_t build_codes_scratch_bytes(int64_t n, int d, int L, int m) {
  if (m > kVecs || n <= 0) return 0;
  if (screened(d, L, m)) return 512 + (size_t)L * 4 + (size_t)L * ((d / L + 15) / 16) * 4 * 32 * 16;
  return 256 + (size_t)edges_grid(n) * kTileWarps * L * kEdgeTile * sizeof(float2);
}

cudaError_t launch_build_codes(const float* X, int64_t n, int d, const int32_t* nbrs, int R, int L, int m,
                               const float* A, const float* B, const float* W16, const float* W16_host,
                               const int32_t* perm, const float* node_proj, int proj_stride, uint8_t* rec,
                               size_t rec_stride, void* scratch, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  if (m <= kVecs) {
    cudaError_t e = cudaMemsetAsync(scratch, 0, sizeof(int), st);
    if (e != cudaSuccess) return e;
    TileArgs a{};
    a.X = X;
    a.n = n;
    a.d = d;
    a.L = L;
    a.m = m;
    a.W = W16;
    a.perm = perm;
    a.node_proj = const_cast<float*>(node_proj);
    a.proj_stride = proj_stride;
    a.nbrs = nbrs;
    a.R = R;
    a.rec = rec;
    a.rec_stride = rec_stride;
    a.bits = code_bits(m);
    a.cpw = codes_per_word(m);
    a.nwords = code_words(L, m);
    a.work = static_cast<int*>(scratch);
    if (screened(d, L, m)) {
      const ScreenTables T = screen_tables(W16_host, d, L);
      unsigned char* w = static_cast<unsigned char*>(scratch) + 256;
      const size_t fb = T.frag.size() * sizeof(uint32_t);
      e = cudaMemcpyAsync(w, T.frag.data(), fb, cudaMemcpyHostToDevice, st);
      if (e == cudaSuccess)
        e = cudaMemcpyAsync(w + fb, T.amax.data(), T.amax.size() * sizeof(float), cudaMemcpyHostToDevice, st);
      // the tables are host vectors of this call: their copies have to be done before it ends
      if (e == cudaSuccess) e = cudaStreamSynchronize(st);
      if (e != cudaSuccess) return e;
      a.frag = reinterpret_cast<const uint4*>(w);
      a.amax = reinterpret_cast<const float*>(w + fb);
      a.ksteps = (d / L + 15) / 16;
      const size_t warps = screen_warp_bytes(d / L) * kScreenWarps;
      const bool fs = fb + warps <= (size_t)220 * 1024;
      const size_t smem = warps + (fs ? fb : 0);
      const int grid = edges_grid(n);
      if (perm) return fs ? launch_screened<true, true>(a, grid, smem, st) : launch_screened<true, false>(a, grid, smem, st);
      return fs ? launch_screened<false, true>(a, grid, smem, st) : launch_screened<false, false>(a, grid, smem, st);
    }
    a.blocks = reinterpret_cast<float2*>(static_cast<unsigned char*>(scratch) + 256);
    return launch_tile_any<0>(a, edges_grid(n), kTileWarps, st);
  }
  const size_t smem = sizeof(float) * ((size_t)R * d + 2 * (size_t)R * L + 4 * (size_t)R +
                                       (size_t)R * (L + 1) * m) +
                      sizeof(int32_t) * ((size_t)R + (size_t)R * (L + 1)) + sizeof(float) * (size_t)(L + 1) * m;
  cudaError_t e = cudaFuncSetAttribute(build_codes_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, build_codes_kernel, kBuildThreads, smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  long long grid = (long long)num_sms() * per_sm;
  if (grid > n) grid = n;
  build_codes_kernel<<<(unsigned)grid, kBuildThreads, smem, st>>>(X, n, d, nbrs, R, L, m, A, B, perm, node_proj,
                                                                  proj_stride, rec, rec_stride, code_bits(m),
                                                                  codes_per_word(m), code_words(L, m));
  return cudaGetLastError();
}

cudaError_t launch_node_proj(const float* X, int64_t n, int d, int L, int m, const float* A, const float* B,
                             const float* W16, const int32_t* perm, float* out, int out_stride, float* norms,
                             cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  if (m <= kVecs) {
    TileArgs a{};
    a.X = X;
    a.n = n;
    a.d = d;
    a.L = L;
    a.m = m;
    a.W = W16;
    a.perm = perm;
    a.node_proj = out;
    a.proj_stride = out_stride;
    a.norms = perm ? nullptr : norms;  // the norm sums the stored order of the coordinates
    const int64_t sms = num_sms();
    const int rows = n >= (int64_t)32 * kRowsPerLane * sms * kTileWarps ? kRowsPerLane : 1;
    const int64_t tiles = (n + 32 * rows - 1) / (32 * rows);
    const int warps = (int)std::min<int64_t>(kTileWarps, (tiles + sms - 1) / sms);
    const int grid = (int)std::min<int64_t>(sms, (tiles + warps - 1) / warps);
    cudaError_t e = rows == 1 ? launch_tile_any<1>(a, grid, warps, st) : launch_tile_any<kRowsPerLane>(a, grid, warps, st);
    if (e != cudaSuccess || !perm) return e;
    return launch_row_norms(X, n, d, norms, st);
  }
  const long long total = n * (long long)out_stride;
  long long grid = (total + 255) / 256;
  const long long cap = (long long)num_sms() * 16;
  if (grid > cap) grid = cap;
  node_proj_kernel<<<(unsigned)grid, 256, 0, st>>>(X, n, d, L, m, A, B, perm, out, out_stride);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? launch_row_norms(X, n, d, norms, st) : e;
}

cudaError_t launch_row_norms(const float* X, int64_t n, int d, float* norms, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  long long grid = (n + 255) / 256;
  const long long cap = (long long)num_sms() * 16;
  if (grid > cap) grid = cap;
  row_norms_kernel<<<(unsigned)grid, 256, 0, st>>>(X, n, d, norms);
  return cudaGetLastError();
}


namespace {
__global__ void wide_flags_kernel(const uint8_t* rec, size_t rec_stride, size_t ids_offset, long long n, int R,
                                  uint8_t* wide) {
  for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (long long)gridDim.x * blockDim.x) {
    const int32_t* ids = reinterpret_cast<const int32_t*>(rec + (size_t)v * rec_stride + ids_offset);
    uint8_t any = 0;
    for (int s = 32; s < R; ++s) any |= (uint8_t)(ids[s] >= 0 && (long long)ids[s] < n);
    wide[v] = any;
  }
}
}  // namespace

cudaError_t launch_wide_flags(const uint8_t* rec, size_t rec_stride, size_t ids_offset, int64_t n, int R,
                              uint8_t* wide, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const long long blocks = std::min<long long>((n + 255) / 256, 4096);
  wide_flags_kernel<<<(unsigned)blocks, 256, 0, st>>>(rec, rec_stride, ids_offset, n, R, wide);
  return cudaGetLastError();
}

}  // namespace peos
