// Brute-force K-NN on the tensor cores (sm_103a tcgen05): graph candidates and ground truth
// for large bases, in two precisions of the scores.
//
//   1. convert: base and queries to BF16 rows (zero-padded to a multiple of 64 elements),
//      and ||x||^2 of every base row in FP32.  The precise form takes a centre of the base
//      off every row and keeps each value as the sum of two BF16 terms, hi and lo, in a row
//      of twice the length.
//   2. candidates: one CTA per SM takes an equal, contiguous share of the (128 queries x 256
//      base rows) tiles, query tile by query tile; a query tile that spans CTAs has one
//      candidate list per CTA (a segment).  A TMA warp brings 128 x 64 query and 256 x 64 base
//      chunks (128-byte swizzled, K-major) through a ring of shared-memory stages behind
//      mbarriers (the query chunks stay resident where they fit); an MMA warp issues
//      tcgen05.mma (BF16 in, FP32 accumulate in tensor memory, M = 128, N = 256, K = 16 per
//      instruction) into one of two accumulators, in the precise form for the products hi hi,
//      lo hi and hi lo; eight epilogue warps (four where the lists are long) read the other
//      accumulator with tcgen05.ld, one query row per thread, and keep the row's best `cand`
//      scores ||x||^2 - 2 q.x (q's own norm does not change the order) in a max-heap in shared
//      memory.  Scores below the heap's worst wait in a short per-row buffer; when a row's
//      buffer is nearly full all rows empty theirs side by side.
//      Where scores are rounded the plain form closes a list at the end of a slice of the base
//      too, so that a query keeps as many rows as it takes to absorb misranked ones, and the
//      CTAs take whole slices where that costs less.
//   3. finalize: the candidates of every segment sorted by score; those that may be among
//      the k nearest (score within twice the error bound of the k-th) get their exact FP32
//      squared distance (sequential over the dimensions), and the k smallest by (dist, id)
//      are the result.
// On integer-valued data below 256 (SIFT-shaped) the BF16 products and their FP32 sums
// are exact, so the candidates are exactly the best rows of each segment.  Otherwise the
// BF16 rounding only reorders near-ties, which the slack of `cand` over k absorbs; the
// final distances are always exact FP32.
//
// The precise form proves its result: a row left out of a full list scored no better than
// that list's worst, so with the score's error bound its distance is known to be above
// the k-th found (rows too long to be near the query aside, whatever their error), or the
// query is handed on to the FFMA kernel (knn.cu).  Norms that vanish
// or come near FP32's range and a CTA that gave up waiting hand every query on.
//
// Every wait on an mbarrier is bounded: after kWaitLimitNs of the global timer (or
// kMaxPolls polls, whichever comes first) the CTA records an error and stops issuing work
// (the host reports PEOS_E_TIMEOUT; the precise form's queries go to the FFMA kernel).
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <float.h>
#include <math.h>

#include <algorithm>
#include <mutex>

#include "device.cuh"
#include "internal.h"

namespace peos {
namespace {

constexpr int kTcM = 128;      // queries per tile: accumulator rows = tensor-memory lanes
constexpr int kTcN = 256;      // base rows per tile: accumulator columns
constexpr int kTcK = 64;       // elements per stage: one 128-byte swizzle atom of BF16
constexpr int kMaxStages = 4;
constexpr int kRows = kTcM;                        // candidate lists per CTA: one per accumulator row
constexpr int kAccCols = 2 * kTcN;                 // two accumulators: all 512 tensor-memory columns
constexpr long long kWaitLimitNs = 2000000000ll;  // 2 s: no wait of a healthy launch comes near it
constexpr long long kMaxPolls = 1ll << 26;
constexpr int kMaxK = 96;          // k peos_knn_tensor serves (candidates per segment: k + 16)
// candidates per query over all segments (finalize's shared memory); the precise form takes up
// to four times as many where more CTAs are worth it (see tc_plan)
constexpr int kMaxCandTotal = 4096;
// Columns screened together, and scores a row buffers before they enter its heap (at least a
// group): 16 and 20 per warp where 8 epilogue warps' buffers fit in shared memory beside the
// lists, 8 and 12 with 4 warps (long lists).
__host__ __device__ constexpr int group_cols(int ew) { return ew == 8 ? 16 : 8; }
__host__ __device__ constexpr int pend_slots(int ew) { return ew == 8 ? 20 : 12; }

constexpr int kABytes = kTcM * kTcK * 2;  // 16 KB
constexpr int kBBytes = kTcN * kTcK * 2;  // 32 KB

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}

// nanoseconds of the GPU's global timer
__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Wait for the phase of `bar` with the given parity; false when `limit_ns` nanoseconds of
// the global timer passed first.  The timer is read only once the first poll failed.
__device__ __forceinline__ bool mbar_wait_n(uint64_t* bar, uint32_t parity, long long limit_ns) {
  const uint32_t a = smem_u32(bar);
  uint64_t t0 = 0;
  for (long long i = 0; i < kMaxPolls; ++i) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(a), "r"(parity)
        : "memory");
    if (done) return true;
    const uint64_t t = global_ns();
    if (i == 0) t0 = t;
    else if ((long long)(t - t0) >= limit_ns) return false;
  }
  return false;
}

__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
  return mbar_wait_n(bar, parity, kWaitLimitNs);
}

// Self-test of the bounded wait: one thread waits on an mbarrier that nothing arrives on;
// the wait gives up after `limit_ns` nanoseconds and the kernel records that it did.
__global__ void bounded_wait_probe_kernel(long long limit_ns, int* gave_up) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    *gave_up = mbar_wait_n(&bar, 0, limit_ns) ? 0 : 1;
  }
}

__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, uint64_t* bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(bar))
      : "memory");
}

// Shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t smem_desc_sw128(const void* p) {
  const uint64_t addr = smem_u32(p);
  uint64_t d = 0;
  d |= (addr >> 4) & 0x3FFFull;            // start address
  d |= (uint64_t)1 << 16;                  // leading byte offset (unused with swizzle)
  d |= (uint64_t)(1024 >> 4) << 32;        // stride byte offset
  d |= (uint64_t)1 << 46;                  // descriptor version
  d |= (uint64_t)2 << 61;                  // 128-byte swizzle
  return d;
}

// Instruction descriptor: BF16 x BF16 -> FP32, A and B K-major, M x N.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// float -> unsigned with the same order (for keys that may be negative)
__device__ __forceinline__ uint32_t ordered(float f) {
  const uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// the score of a candidate key (inverse of ordered on the high word); the largest finite
// value for an empty slot, so that every finite score may enter a list that is not full and
// +inf (a column past the base) never does
__device__ __forceinline__ float key_score(uint64_t key) {
  if (key == kNoKey) return FLT_MAX;
  const uint32_t o = (uint32_t)(key >> 32);
  return __uint_as_float((o & 0x80000000u) ? (o & 0x7fffffffu) : ~o);
}

__device__ __forceinline__ uint32_t bf16_pair(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}

// The precise form works on rows less a centre of the base, so that the score's error is
// relative to the rows' spread and not to a common offset.  Per coordinate the mean of five
// medians of three rows each, which one long row does not move; zero where that is no moderate
// number.  Four coordinates from k on.  Every CTA of the queries' conversion finds it for itself
// (16,384 x 100, one query: 112 us for the call; a launch of its own 117).
__device__ __forceinline__ float median3(float a, float b, float c) { return fmaxf(fminf(a, b), fminf(fmaxf(a, b), c)); }
__device__ __forceinline__ float4 centre_of(const float* __restrict__ X, long long n, int d, int k) {
  float4 m = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int j = 0; j < 15; j += 3) {
    float4 v[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) v[i] = __ldg(reinterpret_cast<const float4*>(X + (size_t)(n * (j + i) / 15) * d + k));
    m.x += median3(v[0].x, v[1].x, v[2].x);
    m.y += median3(v[0].y, v[1].y, v[2].y);
    m.z += median3(v[0].z, v[1].z, v[2].z);
    m.w += median3(v[0].w, v[1].w, v[2].w);
  }
  auto moderate = [](float x) { return fabsf(x) < 1e18f ? 0.2f * x : 0.0f; };
  return make_float4(moderate(m.x), moderate(m.y), moderate(m.z), moderate(m.w));
}

// A warp takes four rows at a time (their loads in flight together), four elements per lane.
// LO: rows less `centre` (FIND, the queries: found here, and stored; the call's flags are
// cleared); the rounding errors' own BF16 values follow the row's hi terms.  norm2: FP32 squared
// norms (base rows); xmax: the largest of them, as its bits (a NaN's bits are larger than any
// number's).  Without LO: `inexact` is set when a score of these rows may be rounded: an
// element that is not an integer of at most 256, or a squared norm of 2^24 / 3 or more (below,
// ||x||^2 + 2 |q.x| and all sums on the way stay under 2^24).
constexpr float kExactNorm2 = 5.5e6f;
constexpr int kConvertThreads = 256;
template <bool LO, bool FIND>
__global__ void convert_bf16_kernel(const float* __restrict__ X, long long n, int d, int pitch,
                                    __nv_bfloat16* __restrict__ out, float* __restrict__ norm2,
                                    unsigned* __restrict__ xmax, unsigned* __restrict__ inexact,
                                    float* __restrict__ centre, const float* __restrict__ base, long long nbase,
                                    int* __restrict__ err) {
  constexpr int kAtOnce = 4;
  constexpr int kWindow = 4 * kConvertThreads;  // FIND (no norms): coordinates whose centre is held at a time
  __shared__ float4 s_centre[FIND ? kConvertThreads : 1];
  const int lane = threadIdx.x & 31;
  const long long w0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
  const size_t row = (size_t)pitch * (LO ? 2 : 1);
  unsigned most = 0;
  bool rounded = false;
  if (FIND && blockIdx.x == 0 && threadIdx.x == 0) {
    xmax[0] = inexact[0] = 0u;
    err[0] = err[1] = 0;
  }
  for (int first = 0; first < pitch; first += kWindow) {
    const int end = FIND ? min(pitch, first + kWindow) : pitch;
    if (FIND) {
      __syncthreads();
      const int k = first + 4 * threadIdx.x;
      if (k < end) {
        const float4 c = k < d ? centre_of(base, nbase, d, k) : make_float4(0.f, 0.f, 0.f, 0.f);
        s_centre[threadIdx.x] = c;
        if (blockIdx.x == 0) *reinterpret_cast<float4*>(centre + k) = c;
      }
      __syncthreads();
    }
    for (long long r0 = w0 * kAtOnce; r0 < n; r0 += nw * kAtOnce) {
      float s[kAtOnce];
#pragma unroll
      for (int j = 0; j < kAtOnce; ++j) s[j] = 0.0f;
      // two steps' loads in flight (1M x 128, 100 queries, the call: 505 us against 532; four 511)
#pragma unroll 2
      for (int k = first + 4 * lane; k < end; k += 128) {
        float4 v[kAtOnce];
#pragma unroll
        for (int j = 0; j < kAtOnce; ++j)
          v[j] = (k < d && r0 + j < n) ? __ldg(reinterpret_cast<const float4*>(X + (size_t)(r0 + j) * d + k))
                                       : make_float4(0.f, 0.f, 0.f, 0.f);
        float4 ce = make_float4(0.f, 0.f, 0.f, 0.f);
        if (FIND) ce = s_centre[(k - first) >> 2];
        else if (LO) ce = __ldg(reinterpret_cast<const float4*>(centre + k));
#pragma unroll
        for (int j = 0; j < kAtOnce; ++j) {
          if (r0 + j >= n) break;
          float4 x = v[j];
          if (LO) x = make_float4(x.x - ce.x, x.y - ce.y, x.z - ce.z, x.w - ce.w);
          const uint2 h = make_uint2(bf16_pair(x.x, x.y), bf16_pair(x.z, x.w));
          __nv_bfloat16* o = out + (size_t)(r0 + j) * row + k;
          *reinterpret_cast<uint2*>(o) = h;
          if (LO) {
            const float4 f = make_float4(__uint_as_float(h.x << 16), __uint_as_float(h.x & 0xffff0000u),
                                         __uint_as_float(h.y << 16), __uint_as_float(h.y & 0xffff0000u));
            *reinterpret_cast<uint2*>(o + pitch) =
                make_uint2(bf16_pair(x.x - f.x, x.y - f.y), bf16_pair(x.z - f.z, x.w - f.w));
          }
          s[j] += x.x * x.x + x.y * x.y + x.z * x.z + x.w * x.w;
          if (!LO) {
            const float top = fmaxf(fmaxf(fabsf(x.x), fabsf(x.y)), fmaxf(fabsf(x.z), fabsf(x.w)));
            // adding 1.5 2^23 rounds to an integer (of small values; larger ones fail the other test)
            const float e = fabsf(((x.x + 12582912.0f) - 12582912.0f) - x.x) + fabsf(((x.y + 12582912.0f) - 12582912.0f) - x.y) +
                            fabsf(((x.z + 12582912.0f) - 12582912.0f) - x.z) + fabsf(((x.w + 12582912.0f) - 12582912.0f) - x.w);
            rounded = rounded || !(e == 0.0f && top <= 256.0f);
          }
        }
      }
      if (norm2 || !LO) {
#pragma unroll
        for (int j = 0; j < kAtOnce; ++j) {
          const float t = warp_sum(s[j]);
          rounded = rounded || !(t < kExactNorm2);
          if (norm2 && r0 + j < n) {
            if (lane == 0) norm2[r0 + j] = t;
            most = max(most, __float_as_uint(t));
          }
        }
      }
    }
    if (!FIND) break;
  }
  if (!LO && __any_sync(kFull, rounded) && lane == 0) *inexact = 1u;
  if (norm2 && lane == 0 && most) atomicMax(xmax, most);
}

// The tiles of one launch: qt x bt, handed out in contiguous shares to G CTAs: equal ones, or
// (`whole`) equal numbers of slices of a query tile's base rows.  A candidate list covers the
// part of one share, one query tile and one slice: a segment.
struct TcShare {
  long long units;  // qt * bt
  int bt, G;
  int Ge;           // CTAs of equal shares (G itself where the shares are not whole slices)
  int st, ns;       // tiles per slice, slices per query tile (st >= bt, 1: not sliced)
  int whole;
  __host__ __device__ long long start(int c, bool by_slices) const {
    if (!by_slices) return units * min(c, Ge) / Ge;
    const long long s = units / bt * ns * min(c, G) / G;  // the share's first slice
    return s / ns * bt + s % ns * st;
  }
  // the CTA whose share holds unit u (equal shares)
  __host__ __device__ int cta_of(long long u) const { return (int)(((u + 1) * Ge - 1) / units); }
  int ctas() const { return G > Ge ? G : Ge; }
  // the list of the segment of CTA c that ends with unit u, among its query tile's lists: from
  // one segment to the next the slice, the CTA or both go up
  __host__ __device__ int list_of(long long u, int c, long long cut, bool by_slices) const {
    const long long q0 = u / bt * bt;
    return (int)((u - q0) / cut) + (by_slices ? 0 : c - cta_of(q0));
  }
  // most lists of one query tile
  __host__ int max_segments() const {
    int most = 1;
    if (!whole)
      for (long long q = 0; q * bt < units; ++q) {
        const int s = cta_of(q * bt + bt - 1) - cta_of(q * bt) + 1;
        if (s > most) most = s;
      }
    return most + ns - 1;
  }
};

struct TcArgs {
  const float* xnorm;
  long long n, nq;
  TcShare share;
  int kchunks;       // pitch / 64
  int cand;          // candidates kept per query per segment
  int stages;        // shared-memory ring depth (2..kMaxStages)
  uint32_t row0;     // id of the launch's first base row
  int nseg, seg0;    // segments per query in `out`, and the launch's first
  uint64_t* out;     // [nq][nseg][cand] (ordered(approx) << 32 | id), prefilled with kNoKey
  const unsigned* inexact;  // 0: no score is rounded, and a list may go on past its slice
  int equal;         // and the shares are equal ones all the same
  int* err;
};

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// the epilogue warps that serve one quarter of the rows (one warp, or two)
template <int EW>
__device__ __forceinline__ void quarter_sync(int quarter) {
  if (EW == 4) __syncwarp();
  else asm volatile("bar.sync %0, 64;" ::"r"(1 + quarter) : "memory");
}

__device__ __forceinline__ void tmem_ld(uint32_t (&v)[8], uint32_t taddr) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld(uint32_t (&v)[16], uint32_t taddr) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr));
}

// Wait for the warp's tensor-memory loads; the registers pass through, so that no use of
// them can be moved above the wait.
__device__ __forceinline__ void tmem_wait(uint32_t (&v)[8]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7])
               :
               : "memory");
}
__device__ __forceinline__ void tmem_wait(uint32_t (&v)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]),
                 "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15])
               :
               : "memory");
}

// A row's candidate list is a max-heap of `cand` keys (root = the worst kept key) and, per
// epilogue warp that serves the row, a buffer of a few (score, id) pairs that were
// below the root's score when they came; all with a stride of one slot per row.  Emptying
// the buffer: the pairs that still beat the root replace it and sift down.  Returns the
// root.  One copy of the code (the screening loop has to stay in the instruction cache).
__device__ __noinline__ uint64_t heap_insert(uint64_t* heap, const uint2* pend, int cand, int waiting) {
  uint64_t worst = heap[0];
  for (int p = 0; p < waiting; ++p) {
    const uint2 w = pend[(size_t)p * kRows];
    const uint64_t key = ((uint64_t)ordered(__uint_as_float(w.x)) << 32) | w.y;
    if (key >= worst) continue;
    int i = 0;
    for (;;) {
      const int l = 2 * i + 1;
      if (l >= cand) break;
      const int r = l + 1;
      const uint64_t hl = heap[(size_t)l * kRows];
      const uint64_t hr = r < cand ? heap[(size_t)r * kRows] : 0ull;
      const bool right = r < cand && hr > hl;
      const uint64_t hc = right ? hr : hl;
      if (hc <= key) break;
      heap[(size_t)i * kRows] = hc;
      i = right ? r : l;
    }
    heap[(size_t)i * kRows] = key;
    worst = heap[0];
  }
  return worst;
}

// The two warps that serve the same 32 rows take turns at their heaps.  The holder never
// waits for anything, so the lock is free again after one emptying; the attempts are
// bounded all the same (false: gave up).
__device__ __forceinline__ bool lock_rows(int* lock, int lane) {
  int got = 0;
  for (int i = 0; i < (1 << 22); ++i) {
    if (lane == 0) got = atomicCAS(lock, 0, 1) == 0;
    got = __shfl_sync(kFull, got, 0);
    if (got) break;
    __nanosleep(64);
  }
  __threadfence_block();
  return got != 0;
}
__device__ __forceinline__ void unlock_rows(int* lock, int lane) {
  __threadfence_block();
  __syncwarp();
  if (lane == 0) atomicExch(lock, 0);
}

// ORDERED: one warp per row, so that the columns arrive in order and a score equal to the
// worst kept one never enters.
template <bool ORDERED>
struct RowList {
  // no score yet: above every finite one, and not passed by +inf (a column past the base)
  static constexpr float kNoWorst = ORDERED ? INFINITY : FLT_MAX;
  uint64_t* heap;
  uint2* pend;
  int* lock;            // null: one warp per row
  volatile int* failed;  // set when a lock could not be had
  int cand;
  int waiting;
  float worst_f;        // the root's score when this warp last saw it (never below the root's now)
  float below_f;        // the next lower score,
  uint32_t worst_id;    // and the root's id

  // warp-wide
  __device__ __forceinline__ void flush() {
    const int lane = threadIdx.x & 31;
    if (lock && !lock_rows(lock, lane)) {
      *failed = 1;
      waiting = 0;
      return;
    }
    const uint64_t worst = heap_insert(heap, pend, cand, waiting);
    waiting = 0;
    worst_f = worst == kNoKey ? kNoWorst : key_score(worst);
    if (!ORDERED) {
      below_f = worst_f == 0.0f ? -FLT_TRUE_MIN : key_score(worst - (1ull << 32));
      worst_id = (uint32_t)worst;
    }
    if (lock) unlock_rows(lock, lane);
  }
};

// One group of scores of the row: a group whose best is not below any row's worst kept score
// costs a fused multiply-add and a minimum per column.  A score equal to the worst kept one
// enters by a lower id (the two halves' columns do not arrive in order); on a base of equal
// rows all others stop here (300,000 x 100, 2,000 queries, k = 10: buffered and refused by
// their keys they took 2.38 ms against 0.54).
template <int kGroup, int kPend, bool ORDERED>
__device__ __forceinline__ void screen(const uint32_t (&v)[kGroup], const float* xn, uint32_t id0, RowList<ORDERED>& L) {
  float sc[kGroup];
#pragma unroll
  for (int u = 0; u < kGroup; u += 4) {
    const float4 x = *reinterpret_cast<const float4*>(xn + u);
    sc[u] = __fmaf_rn(-2.0f, __uint_as_float(v[u]), x.x);  // +inf past the base
    sc[u + 1] = __fmaf_rn(-2.0f, __uint_as_float(v[u + 1]), x.y);
    sc[u + 2] = __fmaf_rn(-2.0f, __uint_as_float(v[u + 2]), x.z);
    sc[u + 3] = __fmaf_rn(-2.0f, __uint_as_float(v[u + 3]), x.w);
  }
  float best = sc[0];
#pragma unroll
  for (int u = 1; u + 1 < kGroup; u += 2) best = fminf(best, fminf(sc[u], sc[u + 1]));
  best = fminf(best, sc[kGroup - 1]);
  if (!__any_sync(kFull, ORDERED ? best < L.worst_f : best <= L.worst_f)) return;
  if (__any_sync(kFull, L.waiting > kPend - kGroup)) L.flush();
  const float most = !ORDERED && id0 > L.worst_id ? L.below_f : L.worst_f;  // equal scores by a lower id only
#pragma unroll
  for (int u = 0; u < kGroup; ++u) {
    if (ORDERED ? sc[u] < most : sc[u] <= most) {
      L.pend[(size_t)L.waiting * kRows] = make_uint2(__float_as_uint(sc[u]), id0 + (uint32_t)u);
      ++L.waiting;
    }
  }
}

// Warp-specialised: EW epilogue warps read the accumulator (warp w the w % 4-th quarter of
// the tensor-memory lanes, one query row per lane; with 8 warps each takes half of the
// columns) and keep the candidates; the next warp issues the TMA loads; the last one the
// MMAs into one of two accumulators (512 tensor-memory columns), so the MMAs of one tile run
// while the epilogue reads the tile before.  ARES: the query tile's chunks are loaded once
// per segment and stay in shared memory.
//
// What bounds it (1M x 128 rows, 10,000 queries, k = 10: 309k tiles, 0.57 us each at the
// measured BF16 rate): the whole call takes 4.5 ms, 3.2 ms with nothing ever entering a list;
// before, one tile at a time per SM behind one row of insertions, 9.2 ms.  Screening has to
// stay in the instruction cache (all insertion code in one place: 13.3 -> 5.9 ms), two
// epilogue warps per scheduler hide each other's tensor-memory loads (5.9 -> 5.3), and
// without a barrier per tile they drift past each other's insertions (5.3 -> 4.5).  Equal
// shares of the tiles replace whole query tiles x base slices, whose last wave was half
// empty.  16 epilogue warps measured 4.7 ms, groups of 8 / 32 columns 5.4 / 4.6.
template <bool PRECISE, bool ARES, int EW>
__global__ void __launch_bounds__((EW + 2) * 32, 1) knn_tc_kernel(const __grid_constant__ CUtensorMap tq,
                                                                const __grid_constant__ CUtensorMap tx, TcArgs a) {
  constexpr int kEpi = EW * 32, kHalves = EW / 4, kTmaWarp = EW, kMmaWarp = EW + 1;
  constexpr int kGroup = group_cols(EW), kPend = pend_slots(EW);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  // 1024-byte alignment for the swizzled tiles
  unsigned char* sm = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
  const int S = a.stages, KC = a.kchunks;
  const int na = ARES ? KC * (PRECISE ? 2 : 1) : S;        // query chunks in shared memory
  unsigned char* sA = sm;                                  // na x 16 KB
  unsigned char* sB = sA + na * kABytes;                   // S x 32 KB
  uint64_t* keys = reinterpret_cast<uint64_t*>(sB + S * kBBytes);  // [cand][128]
  uint2* pend = reinterpret_cast<uint2*>(keys + (size_t)a.cand * kRows);            // [kHalves][kPend][128]
  uint64_t* bars = reinterpret_cast<uint64_t*>(pend + (size_t)kHalves * kPend * kRows);  // full[S], empty[S], acc_full[2], acc_empty[2], a_full, a_empty
  uint64_t* full = bars;
  uint64_t* empty = bars + S;
  uint64_t* accf = bars + 2 * S;
  uint64_t* acce = accf + 2;
  uint64_t* afull = acce + 2;
  uint64_t* aempty = afull + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(aempty + 1);
  __shared__ volatile int s_fail;
  __shared__ int s_lock[4];            // heaps of each quarter's rows
  __shared__ __align__(16) float s_xn[EW][kTcN / kHalves];  // per epilogue warp: ||x||^2 of its columns' base rows

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int bt = a.share.bt;
  const bool exact = PRECISE || __ldg(a.inexact) == 0u;
  const bool by_slices = !PRECISE && a.share.whole && !(exact && a.equal);
  const long long u0 = a.share.start(blockIdx.x, by_slices), u1 = a.share.start(blockIdx.x + 1, by_slices);

  if (tid == 0) {
    s_fail = 0;
    for (int l = 0; l < 4; ++l) s_lock[l] = 0;
    for (int s = 0; s < S; ++s) {
      mbar_init(full + s, 1);
      mbar_init(empty + s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(accf + b, 1);
      mbar_init(acce + b, EW);
    }
    mbar_init(afull, 1);
    mbar_init(aempty, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(kAccCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  // the steps of one 64-element chunk: which query part (hi 0, lo 1) meets which base part;
  // with the query chunks resident a base chunk serves every query part it meets
  constexpr int kSteps = PRECISE ? (ARES ? 2 : 3) : 1;
  if (warp == kTmaWarp) {
    if (lane == 0) {
      uint32_t it = 0, seg = 0;
      bool ok = true;
      for (long long u = u0; u < u1 && ok; ++seg) {
        const long long qt = u / bt, ue = min(u1, (qt + 1) * bt);
        if (ARES) {
          if (seg > 0 && !mbar_wait(aempty, (seg - 1) & 1)) {
            ok = false;
            break;
          }
          mbar_expect_tx(afull, (uint32_t)(na * kABytes));
          for (int c = 0; c < na; ++c) tma_load_2d(sA + c * kABytes, &tq, afull, c * kTcK, (int)(qt * kTcM));
        }
        for (; u < ue && ok; ++u) {
          if (s_fail) {
            ok = false;
            break;
          }
          const int r0 = (int)((u - qt * bt) * kTcN);
          for (int kc = 0; kc < KC && ok; ++kc) {
#pragma unroll
            for (int st = 0; st < kSteps; ++st, ++it) {
              const int s = it % S;
              const uint32_t use = it / S;
              if (use > 0 && !mbar_wait(empty + s, (use - 1) & 1)) {
                ok = false;
                break;
              }
              const int xpart = PRECISE ? (ARES ? st : st == 2) : 0;
              const int qpart = PRECISE && !ARES && st == 1;
              mbar_expect_tx(full + s, ARES ? kBBytes : kABytes + kBBytes);
              if (!ARES) tma_load_2d(sA + s * kABytes, &tq, full + s, (qpart * KC + kc) * kTcK, (int)(qt * kTcM));
              tma_load_2d(sB + s * kBBytes, &tx, full + s, (xpart * KC + kc) * kTcK, r0);
            }
          }
        }
        u = ue;
      }
      if (!ok) s_fail = 1;
    }
  } else if (warp == kMmaWarp) {
    if (lane == 0) {
      const uint32_t idesc = idesc_bf16(kTcM, kTcN);
      uint32_t it = 0, seg = 0, t = 0;
      bool ok = true;
      for (long long u = u0; u < u1 && ok; ++seg) {
        const long long qt = u / bt, ue = min(u1, (qt + 1) * bt);
        if (ARES && !mbar_wait(afull, seg & 1)) {
          ok = false;
          break;
        }
        for (; u < ue && ok; ++u, ++t) {
          const uint32_t b = t & 1, ub = t >> 1;
          if (s_fail || (ub > 0 && !mbar_wait(acce + b, (ub - 1) & 1))) {  // the epilogue is done with this accumulator
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t dacc = tmem + b * kTcN;
          uint32_t acc = 0;  // the tile's first MMA overwrites the accumulator
          auto mma = [&](const unsigned char* pa, const unsigned char* pb) {
#pragma unroll
            for (int k16 = 0; k16 < kTcK / 16; ++k16) {
              const uint64_t da = smem_desc_sw128(pa + k16 * 32);
              const uint64_t db = smem_desc_sw128(pb + k16 * 32);
              asm volatile(
                  "{\n\t.reg .pred p;\n\t"
                  "setp.ne.b32 p, %4, 0;\n\t"
                  "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(dacc),
                  "l"(da), "l"(db), "r"(idesc), "r"(acc));
              acc = 1;
            }
          };
          for (int kc = 0; kc < KC && ok; ++kc) {
#pragma unroll
            for (int st = 0; st < kSteps; ++st, ++it) {
              const int s = it % S;
              if (!mbar_wait(full + s, (it / S) & 1)) {
                ok = false;
                break;
              }
              asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
              if (ARES) {
                mma(sA + kc * kABytes, sB + s * kBBytes);
                if (PRECISE && st == 0) mma(sA + (KC + kc) * kABytes, sB + s * kBBytes);
              } else {
                mma(sA + s * kABytes, sB + s * kBBytes);
              }
              asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                               smem_u32(empty + s))
                           : "memory");
            }
          }
          if (!ok) break;
          asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                           smem_u32(accf + b))
                       : "memory");
        }
        if (ARES && ok && ue < u1)  // the segment's MMAs are done with the query chunks
          asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                           smem_u32(aempty))
                       : "memory");
        u = ue;
      }
      if (!ok) s_fail = 1;
    }
  } else {
    // epilogue: a lane owns accumulator row `row` (query qt * 128 + row), shared with the
    // warp of the other half
    const int quarter = warp & 3, half = warp >> 2, row = quarter * 32 + lane;
    constexpr int kCols = kTcN / kHalves;
    using List = RowList<kHalves == 1>;
    List list{keys + row, pend + (size_t)half * kPend * kRows + row, kHalves > 1 ? &s_lock[quarter] : nullptr,
              &s_fail, a.cand, 0, List::kNoWorst, List::kNoWorst, 0xffffffffu};
    uint32_t t = 0;
    bool ok = true;
    // ||x||^2 of the warp's columns of the next tile, loaded a tile ahead
    constexpr int kNorms = kCols / 32;
    float xn[kNorms];
    float* my_xn = s_xn[warp];
    auto load_norms = [&](int tile) {  // tile of the base
      const long long r = (long long)tile * kTcN + half * kCols + lane;
#pragma unroll
      for (int j = 0; j < kNorms; ++j) xn[j] = r + 32 * j < a.n ? __ldg(a.xnorm + r + 32 * j) : INFINITY;
    };
    if (u0 < u1) load_norms((int)(u0 % bt));
    const long long st = exact ? bt : a.share.st;
    for (long long u = u0; u < u1;) {
      const long long qt = u / bt, qe = (qt + 1) * bt;
      const long long ue = min(min(u1, qe), qt * bt + ((u - qt * bt) / st + 1) * st);
      for (int i = half; i < a.cand; i += kHalves) list.heap[(size_t)i * kRows] = kNoKey;
      list.worst_f = List::kNoWorst;
      list.worst_id = 0xffffffffu;
      quarter_sync<EW>(quarter);
      // after a failed wait the warp only keeps up with its barriers
      for (; u < ue && ok; ++u, ++t) {
        const uint32_t b = t & 1;
        const uint32_t id0 = a.row0 + (uint32_t)((u - qt * bt) * kTcN) + half * kCols;
#pragma unroll
        for (int j = 0; j < kNorms; ++j) my_xn[lane + 32 * j] = xn[j];
        if (u + 1 < u1) load_norms(u + 1 < qe ? (int)(u + 1 - qt * bt) : 0);
        if (!mbar_wait(accf + b, (t >> 1) & 1)) s_fail = 1;
        __syncwarp();
        ok = !__any_sync(kFull, s_fail != 0);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16) + b * kTcN + half * kCols;
        // two loads in flight: one is screened while the next arrives
        uint32_t va[kGroup], vb[kGroup];
        tmem_ld(va, taddr);  // warp-collective
        tmem_wait(va);
#pragma unroll 1
        for (int c0 = 0; c0 < kCols; c0 += 2 * kGroup) {
          tmem_ld(vb, taddr + c0 + kGroup);
          screen<kGroup, kPend, kHalves == 1>(va, my_xn + c0, id0 + c0, list);
          __syncwarp();
          tmem_wait(vb);
          if (c0 + 2 * kGroup < kCols) tmem_ld(va, taddr + c0 + 2 * kGroup);
          screen<kGroup, kPend, kHalves == 1>(vb, my_xn + c0 + kGroup, id0 + c0 + kGroup, list);
          __syncwarp();
          tmem_wait(va);
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(acce + b);  // this warp is done with the accumulator
      }
      u = ue;
      list.flush();
      quarter_sync<EW>(quarter);
      if (ok && qt * kTcM + row < a.nq) {
        const int seg = a.seg0 + a.share.list_of(ue - 1, blockIdx.x, by_slices ? a.share.st : st, by_slices);
        uint64_t* o = a.out + ((size_t)(qt * kTcM + row) * a.nseg + seg) * a.cand;
        for (int i = half; i < a.cand; i += kHalves) o[i] = list.heap[(size_t)i * kRows];
      }
      quarter_sync<EW>(quarter);  // the lists are written before they are emptied for the next query tile
    }
  }
  __syncthreads();
  if (s_fail && tid == 0) atomicExch(a.err, 1);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == kMmaWarp)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kAccCols));
}

struct FinArgs {
  const float* X;
  const float* Q;
  long long nq;
  int d;
  const uint64_t* cand;  // [nq][nseg][cand]
  int nseg, ncand1;      // segments, candidates per segment
  int P;                 // power of two >= nseg * ncand1
  int k;
  int32_t* ids_out;
  float* dists_out;
  const unsigned* xmax;  // bits of the largest ||x||^2
  const float* centre;   // precise form: what was taken off rows and queries
  float c_dot;           // |score error| <= c_dot ||q|| ||x|| + c_norm ||x||^2 + c_q ||q||^2
  float c_norm, c_q;
  float reach;           // see `radius` below
  // precise form: queries whose result is not proven
  const int* err;
  int* left_count;
  int32_t* left;
};

// One group of WPQ warps per query.
template <int WPQ>
__device__ __forceinline__ void group_sync() {
  if (WPQ == 1) __syncwarp();
  else __syncthreads();
}

template <int WPQ>
__device__ __forceinline__ void group_sort(uint64_t* key, int P, int t) {
  for (int size = 2; size <= P; size <<= 1) {
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      for (int i = t; i < (P >> 1); i += WPQ * 32) {
        const int lo = 2 * i - (i & (stride - 1));
        const int hi = lo + stride;
        const uint64_t x = key[lo], y = key[hi];
        if ((x > y) == ((lo & size) == 0)) {
          key[lo] = y;
          key[hi] = x;
        }
      }
      group_sync<WPQ>();
    }
  }
}

constexpr int kFinWarps = 4;      // warps per CTA where a warp takes a query
constexpr int kFinGroupWarps = 8;  // where a CTA takes one
template <int WPQ, bool PRECISE>
__global__ void __launch_bounds__((WPQ == 1 ? kFinWarps : WPQ) * 32) knn_tc_finalize(FinArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int kQueries = WPQ == 1 ? kFinWarps : 1;  // per CTA
  // 16-byte pieces of a candidate's row loaded at a time, 4 / 8: a warp per query 1.32 / 1.42 ms
  // (65,536 x 960, 10,000 queries, k = 100; 1.3 to 2.3 where the compiler chooses), a CTA per query
  // 0.239 / 0.219 (300,000 x 100, 2,000 queries, k = 100)
  constexpr int kAhead = WPQ == 1 ? 4 : 8;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t = WPQ == 1 ? lane : threadIdx.x;
  uint64_t* s_key = reinterpret_cast<uint64_t*>(smem_raw) + (size_t)(WPQ == 1 ? warp : 0) * a.P;
  const int d = a.d, d4 = d >> 2, ncand = a.nseg * a.ncand1;
  const float xm2 = __uint_as_float(*a.xmax), xm = 1.00001f * sqrtf(xm2);
  for (long long q = (long long)blockIdx.x * kQueries + (WPQ == 1 ? warp : 0); q < a.nq; q += (long long)gridDim.x * kQueries) {
    const float4* qv = reinterpret_cast<const float4*>(a.Q + (size_t)q * d);
    // ||q||^2 (less the centre), the same in every warp
    double q2 = 0.0;
    for (int c = lane; c < d4; c += 32) {
      float4 v = __ldg(qv + c);
      if (PRECISE) {
        const float4 ce = __ldg(reinterpret_cast<const float4*>(a.centre) + c);
        v = make_float4(v.x - ce.x, v.y - ce.y, v.z - ce.z, v.w - ce.w);
      }
      q2 += (double)v.x * v.x + (double)v.y * v.y + (double)v.z * v.z + (double)v.w * v.w;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) q2 += __shfl_xor_sync(kFull, q2, o);
    const float qn = 1.00001f * sqrtf((float)q2);
    // The score's error for a row of norm up to r.  Only rows near the query matter: one of norm
    // N > 2 (||q|| + sqrt(D)) lies N / 2 + sqrt(D) or more from the query, beyond a distance of D
    // whatever its score's error, and scores above D - ||q||^2 as long as that error is below
    // N^2 / 4 (reach: 2, or infinity where it may not be).  So one long row does not widen the bound.
    // Both in FP32, rounded up, with room for values that underflow (in FP64, which is slow here,
    // 6.27 ms against 6.10: 65,536 x 960, 10,000 queries, k = 100).
    auto error_to = [&](float r) { return 1.0001f * (a.c_dot * qn * r + a.c_norm * r * r + a.c_q * qn * qn) + 1e-30f; };
    auto radius = [&](double D) { return fminf(xm, a.reach * (qn + 1.0001f * sqrtf(fmaxf((float)D, 0.0f))) + 1e-12f); };
    const uint64_t* src = a.cand + (size_t)q * ncand;
    int P = a.P;
    if (WPQ == 1 && !PRECISE) {  // the filled slots alone
      int have = 0;
      for (int i0 = 0; i0 < ncand; i0 += 32) {
        const uint64_t key = i0 + lane < ncand ? src[i0 + lane] : kNoKey;
        const unsigned m = __ballot_sync(kFull, key != kNoKey);
        if (key != kNoKey) s_key[have + __popc(m & ((1u << lane) - 1u))] = key;
        have += __popc(m);
      }
      P = 1;
      while (P < have || P < a.k) P <<= 1;
      for (int i = have + lane; i < P; i += 32) s_key[i] = kNoKey;
    } else {
      for (int i = t; i < P; i += WPQ * 32) s_key[i] = i < ncand ? src[i] : kNoKey;
    }
    // the smallest root of a full list: no row left out scored below it
    uint64_t left_out = kNoKey;
    if (PRECISE) {
      for (int i = lane; i < a.nseg; i += 32) left_out = min(left_out, src[(size_t)i * a.ncand1]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) left_out = min(left_out, (uint64_t)__shfl_xor_sync(kFull, (unsigned long long)left_out, o));
    }
    group_sync<WPQ>();
    group_sort<WPQ>(s_key, P, t);
    // a candidate more than two error bounds above the k-th score is farther than k others,
    // also in FP32
    const double fp = (double)(d + 4) * 0x1p-23;
    const uint64_t kth = s_key[a.k - 1];
    double thr = INFINITY;
    if (kth != kNoKey) {
      const double S = (double)key_score(kth), err = (double)error_to(radius(S + q2)), D = S + err + q2;
      thr = S + err + (double)error_to(radius(D)) + fp * fabs(D);
    }
    int m = 0;  // candidates to measure: the first m
    {
      int lo = 0, hi = P;
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        const uint64_t key = s_key[mid];
        if (key != kNoKey && !((double)key_score(key) > thr)) lo = mid + 1; else hi = mid;
      }
      m = lo;
    }
    int P2 = 1;
    while (P2 < m) P2 <<= 1;
    if (P2 < a.k) {
      while (P2 < a.k) P2 <<= 1;
      P2 = min(P2, P);
    }
    group_sync<WPQ>();
    for (int i = t; i < P2; i += WPQ * 32) {
      uint64_t key = kNoKey;
      if (i < m) {
        const uint32_t id = (uint32_t)(s_key[i] & 0xffffffffu);
        const float4* xv = reinterpret_cast<const float4*>(a.X + (size_t)id * d);
        float acc = 0.0f;
        auto add = [&](const float4& x, const float4& y) {
          const float e0 = y.x - x.x, e1 = y.y - x.y, e2 = y.z - x.z, e3 = y.w - x.w;
          if (PRECISE) {  // the FFMA kernel's sum
            acc = fmaf(e0, e0, acc);
            acc = fmaf(e1, e1, acc);
            acc = fmaf(e2, e2, acc);
            acc = fmaf(e3, e3, acc);
          } else {
            acc = acc + e0 * e0;
            acc = acc + e1 * e1;
            acc = acc + e2 * e2;
            acc = acc + e3 * e3;
          }
        };
        int c = 0;
        for (; c + kAhead <= d4; c += kAhead) {  // the row's pieces in flight together
          float4 x[kAhead];
#pragma unroll
          for (int j = 0; j < kAhead; ++j) x[j] = __ldg(xv + c + j);
#pragma unroll
          for (int j = 0; j < kAhead; ++j) add(x[j], __ldg(qv + c + j));
        }
        for (; c < d4; ++c) add(__ldg(xv + c), __ldg(qv + c));
        key = pack_key(acc, (int32_t)id);
      }
      s_key[i] = key;
    }
    group_sync<WPQ>();
    group_sort<WPQ>(s_key, P2, t);
    for (int j = t; j < a.k; j += WPQ * 32) {
      const uint64_t key = j < P2 ? s_key[j] : kNoKey;
      a.ids_out[(size_t)q * a.k + j] = key == kNoKey ? -1 : key_id(key);
      a.dists_out[(size_t)q * a.k + j] = key == kNoKey ? INFINITY : key_dist(key);
    }
    if (PRECISE && t == 0) {
      // below 1e37 no score, no BF16 term and no distance overflows (|q.x| <= ||q|| ||x||); a
      // score that did would have entered no list
      bool proven = *a.err == 0 && xm2 >= 1e-24f && xm2 < 1e37f && (q2 >= 1e-24 || q2 == 0.0) && q2 < 1e37;
      if (left_out != kNoKey) {
        const uint64_t last = s_key[a.k - 1];
        proven = proven && last != kNoKey &&
                 ((double)key_score(left_out) - (double)error_to(radius((double)key_dist(last))) + q2) * (1.0 - fp) >
                     (double)key_dist(last) * (1.0 + 0x1p-20);
      }
      if (!proven) a.left[atomicAdd(a.left_count, 1)] = (int32_t)q;
    }
    group_sync<WPQ>();
  }
}

using EncodeTiled = PFN_cuTensorMapEncodeTiled_v12000;

EncodeTiled encode_fn() {
  static std::mutex mu;
  static EncodeTiled fn = nullptr;
  std::lock_guard<std::mutex> lock(mu);
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiled>(p);
  }
  return fn;
}

// 2-D tensor map over a BF16 matrix of `rows` rows of `pitch` elements; box = box_k x box_rows,
// 128-byte swizzle.
bool make_map(CUtensorMap* m, const void* base, long long rows, int pitch, int box_rows) {
  EncodeTiled enc = encode_fn();
  if (!enc) return false;
  cuuint64_t dims[2] = {(cuuint64_t)pitch, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)pitch * 2};
  cuuint32_t box[2] = {(cuuint32_t)kTcK, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

namespace {

constexpr size_t kTcPad = 256;
size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }
int tc_pitch(int d) { return (d + kTcK - 1) / kTcK * kTcK; }

// The plan of one call: how the tiles are shared and what the scratch holds.
struct TcPlan {
  int pitch, cand, nseg, slabs, most_cand;
  long long slab_rows;  // base rows converted at a time
  TcShare share;        // of a full slab
  int equal;            // see equal_if_exact
  size_t xb, qb, xnorm, cand_buf, centre, flags, total;  // scratch offsets
};

// cost of a list's start in tiles: it takes about cand (1 + ln(rows / cand)) insertions
double list_tiles(double rows, int cand) { return 64.0 * (rows > cand ? 1.0 + log(rows / cand) : 1.0); }

// The slices of the base whose best `cand` rows a query keeps where scores are rounded (that
// many lists are what absorbs misranked rows; with the lists of the CTAs' shares alone, as few
// as one, 6 of 20,000 queries over 1M x 100 unit vectors lost one of their 10 nearest): the
// number that would be quickest with a CTA per slice and query tile, among slices of at least
// 4 tiles.
int tc_slices(long long n, long long qt, int cand, int sms) {
  const long long most = std::max(1LL, std::min((n + 4LL * kTcN - 1) / (4LL * kTcN), (long long)kMaxCandTotal / cand));
  long long best = 1;
  double best_cost = -1.0;
  for (long long s = 1; s <= most; ++s) {
    const double rows = (double)((n + s - 1) / s);
    const double cost = (double)((qt * s + sms - 1) / sms) * (ceil(rows / kTcN) + list_tiles(rows, cand));
    if (best_cost < 0.0 || cost < best_cost) {
      best_cost = cost;
      best = s;
    }
  }
  return (int)best;
}

TcShare tc_share(long long n, long long nq, int cand, int slabs, bool precise, int most_cand, int sms) {
  TcShare s;
  const long long qt = (nq + kTcM - 1) / kTcM;
  s.bt = (int)((n + kTcN - 1) / kTcN);
  s.units = qt * s.bt;
  s.st = s.bt;
  s.ns = 1;
  s.whole = 0;
  if (!precise) {
    const int want = tc_slices(n, qt, cand, sms);
    s.st = (int)(((n + want - 1) / want + kTcN - 1) / kTcN);
    s.ns = (s.bt + s.st - 1) / s.st;
  }
  // one CTA per SM; no more than most_cand candidates per query over its segments (a
  // query tile's share spans at most ceil(G / qt) + 1 CTAs), and segments of at least 4
  // tiles, below which the lists' start-up would outweigh the tiles
  long long G = sms;
  const long long most = most_cand / ((long long)cand * slabs);
  const long long room = most - s.ns + 1;  // lists of a query tile beside its slices' own
  if (room >= 2) G = std::min(G, std::max(1LL, (room - 1) * qt));
  else G = std::min(G, qt);
  G = std::min(G, std::max(1LL, s.units / 4));
  s.G = s.Ge = (int)std::max(1LL, G);
  if (s.ns > 1) {
    // whole slices where their uneven numbers cost less than the lists cut by equal shares
    const double start = list_tiles(256.0 * s.st, cand), slices = (double)(qt * s.ns);
    const int gw = (int)std::min<long long>(sms, qt * s.ns);
    if (room < 2 || ceil(slices / gw) * (s.st + start) <= (double)s.units / s.G + (slices / s.G + 1.0) * start) {
      s.whole = 1;
      s.G = gw;
      // without slices
      s.Ge = (int)std::max(1LL, std::min({(long long)sms, std::max(1LL, (most - 1) * qt), s.units / 4}));
    }
  }
  return s;
}

// Whole slices are for scores that are rounded.  Where none is (the kernel finds out) a list goes
// on past its slice, and equal shares are taken after all if the CTA that has most to do then has
// less: its tiles and its lists' insertions, each about 1.2 tiles' time (integer rows of 128:
// 606,000, 11,863 queries, k = 1 1,580 tiles at most against 1,449, 3,227 us against 3,033;
// 314,000, 6,681 queries, k = 1 614 tiles and one list against 428 and two, 1,399 us against 1,336).
double busiest(const TcShare& s, bool by_slices, int cand) {
  double most = 0.0;
  for (int c = 0; c < s.ctas(); ++c) {
    const long long u1 = s.start(c + 1, by_slices);
    double cost = 0.0;
    for (long long u = s.start(c, by_slices); u < u1;) {
      const long long ue = std::min(u1, (u / s.bt + 1) * s.bt);
      const double rows = 256.0 * (ue - u);
      cost += (double)(ue - u) + 1.2 * cand * (rows > cand ? 1.0 + log(rows / cand) : 1.0);
      u = ue;
    }
    most = std::max(most, cost);
  }
  return most;
}
int equal_segments(TcShare s) {
  s.whole = 0;
  s.ns = 1;
  return s.max_segments();
}
int equal_if_exact(const TcShare& s, int cand, int most_cand) {
  // looked at where the slices' uneven numbers cost 4% of at least 256 tiles a CTA (the sums
  // take some 8 us of the host)
  const long long slices = s.units / s.bt * s.ns, least = (s.units + s.Ge - 1) / s.Ge;
  if (!s.whole || least < 256 || (slices + s.G - 1) / s.G * s.st * 100 < least * 104) return 0;
  return equal_segments(s) * cand <= most_cand && busiest(s, false, cand) < busiest(s, true, cand);
}

// The longest list whose launch fits in shared memory (4 epilogue warps, two stages of query
// and base chunks).  The precise form serves k up to 8 below it: its lists hold 16 more than
// k, fewer where shared memory ends (a shorter slack only proves fewer queries).
constexpr int kMaxCand = 113;

// The precise form's scratch stays within 1 GiB (the bound that peos_knn_bruteforce states):
// the base is converted in slabs of at most 768 MiB, the rest holds queries and lists.
constexpr size_t kExactBytes = (size_t)1 << 30, kExactSlabBytes = (size_t)768 << 20;

// Estimated times of the exact brute force in us, from the measured rates of both forms: per
// tile of 256 rows and 128 queries 0.9 + 2.1 us for every 128 elements of a row (a fifth more
// where the query tile does not stay in shared memory, 1.4 times with 4 epilogue warps), 0.7 us
// per insertion into a list, finalize's sort in steps of 512 keys, and the conversion at
// 5.5 TB/s; a FFMA chunk of 16,384 rows by its 10.4 us per element, by its insertions, and 1.25
// of them at once on an SM.  Against 94 measured shapes (2,048..10M rows, d = 4..960, 1..10,000
// queries, k = 1..105) the FFMA estimates are 0.68..1.30 of the time and the scores' 0.36..1.72
// (lowest for 10,000 queries over few rows, where the other form is far off), and the quicker
// form is chosen in all but one (2,048 x 4, one query, k = 10: 112 us against 94).
double exact_us(const TcPlan& p, long long n, long long nq, int d, int k, int sms) {
  const double qt = (double)((nq + kTcM - 1) / kTcM), G = p.share.G;
  const double wide = p.cand > 84 ? 1.4 : 1.0;  // 4 epilogue warps beside lists that long
  const double tile = (0.9 + 2.1 * p.pitch / 128 * (p.pitch > 256 ? 1.2 : 1.0)) * wide;
  const double rows = std::min((double)p.slab_rows, std::max(256.0, p.slab_rows * qt / G));
  const double ins = p.cand * (1.0 + log(std::max(1.0, rows / p.cand)));
  int lg = 1;
  while ((1 << lg) < p.nseg * p.cand) ++lg;
  const double sort = 0.5 * lg * (lg + 1) * (1 << lg) / 512 * std::max(1.0, (double)nq / sms);
  const double finalize = lg <= 10 && nq >= 2LL * sms ? 0.025 * sort : 0.05 * sort;
  return 65.0 + n * (4.0 * d + 4.0 * p.pitch) / 5.5e6 +
         p.slabs * (p.share.units / G * tile + (G + qt - 1.0) / G * 0.7 * ins) + finalize;
}
double ffma_us(long long n, long long nq, int d, int k, int sms) {
  const double rows = (double)std::min(n, 16384LL), ctas = (double)((n + 16383) / 16384) * ((nq + 31) / 32);
  const double chunk = rows / 16384 * (10.4 * d + 90.0) + k * (1.0 + log(std::max(1.0, rows / k))) * (0.6 + 0.008 * k);
  return 45.0 + chunk * std::max(1.0, ctas / sms / 1.25);
}

// False: not served.
bool tc_plan(long long n, long long nq, int d, int k, bool precise, int sms, TcPlan* p) {
  p->pitch = tc_pitch(d);
  p->cand = precise ? std::min(k + 16, kMaxCand) : k + 16;
  if (p->cand < k + 8 || p->cand > kMaxCand) return false;
  const size_t row = (size_t)p->pitch * 2 * (precise ? 2 : 1);
  p->slab_rows = n;
  p->slabs = 1;
  if (precise) {
    const long long fit = std::max<long long>(kTcN, (long long)(kExactSlabBytes / row) / kTcN * kTcN);
    p->slabs = (int)((n + fit - 1) / fit);
    p->slab_rows = p->slabs > 1 ? fit : n;
  }
  bool served = false;
  TcPlan best = *p;
  for (int most = kMaxCandTotal; most <= (precise ? 4 : 1) * kMaxCandTotal; most *= 2) {
    p->most_cand = most;
    p->share = tc_share(p->slab_rows, nq, p->cand, p->slabs, precise, most, sms);
    p->equal = equal_if_exact(p->share, p->cand, most);
    int seg = std::max(p->share.max_segments(), p->equal ? equal_segments(p->share) : 0);
    if (p->slabs > 1) {
      const TcShare last = tc_share(n - (long long)(p->slabs - 1) * p->slab_rows, nq, p->cand, p->slabs, precise, most, sms);
      seg = std::max(seg, last.max_segments());
    }
    p->nseg = seg * p->slabs;
    if ((long long)p->nseg * p->cand > most && p->nseg > 1) continue;
    if (!served || exact_us(*p, n, nq, d, k, sms) < exact_us(best, n, nq, d, k, sms)) best = *p;
    served = true;
  }
  if (!served) return false;
  *p = best;
  size_t o = 0;
  p->xb = o;
  o += up256((size_t)p->slab_rows * row);
  p->qb = o;
  o += up256((size_t)nq * row);
  p->xnorm = o;
  o += up256((size_t)p->slab_rows * 4);
  p->cand_buf = o;
  o += up256((size_t)nq * p->nseg * p->cand * 8);
  p->centre = o;
  if (precise) o += up256((size_t)p->pitch * 4);
  p->flags = o;  // xmax, inexact
  o += kTcPad;
  p->total = o;
  return true;
}

template <bool PRECISE, bool ARES, int EW>
cudaError_t launch_tc(const CUtensorMap& mq, const CUtensorMap& mx, TcArgs ta, int maxsm, cudaStream_t st, bool* fits) {
  auto fn = knn_tc_kernel<PRECISE, ARES, EW>;
  cudaFuncAttributes fa;
  cudaError_t e = cudaFuncGetAttributes(&fa, fn);
  if (e != cudaSuccess) return e;
  const size_t room = (size_t)maxsm - fa.sharedSizeBytes;  // the kernel's static shared memory comes off the top
  // as many ring stages as fit beside the lists and the resident query chunks (one CTA per SM
  // either way: the two accumulators take all 512 tensor-memory columns)
  const size_t fixed = 1024 + (size_t)(ta.cand + EW / 4 * pend_slots(EW)) * kRows * 8 + (2 * kMaxStages + 6) * 8 + 16 +
                       (ARES ? (size_t)ta.kchunks * (PRECISE ? 2 : 1) * kABytes : 0);
  const size_t stage = kBBytes + (ARES ? 0 : kABytes);
  int stages = kMaxStages;
  const int least = ARES ? 3 : 2;
  while (stages > least && fixed + (size_t)stages * stage > room) --stages;
  size_t smem = fixed + (size_t)stages * stage;
  *fits = smem <= room;
  if (!*fits) return cudaSuccess;
  const size_t one_per_sm = ((size_t)maxsm) / 2 + 1024;  // never two CTAs on one SM
  if (smem < one_per_sm) smem = one_per_sm;
  ta.stages = stages;
  e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  fn<<<(unsigned)ta.share.ctas(), (EW + 2) * 32, smem, st>>>(mq, mx, ta);
  return cudaGetLastError();
}

// The candidate lists and their evaluation; `left` / `left_count` (precise): the queries
// whose result is not proven.
template <bool PRECISE>
cudaError_t run_tc(const TcPlan& p, const float* X, long long n, int d, const float* Q, long long nq, int k,
                   int32_t* ids_out, float* dists_out, unsigned char* w, int* err, int* left_count, int32_t* left,
                   int sms, cudaStream_t st) {
  int dev = 0, maxsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&maxsm, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  __nv_bfloat16* xb = reinterpret_cast<__nv_bfloat16*>(w + p.xb);
  __nv_bfloat16* qb = reinterpret_cast<__nv_bfloat16*>(w + p.qb);
  float* xnorm = reinterpret_cast<float*>(w + p.xnorm);
  uint64_t* cand_buf = reinterpret_cast<uint64_t*>(w + p.cand_buf);
  unsigned* xmax = reinterpret_cast<unsigned*>(w + p.flags);
  float* centre = PRECISE ? reinterpret_cast<float*>(w + p.centre) : nullptr;
  cudaError_t e = cudaMemsetAsync(cand_buf, 0xff, (size_t)nq * p.nseg * p.cand * 8, st);
  if (!PRECISE && e == cudaSuccess) e = cudaMemsetAsync(xmax, 0, 2 * sizeof(unsigned), st);
  if (e != cudaSuccess) return e;
  const int cols = p.pitch * (PRECISE ? 2 : 1);
  const int cg = sms * 8;
  convert_bf16_kernel<PRECISE, PRECISE><<<(unsigned)std::min<long long>(cg, (nq + 31) / 32), kConvertThreads, 0, st>>>(
      Q, nq, d, p.pitch, qb, nullptr, xmax, xmax + 1, centre, X, n, err);
  CUtensorMap mq;
  if (!make_map(&mq, qb, nq, cols, kTcM)) return cudaErrorNotSupported;
  for (int s = 0; s < p.slabs; ++s) {
    const long long r0 = (long long)s * p.slab_rows, rows = std::min(p.slab_rows, n - r0);
    convert_bf16_kernel<PRECISE, false><<<(unsigned)std::min<long long>(cg, (rows + 31) / 32), kConvertThreads, 0, st>>>(
        X + (size_t)r0 * d, rows, d, p.pitch, xb, xnorm, xmax, xmax + 1, centre, nullptr, 0, nullptr);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    CUtensorMap mx;
    if (!make_map(&mx, xb, rows, cols, kTcN)) return cudaErrorNotSupported;
    TcArgs ta;
    ta.xnorm = xnorm;
    ta.n = rows;
    ta.nq = nq;
    ta.share = rows == p.slab_rows ? p.share : tc_share(rows, nq, p.cand, p.slabs, PRECISE, p.most_cand, sms);
    ta.kchunks = p.pitch / kTcK;
    ta.cand = p.cand;
    ta.row0 = (uint32_t)r0;
    ta.nseg = p.nseg;
    ta.seg0 = s * (p.nseg / p.slabs);
    ta.out = cand_buf;
    ta.inexact = xmax + 1;
    ta.equal = p.equal;
    ta.err = err;
    bool fits = false;
    e = launch_tc<PRECISE, true, 8>(mq, mx, ta, maxsm, st, &fits);
    if (e == cudaSuccess && !fits) e = launch_tc<PRECISE, false, 8>(mq, mx, ta, maxsm, st, &fits);
    if (e == cudaSuccess && !fits) e = launch_tc<PRECISE, false, 4>(mq, mx, ta, maxsm, st, &fits);
    if (e == cudaSuccess && !fits) e = cudaErrorInvalidConfiguration;
    if (e != cudaSuccess) return e;
  }
  FinArgs fa{};
  fa.X = X;
  fa.Q = Q;
  fa.nq = nq;
  fa.d = d;
  fa.cand = cand_buf;
  fa.nseg = p.nseg;
  fa.ncand1 = p.cand;
  fa.P = 1;
  while (fa.P < p.nseg * p.cand || fa.P < k) fa.P <<= 1;
  fa.k = k;
  fa.ids_out = ids_out;
  fa.dists_out = dists_out;
  fa.xmax = xmax;
  fa.centre = centre;
  // Score error, relative to ||q|| ||x||: the terms dropped or rounded (BF16's unit roundoff
  // is 2^-8: 2 (2^-8 + 2^-18) alone, 3.05 2^-16 for the two-term sums), and the FP32
  // accumulation, at most 2^-23 per product (each step of 16 aligns its products and the
  // accumulator to the largest and truncates); times 2 for -2 q.x, plus the last rounding.
  // Taking the centre off rounds every element once: x and q move by at most 2^-24 of their
  // norms, their squared distance by 2^-23 (||x|| + ||q||)^2.
  const double products = (double)p.pitch * (PRECISE ? 3 : 1);
  fa.c_dot = (float)(2.0 * ((PRECISE ? 3.05 * 0x1p-16 : 2.02 * 0x1p-8) + products * 0x1p-23) + 0x1p-21);
  fa.c_norm = (float)((d / 32 + 10) * 0x1p-23);
  if (PRECISE) {
    fa.c_dot += 1.01f * 0x1p-22f;
    fa.c_norm += 1.01f * 0x1p-23f;
    fa.c_q = 1.01f * 0x1p-23f;
  }
  fa.reach = 0.5f * fa.c_dot + fa.c_norm + fa.c_q < 0.2f ? 2.0f : INFINITY;
  fa.err = err;
  fa.left_count = left_count;
  fa.left = left;
  // a warp per query, or a CTA per query where the lists are long or the queries few
  if (fa.P <= 1024 && nq >= 2LL * sms) {
    const size_t sm = (size_t)fa.P * 8 * kFinWarps;
    e = cudaFuncSetAttribute(knn_tc_finalize<1, PRECISE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    const long long g = std::min<long long>((nq + kFinWarps - 1) / kFinWarps, (long long)sms * 16);
    knn_tc_finalize<1, PRECISE><<<(unsigned)g, kFinWarps * 32, sm, st>>>(fa);
  } else {
    const size_t sm = (size_t)fa.P * 8;
    e = cudaFuncSetAttribute(knn_tc_finalize<kFinGroupWarps, PRECISE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    const long long g = std::min<long long>(nq, (long long)sms * 8);
    knn_tc_finalize<kFinGroupWarps, PRECISE><<<(unsigned)g, kFinGroupWarps * 32, sm, st>>>(fa);
  }
  return cudaGetLastError();
}

}  // namespace

int knn_tc_max_k() { return kMaxK; }

size_t knn_tc_scratch_bytes(long long n, long long nq, int d, int k, int sms) {
  TcPlan p;
  return tc_plan(n, nq, d, k, false, sms, &p) ? p.total : 0;
}

cudaError_t launch_knn_tc(const float* X, long long n, int d, const float* Q, long long nq, int k, int32_t* ids_out,
                          float* dists_out, void* scratch, int* err_flag, cudaStream_t st) {
  (void)cudaGetLastError();  // start from a clean error state: the launch checks below read it
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  TcPlan p;
  if (!tc_plan(n, nq, d, k, false, sms, &p)) return cudaErrorInvalidConfiguration;
  return run_tc<false>(p, X, n, d, Q, nq, k, ids_out, dists_out, static_cast<unsigned char*>(scratch), err_flag, nullptr,
                       nullptr, sms, st);
}

// ---- exact brute force: the precise form, and the FFMA kernel for what it leaves -----------

namespace {
// the length of the list's part from query `first` on, at most `most`
__global__ void part_count_kernel(const int* __restrict__ count, long long first, long long most, int* __restrict__ part) {
  *part = (int)max(0ll, min(most, *count - first));
}

// what has to outlast the scores: the list of queries left over and its length
size_t left_bytes(long long nq) { return kTcPad + up256((size_t)nq * 4); }
}  // namespace

// Where the FFMA form is quicker the scores do not serve: a few queries over a large base (their
// lists limit the CTAs: 10M x 128, k = 100, 1 / 32 queries 13.1 / 18.2 ms against 8.5 / 8.6;
// 10M x 960, k = 10, one query 76 against 41), and short rows of a small one (2,048 x 4, k = 10,
// 1 / 500 / 10,000 queries 94 / 161 / 284 us against 112 / 130 / 170).
size_t knn_exact_scratch_bytes(long long n, long long nq, int d, int k, int sms) {
  TcPlan p;
  if (!tc_plan(n, nq, d, k, true, sms, &p) || exact_us(p, n, nq, d, k, sms) >= ffma_us(n, nq, d, k, sms)) return 0;
  return left_bytes(nq) + p.total;
}

long long knn_exact_slice(long long n, long long nq, int d, int k, int sms) {
  for (long long parts = 1;; parts *= 2) {
    long long slice = (nq + parts - 1) / parts;
    if (parts > 1) slice = (slice + kTcM - 1) / kTcM * kTcM;
    const size_t bytes = knn_exact_scratch_bytes(n, slice, d, k, sms);
    if (!bytes || bytes <= kExactBytes || slice <= kTcM) return bytes ? slice : 0;
  }
}

cudaError_t launch_knn_exact(const float* X, long long n, int d, const float* Q, long long nq, int k, int32_t* ids_out,
                             float* dists_out, void* scratch, long long ffma_slice, int sms, cudaStream_t st) {
  TcPlan p;
  if (!tc_plan(n, nq, d, k, true, sms, &p)) return cudaErrorInvalidConfiguration;
  int* err = static_cast<int*>(scratch);
  int* left_count = err + 1;
  int32_t* left = reinterpret_cast<int32_t*>(static_cast<unsigned char*>(scratch) + kTcPad);
  unsigned char* w = static_cast<unsigned char*>(scratch) + left_bytes(nq);
  cudaError_t e = run_tc<true>(p, X, n, d, Q, nq, k, ids_out, dists_out, w, err, left_count, left, sms, st);
  // the scores are done with w when these run.  A list that may exceed the FFMA lists' slice is
  // taken part by part, its length in a launch of its own (with the first position as an argument
  // of the FFMA kernel its inner loop came out slower: 32,113 x 960, 1,217 queries, k = 121,
  // 12.38 -> 13.68 ms); parts past the list are empty launches
  if (nq <= ffma_slice)
    return e == cudaSuccess ? launch_knn(X, n, d, Q, nq, k, ids_out, dists_out, w, st, left, left_count) : e;
  int* part = left_count + 1;
  for (long long q = 0; q < nq && e == cudaSuccess; q += ffma_slice) {
    const long long most = std::min(ffma_slice, nq - q);
    part_count_kernel<<<1, 1, 0, st>>>(left_count, q, most, part);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = launch_knn(X, n, d, Q, most, k, ids_out, dists_out, w, st, left + q, part);
  }
  return e;
}

size_t knn_exact_left_bytes(long long nq) { return left_bytes(nq); }

cudaError_t launch_bounded_wait_probe(long long limit_ns, int* gave_up, cudaStream_t st) {
  bounded_wait_probe_kernel<<<1, 32, 0, st>>>(limit_ns, gave_up);
  return cudaGetLastError();
}

}  // namespace peos
