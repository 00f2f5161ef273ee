// FP64 tall-skinny products of the iteration (Sec. 3's O(np^2) part):
//   gram:     out = A^T B (p x q Grams such as E_X^T X, D^T M D, X^T M X),
//             split over row chunks; partial tiles are summed in chunk
//             order, so the result is deterministic;
//   combine:  out = A1 C1 + A2 C2 + beta B (the retraction updates
//             X+ = X C1 + D C2 of Eq. QR / Eq. WY3 and D = G - X S).
// FP64 arithmetic is the bound of both on GB300 (n p^2 FMAs against n p
// words of traffic); tiles are 64 x 64 with a 4 x 4 register block per
// thread, strided so that shared-memory reads are conflict-free.
#include <mutex>

#include "ks_async.cuh"
#include "ks_device.cuh"
#include "ks_steps.h"

namespace ks {

// 16-byte global -> shared copy (cp.async, L2 only); src_bytes = 0 copies
// nothing and zero-fills the 16 bytes.
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, uint32_t src_bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src),
               "r"(src_bytes)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
  asm volatile("cp.async.commit_group;\n" ::: "memory");
}

// Tensor cores for the FP32 phase when the products are wide enough for the
// SIMT FP32 pipes to be the bound (use_tc = 1: from 256 columns; 2: always;
// 0: never).  Below, the line is one of accuracy: three TF32 products leave an error
// of 2e-7 of sum |a||c| (rms; SIMT 2.8e-8) in an update and 4e-8 (2e-9) in a Gram,
// although they are the faster ones from 96 columns on.  64^3, update of two blocks /
// Gram, SIMT against tensor cores: p = 64 138 / 86 against 251 / 186 us, p = 96
// 460 / 267 against 310 / 188, p = 128 601 / 273 against 373 / 201, p = 256
// 2234 / 942 against 835 / 385.
static bool use_tensor_cores(const Problem &P, int a, int b) {
  if (P.use_tc == 0 || a <= 8 || b <= 8) return false;
  return P.use_tc == 2 || (a >= 256 && b >= 256);
}

static int gram_chunks(const Problem &P, int pa, int qb) {
  const int tiles = ((pa + kTile - 1) / kTile) * ((qb + kTile - 1) / kTile);
  // (the small and mid kernels run one block per chunk: tiles = 1 there too)
  int chunks = (4 * P.sms + tiles - 1) / tiles;
  // at least 256 rows per chunk, so small problems do not pay for many
  // partial tiles
  const int maxc = (P.n + 255) / 256;
  if (chunks > maxc) chunks = maxc;
  if (chunks < 1) chunks = 1;
  return chunks;
}

// T = double, or float for the mixed path (FP32 products and per-chunk
// FP32 sums, chunk partials summed in FP64).
// K-values per stage of the 64-tile update: 32 in FP32 (more bytes in
// flight per thread), 16 in FP64 (FP64-pipe-bound; keeps the two stage
// buffers within the 48 KiB of static shared memory).  The Gram stages
// kTileK rows (measured faster than 32 at p = 64).
template <typename T>
__host__ __device__ constexpr int stage_k() { return sizeof(T) == 4 ? 32 : 16; }

// Vector of 4 consecutive T in shared memory (16- or 32-byte aligned).
template <typename T>
__device__ __forceinline__ void ld4(const T *p, T (&v)[4]) {
  if constexpr (sizeof(T) == 4) {
    const float4 q = *reinterpret_cast<const float4 *>(p);
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
  } else {
    const double2 q0 = reinterpret_cast<const double2 *>(p)[0];
    const double2 q1 = reinterpret_cast<const double2 *>(p)[1];
    v[0] = q0.x; v[1] = q0.y; v[2] = q1.x; v[3] = q1.y;
  }
}

// One 64 x 64 output tile (index `tile`, row-major over the tile grid) of
// one row chunk.  Thread (ty, tx) of 16 x 16 owns the contiguous 4 x 4 block
// a0 + 4ty + i, b0 + 4tx + j, so a row step costs two vector shared-memory
// loads for 16 FMAs; the next stage of rows is loaded into registers while
// the current one is consumed, and two shared buffers alternate (one
// barrier per stage).  Each entry is the same row-ascending FMA chain as a
// one-output-per-thread loop.
template <typename T>
__device__ __forceinline__ void gram_tile_body(long long n, int pa, int qb, long long rows_per,
                                               const T *__restrict__ A, const T *__restrict__ B,
                                               double *__restrict__ part, int tile, int chunk) {
  constexpr int SK = kTileK;
  __shared__ __align__(16) T As[2][SK][kTile];
  __shared__ __align__(16) T Bs[2][SK][kTile];
  const int tq = (qb + kTile - 1) / kTile;
  const int ta = tile / tq, tb = tile % tq;
  const long long r0 = chunk * rows_per;
  long long r1 = r0 + rows_per;
  if (r1 > n) r1 = n;
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  const int a0 = ta * kTile, b0 = tb * kTile;
  T acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0;
  constexpr int kPer = SK * kTile / 256;         // staged values per thread and operand
  T ra[kPer], rb[kPer];
  auto fetch = [&](long long r) {
#pragma unroll
    for (int t = 0; t < kPer; ++t) {
      const int idx = tid + t * 256;
      const int rr = idx >> 6, cc = idx & 63;
      const long long row = r + rr;
      const bool rowok = row < r1;
      ra[t] = (rowok && a0 + cc < pa) ? A[row * pa + a0 + cc] : (T)0;
      rb[t] = (rowok && b0 + cc < qb) ? B[row * qb + b0 + cc] : (T)0;
    }
  };
  auto stash = [&](int buf) {
#pragma unroll
    for (int t = 0; t < kPer; ++t) {
      const int idx = tid + t * 256;
      As[buf][idx >> 6][idx & 63] = ra[t];
      Bs[buf][idx >> 6][idx & 63] = rb[t];
    }
  };
  if (r0 < r1) {
    fetch(r0);
    stash(0);
  }
  __syncthreads();
  int buf = 0;
  for (long long r = r0; r < r1; r += SK, buf ^= 1) {
    const bool more = r + SK < r1;
    if (more) fetch(r + SK);
#pragma unroll
    for (int rr = 0; rr < SK; ++rr) {
      T av[4], bv[4];
      ld4(&As[buf][rr][4 * ty], av);
      ld4(&Bs[buf][rr][4 * tx], bv);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma(av[i], bv[j], acc[i][j]);
    }
    if (more) stash(buf ^ 1);
    __syncthreads();
  }
  double *dst = part + (long long)chunk * pa * qb;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int a = a0 + 4 * ty + i;
    if (a >= pa) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int b = b0 + 4 * tx + j;
      if (b < qb) dst[(long long)a * qb + b] = (double)acc[i][j];
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(256) gram_kernel(long long n, int pa, int qb, long long rows_per,
                                                   const T *__restrict__ A,
                                                   const T *__restrict__ B,
                                                   double *__restrict__ part) {
  gram_tile_body<T>(n, pa, qb, rows_per, A, B, part, blockIdx.x, blockIdx.y);
}

// out[e] = sum over chunks of part[c * len + e]: 8 threads per output, each
// summing a strided eighth of the chunks, then a fixed butterfly (the order
// is the same on every run).
__global__ void gram_reduce_kernel(int chunks, long long len, const double *__restrict__ part,
                                   double *__restrict__ out) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long e = t >> 3;
  const int sub = (int)(t & 7);
  double acc = 0.0;
  if (e < len)
    for (int c = sub; c < chunks; c += 8) acc += part[(long long)c * len + e];
  acc += __shfl_xor_sync(0xffffffffu, acc, 1);
  acc += __shfl_xor_sync(0xffffffffu, acc, 2);
  acc += __shfl_xor_sync(0xffffffffu, acc, 4);
  if (sub == 0 && e < len) out[e] = acc;
}

// Small Grams (pa, qb <= kSmallPQ): each thread accumulates the whole pa x qb
// outer-product sum of its rows in registers, so no arithmetic is spent on
// padding (on GB300 every wasted FP64 FMA costs as much as a useful one);
// warp butterflies then a fixed-order sum over the warps give the chunk
// partial.
constexpr int kSmallPQ = 8;

// Sums v[0 .. V) over the 32 lanes, the results spread over them: each round
// a lane keeps half of its values and gets its partner's share of that half, so
// 16 values take 16 FP64 adds (a butterfly per value: 80) and 64 take 62.  Lane
// holds the sum of index i (returned) in v[0] (V = 16; both lanes of a pair) or
// of i and i + 1 in v[0], v[1] (V = 64).
template <int V>
__device__ __forceinline__ int warp_scatter_sum(double (&v)[V], int lane) {
  int idx = 0, m = V / 2;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    if (m >= 1) {
      const bool up = (lane & o) != 0;
#pragma unroll
      for (int i = 0; i < V / 2; ++i)
        if (i < m) {
          const double keep = up ? v[i + m] : v[i], send = up ? v[i] : v[i + m];
          v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
      if (up) idx += m;
      m >>= 1;
    } else {
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    }
  }
  return idx;
}

template <typename T>
__device__ __forceinline__ void gram_small_body(long long n, int pa, int qb, long long rows_per,
                                                const T *__restrict__ A, const T *__restrict__ B,
                                                double *__restrict__ part, int chunk) {
  __shared__ double red[8][kSmallPQ * kSmallPQ];
  const long long r0 = chunk * rows_per;
  long long r1 = r0 + rows_per;
  if (r1 > n) r1 = n;
  T acc[kSmallPQ][kSmallPQ];
#pragma unroll
  for (int a = 0; a < kSmallPQ; ++a)
#pragma unroll
    for (int b = 0; b < kSmallPQ; ++b) acc[a][b] = 0;
  for (long long r = r0 + threadIdx.x; r < r1; r += blockDim.x) {
    T av[kSmallPQ], bv[kSmallPQ];
#pragma unroll
    for (int a = 0; a < kSmallPQ; ++a) av[a] = a < pa ? A[r * pa + a] : (T)0;
#pragma unroll
    for (int b = 0; b < kSmallPQ; ++b) bv[b] = b < qb ? B[r * qb + b] : (T)0;
#pragma unroll
    for (int a = 0; a < kSmallPQ; ++a) {
      if (a >= pa) break;
#pragma unroll
      for (int b = 0; b < kSmallPQ; ++b) {
        if (b >= qb) break;
        acc[a][b] = fma(av[a], bv[b], acc[a][b]);
      }
    }
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (pa * qb == 1) {
    // one value (the orbital-free model): five adds, not the 16 of the spread sum.  An
    // FP64 add holds the SM's pipe for 16 clocks per warp, 32 of them share it
    double v = (double)acc[0][0];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) red[warp][0] = v;
  } else if (pa <= 4 && qb <= 4) {
    double v[16];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) v[4 * a + b] = (double)acc[a][b];
    const int i = warp_scatter_sum<16>(v, lane);
    if ((lane & 1) == 0) red[warp][(i >> 2) * kSmallPQ + (i & 3)] = v[0];
  } else {
    double v[64];
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
      for (int b = 0; b < 8; ++b) v[8 * a + b] = (double)acc[a][b];
    const int i = warp_scatter_sum<64>(v, lane);
    red[warp][i] = v[0];
    red[warp][i + 1] = v[1];
  }
  __syncthreads();
  for (int e = threadIdx.x; e < pa * qb; e += blockDim.x) {
    const int a = e / qb, b = e % qb;
    double v = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v += red[w][a * kSmallPQ + b];
    part[(long long)chunk * pa * qb + e] = v;
  }
}

// Mid-size Grams (kSmallPQ < pa, qb <= kMidPQ): the block keeps the whole
// pa x qb result of its row chunk, staging kMidRows rows of A and B in shared
// memory at a time.  Threads map onto the outputs with no padding beyond one row
// and column, so no FMA is spent on entries outside the Gram (the 64-wide tile
// would spend (64/p)^2 times the work at p = 16).  Up to 256 outputs: one per
// thread.  Above, in FP32 a 2 x 2 block per thread: four shared values for four
// FMAs where one output per thread reads eight, which bound the kernel (two reads
// per FMA).  Measured, the Grams of 24 batched jobs (N 20 to 38, p 4 to 32):
// 123 -> 71 us per launch.  FP64 keeps single outputs, every 256th to a thread: its
// pipe is the bound, and 2 x 2 blocks leave warps idle (81 threads at p = 17).  One
// step_gram call at 48^3, single against 2 x 2: p = 17 95 / 111 us, p = 20 112 / 134,
// p = 29 199 / 233, p = 32 230 / 232; in FP32 at p = 29 63 / 48, p = 32 71 / 48.
// Every output is the same row-ascending chain in all.
constexpr int kMidPQ = 32, kMidRows = 32;
static_assert(kMidRows * kMidPQ <= 4 * 256, "a stage is 4 values per thread of a 256-thread block");

template <typename T>
__device__ __forceinline__ void gram_mid_body(long long n, int pa, int qb, long long rows_per,
                                              const T *__restrict__ A, const T *__restrict__ B,
                                              double *__restrict__ part, int chunk) {
  // (an odd width's last block reads one value past its row: the next row's, or
  // up to one value past the stage, so a few spare entries)
  __shared__ __align__(16) T As[kMidRows * kMidPQ + 4];
  __shared__ __align__(16) T Bs[kMidRows * kMidPQ + 4];
  const long long r0 = chunk * rows_per;
  long long r1 = r0 + rows_per;
  if (r1 > n) r1 = n;
  const int outs = pa * qb;
  const bool wide = sizeof(T) == 4 && outs > 256;
  const int tb = (qb + 1) / 2, ta = (pa + 1) / 2;
  const bool work = (int)threadIdx.x < (wide ? ta * tb : outs);
  // this thread's outputs (row, column): a 2 x 2 block, or every 256th
  int oa[4], ob[4];
  bool own[4];
  T acc[4] = {0, 0, 0, 0};
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int e = threadIdx.x + u * blockDim.x;
    oa[u] = !work ? 0 : wide ? 2 * ((int)threadIdx.x / tb) + (u >> 1) : e / qb;
    ob[u] = !work ? 0 : wide ? 2 * ((int)threadIdx.x % tb) + (u & 1) : e % qb;
    own[u] = work && oa[u] < pa && ob[u] < qb;
  }
  // the next stage's values travel in registers while this stage computes
  // (256 threads x 4 cover a stage of kMidRows x kMidPQ)
  T ra[4], rb[4];
  auto fetch = [&](long long r) {
    const int rows = (int)min((long long)kMidRows, r1 - r);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int t = threadIdx.x + u * blockDim.x;
      ra[u] = t < rows * pa ? A[r * pa + t] : (T)0;
      rb[u] = t < rows * qb ? B[r * qb + t] : (T)0;
    }
  };
  if (r0 < r1) fetch(r0);
  for (long long r = r0; r < r1; r += kMidRows) {
    const int rows = (int)min((long long)kMidRows, r1 - r);
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int t = threadIdx.x + u * blockDim.x;
      if (t < rows * pa) As[t] = ra[u];
      if (t < rows * qb) Bs[t] = rb[u];
    }
    __syncthreads();
    if (r + kMidRows < r1) fetch(r + kMidRows);
    if (!work) continue;
    if (!wide) {
      // (up to 256 outputs: the first only)
#pragma unroll
      for (int u = 0; u < (sizeof(T) == 8 ? 4 : 1); ++u) {
        if (u > 0 && !own[u]) break;
        T a = acc[u];
#pragma unroll 8
        for (int k = 0; k < rows; ++k) a = fma(As[k * pa + oa[u]], Bs[k * qb + ob[u]], a);
        acc[u] = a;
      }
    } else {
      const T *as = As + oa[0], *bs = Bs + ob[0];
#pragma unroll 8
      for (int k = 0; k < rows; ++k) {
        const T a0 = as[k * pa], a1 = as[k * pa + 1], b0 = bs[k * qb], b1 = bs[k * qb + 1];
        acc[0] = fma(a0, b0, acc[0]);
        acc[1] = fma(a0, b1, acc[1]);
        acc[2] = fma(a1, b0, acc[2]);
        acc[3] = fma(a1, b1, acc[3]);
      }
    }
  }
  double *dst = part + (long long)chunk * outs;
#pragma unroll
  for (int u = 0; u < 4; ++u)
    if (own[u]) dst[oa[u] * qb + ob[u]] = (double)acc[u];
}

template <typename T>
__global__ void __launch_bounds__(256) gram_mid_kernel(long long n, int pa, int qb,
                                                       long long rows_per,
                                                       const T *__restrict__ A,
                                                       const T *__restrict__ B,
                                                       double *__restrict__ part) {
  gram_mid_body<T>(n, pa, qb, rows_per, A, B, part, blockIdx.x);
}

// out (null: left to the reduction kernel): the last block to finish sums the
// chunks, in chunk order, and re-arms the counter.
template <typename T>
__global__ void __launch_bounds__(256) gram_small_kernel(long long n, int pa, int qb,
                                                         long long rows_per,
                                                         const T *__restrict__ A,
                                                         const T *__restrict__ B,
                                                         double *__restrict__ part,
                                                         double *__restrict__ out,
                                                         unsigned int *counter) {
  gram_small_body<T>(n, pa, qb, rows_per, A, B, part, blockIdx.x);
  if (!out) return;
  __shared__ int s_last;
  __shared__ double sums[256];
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(counter, 1u) == gridDim.x - 1u;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  constexpr int kLen = kSmallPQ * kSmallPQ, kSubs = 256 / kLen;
  const int e = threadIdx.x % kLen, sub = threadIdx.x / kLen, len = pa * qb;
  double v = 0.0;
  if (e < len)
    for (int c = sub; c < (int)gridDim.x; c += kSubs) v += ldcg(part + (long long)c * len + e);
  sums[threadIdx.x] = v;
  __syncthreads();
  if (sub == 0 && e < len) {
#pragma unroll
    for (int s = 1; s < kSubs; ++s) v += sums[s * kLen + e];
    out[e] = v;
  }
  if (threadIdx.x == 0) *counter = 0u;
}

// Pipelined FP32 Grams for 32 < max(pa, qb) <= 64 and 16-byte-aligned
// operands (widths multiples of 4).  Two forms:
//   pair   (Dual = false): out = A1^T B1 + A2^T B2 -- the rows of the second
//          pair follow those of the first (A2 null: one Gram);
//   shared (Dual = true):  out1 = A1^T B, out2 = A2^T B (even warps take A1,
//          odd warps A2, on the same rows, so B comes from DRAM once).
// FP32 FMAs bound it, and next to them shared memory (128 bytes per clock):
// a 4 x 4 block of outputs per thread reads two bytes per FMA, the 8 x 16
// block per lane here three quarters of one.  A warp keeps the whole 64 x 64
// tile and runs alone on stages of kGaRows rows (a ring of kGaStages, cp.async
// 16 bytes per copy, zero-filled past the last row and past pa, qb); lane
// (ty, tx) of 8 x 4 owns columns 4 ty + 32 h of A and 4 tx + 16 j of B.  The
// warps' tiles (chains of about 200 rows at 64^3) are added in pairs in FP32 with
// the error of every sum kept (two-sum, Knuth), so nothing of a tile is rounded
// away: a partial is the sum and its error, 48 bits (in FP64 those 4096 x 8 adds
// per block took 17 us).  The blocks' sums are added in FP64 in block order.  One
// Gram at 64^3 x 64: 63 us for 4 x 4 per thread (34 TF/s), 56 here (38); packed FMAs
// cost more in duplicating A than they save (65).
constexpr int kGaStages = 3, kGaRows = 16, kGaWarps = 8;

constexpr size_t gram_wa_smem() {
  // the rings; the same memory then holds the warps' tiles
  constexpr size_t ring = (size_t)kGaWarps * kGaStages * 2 * kGaRows * kTile * sizeof(float);
  static_assert(ring >= (size_t)kGaWarps * kTile * kTile * sizeof(float), "the tiles fit");
  return ring;
}

template <bool Dual>
__global__ void __launch_bounds__(32 * kGaWarps, 1) gram2_wa_kernel(
    long long n, int pa, int qb, const float *__restrict__ A1, const float *__restrict__ B1,
    const float *__restrict__ A2, const float *__restrict__ B2, float2 *__restrict__ part) {
  extern __shared__ __align__(16) float ga_smem[];
  constexpr int kStage = 2 * kGaRows * kTile;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, ty = lane >> 2, tx = lane & 3;
  float *ring = ga_smem + (size_t)warp * kGaStages * kStage;
  const long long nv = (!Dual && A2) ? 2 * n : n;    // rows streamed (both pairs)
  const long long nst = (nv + kGaRows - 1) / kGaRows;
  // stages of this warp (of this warp's pair in the shared form)
  const long long first = (long long)(Dual ? warp >> 1 : warp) * gridDim.x + blockIdx.x;
  const long long step = (long long)(Dual ? kGaWarps / 2 : kGaWarps) * gridDim.x;
  const long long W = nst > first ? (nst - first + step - 1) / step : 0;
  const float *Aw = Dual && (warp & 1) ? A2 : A1;
  auto issue = [&](long long w) {
    const long long r0 = (first + w * step) * kGaRows;
    float *dst = ring + (w % kGaStages) * kStage;
#pragma unroll
    for (int t = 0; t < kStage / 128; ++t) {           // operand, row, 4-column chunk
      const int idx = lane + 32 * t, op = idx / (kGaRows * 16);
      const int rr = idx / 16 % kGaRows, c4 = idx % 16 * 4;
      long long row = r0 + rr;
      const int w_ = op == 1 ? qb : pa;
      const float *M = op == 0 ? Aw : B1;
      if (!Dual && row >= n) {
        M = op == 0 ? A2 : B2;
        row -= n;
      }
      const float *src = A1;
      uint32_t bytes = 0;
      if (row < n && r0 + rr < nv && c4 < w_ && KS_IN(row * w_ + c4 + 3, n * w_)) {
        src = M + row * w_ + c4;
        bytes = 16;
      }
      const int di = op * kGaRows * kTile + rr * kTile + c4;
      if (KS_IN(di + 3, kStage)) cp_async16(smem_addr(dst + di), src, bytes);
    }
  };
  float acc[8][16];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 16; ++j) acc[i][j] = 0.f;
  for (int st = 0; st < kGaStages - 1; ++st) {
    if (st < W) issue(st);
    cp_async_commit();
  }
  for (long long w = 0; w < W; ++w) {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(kGaStages - 2) : "memory");
    __syncwarp();
    if (w + kGaStages - 1 < W) issue(w + kGaStages - 1);
    cp_async_commit();
    const float *As = ring + (w % kGaStages) * kStage + 4 * ty;
    const float *Bs = ring + (w % kGaStages) * kStage + kGaRows * kTile + 4 * tx;
#pragma unroll 2
    for (int r = 0; r < kGaRows; ++r) {
      float av[8], bv[16];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float4 v = *reinterpret_cast<const float4 *>(As + r * kTile + 32 * h);
        av[4 * h] = v.x; av[4 * h + 1] = v.y; av[4 * h + 2] = v.z; av[4 * h + 3] = v.w;
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float4 v = *reinterpret_cast<const float4 *>(Bs + r * kTile + 16 * j);
        bv[4 * j] = v.x; bv[4 * j + 1] = v.y; bv[4 * j + 2] = v.z; bv[4 * j + 3] = v.w;
      }
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 16; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
    }
  }
  asm volatile("cp.async.wait_all;\n" ::: "memory");
  __syncthreads();
  float *tile = ga_smem + (size_t)warp * kTile * kTile;
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
      *reinterpret_cast<float4 *>(tile + (32 * (i >> 2) + 4 * ty + (i & 3)) * kTile + 16 * j +
                                  4 * tx) =
          make_float4(acc[i][4 * j], acc[i][4 * j + 1], acc[i][4 * j + 2], acc[i][4 * j + 3]);
  __syncthreads();
  const int len = pa * qb;
  float2 *dst = part + (long long)blockIdx.x * (Dual ? 2 : 1) * len;
  for (int e = threadIdx.x; e < (Dual ? 2 : 1) * len; e += 32 * kGaWarps) {
    const int which = e >= len ? 1 : 0, f = e - which * len, at = f / qb * kTile + f % qb;
    constexpr int kTiles = Dual ? kGaWarps / 2 : kGaWarps;
    float v[kTiles], lo = 0.f;
#pragma unroll
    for (int s = 0; s < kTiles; ++s)
      v[s] = ga_smem[(size_t)(s * (Dual ? 2 : 1) + which) * kTile * kTile + at];
#pragma unroll
    for (int o = kTiles / 2; o > 0; o >>= 1)
#pragma unroll
      for (int s = 0; s < o; ++s) {
        const float x = v[s], y = v[s + o], sum = __fadd_rn(x, y);
        const float yy = __fsub_rn(sum, x);
        lo += __fadd_rn(__fsub_rn(x, __fsub_rn(sum, yy)), __fsub_rn(y, yy));
        v[s] = sum;
      }
    if (KS_IN((long long)blockIdx.x * (Dual ? 2 : 1) * len + e,
              (long long)gridDim.x * (Dual ? 2 : 1) * len))
      dst[e] = make_float2(v[0], isfinite(v[0]) ? lo : 0.f);
  }
}

// FP64 sums of the blocks' partials (sum and error) in block order: element e <
// len1 of each goes to out1[e], the rest to out2[e - len1]; out32 (optional) gets
// every sum rounded to FP32 at index e.  The errors, 2^-24 of the sums, are added in
// FP32 first.
__global__ void gram_reduce2_kernel(int chunks, long long len, long long len1,
                                    const float2 *__restrict__ part, double *__restrict__ out1,
                                    double *__restrict__ out2, float *__restrict__ out32) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long e = t >> 3;
  const int sub = (int)(t & 7);
  double acc = 0.0;
  float lo = 0.f;
  if (e < len)
    for (int c = sub; c < chunks; c += 8) {
      const float2 v = part[(long long)c * len + e];
      acc += (double)v.x;
      lo += v.y;
    }
  acc += (double)lo;
  acc += __shfl_xor_sync(0xffffffffu, acc, 1);
  acc += __shfl_xor_sync(0xffffffffu, acc, 2);
  acc += __shfl_xor_sync(0xffffffffu, acc, 4);
  if (sub == 0 && e < len) {
    if (e < len1) out1[e] = acc;
    else out2[e - len1] = acc;
    if (out32) out32[e] = (float)acc;
  }
}

// The pipelined Gram kernels apply: FP32, 32 < max(pa, qb) <= 64, widths
// multiples of 4 and 16-byte-aligned operands.
static bool gram_wa_applies(int pa, int qb, std::initializer_list<const float *> ops) {
  if (pa > kTile || qb > kTile || (pa <= kMidPQ && qb <= kMidPQ) || pa % 4 || qb % 4) return false;
  for (const float *A : ops)
    if (reinterpret_cast<uintptr_t>(A) % 16) return false;
  return true;
}

template <bool Dual>
static ks_status launch_gram2_wa(Problem &P, int pa, int qb, const float *A1, const float *B1,
                                 const float *A2, const float *B2, double *out1, double *out2,
                                 float *out32 = nullptr) {
  const long long nv = (!Dual && A2) ? 2 * P.n : P.n;
  const long long nst = (nv + kGaRows - 1) / kGaRows;
  long long blocks = P.sms;
  if (blocks > nst) blocks = nst;
  const long long len = (long long)pa * qb * (Dual ? 2 : 1);
  if ((size_t)blocks * len > P.partials_len)
    return set_error(KS_EINVAL, "gram: partial buffer too small");
  float2 *part = reinterpret_cast<float2 *>(P.partials);
  {
    ProfScope ps_(P.stream, KP_GRAM, 2.0 * nv * pa * qb * (Dual ? 2 : 1),
                  (double)nv * (pa + qb + (Dual ? pa : 0)) * sizeof(float));
    gram2_wa_kernel<Dual><<<(int)blocks, 32 * kGaWarps, gram_wa_smem(), P.stream>>>(
        P.n, pa, qb, A1, B1, A2, B2, part);
  }
  KS_CUDA_TRY(cudaGetLastError());
  {
    ProfScope ps_(P.stream, KP_REDUCE);
    gram_reduce2_kernel<<<(int)((8 * len + kThreads - 1) / kThreads), kThreads, 0, P.stream>>>(
        (int)blocks, len, (long long)pa * qb, part, out1, out2, out32);
  }
  KS_CUDA_TRY(cudaGetLastError());
  return KS_OK;
}

template <typename T>
ks_status launch_gram(Problem &P, const T *A, int pa, const T *B, int qb, double *out) {
  if (sizeof(T) == 8 && P.use_oz > 0 && pa + qb <= P.oz_emax_len &&
      (P.use_oz == 2 || (pa >= 48 && qb >= 48))) {
    // FP64: digit-split products on the tensor cores, FP64 chunk partials
    const int chunks = gram_oz_chunks(P, pa, qb);
    if ((size_t)chunks * pa * qb > P.partials_len)
      return set_error(KS_EINVAL, "gram: partial buffer too small");
    KS_TRY(launch_gram_oz(P, (const double *)A, pa, (const double *)B, qb, P.oz_emax, P.partials,
                          chunks));
    const long long len = (long long)pa * qb;
    {
      ProfScope ps_(P.stream, KP_REDUCE);
      gram_reduce_kernel<<<(int)((8 * len + kThreads - 1) / kThreads), kThreads, 0, P.stream>>>(
          chunks, len, P.partials, out);
    }
    KS_CUDA_TRY(cudaGetLastError());
    return KS_OK;
  }
  if (sizeof(T) == 4 && use_tensor_cores(P, pa, qb)) {
    // FP32 phase: tensor cores (3 x TF32), FP64 chunk partials
    const int chunks = gram_tc_chunks(P, pa, qb);
    if ((size_t)chunks * pa * qb > P.partials_len)
      return set_error(KS_EINVAL, "gram: partial buffer too small");
    KS_TRY(launch_gram_tc(P, (const float *)A, pa, (const float *)B, qb, P.partials, chunks));
    const long long len = (long long)pa * qb;
    {
      ProfScope ps_(P.stream, KP_REDUCE);
      gram_reduce_kernel<<<(int)((8 * len + kThreads - 1) / kThreads), kThreads, 0, P.stream>>>(
          chunks, len, P.partials, out);
    }
    KS_CUDA_TRY(cudaGetLastError());
    return KS_OK;
  }
  if (sizeof(T) == 4 && gram_wa_applies(pa, qb, {(const float *)A, (const float *)B}))
    return launch_gram2_wa<false>(P, pa, qb, (const float *)A, (const float *)B, nullptr, nullptr,
                                  out, nullptr);
  const int chunks = gram_chunks(P, pa, qb);
  long long rows_per = (P.n + chunks - 1) / chunks;
  rows_per = (rows_per + kTileK - 1) / kTileK * kTileK;
  const int tiles = ((pa + kTile - 1) / kTile) * ((qb + kTile - 1) / kTile);
  const size_t need = (size_t)chunks * pa * qb;
  if (need > P.partials_len)
    return set_error(KS_EINVAL, "gram: partial buffer too small (%zu > %zu)", need, P.partials_len);
  // few chunks of a small Gram are summed by the last block (a launch less); many
  // take too long in one block.  step_gram by a reduction launch against the last
  // block: 20^3 (32 chunks) p = 2 33.5 / 32.8 us, p = 8 36.5 / 35.4; 28^3 (86) p = 4
  // 34.2 / 33.4, p = 8 37.5 / 37.6; 32^3 (128) p = 1 30.0 / 33.6, p = 8 37.5 / 42.6;
  // 48^3 (432) p = 1 34.6 / 46.6
  const bool tail = pa <= kSmallPQ && qb <= kSmallPQ && chunks <= 96;
  {
    ProfScope ps_(P.stream, KP_GRAM, 2.0 * P.n * pa * qb, (double)P.n * (pa + qb) * sizeof(T));
    if (pa <= kSmallPQ && qb <= kSmallPQ)
      gram_small_kernel<T><<<chunks, 256, 0, P.stream>>>(P.n, pa, qb, rows_per, A, B, P.partials,
                                                         tail ? out : nullptr, P.red_counter);
    else if (pa <= kMidPQ && qb <= kMidPQ)
      gram_mid_kernel<T><<<chunks, 256, 0, P.stream>>>(P.n, pa, qb, rows_per, A, B, P.partials);
    else
      gram_kernel<T><<<dim3(tiles, chunks), 256, 0, P.stream>>>(P.n, pa, qb, rows_per, A, B,
                                                                P.partials);
  }
  KS_CUDA_TRY(cudaGetLastError());
  if (tail) return KS_OK;
  const long long len = (long long)pa * qb;
  {
    ProfScope ps_(P.stream, KP_REDUCE);
    gram_reduce_kernel<<<(int)((8 * len + kThreads - 1) / kThreads), kThreads, 0, P.stream>>>(
        chunks, len, P.partials, out);
  }
  KS_CUDA_TRY(cudaGetLastError());
  return KS_OK;
}

ks_status launch_gram_pair(Problem &P, const float *A1, const float *B1, const float *A2,
                           const float *B2, int pa, int qb, double *out, double *tmp) {
  if (gram_wa_applies(pa, qb, {A1, B1, A2, B2}))
    return launch_gram2_wa<false>(P, pa, qb, A1, B1, A2, B2, out, nullptr, nullptr);
  KS_TRY(launch_gram<float>(P, A1, pa, B1, qb, out));
  KS_TRY(launch_gram<float>(P, A2, pa, B2, qb, tmp));
  return launch_add_pp(P, out, 1.0, tmp, out);
}

// FP32 copies of two p x p FP64 matrices, one after the other.
__global__ void pair_to_f32_kernel(long long len, const double *__restrict__ a,
                                   const double *__restrict__ b, float *__restrict__ out) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e < len) out[e] = (float)a[e];
  else if (e < 2 * len) out[e] = (float)b[e - len];
}

ks_status launch_gram_dual(Problem &P, const float *A1, const float *A2, const float *B, int pa,
                           int qb, double *out1, double *out2, float *out32) {
  if (gram_wa_applies(pa, qb, {A1, A2, B}))
    return launch_gram2_wa<true>(P, pa, qb, A1, B, A2, nullptr, out1, out2, out32);
  KS_TRY(launch_gram<float>(P, A1, pa, B, qb, out1));
  KS_TRY(launch_gram<float>(P, A2, pa, B, qb, out2));
  if (out32) {
    const long long len = (long long)pa * qb;
    {
      ProfScope ps_(P.stream, KP_REDUCE);
      pair_to_f32_kernel<<<(int)((2 * len + kThreads - 1) / kThreads), kThreads, 0, P.stream>>>(
          len, out1, out2, out32);
    }
    KS_CUDA_TRY(cudaGetLastError());
  }
  return KS_OK;
}

// TC is the type of the coefficients C1, C2: double, or float copies made
// once per update for the FP32 phase (converting in every block would put
// a conversion per staged element on the FP64 pipe).
// One 64 x 64 output tile: thread (ty, tx) owns rows r0 + 4ty + i and
// columns c0 + 4tx + j.  The A slice is stored transposed (K-rows of 64
// rows, padded to keep the vector loads aligned) and the C slice as is, so a
// K-step costs two vector loads for 16 FMAs; stages of K-values run over
// A1 C1 then A2 C2, the next one loaded into registers while the current
// one is consumed (two shared buffers, one barrier per stage).  Each entry
// is the same K-ascending FMA chain as before.
constexpr int kAtLd = kTile + 4;

template <typename T, typename TC>
__device__ __forceinline__ void combine_tile_body(long long n, int q, const T *__restrict__ A1,
                                                  int k1, const TC *__restrict__ C1,
                                                  const T *__restrict__ A2, int k2,
                                                  const TC *__restrict__ C2, double alpha_d,
                                                  double beta_d, const T *__restrict__ Bm,
                                                  T *__restrict__ out, int bx, int by) {
  constexpr int SK = stage_k<T>();
  __shared__ __align__(16) T At[2][SK][kAtLd];
  __shared__ __align__(16) T Cs[2][SK][kTile];
  const T alpha = (T)alpha_d, beta = (T)beta_d;
  const long long r0 = (long long)bx * kTile;
  const int c0 = by * kTile;
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  T acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0;
  const int s1 = (k1 + SK - 1) / SK;
  const int s2 = A2 ? (k2 + SK - 1) / SK : 0;
  const int stages = s1 + s2;
  constexpr int kPer = SK * kTile / 256;         // staged values per thread and operand
  T ra[kPer], rc[kPer];
  auto fetch = [&](int s) {
    const bool first = s < s1;
    const T *A = first ? A1 : A2;
    const TC *C = first ? C1 : C2;
    const int kk = first ? k1 : k2;
    const int k0 = (first ? s : s - s1) * SK;
#pragma unroll
    for (int t = 0; t < kPer; ++t) {
      const int idx = tid + t * 256;
      const int rr = idx / SK, cc = idx % SK;              // A slice: 64 rows x SK
      const long long row = r0 + rr;
      ra[t] = (row < n && k0 + cc < kk) ? A[row * kk + k0 + cc] : (T)0;
      const int cr = idx >> 6, ccol = idx & 63;            // C slice: SK x 64
      rc[t] = (k0 + cr < kk && c0 + ccol < q) ? (T)C[(long long)(k0 + cr) * q + c0 + ccol] : (T)0;
    }
  };
  auto stash = [&](int buf) {
#pragma unroll
    for (int t = 0; t < kPer; ++t) {
      const int idx = tid + t * 256;
      At[buf][idx % SK][idx / SK] = ra[t];
      Cs[buf][idx >> 6][idx & 63] = rc[t];
    }
  };
  if (stages > 0) {
    fetch(0);
    stash(0);
  }
  __syncthreads();
  for (int s = 0; s < stages; ++s) {
    const int buf = s & 1;
    const bool more = s + 1 < stages;
    if (more) fetch(s + 1);
#pragma unroll
    for (int t = 0; t < SK; ++t) {
      T av[4], cv[4];
      ld4(&At[buf][t][4 * ty], av);
      ld4(&Cs[buf][t][4 * tx], cv);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma(av[i], cv[j], acc[i][j]);
    }
    if (more) stash(buf ^ 1);
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const long long row = r0 + 4 * ty + i;
    if (row >= n) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int col = c0 + 4 * tx + j;
      if (col >= q) continue;
      T v = alpha * acc[i][j];
      if (Bm) v = fma(beta, Bm[row * q + col], v);
      out[row * q + col] = v;
    }
  }
}

template <typename T, typename TC>
__global__ void __launch_bounds__(256) combine_kernel(long long n, int q, const T *__restrict__ A1,
                                                      int k1, const TC *__restrict__ C1,
                                                      const T *__restrict__ A2, int k2,
                                                      const TC *__restrict__ C2, double alpha_d,
                                                      double beta_d,
                                                      const T *__restrict__ Bm,
                                                      T *__restrict__ out) {
  combine_tile_body<T, TC>(n, q, A1, k1, C1, A2, k2, C2, alpha_d, beta_d, Bm, out, blockIdx.x,
                           blockIdx.y);
}

// Narrow updates (q <= kNarrowQ): a thread takes 4 consecutive columns, the small
// C matrices in shared memory, no padded arithmetic.  One row per thread, A read
// from L1 (combine_narrow_body): FP64, bound by its pipe, and FP32 launches that do
// not fill the chip with threads.  The other FP32 ones: combine_rows_body.
constexpr int kNarrowQ = 32;
constexpr int kNarrowK = 2 * kNarrowQ;
constexpr int kNarrowCols = 4;                     // output columns per thread

// FP32 form: 4 rows x 4 columns per thread.  A tile's rows (as many as the
// threads cover; 144 at q = 26) are staged up to 32 columns at a time, read and
// written as contiguous memory; four k of A and of C are one 16-byte shared read
// each, 8 reads for 64 FMAs (one row per thread and scalar reads: 5 per 4), and
// the rounding of C to FP32, on the FP64 pipe, is per tile of rows instead of per
// 1024 outputs.  Rows of a thread lie `groups` apart: a warp's groups read
// consecutive rows, whose odd multiple of 16 bytes misses no bank.  Every output
// keeps its chain over k and its last step.  Measured, 24 batched jobs (N 20 to
// 38, p 4 to 32): 119 -> 93 us per update of one or two blocks.  What is left is
// latency: a tile loads, computes and writes in turn, four blocks to an SM.
constexpr int kNrK = 32;                           // columns of A per stage
constexpr int kNrStage = 6144;                     // floats of a stage: 1024 rows x 4 .. 128 x 36

__device__ __forceinline__ int nr_pitch(int kc) {  // odd multiple of 4 floats
  const int v = (kc + 3) / 4;
  return 4 * (v | 1);
}

__device__ __forceinline__ void combine_rows_body(
    long long n, int q, const float *__restrict__ A1, int k1, const double *__restrict__ C1,
    const float *__restrict__ A2, int k2, const double *__restrict__ C2, float alpha, float beta,
    const float *__restrict__ Bm, float *__restrict__ out, int vb, int vnb) {
  __shared__ __align__(16) float Cs[2 * kNarrowK * kNarrowQ];
  __shared__ __align__(16) float As[kNrStage];
  const int K = k1 + (A2 ? k2 : 0);
  const int ncg = (q + 3) / 4, ldc = 4 * ncg;
  const int groups = min(256 / ncg, kNrStage / (4 * nr_pitch(min(max(k1, A2 ? k2 : 0), kNrK))));
  const int tr = 4 * groups;                       // rows of a tile
  const long long ntiles = (n + tr - 1) / tr;
  if (vb >= ntiles) return;
  for (int e = threadIdx.x; e < K * ldc; e += blockDim.x) {
    const int k = e / ldc, c = e - k * ldc;
    Cs[e] = c >= q ? 0.f : (float)(k < k1 ? C1[k * q + c] : C2[(k - k1) * q + c]);
  }
  const int g = threadIdx.x / ncg, col0 = 4 * (threadIdx.x % ncg);
  const bool work = g < groups;
  for (long long t = vb; t < ntiles; t += vnb) {
    const long long r0 = t * tr;
    const int rows = (int)min((long long)tr, n - r0);
    float acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int u = 0; u < 4; ++u) acc[i][u] = 0.f;
    for (int s = 0; s < (A2 ? 2 : 1); ++s) {
      const int ks = s ? k2 : k1;
      const float *A = (s ? A2 : A1) + r0 * ks;
      for (int kb = 0; kb < ks; kb += kNrK) {
        const int kc = min(kNrK, ks - kb), ld = nr_pitch(kc);
        __syncthreads();                           // (the stage, and Cs the first time)
        // element e = row kc + k of the stage, advanced without a division
        const int dr = 256 / kc, dk = 256 - dr * kc;
        int row = threadIdx.x / kc, k = threadIdx.x - row * kc;
        const int cnt = rows * kc;
        for (int e0 = threadIdx.x; e0 < cnt; e0 += 8 * 256) {
          float v[8];
          int at[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const bool in = e0 + u * 256 < cnt;
            at[u] = in ? row * ld + k : -1;
            v[u] = in ? A[(long long)row * ks + kb + k] : 0.f;
            row += dr;
            k += dk;
            if (k >= kc) {
              k -= kc;
              ++row;
            }
          }
#pragma unroll
          for (int u = 0; u < 8; ++u)
            if (at[u] >= 0) As[at[u]] = v[u];
        }
        __syncthreads();
        if (work) {
          const float *a0 = As + g * ld;
          const float *c0 = Cs + ((s ? k1 : 0) + kb) * ldc + col0;
          int kk = 0;
          for (; kk + 4 <= kc; kk += 4) {
            float a[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const float4 w = *reinterpret_cast<const float4 *>(a0 + i * groups * ld + kk);
              a[i][0] = w.x; a[i][1] = w.y; a[i][2] = w.z; a[i][3] = w.w;
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float4 c = *reinterpret_cast<const float4 *>(c0 + (kk + j) * ldc);
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                acc[i][0] = fma(a[i][j], c.x, acc[i][0]);
                acc[i][1] = fma(a[i][j], c.y, acc[i][1]);
                acc[i][2] = fma(a[i][j], c.z, acc[i][2]);
                acc[i][3] = fma(a[i][j], c.w, acc[i][3]);
              }
            }
          }
          for (; kk < kc; ++kk) {
            const float4 c = *reinterpret_cast<const float4 *>(c0 + kk * ldc);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const float a = a0[i * groups * ld + kk];
              acc[i][0] = fma(a, c.x, acc[i][0]);
              acc[i][1] = fma(a, c.y, acc[i][1]);
              acc[i][2] = fma(a, c.z, acc[i][2]);
              acc[i][3] = fma(a, c.w, acc[i][3]);
            }
          }
        }
      }
    }
    // the tile's outputs leave through the stage: contiguous rows x q
    __syncthreads();
    if (work)
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (col0 + u < q) As[(g + i * groups) * q + col0 + u] = acc[i][u];
    __syncthreads();
    const long long o0 = r0 * q;
#pragma unroll 4
    for (int e = threadIdx.x; e < rows * q; e += 256) {
      float v = alpha * As[e];
      if (Bm) v = fma(beta, Bm[o0 + e], v);
      out[o0 + e] = v;
    }
  }
}

template <typename T>
__device__ __forceinline__ void combine_narrow_body(
    long long n, int q, const T *__restrict__ A1, int k1, const double *__restrict__ C1,
    const T *__restrict__ A2, int k2, const double *__restrict__ C2, double alpha_d,
    double beta_d, const T *__restrict__ Bm, T *__restrict__ out, int vb, int vnb) {
  __shared__ T Cs[2][kNarrowK * kNarrowQ];
  for (int e = threadIdx.x; e < k1 * q; e += blockDim.x) Cs[0][e] = (T)C1[e];
  if (A2)
    for (int e = threadIdx.x; e < k2 * q; e += blockDim.x) Cs[1][e] = (T)C2[e];
  __syncthreads();
  const T alpha = (T)alpha_d, beta = (T)beta_d;
  // a thread takes kNarrowCols consecutive columns of one row, so each value
  // of the row of A is loaded once for kNarrowCols FMAs (each output's FMA
  // chain runs over k in ascending order, as with one output per thread)
  const int ncg = (q + kNarrowCols - 1) / kNarrowCols;
  const long long total = n * ncg;
  for (long long e = (long long)vb * blockDim.x + threadIdx.x; e < total;
       e += (long long)vnb * blockDim.x) {
    const long long row = e / ncg;
    const int col0 = (int)(e - row * ncg) * kNarrowCols;
    const int nc = q - col0 < kNarrowCols ? q - col0 : kNarrowCols;
    T acc[kNarrowCols];
#pragma unroll
    for (int u = 0; u < kNarrowCols; ++u) acc[u] = 0;
    const T *a1 = A1 + row * k1;
    for (int k = 0; k < k1; ++k) {
      const T a = a1[k];
#pragma unroll
      for (int u = 0; u < kNarrowCols; ++u)
        if (u < nc) acc[u] = fma(a, Cs[0][k * q + col0 + u], acc[u]);
    }
    if (A2) {
      const T *a2 = A2 + row * k2;
      for (int k = 0; k < k2; ++k) {
        const T a = a2[k];
#pragma unroll
        for (int u = 0; u < kNarrowCols; ++u)
          if (u < nc) acc[u] = fma(a, Cs[1][k * q + col0 + u], acc[u]);
      }
    }
#pragma unroll
    for (int u = 0; u < kNarrowCols; ++u) {
      if (u >= nc) break;
      const long long o = row * q + col0 + u;
      T v = alpha * acc[u];
      if (Bm) v = fma(beta, Bm[o], v);
      out[o] = v;
    }
  }
}

template <typename T, bool Rows>
__global__ void __launch_bounds__(256) combine_narrow_kernel(
    long long n, int q, const T *__restrict__ A1, int k1, const double *__restrict__ C1,
    const T *__restrict__ A2, int k2, const double *__restrict__ C2, double alpha_d,
    double beta_d, const T *__restrict__ Bm, T *__restrict__ out) {
  if constexpr (Rows)
    combine_rows_body(n, q, A1, k1, C1, A2, k2, C2, (float)alpha_d, (float)beta_d, Bm, out,
                      blockIdx.x, gridDim.x);
  else
    combine_narrow_body<T>(n, q, A1, k1, C1, A2, k2, C2, alpha_d, beta_d, Bm, out, blockIdx.x,
                           gridDim.x);
}

// Staged tiles of rows for an FP32 narrow update of one system (job tables always
// take them: their jobs fill the chip together): from 16 columns on where the
// one-row form's threads would fill the chip (2048 per SM), or where its chain over k
// is longer than a stage.  Below, a tile of up to 1024 rows leaves most SMs without
// one; on few columns the two are even, or the one-row form is ahead, which skips
// what a ragged group of four pads.  step_combine_f32 with two blocks and Bm, one-row
// against staged: 20^3, p = 5 25 / 33 us; 48^3, p = 15 36 / 38; 64^3, p = 9 37 / 46;
// 80^3, p = 13 62 / 71; 48^3, p = 16 47 / 38; 64^3, p = 16 59 / 48, p = 32 158 / 94.
static bool narrow_rows_applies(const Problem &P, int K, int q) {
  const long long threads = (long long)P.n * ((q + kNarrowCols - 1) / kNarrowCols);
  return (q >= 16 && threads >= 2048LL * P.sms) || K > kNrK;
}

// Tall-skinny FP32 update, q <= 64 output columns and K = k1 + k2 + k3 <= 192
// (the retraction and projection updates of the FP32 phase at p <= 64):
// persistent blocks keep the whole coefficient matrix [C1; C2] (K x 64, zero
// padded) in shared memory for the life of the block and stream row tiles
// of 128 rows of [A1, A2] through a double-buffered stage of 32 K-values,
// the next stage (of this tile or of the block's next tile) loaded into
// registers while the current one is consumed.  Thread (ty, tx) of 16 x 16
// owns rows 8 ty .. 8 ty + 7 and columns 4 tx .. 4 tx + 3 of a tile: 32 FMAs
// per three vector shared-memory loads.  Each output is the same K-ascending
// FMA chain (A1 C1, then A2 C2) and the same final alpha/beta step as
// combine_tile_body, so the two kernels give bitwise-equal results for two
// blocks.  A third block (A3 C3) and a second output out2 = add2 + out
// serve the increment form's retraction in one pass.
constexpr int kTsRows = 128, kTsK = 32, kTsMaxK = 192, kTsLd = kTsRows + 4;

size_t combine_ts_smem(int K) {
  const int nst = (K + kTsK - 1) / kTsK;
  return ((size_t)nst * kTsK * kTile + (size_t)2 * kTsK * kTsLd) * sizeof(float);
}

// Optional outputs of the tall-skinny update's epilogue: the density of the
// new iterate (rho set) and whether every array allows 16-byte accesses.
struct TsDensity {
  const double *rho_b = nullptr;
  double *rho = nullptr;
  double occ = 0.0;
  int vec = 0;
};

// Epilogue of the tall-skinny update for one thread's 8 rows (row0 ..
// row0 + 7) x 4 columns (4 tx .. 4 tx + 3): out = alpha acc + beta Bm and
// out2 = add2 + out, 16-byte accesses when the four columns are in range and
// every array is 16-byte aligned.  With dn.rho set (out2 the FP32 copy of
// X_b + delta, add2 = X_b, out = delta) it also forms the density of the
// new iterate in the increment form, rho = rho_b + f sum delta (2 X_b +
// delta) (Sec. 2.3, rho = diag(X X^T) per occupied orbital): the 16 threads
// of a row (the lanes tx of one half-warp) sum their columns by a butterfly.
// The accumulators are cleared for the next tile.
__device__ __forceinline__ void ts_epilogue(long long n, int q, long long row0, int tx,
                                            float (&acc)[8][4], float alpha, float beta,
                                            const float *__restrict__ Bm, float *__restrict__ out,
                                            const float *__restrict__ add2,
                                            float *__restrict__ out2, const TsDensity &dn) {
  const int col0 = 4 * tx;
  const bool vec = dn.vec && col0 + 3 < q;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const long long row = row0 + i;
    float dsum = 0.f;
    if (row < n) {
      const long long o = row * q + col0;
      if (vec && KS_IN(o + 3, n * q)) {
        float4 v = make_float4(alpha * acc[i][0], alpha * acc[i][1], alpha * acc[i][2],
                               alpha * acc[i][3]);
        if (Bm) {
          const float4 b = *reinterpret_cast<const float4 *>(Bm + o);
          v.x = fmaf(beta, b.x, v.x); v.y = fmaf(beta, b.y, v.y);
          v.z = fmaf(beta, b.z, v.z); v.w = fmaf(beta, b.w, v.w);
        }
        *reinterpret_cast<float4 *>(out + o) = v;
        if (out2) {
          const float4 h = *reinterpret_cast<const float4 *>(add2 + o);
          *reinterpret_cast<float4 *>(out2 + o) =
              make_float4(h.x + v.x, h.y + v.y, h.z + v.z, h.w + v.w);
          if (dn.rho) {
            dsum = fmaf(v.x, fmaf(2.f, h.x, v.x), dsum);
            dsum = fmaf(v.y, fmaf(2.f, h.y, v.y), dsum);
            dsum = fmaf(v.z, fmaf(2.f, h.z, v.z), dsum);
            dsum = fmaf(v.w, fmaf(2.f, h.w, v.w), dsum);
          }
        }
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          if (col0 + j < q && KS_IN(o + j, n * q)) {
            float v = alpha * acc[i][j];
            if (Bm) v = fmaf(beta, Bm[o + j], v);
            out[o + j] = v;
            if (out2) {
              const float h = add2[o + j];
              out2[o + j] = h + v;
              if (dn.rho) dsum = fmaf(v, fmaf(2.f, h, v), dsum);
            }
          }
        }
      }
    }
    if (dn.rho) {
#pragma unroll
      for (int s = 8; s > 0; s >>= 1) dsum += __shfl_xor_sync(0xffffffffu, dsum, s);
      if (tx == 0 && row < n) dn.rho[row] = dn.rho_b[row] + dn.occ * (double)dsum;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
  }
}

__global__ void __launch_bounds__(256, 2) combine_ts_kernel(
    long long n, int q, const float *__restrict__ A1, int k1, const float *__restrict__ c1,
    const float *__restrict__ A2, int k2, const float *__restrict__ c2,
    const float *__restrict__ A3, int k3, const float *__restrict__ c3, float alpha, float beta,
    const float *__restrict__ Bm, float *__restrict__ out, const float *__restrict__ add2,
    float *__restrict__ out2, long long ntiles, TsDensity dn) {
  extern __shared__ __align__(16) float ts_smem[];
  const int k12 = k1 + (A2 ? k2 : 0);
  const int K = k12 + (A3 ? k3 : 0);
  const int nst = (K + kTsK - 1) / kTsK;
  float *Cs = ts_smem;                              // [nst * kTsK][64]
  float *As = ts_smem + (size_t)nst * kTsK * kTile;  // [2][kTsK][kTsLd]
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  for (int e = tid; e < nst * kTsK * kTile; e += 256) {
    const int r = e / kTile, c = e % kTile;
    float v = 0.f;
    if (c < q) {
      if (r < k1) v = c1[(long long)r * q + c];
      else if (r < k12) v = c2[(long long)(r - k1) * q + c];
      else if (r < K) v = c3[(long long)(r - k12) * q + c];
    }
    Cs[e] = v;
  }
  const long long mine = ntiles > blockIdx.x ? (ntiles - blockIdx.x + gridDim.x - 1) / gridDim.x : 0;
  const long long W = mine * nst;                   // (tile, stage) steps of this block
  constexpr int kPer = kTsRows * kTsK / 256;       // staged A values per thread
  float ra[kPer];
  auto fetch = [&](long long w) {
    const long long tile = blockIdx.x + (w / nst) * gridDim.x;
    const int k0 = (int)(w % nst) * kTsK;
#pragma unroll
    for (int t = 0; t < kPer; ++t) {
      const int idx = tid + t * 256;
      const int rr = idx / kTsK, kk = idx % kTsK;
      const long long row = tile * kTsRows + rr;
      const int k = k0 + kk;
      float v = 0.f;
      if (row < n) {
        if (k < k1) v = A1[row * k1 + k];
        else if (k < k12) v = A2[row * k2 + (k - k1)];
        else if (k < K) v = A3[row * k3 + (k - k12)];
      }
      ra[t] = v;
    }
  };
  auto stash = [&](int buf) {
#pragma unroll
    for (int t = 0; t < kPer; ++t) {
      const int idx = tid + t * 256;
      As[((size_t)buf * kTsK + idx % kTsK) * kTsLd + idx / kTsK] = ra[t];
    }
  };
  float acc[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
  if (W > 0) {
    fetch(0);
    stash(0);
  }
  __syncthreads();
  for (long long w = 0; w < W; ++w) {
    const int buf = (int)(w & 1);
    const bool more = w + 1 < W;
    if (more) fetch(w + 1);
    const int k0 = (int)(w % nst) * kTsK;
    const float *Ab = As + (size_t)buf * kTsK * kTsLd;
#pragma unroll 8
    for (int k = 0; k < kTsK; ++k) {
      const float4 a0 = *reinterpret_cast<const float4 *>(Ab + k * kTsLd + 8 * ty);
      const float4 a1 = *reinterpret_cast<const float4 *>(Ab + k * kTsLd + 8 * ty + 4);
      const float4 cv = *reinterpret_cast<const float4 *>(Cs + (size_t)(k0 + k) * kTile + 4 * tx);
      const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      const float cc[4] = {cv.x, cv.y, cv.z, cv.w};
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], cc[j], acc[i][j]);
    }
    if (w % nst == nst - 1) {
      const long long tile = blockIdx.x + (w / nst) * gridDim.x;
      ts_epilogue(n, q, tile * kTsRows + 8 * ty, tx, acc, alpha, beta, Bm, out, add2, out2, dn);
    }
    if (more) stash(buf ^ 1);
    __syncthreads();
  }
}

static void launch_ts(Problem &P, int q, const float *A1, int k1, const float *c1,
                      const float *A2, int k2, const float *c2, const float *A3, int k3,
                      const float *c3, float alpha, float beta, const float *Bm, float *out,
                      const float *add2, float *out2, TsDensity dn = TsDensity());

// FP32 copies of the update coefficients (one launch for both matrices).
__global__ void coef_convert_kernel(long long len1, const double *__restrict__ C1,
                                    float *__restrict__ c1, long long len2,
                                    const double *__restrict__ C2, float *__restrict__ c2) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e < len1) c1[e] = (float)C1[e];
  else if (e < len1 + len2) c2[e - len1] = (float)C2[e - len1];
}

template <typename T>
ks_status launch_combine(Problem &P, const T *A1, int k1, const double *C1, const T *A2, int k2,
                         const double *C2, double alpha, double beta, const T *Bm, T *out, int q) {
  if (sizeof(T) == 8 && combine_oz_applies(P, k1, A2 ? k2 : 0, q))
    return launch_combine_oz(P, (const double *)A1, k1, C1, (const double *)A2, k2, C2, alpha,
                             beta, (const double *)Bm, (double *)out, q);
  if (sizeof(T) == 4 && q > kNarrowQ && use_tensor_cores(P, k1, q))
    return launch_combine_tc(P, (const float *)A1, k1, C1, (const float *)A2, k2, C2, alpha, beta,
                             (const float *)Bm, (float *)out, q);
  if (q <= kNarrowQ && k1 <= kNarrowK && (!A2 || k2 <= kNarrowK)) {
    const long long total = (long long)P.n * ((q + kNarrowCols - 1) / kNarrowCols);
    long long nb = (total + 255) / 256;
    if (nb > 32LL * P.sms) nb = 32LL * P.sms;
    {
      ProfScope ps_(P.stream, KP_COMBINE, 2.0 * P.n * q * (k1 + (A2 ? k2 : 0)),
                    (double)P.n * ((k1 + (A2 ? k2 : 0)) + q * (Bm ? 2 : 1)) * sizeof(T));
      bool rows = false;
      if constexpr (sizeof(T) == 4) {
        rows = narrow_rows_applies(P, k1 + (A2 ? k2 : 0), q);
        if (rows)
          combine_narrow_kernel<T, true><<<(int)nb, 256, 0, P.stream>>>(
              P.n, q, A1, k1, C1, A2, k2, C2, alpha, beta, Bm, out);
      }
      if (!rows)
        combine_narrow_kernel<T, false><<<(int)nb, 256, 0, P.stream>>>(
            P.n, q, A1, k1, C1, A2, k2, C2, alpha, beta, Bm, out);
    }
    KS_CUDA_TRY(cudaGetLastError());
    return KS_OK;
  }
  dim3 grid((unsigned)((P.n + kTile - 1) / kTile), (unsigned)((q + kTile - 1) / kTile));
  if (sizeof(T) == 4) {
    float *c1 = P.cf, *c2 = P.cf + (size_t)P.p * P.p;
    const long long len1 = (long long)k1 * q, len2 = A2 ? (long long)k2 * q : 0;
    {
      ProfScope ps_(P.stream, KP_REDUCE);
      coef_convert_kernel<<<(int)((len1 + len2 + 255) / 256), 256, 0, P.stream>>>(
          len1, C1, c1, len2, C2, c2);
    }
    KS_CUDA_TRY(cudaGetLastError());
    const int K = k1 + (A2 ? k2 : 0);
    // tensor cores: beta Bm enters as a third operand with the coefficient
    // beta I, alpha scales the other coefficients
    if (combine_tc64_applies(P, q, {k1, A2 ? k2 : 0, Bm ? q : 0}, {A1, A2, Bm, out}))
      return launch_combine_tc64(P, q, (const float *)A1, k1, c1, (float)alpha,
                                 (const float *)A2, k2, A2 ? c2 : nullptr, (float)alpha,
                                 (const float *)Bm, q, nullptr, (float)beta, (float *)out,
                                 nullptr, nullptr, nullptr);
    if (q <= kTile && K <= kTsMaxK) {
      ProfScope ps_(P.stream, KP_COMBINE, 2.0 * P.n * q * K,
                    (double)P.n * (K + q * (Bm ? 2 : 1)) * sizeof(T));
      launch_ts(P, q, (const float *)A1, k1, c1, (const float *)A2, k2, A2 ? c2 : nullptr, nullptr,
                0, nullptr, (float)alpha, (float)beta, (const float *)Bm, (float *)out, nullptr,
                nullptr);
      KS_CUDA_TRY(cudaGetLastError());
      return KS_OK;
    }
    ProfScope ps_(P.stream, KP_COMBINE, 2.0 * P.n * q * (k1 + (A2 ? k2 : 0)),
                  (double)P.n * ((k1 + (A2 ? k2 : 0)) + q * (Bm ? 2 : 1)) * sizeof(T));
    combine_kernel<T, float><<<grid, 256, 0, P.stream>>>(P.n, q, A1, k1, c1, A2, k2,
                                                         A2 ? c2 : nullptr, alpha, beta, Bm, out);
  } else {
    ProfScope ps_(P.stream, KP_COMBINE, 2.0 * P.n * q * (k1 + (A2 ? k2 : 0)),
                  (double)P.n * ((k1 + (A2 ? k2 : 0)) + q * (Bm ? 2 : 1)) * sizeof(T));
    combine_kernel<T, double><<<grid, 256, 0, P.stream>>>(P.n, q, A1, k1, C1, A2, k2, C2, alpha,
                                                          beta, Bm, out);
  }
  KS_CUDA_TRY(cudaGetLastError());
  return KS_OK;
}

// ---------------------------------------------------------------- batched
// Grams of every active job: tiles x chunks blocks per job (64-tile kernel)
// or chunks blocks (p <= kSmallPQ), then the chunk sums into pp + smOut p^2.
template <typename T>
__global__ void __launch_bounds__(256) gram_batch_kernel(const BJob *__restrict__ jobs,
                                                         const int *__restrict__ start, int J,
                                                         const unsigned char *__restrict__ active,
                                                         int sA, int sB, int small) {
  const int j = batch_job_of(start, J, blockIdx.x);
  if (!active[j]) return;
  const BJob &b = jobs[j];
  const int vb = blockIdx.x - start[j];
  const T *A = (const T *)b.blk[sA], *Bp = (const T *)b.blk[sB];
  if (small == 1) {
    gram_small_body<T>(b.n, b.p, b.p, b.gram_rows_per, A, Bp, b.partials, vb);
  } else if (small == 2) {
    gram_mid_body<T>(b.n, b.p, b.p, b.gram_rows_per, A, Bp, b.partials, vb);
  } else {
    const int tiles = ((b.p + kTile - 1) / kTile) * ((b.p + kTile - 1) / kTile);
    gram_tile_body<T>(b.n, b.p, b.p, b.gram_rows_per, A, Bp, b.partials, vb % tiles, vb / tiles);
  }
}

__global__ void gram_reduce_batch_kernel(const BJob *__restrict__ jobs,
                                         const int *__restrict__ start, int J,
                                         const unsigned char *__restrict__ active, int smOut) {
  const int j = batch_job_of(start, J, blockIdx.x);
  if (!active[j]) return;
  const BJob &b = jobs[j];
  const long long t = (long long)(blockIdx.x - start[j]) * blockDim.x + threadIdx.x;
  const long long len = (long long)b.p * b.p;
  const long long e = t >> 3;
  const int sub = (int)(t & 7);
  double acc = 0.0;
  if (e < len)
    for (int c = sub; c < b.gram_chunks; c += 8) acc += b.partials[(long long)c * len + e];
  acc += __shfl_xor_sync(0xffffffffu, acc, 1);
  acc += __shfl_xor_sync(0xffffffffu, acc, 2);
  acc += __shfl_xor_sync(0xffffffffu, acc, 4);
  if (sub == 0 && e < len) b.pp[(size_t)smOut * len + e] = acc;
}

template <typename T>
ks_status batch_gram(Batch &B, int sA, int sB, int smOut) {
  for (int small = 2; small >= 0; --small) {
    const int m = small == 2 ? BM_GRAM_MID : small == 1 ? BM_GRAM_SMALL : BM_GRAM_TILED;
    const int nb = B.total(m);
    if (nb == 0) continue;
    {
      ProfScope ps_(B.stream, KP_GRAM);
      gram_batch_kernel<T><<<nb, 256, 0, B.stream>>>(B.jobs_dev, B.map(m), B.J, B.active_dev, sA,
                                                     sB, small);
    }
    KS_CUDA_TRY(cudaGetLastError());
  }
  const int nr = B.total(BM_GRAM_REDUCE);
  {
    ProfScope ps_(B.stream, KP_REDUCE);
    gram_reduce_batch_kernel<<<nr, kThreads, 0, B.stream>>>(B.jobs_dev, B.map(BM_GRAM_REDUCE), B.J,
                                                            B.active_dev, smOut);
  }
  KS_CUDA_TRY(cudaGetLastError());
  return KS_OK;
}

// out = alpha (A1 C1 + A2 C2) + beta Bm with q = k1 = k2 = p per job; C from
// pp (FP64; the 64-tile form of the FP32 phase reads the FP32 copies that
// coef_batch_kernel leaves in cf).
struct CombSlots {
  int a1, c1, a2, c2, bm, out;
  double alpha, beta;
};

__global__ void coef_batch_kernel(const BJob *__restrict__ jobs, const int *__restrict__ start,
                                  int J, const unsigned char *__restrict__ active, int smC1,
                                  int smC2) {
  const int j = batch_job_of(start, J, blockIdx.x);
  if (!active[j]) return;
  const BJob &b = jobs[j];
  const long long len = (long long)b.p * b.p;
  const long long e = (long long)(blockIdx.x - start[j]) * blockDim.x + threadIdx.x;
  if (e < len) b.cf[e] = (float)b.pp[(size_t)smC1 * len + e];
  else if (smC2 >= 0 && e < 2 * len) b.cf[e] = (float)b.pp[(size_t)smC2 * len + e - len];
}

// (two kernels, so that each form has its own registers and shared memory)
template <typename T, bool Narrow>
__global__ void __launch_bounds__(256) combine_batch_kernel(const BJob *__restrict__ jobs,
                                                            const int *__restrict__ start, int J,
                                                            const unsigned char *__restrict__ active,
                                                            CombSlots sl) {
  const int j = batch_job_of(start, J, blockIdx.x);
  if (!active[j]) return;
  const BJob &b = jobs[j];
  const int p = b.p;
  const long long len = (long long)p * p;
  const int vb = blockIdx.x - start[j];
  const T *A1 = (const T *)b.blk[sl.a1];
  const T *A2 = sl.a2 >= 0 ? (const T *)b.blk[sl.a2] : nullptr;
  const T *Bm = sl.bm >= 0 ? (const T *)b.blk[sl.bm] : nullptr;
  T *out = (T *)b.blk[sl.out];
  const double *C1 = b.pp + (size_t)sl.c1 * len;
  const double *C2 = sl.c2 >= 0 ? b.pp + (size_t)sl.c2 * len : nullptr;
  if constexpr (Narrow) {
    if constexpr (sizeof(T) == 4)
      combine_rows_body(b.n, p, A1, p, C1, A2, p, C2, (float)sl.alpha, (float)sl.beta, Bm, out,
                        vb, b.comb_nb);
    else
      combine_narrow_body<T>(b.n, p, A1, p, C1, A2, p, C2, sl.alpha, sl.beta, Bm, out, vb,
                             b.comb_nb);
  } else {
    const int ct = (p + kTile - 1) / kTile;
    if (sizeof(T) == 4)
      combine_tile_body<T, float>(b.n, p, A1, p, b.cf, A2, p, C2 ? b.cf + len : nullptr,
                                  sl.alpha, sl.beta, Bm, out, vb / ct, vb % ct);
    else
      combine_tile_body<T, double>(b.n, p, A1, p, C1, A2, p, C2, sl.alpha, sl.beta, Bm, out,
                                   vb / ct, vb % ct);
  }
}

template <typename T>
ks_status batch_combine(Batch &B, int sA1, int smC1, int sA2, int smC2, double alpha, double beta,
                        int sBm, int sOut) {
  const CombSlots sl{sA1, smC1, sA2, smC2, sBm, sOut, alpha, beta};
  const int nt = B.total(BM_COMB_TILED);
  if (sizeof(T) == 4 && nt > 0) {
    {
      ProfScope ps_(B.stream, KP_REDUCE);
      coef_batch_kernel<<<B.total(BM_COEF), kThreads, 0, B.stream>>>(
          B.jobs_dev, B.map(BM_COEF), B.J, B.active_dev, smC1, sA2 >= 0 ? smC2 : -1);
    }
    KS_CUDA_TRY(cudaGetLastError());
  }
  for (int narrow = 1; narrow >= 0; --narrow) {
    const int m = narrow ? BM_COMB_NARROW : BM_COMB_TILED;
    const int nb = B.total(m);
    if (nb == 0) continue;
    {
      ProfScope ps_(B.stream, KP_COMBINE);
      if (narrow)
        combine_batch_kernel<T, true><<<nb, 256, 0, B.stream>>>(B.jobs_dev, B.map(m), B.J,
                                                                B.active_dev, sl);
      else
        combine_batch_kernel<T, false><<<nb, 256, 0, B.stream>>>(B.jobs_dev, B.map(m), B.J,
                                                                 B.active_dev, sl);
    }
    KS_CUDA_TRY(cudaGetLastError());
  }
  return KS_OK;
}

// Precision conversion / copy of a block of every active job.
template <typename A, typename Bt>
__global__ void convert_batch_kernel(const BJob *__restrict__ jobs, const int *__restrict__ start,
                                     int J, const unsigned char *__restrict__ active, int sIn,
                                     int sOut) {
  const int j = batch_job_of(start, J, blockIdx.x);
  if (!active[j]) return;
  const BJob &b = jobs[j];
  const long long total = b.n * b.p;
  const A *in = (const A *)b.blk[sIn];
  Bt *out = (Bt *)b.blk[sOut];
  const long long base = (long long)(blockIdx.x - start[j]) * blockDim.x * 4 + threadIdx.x;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const long long e = base + (long long)u * blockDim.x;
    if (e < total) out[e] = (Bt)in[e];
  }
}

template <typename Tin, typename Tout>
ks_status batch_convert(Batch &B, int sIn, int sOut) {
  {
    ProfScope ps_(B.stream, KP_OTHER);
    convert_batch_kernel<Tin, Tout><<<B.total(BM_COPY), kThreads, 0, B.stream>>>(
        B.jobs_dev, B.map(BM_COPY), B.J, B.active_dev, sIn, sOut);
  }
  KS_CUDA_TRY(cudaGetLastError());
  return KS_OK;
}

// ||O - I||_F^2 of every active job into its scalar row.
__global__ void ortho_err_batch_kernel(const BJob *__restrict__ jobs,
                                       const unsigned char *__restrict__ active, int smO) {
  const int j = blockIdx.x;
  if (!active[j]) return;
  const BJob &b = jobs[j];
  __shared__ double smem[33];
  const int p = b.p;
  const double *O = b.pp + (size_t)smO * p * p;
  double acc = 0.0;
  for (int e = threadIdx.x; e < p * p; e += blockDim.x) {
    const int i = e / p, k = e % p;
    const double d = O[e] - (i == k ? 1.0 : 0.0);
    acc = fma(d, d, acc);
  }
  const double s = block_sum(acc, smem);
  if (threadIdx.x == 0) b.scal[SC_ORTHO] = s;
}

ks_status batch_ortho_err(Batch &B, int smO) {
  {
    ProfScope ps_(B.stream, KP_REDUCE);
    ortho_err_batch_kernel<<<B.J, kThreads, 0, B.stream>>>(B.jobs_dev, B.active_dev, smO);
  }
  KS_CUDA_TRY(cudaGetLastError());
  return KS_OK;
}

template ks_status batch_gram<double>(Batch &, int, int, int);
template ks_status batch_gram<float>(Batch &, int, int, int);
template ks_status batch_combine<double>(Batch &, int, int, int, int, double, double, int, int);
template ks_status batch_combine<float>(Batch &, int, int, int, int, double, double, int, int);
template ks_status batch_convert<double, float>(Batch &, int, int);
template ks_status batch_convert<float, double>(Batch &, int, int);
template ks_status batch_convert<double, double>(Batch &, int, int);
template ks_status batch_convert<float, float>(Batch &, int, int);

template ks_status launch_gram<double>(Problem &, const double *, int, const double *, int,
                                       double *);
template ks_status launch_gram<float>(Problem &, const float *, int, const float *, int, double *);
// Warp form of the tall-skinny update (combine_wa_kernel below).
constexpr int kWaStages = 3, kWaR = 8, kWaRows = 4 * kWaR, kWaK = 32, kWaLd = kWaK + 4;
constexpr int kWaWarps = 12;

// Half h of the epilogue for one lane: rows row0 + 4 i, columns 32 h + 4 tx ..
// + 3 of out = alpha acc + beta Bm and out2 = add2 + out; `staged` holds this
// half of Bm or add2 in shared memory (row stride kWaLd).  dsum[i] gathers
// the row's density increment (ts_epilogue).
__device__ __forceinline__ void wa_half(long long n, int q, long long row0, int tx, int h,
                                        f2_t (&acc)[kWaR][4], float alpha, float beta,
                                        const float *staged, bool with_b, float *__restrict__ out,
                                        float *__restrict__ out2, bool vec, bool dens,
                                        float (&dsum)[kWaR]) {
  const int col0 = 32 * h + 4 * tx;
#pragma unroll
  for (int i = 0; i < kWaR; ++i) {
    const long long row = row0 + 4 * i, o = row * q + col0;
    const float4 s4 = staged ? *reinterpret_cast<const float4 *>(staged + 4 * i * kWaLd)
                             : make_float4(0.f, 0.f, 0.f, 0.f);
    const float s[4] = {s4.x, s4.y, s4.z, s4.w};
    float v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float lo, hi;
      f2_split(acc[i][2 * h + (j >> 1)], lo, hi);
      v[j] = alpha * ((j & 1) ? hi : lo);
      if (with_b) v[j] = fmaf(beta, s[j], v[j]);
    }
    if (row < n && vec && col0 + 3 < q && KS_IN(o + 3, n * q)) {
      *reinterpret_cast<float4 *>(out + o) = make_float4(v[0], v[1], v[2], v[3]);
      if (out2)
        *reinterpret_cast<float4 *>(out2 + o) =
            make_float4(s[0] + v[0], s[1] + v[1], s[2] + v[2], s[3] + v[3]);
    } else if (row < n) {
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (col0 + j < q && KS_IN(o + j, n * q)) {
          out[o + j] = v[j];
          if (out2) out2[o + j] = s[j] + v[j];
        }
    }
    if (dens)
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (col0 + j < q) dsum[i] = fmaf(v[j], fmaf(2.f, s[j], v[j]), dsum[i]);
  }
}

// Pipelined form of combine_ts_kernel for 16-byte-aligned operands (every k
// a multiple of 4 and every A base 16-byte aligned).  FP32 FMAs bound it
// (6.4 GFLOP against 336 MB for the retraction at 64^3 x 64), and next to them
// shared memory, which delivers 128 bytes per clock against 128 FMAs: an
// 8 x 4 block of outputs per thread reads 1.5 bytes per FMA, the 8 x 8 block
// per lane here one.  Each warp runs alone on tiles of 32 rows, with its own
// ring of kWaStages stages (32 rows x kWaK K-values, cp.async 16 bytes per copy,
// zero-filled past the last row and past K) and no block barrier, so one warp's
// epilogue overlaps the others' products.  The epilogue's operand (Bm or
// add2) follows the K stages through the ring as two more stages: read from
// global memory in the epilogue, its 16 loads per lane waited one by one (one
// stage where q <= kWaK).  A lane owns rows ty + 4 i (i < 8) and columns 4 tx .. + 3
// and 32 + 4 tx .. + 3 (ty = lane / 8, tx = lane % 8).  The coefficient image (K x
// 64, zero padded) is shared by the block's warps, and the FMAs are packed pairs of
// columns
// (f2_fma: the scalar outer product stops at 49 of 76 TF/s).  Update with Bm at
// 64^3, K = 128: 134 us for the block-synchronous 8 x 4 form (32 TF/s), 107 us
// here (40 TF/s); 16 x 8 per lane (8 warps) took 168 us.
// The FMA chains and the final step are those of combine_ts_kernel (K
// ascending).

size_t combine_wa_smem(int K) {
  const int nst = (K + kWaK - 1) / kWaK;
  return ((size_t)nst * kWaK * kTile + (size_t)kWaWarps * kWaStages * kWaRows * kWaLd) *
         sizeof(float);
}

__global__ void __launch_bounds__(32 * kWaWarps, 1) combine_wa_kernel(
    long long n, int q, const float *__restrict__ A1, int k1, const float *__restrict__ c1,
    const float *__restrict__ A2, int k2, const float *__restrict__ c2,
    const float *__restrict__ A3, int k3, const float *__restrict__ c3, float alpha, float beta,
    const float *__restrict__ Bm, float *__restrict__ out, const float *__restrict__ add2,
    float *__restrict__ out2, long long ntiles, TsDensity dn) {
  extern __shared__ __align__(16) float wa_smem[];
  const int k12 = k1 + (A2 ? k2 : 0);
  const int K = k12 + (A3 ? k3 : 0);
  const int nst = (K + kWaK - 1) / kWaK;
  // the epilogue's operand: at most one of Bm (added) and add2 (to out2)
  const float *Es = Bm ? Bm : add2;
  // one stage per kWaK of its q columns: for q <= kWaK a second one would lie
  // past its rows
  const int ntot = nst + (Es ? (q + kWaK - 1) / kWaK : 0);
  float *Cs = wa_smem;                                  // [nst * kWaK][64]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, ty = lane >> 3, tx = lane & 7;
  constexpr int kRing = kWaStages * kWaRows * kWaLd;
  float *As = wa_smem + (size_t)nst * kWaK * kTile + (size_t)warp * kRing;
  for (int e = threadIdx.x; e < nst * kWaK * kTile; e += 32 * kWaWarps) {
    const int r = e / kTile, c = e % kTile;
    float v = 0.f;
    if (c < q) {
      if (r < k1) v = c1[(long long)r * q + c];
      else if (r < k12) v = c2[(long long)(r - k1) * q + c];
      else if (r < K) v = c3[(long long)(r - k12) * q + c];
    }
    Cs[e] = v;
  }
  // this warp's tiles: (warp + kWaWarps j) gridDim + block, so that the tiles
  // spread evenly over the blocks
  const long long first = (long long)warp * gridDim.x + blockIdx.x;
  const long long step = (long long)kWaWarps * gridDim.x;
  const long long mine = ntiles > first ? (ntiles - first + step - 1) / step : 0;
  const long long W = mine * ntot;
  int istage = 0;                                       // K stage and tile of the next issue
  long long itile = first;
  int ibuf = 0;
  // widths that are multiples of kWaK (q = 32 or 64): a stage lies in one operand, so
  // its copies share one base and one bound.  step_combine_f32 with Bm at 64^3, each copy
  // looking for its operand against this: k = 64, q = 64 97 / 88 us, 64 + 64, 64 142 /
  // 138, 96, 32 112 / 105; at 32^3 even
  const bool whole = k1 % kWaK == 0 && k12 % kWaK == 0 && K % kWaK == 0 && q % kWaK == 0;
  auto issue = [&]() {
    const int k0 = istage * kWaK;
    float *dst = As + ibuf * (kWaRows * kWaLd);
    if (whole) {
      const float *M = Es;
      int ld = q, kc = k0 - K;
      if (k0 < k1) { M = A1; ld = k1; kc = k0; }
      else if (k0 < k12) { M = A2; ld = k2; kc = k0 - k1; }
      else if (k0 < K) { M = A3; ld = k3; kc = k0 - k12; }
      const long long row0 = itile * kWaRows + (lane >> 3);
      const float *src = M + row0 * ld + kc + (lane & 7) * 4;
      const uint32_t d0 = smem_addr(dst + (lane >> 3) * kWaLd + (lane & 7) * 4);
#pragma unroll
      for (int t = 0; t < kWaRows / 4; ++t) {
        const bool in = row0 + 4 * t < n && KS_IN(kc + (lane & 7) * 4 + 3, ld);
        cp_async16(d0 + t * 4 * kWaLd * 4, in ? src + (long long)4 * t * ld : M, in ? 16u : 0u);
      }
    } else
#pragma unroll
    for (int t = 0; t < kWaRows * kWaK / 128; ++t) {
      const int rr = (lane >> 3) + 4 * t, kq = (lane & 7) * 4;
      const long long row = itile * kWaRows + rr;
      const int k = k0 + kq;
      const float *src = A1;
      uint32_t bytes = 0;
      if (istage >= nst) {
        const int c = (istage - nst) * kWaK + kq;
        if (row < n && c < q && KS_IN(row * q + c + 3, n * q)) { src = Es + row * q + c; bytes = 16; }
      } else if (row < n) {
        if (k < k1) {
          if (KS_IN(row * k1 + k + 3, n * k1)) { src = A1 + row * k1 + k; bytes = 16; }
        } else if (k < k12) {
          if (KS_IN(row * k2 + (k - k1) + 3, n * k2)) { src = A2 + row * k2 + (k - k1); bytes = 16; }
        } else if (k < K) {
          if (KS_IN(row * k3 + (k - k12) + 3, n * k3)) { src = A3 + row * k3 + (k - k12); bytes = 16; }
        }
      }
      const int di = rr * kWaLd + kq;
      if (KS_IN(di + 3, kWaRows * kWaLd)) cp_async16(smem_addr(dst + di), src, bytes);
    }
    if (++istage == ntot) {
      istage = 0;
      itile += step;
    }
    if (++ibuf == kWaStages) ibuf = 0;
  };
  f2_t acc[kWaR][4];
  float dsum[kWaR];
#pragma unroll
  for (int i = 0; i < kWaR; ++i) dsum[i] = 0.f;
#pragma unroll
  for (int i = 0; i < kWaR; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
  for (int st = 0; st < kWaStages - 1; ++st) {
    if (st < W) issue();
    cp_async_commit();
  }
  __syncthreads();                                      // C staged
  int stage = 0, buf = 0;
  long long tile = first;
  for (long long w = 0; w < W; ++w) {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(kWaStages - 2) : "memory");  // stage w landed
    __syncwarp();                                       // ... every lane's; stage w - 1 consumed
    if (w + kWaStages - 1 < W) issue();
    cp_async_commit();
    const float *Ab = As + buf * (kWaRows * kWaLd) + ty * kWaLd;
    if (stage < nst) {
      const float *Cb = Cs + (size_t)stage * kWaK * kTile + 4 * tx;
#pragma unroll 1
      for (int kq = 0; kq < kWaK; kq += 4) {
        float4 a[kWaR];
#pragma unroll
        for (int i = 0; i < kWaR; ++i)
          a[i] = *reinterpret_cast<const float4 *>(Ab + 4 * i * kWaLd + kq);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          const ulonglong2 lo = *reinterpret_cast<const ulonglong2 *>(Cb + (kq + kk) * kTile);
          const ulonglong2 hi = *reinterpret_cast<const ulonglong2 *>(Cb + (kq + kk) * kTile + 32);
          const f2_t cc[4] = {lo.x, lo.y, hi.x, hi.y};
#pragma unroll
          for (int i = 0; i < kWaR; ++i) {
            const f2_t av = f2_dup(kk == 0 ? a[i].x : kk == 1 ? a[i].y : kk == 2 ? a[i].z : a[i].w);
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = f2_fma(av, cc[j], acc[i][j]);
          }
        }
      }
    }
    const long long row0 = tile * kWaRows + ty;
    if (Es ? stage >= nst : stage == nst - 1) {
#pragma unroll
      for (int h = 0; h < 2; ++h)
        if (!Es || stage == nst + h)
          wa_half(n, q, row0, tx, h, acc, alpha, beta, Es ? Ab + 4 * tx : nullptr, Bm != nullptr,
                  out, out2, dn.vec != 0, dn.rho != nullptr, dsum);
    }
    if (++buf == kWaStages) buf = 0;
    if (++stage == ntot) {
      if (dn.rho) {
        // the eight lanes of a row; lane tx keeps row row0 + 4 tx, so the FP64 tail
        // is one instruction per tile
        float mine_ = 0.f;
#pragma unroll
        for (int i = 0; i < kWaR; ++i) {
#pragma unroll
          for (int s = 4; s > 0; s >>= 1) dsum[i] += __shfl_xor_sync(0xffffffffu, dsum[i], s);
          if (tx == i) mine_ = dsum[i];
          dsum[i] = 0.f;
        }
        const long long row = row0 + 4 * tx;
        if (row < n) dn.rho[row] = dn.rho_b[row] + dn.occ * (double)mine_;
      }
#pragma unroll
      for (int i = 0; i < kWaR; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
      stage = 0;
      tile += step;
    }
  }
  asm volatile("cp.async.wait_all;\n" ::: "memory");
}

// The pipelined kernel applies when every 16-byte copy of A stays inside one
// row of one operand: each width a multiple of 4 and each base 16-byte aligned.
static bool ta_aligned(const float *A1, int k1, const float *A2, int k2, const float *A3, int k3) {
  auto ok = [](const float *A, int k) {
    return !A || (k % 4 == 0 && reinterpret_cast<uintptr_t>(A) % 16 == 0);
  };
  return ok(A1, k1) && ok(A2, k2) && ok(A3, k3);
}

// Launch of the tall-skinny update (pipelined when aligned).
static void launch_ts(Problem &P, int q, const float *A1, int k1, const float *c1,
                      const float *A2, int k2, const float *c2, const float *A3, int k3,
                      const float *c3, float alpha, float beta, const float *Bm, float *out,
                      const float *add2, float *out2, TsDensity dn) {
  auto al16 = [](const void *ptr) { return reinterpret_cast<uintptr_t>(ptr) % 16 == 0; };
  dn.vec = q % 4 == 0 && al16(out) && al16(Bm) && al16(add2) && al16(out2) ? 1 : 0;
  const int K = k1 + (A2 ? k2 : 0) + (A3 ? k3 : 0);
  // (the staged epilogue operand: one of Bm and add2, in 16-byte copies)
  const float *es = Bm ? Bm : add2;
  if (ta_aligned(A1, k1, A2, k2, A3, k3) && !(Bm && add2) && ta_aligned(es, q, es, q, es, q)) {
    const long long ntiles = (P.n + kWaRows - 1) / kWaRows;
    const long long nb = ntiles < P.sms ? ntiles : P.sms;
    combine_wa_kernel<<<(int)nb, 32 * kWaWarps, combine_wa_smem(K), P.stream>>>(
        P.n, q, A1, k1, c1, A2, k2, c2, A3, k3, c3, alpha, beta, Bm, out, add2, out2, ntiles, dn);
    return;
  }
  const long long ntiles = (P.n + kTsRows - 1) / kTsRows;
  long long nb = 2LL * P.sms;
  if (nb > ntiles) nb = ntiles;
  combine_ts_kernel<<<(int)nb, 256, combine_ts_smem(K), P.stream>>>(
      P.n, q, A1, k1, c1, A2, k2, c2, A3, k3, c3, alpha, beta, Bm, out, add2, out2, ntiles, dn);
}

// out = A1 C1 + A2 C2 + A3 C3 and out2 = add2 + out in one pass of the
// tall-skinny FP32 kernel (n x q blocks, q <= 64, k1 + k2 + k3 <= 192); false
// (nothing launched) for other shapes or when the tensor cores take the
// products.
bool combine3_f32_applies(const Problem &P, int k1, int k2, int k3, int q) {
  return q <= kTile && k1 + k2 + k3 <= kTsMaxK && !use_tensor_cores(P, k1, q);
}

ks_status launch_combine3_f32(Problem &P, const float *A1, int k1, const double *C1,
                              const float *A2, int k2, const double *C2, const float *A3, int k3,
                              const double *C3, float *out, const float *add2, float *out2, int q,
                              const double *rho_b, double *rho, bool images_ready) {
  if (!combine3_f32_applies(P, k1, k2, k3, q))
    return set_error(KS_EINVAL, "combine3: shape outside the tall-skinny kernel");
  // FP32 images of C1, C2, C3 one after the other in P.cf (3 p^2 floats)
  float *c1 = P.cf, *c2 = P.cf + (size_t)k1 * q, *c3 = c2 + (size_t)k2 * q;
  if ((size_t)(k1 + k2 + k3) * q > (size_t)3 * P.p * P.p)
    return set_error(KS_EINVAL, "combine3: coefficient image too small");
  const long long len1 = (long long)k1 * q, len2 = (long long)k2 * q, len3 = (long long)k3 * q;
  if (!images_ready) {
    ProfScope ps_(P.stream, KP_REDUCE);
    coef_convert_kernel<<<(int)((len1 + len2 + 255) / 256), 256, 0, P.stream>>>(len1, C1, c1,
                                                                                len2, C2, c2);
    coef_convert_kernel<<<(int)((len3 + 255) / 256), 256, 0, P.stream>>>(len3, C3, c3, 0,
                                                                         nullptr, nullptr);
  }
  KS_CUDA_TRY(cudaGetLastError());
  const int K = k1 + k2 + k3;
  // tensor cores when out2 adds A1 (the retraction: A1 = X_b): A1 goes last,
  // where the epilogue reads it back from the ring
  if (combine_tc64_applies(P, q, {k1, k2, k3}, {A1, A2, A3, out, out2}) &&
      (!out2 || (add2 == A1 && k1 == q))) {
    const bool dens = rho && out2 && q == P.p;
    return launch_combine_tc64(P, q, A2, k2, c2, 1.0f, A3, k3, c3, 1.0f, A1, k1, c1, 1.0f, out,
                               out2, dens ? rho_b : nullptr, dens ? rho : nullptr);
  }
  {
    ProfScope ps_(P.stream, KP_COMBINE, 2.0 * P.n * q * K,
                  (double)P.n * (K + q * (out2 ? 3 : 1)) * sizeof(float));
    TsDensity dn;
    if (rho && add2 && out2 && q == P.p) {
      dn.rho_b = rho_b;
      dn.rho = rho;
      dn.occ = P.occ;
    }
    launch_ts(P, q, A1, k1, c1, A2, k2, c2, A3, k3, c3, 1.0f, 0.0f, nullptr, out, add2, out2, dn);
  }
  KS_CUDA_TRY(cudaGetLastError());
  return KS_OK;
}

// Dynamic shared memory of the tall-skinny update beyond the default 48 KiB
// (on the current device; called when a problem is created).
ks_status configure_blas_kernels() {
  KS_CUDA_TRY(cudaFuncSetAttribute(gram2_wa_kernel<true>,
                                   cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)gram_wa_smem()));
  KS_CUDA_TRY(cudaFuncSetAttribute(gram2_wa_kernel<false>,
                                   cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)gram_wa_smem()));
  KS_CUDA_TRY(cudaFuncSetAttribute(combine_ts_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)combine_ts_smem(kTsMaxK)));
  KS_CUDA_TRY(cudaFuncSetAttribute(combine_wa_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)combine_wa_smem(kTsMaxK)));
  return KS_OK;
}

template ks_status launch_combine<double>(Problem &, const double *, int, const double *,
                                          const double *, int, const double *, double, double,
                                          const double *, double *, int);
template ks_status launch_combine<float>(Problem &, const float *, int, const double *,
                                         const float *, int, const double *, double, double,
                                         const float *, float *, int);

template <typename A, typename B>
__global__ void convert_kernel(long long total, const A *__restrict__ in, B *__restrict__ out) {
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x)
    out[e] = (B)in[e];
}

template <typename A, typename B>
static ks_status convert_impl(Problem &P, const A *in, B *out) {
  const long long total = (long long)P.n * P.p;
  const int nb = reduce_blocks(P, total);
  {
    ProfScope ps_(P.stream, KP_OTHER);
    convert_kernel<A, B><<<nb, kThreads, 0, P.stream>>>(total, in, out);
  }
  KS_CUDA_TRY(cudaGetLastError());
  return KS_OK;
}

ks_status launch_convert(Problem &P, const double *in, float *out) { return convert_impl(P, in, out); }
ks_status launch_convert(Problem &P, const float *in, double *out) { return convert_impl(P, in, out); }

__global__ void ortho_err_kernel(int p, const double *__restrict__ O, double *out) {
  __shared__ double smem[33];
  double acc = 0.0;
  for (int e = threadIdx.x; e < p * p; e += blockDim.x) {
    const int i = e / p, j = e % p;
    const double d = O[e] - (i == j ? 1.0 : 0.0);
    acc = fma(d, d, acc);
  }
  const double s = block_sum(acc, smem);
  if (threadIdx.x == 0) *out = s;
}

ks_status launch_ortho_err(Problem &P, const double *O, double *out) {
  {
    ProfScope ps_(P.stream, KP_REDUCE);
    ortho_err_kernel<<<1, kThreads, 0, P.stream>>>(P.p, O, out);
  }
  KS_CUDA_TRY(cudaGetLastError());
  return KS_OK;
}

// ---------------------------------------------------------------- no-alloc
// Scratch of ks_gram_noalloc: the per-chunk partial Grams live in this
// file-scope device array instead of memory from cudaMalloc.  Every GPU that
// loads the library holds it (16 MiB) until the process exits.
constexpr size_t kNoAllocDoubles = size_t(1) << 21;
static __device__ __align__(256) double g_noalloc_scratch[kNoAllocDoubles];

namespace {
std::mutex g_noalloc_mu;
constexpr int kMaxDevices = 64;
double *g_noalloc_ptr[kMaxDevices] = {};
}  // namespace

KS_OOB_READER(blas)

}  // namespace ks

extern "C" ks_status ks_gram_noalloc(const double *A, int pa, const double *B, int qb,
                                     long long n, double *out, void *stream) {
  using namespace ks;
  if (!A || !B || !out) return set_error(KS_EINVAL, "null argument");
  if (pa < 1 || qb < 1 || n < 1) return set_error(KS_EINVAL, "bad sizes");
  if ((size_t)pa * (size_t)qb > kNoAllocDoubles)
    return set_error(KS_EINVAL, "ks_gram_noalloc: pa * qb = %zu exceeds the scratch capacity %zu",
                     (size_t)pa * qb, kNoAllocDoubles);
  int dev = 0;
  KS_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return set_error(KS_EINVAL, "device index out of range");
  double *scratch = nullptr;
  {
    // first call on this device: translate the array's host-side name into
    // its device address (with this device current)
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
      void *ptr = nullptr;
      KS_CUDA_TRY(cudaGetSymbolAddress(&ptr, g_noalloc_scratch));
      g_noalloc_ptr[dev] = (double *)ptr;
    }
    scratch = g_noalloc_ptr[dev];
  }
  int sms = 0;
  KS_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int tiles = ((pa + kTile - 1) / kTile) * ((qb + kTile - 1) / kTile);
  long long chunks = (4LL * sms + tiles - 1) / tiles;
  const long long maxc = (n + kTileK - 1) / kTileK;
  const long long capc = (long long)(kNoAllocDoubles / ((size_t)pa * qb));
  if (chunks > maxc) chunks = maxc;
  if (chunks > capc) chunks = capc;
  if (chunks < 1) chunks = 1;
  long long rows_per = (n + chunks - 1) / chunks;
  rows_per = (rows_per + kTileK - 1) / kTileK * kTileK;
  cudaStream_t s = (cudaStream_t)stream;
  {
    // every partial tile is written in full (zeros for empty row ranges)
    // before the reduction reads it, so nothing needs clearing
    ProfScope ps_(s, KP_GRAM, 2.0 * n * pa * qb, (double)n * (pa + qb) * sizeof(double));
    gram_kernel<double><<<dim3(tiles, (unsigned)chunks), 256, 0, s>>>(n, pa, qb, rows_per, A, B,
                                                                       scratch);
  }
  KS_CUDA_TRY(cudaGetLastError());
  const long long len = (long long)pa * qb;
  {
    ProfScope ps_(s, KP_REDUCE);
    gram_reduce_kernel<<<(int)((8 * len + kThreads - 1) / kThreads), kThreads, 0, s>>>(
        (int)chunks, len, scratch, out);
  }
  KS_CUDA_TRY(cudaGetLastError());
  return KS_OK;
}
