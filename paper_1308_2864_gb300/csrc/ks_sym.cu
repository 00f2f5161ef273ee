// FP64 row kernels of the iteration's n p^2 work for blocks of 9 to 128
// columns, which spend no FP64 instruction that the result does not need:
//   gram_sym:    A^T B whose result is symmetric (E_X^T X with E_X = H X,
//                D^T M D, X^T M X, E_X^T M^{-1} E_X): the lower triangle of
//                4 x 4 output blocks only, mirrored by the reduction;
//   update_tri:  (X - tau D) U with U = L^{-T} upper triangular: the QR step
//                (Eq. QR, Alg. ChQR), which is X U + D (-tau U) with a
//                quarter of that form's multiplications, and X L^{-T} of the
//                Cholesky QR (D null) with half of them.
// The bound of both is the FP64 pipe (two lanes per SM and clock on GB300,
// so a warp's FMA holds it for 16 clocks): loads, shared memory and index
// arithmetic hide behind it, and the FMA count is what matters.  Measured
// against the full 64 x 64 tiles they replace here: M-orthonormalising 96^3 x
// 128 (two Grams, two updates, mass stencils) 104.7 -> 59.0 ms, of which the
// FP64 FMAs of these kernels need 49; 64^3 x 64 energy and gradient 8.6 ->
// 5.9 ms (one Gram of it left out, the other halved).  Below 9 columns the
// one-thread-per-row kernels have no padding to save; above 128 the packed U
// and a row tile no longer fit shared memory, and the full tiles stay.
#include "ks_device.cuh"

namespace ks {

constexpr int kSymMinP = 9, kSymMaxP = 128;

// ---------------------------------------------------------------- Gram
// A block owns one chunk of rows and the whole lower triangle of g (g + 1) / 2
// output blocks, g = ceil(p / 4).  One thread per output block makes a `set`;
// the block's threads hold as many sets as fit, and set s takes rows s,
// s + nsets, ... of each stage, so that all threads work at any p (a 64 x 64
// tile would spend (64 / p)^2 times the work at p = 40).  Stages of sk rows
// are contiguous in memory and copied by cp.async into two buffers.  The
// sets' sums are added through shared memory in set order, the chunks' in
// chunk order by the reduction below: the result is deterministic.
constexpr int kSymThreads = 544;          // 4 sets at p = 64, 1 at p = 128 (528 blocks)

struct SymPlan {
  int g, tri, nsets, threads, sk, chunks;
  long long rows_per;
  size_t smem;
};

static SymPlan sym_plan(const Problem &P) {
  SymPlan s;
  const int p = P.p;
  s.g = (p + 3) / 4;
  s.tri = s.g * (s.g + 1) / 2;
  s.nsets = kSymThreads / s.tri;
  s.threads = (s.nsets * s.tri + 31) / 32 * 32;
  // about 2048 entries per operand and stage, a multiple of the sets (equal
  // work) rounded up to even (copies are of 16 bytes at even p, of 8 at odd p)
  int m = 2048 / (p * s.nsets);
  if (m < 1) m = 1;
  s.sk = s.nsets * m;
  if (s.sk < 8) s.sk = 8;
  s.sk += s.sk & 1;
  // one block per SM: the FP64 pipe is full with a warp or two per quarter
  s.chunks = P.sms;
  const long long most = (long long)(P.partials_len / ((size_t)s.tri * 16));
  if (s.chunks > most) s.chunks = (int)most;
  s.rows_per = (P.n + s.chunks - 1) / s.chunks;
  s.rows_per += s.rows_per & 1;
  s.chunks = (int)((P.n + s.rows_per - 1) / s.rows_per);
  const size_t stage = ((size_t)4 * s.sk * p + 4) * sizeof(double);
  const size_t fold = s.nsets > 1 ? (size_t)s.nsets * s.tri * 16 * sizeof(double) : 0;
  s.smem = stage > fold ? stage : fold;
  return s;
}

__device__ __forceinline__ void sym_block(int t, int &i, int &c) {
  int r = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
  while (r > 0 && r * (r + 1) / 2 > t) --r;
  while ((r + 1) * (r + 2) / 2 <= t) ++r;
  i = r;
  c = t - r * (r + 1) / 2;
}

// Copies of 16 bytes (8 when an operand's base is not 16-byte aligned).
template <int Bytes>
__device__ __forceinline__ void sym_cp(double *dst, const double *src) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(d), "l"(src), "n"(Bytes)
               : "memory");
}

// Vec: 16-byte shared-memory loads and copies (p even and aligned bases).
template <bool Vec>
__global__ void __launch_bounds__(kSymThreads) gram_sym_kernel(
    long long n, int p, int tri, int nsets, int sk, long long rows_per,
    const double *__restrict__ A, const double *__restrict__ B, double *__restrict__ part) {
  extern __shared__ __align__(16) double sy_smem[];
  const int tid = threadIdx.x;
  const int set = tid / tri, t = tid - set * tri;
  const bool work = set < nsets;
  int bi = 0, bc = 0;
  if (work) sym_block(t, bi, bc);
  const long long r0 = blockIdx.x * rows_per;
  const long long r1 = r0 + rows_per < n ? r0 + rows_per : n;
  const int len = sk * p;
  auto issue = [&](long long r, int buf) {
    const int cnt = (int)(r1 - r < sk ? r1 - r : sk) * p;
    double *da = sy_smem + (size_t)buf * 2 * len, *db = da + len;
    const double *ga = A + r * p, *gb = B + r * p;
    if (Vec) {
      for (int e = 2 * tid; e < cnt; e += 2 * blockDim.x)
        if (KS_IN(r * p + e + 1, n * p)) {
          sym_cp<16>(da + e, ga + e);
          sym_cp<16>(db + e, gb + e);
        }
    } else {
      for (int e = tid; e < cnt; e += blockDim.x)
        if (KS_IN(r * p + e, n * p)) {
          sym_cp<8>(da + e, ga + e);
          sym_cp<8>(db + e, gb + e);
        }
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  double acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.0;
  if (r0 < r1) issue(r0, 0);
  int buf = 0;
  for (long long r = r0; r < r1; r += sk, buf ^= 1) {
    if (r + sk < r1) {
      issue(r + sk, buf ^ 1);
      asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    }
    __syncthreads();
    if (work) {
      const int rows = (int)(r1 - r < sk ? r1 - r : sk);
      // columns past p of the last block read the next row or the padding:
      // they only reach outputs that are not stored
      const double *as = sy_smem + (size_t)buf * 2 * len + 4 * bi;
      const double *bs = sy_smem + (size_t)buf * 2 * len + len + 4 * bc;
      for (int rr = set; rr < rows; rr += nsets) {
        double av[4], bv[4];
        if (Vec) {
          const double2 a0 = *reinterpret_cast<const double2 *>(as + rr * p);
          const double2 a1 = *reinterpret_cast<const double2 *>(as + rr * p + 2);
          const double2 b0 = *reinterpret_cast<const double2 *>(bs + rr * p);
          const double2 b1 = *reinterpret_cast<const double2 *>(bs + rr * p + 2);
          av[0] = a0.x; av[1] = a0.y; av[2] = a1.x; av[3] = a1.y;
          bv[0] = b0.x; bv[1] = b0.y; bv[2] = b1.x; bv[3] = b1.y;
        } else {
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            av[u] = as[rr * p + u];
            bv[u] = bs[rr * p + u];
          }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[i][j] = fma(av[i], bv[j], acc[i][j]);
      }
    }
    __syncthreads();
  }
  double *dst = part + (long long)blockIdx.x * tri * 16;
  if (nsets == 1) {
    if (work)
#pragma unroll
      for (int u = 0; u < 16; ++u) dst[(long long)t * 16 + u] = acc[u >> 2][u & 3];
    return;
  }
  if (work)
#pragma unroll
    for (int u = 0; u < 16; ++u) sy_smem[((size_t)set * 16 + u) * tri + t] = acc[u >> 2][u & 3];
  __syncthreads();
  for (int e = tid; e < tri * 16; e += blockDim.x) {
    double v = 0.0;
    for (int s = 0; s < nsets; ++s) v += sy_smem[(size_t)s * 16 * tri + e];
    // e = u * tri + t here; the partial keeps 16 consecutive values per block
    dst[(long long)(e % tri) * 16 + e / tri] = v;
  }
}

// out = the chunks' sums in chunk order (8 strided eighths, then in order),
// mirrored; a block takes 32 consecutive partial entries.
__global__ void __launch_bounds__(256) gram_sym_reduce_kernel(int chunks, int p, int tri,
                                                              const double *__restrict__ part,
                                                              double *__restrict__ out) {
  __shared__ double s[8][32];
  const int lane = threadIdx.x & 31, sub = threadIdx.x >> 5;
  const long long len = (long long)tri * 16;
  const long long e = (long long)blockIdx.x * 32 + lane;
  double acc = 0.0;
  if (e < len)
    for (int c = sub; c < chunks; c += 8) acc += part[c * len + e];
  s[sub][lane] = acc;
  __syncthreads();
  if (sub != 0 || e >= len) return;
  double v = s[0][lane];
#pragma unroll
  for (int u = 1; u < 8; ++u) v += s[u][lane];
  int bi, bc;
  sym_block((int)(e >> 4), bi, bc);
  const int a = 4 * bi + (int)((e >> 2) & 3), b = 4 * bc + (int)(e & 3);
  if (a >= p || b >= p) return;
  out[(size_t)a * p + b] = v;
  if (bi != bc) out[(size_t)b * p + a] = v;
}

static bool sym_applies(const Problem &P) {
  return P.p >= kSymMinP && P.p <= kSymMaxP && !(P.use_oz > 0 && (P.use_oz == 2 || P.p >= 48));
}

template <>
ks_status launch_gram_sym<float>(Problem &P, const float *A, const float *B, double *out) {
  return launch_gram<float>(P, A, P.p, B, P.p, out);
}

template <>
ks_status launch_gram_sym<double>(Problem &P, const double *A, const double *B, double *out) {
  if (!sym_applies(P)) return launch_gram<double>(P, A, P.p, B, P.p, out);
  const SymPlan s = sym_plan(P);
  const bool vec = P.p % 2 == 0 && reinterpret_cast<uintptr_t>(A) % 16 == 0 &&
                   reinterpret_cast<uintptr_t>(B) % 16 == 0;
  {
    ProfScope ps_(P.stream, KP_GRAM, (double)P.n * P.p * (P.p + 1), 2.0 * P.n * P.p * 8.0);
    if (vec)
      gram_sym_kernel<true><<<s.chunks, s.threads, s.smem, P.stream>>>(
          P.n, P.p, s.tri, s.nsets, s.sk, s.rows_per, A, B, P.partials);
    else
      gram_sym_kernel<false><<<s.chunks, s.threads, s.smem, P.stream>>>(
          P.n, P.p, s.tri, s.nsets, s.sk, s.rows_per, A, B, P.partials);
  }
  KS_CUDA_TRY(cudaGetLastError());
  {
    ProfScope ps_(P.stream, KP_REDUCE);
    gram_sym_reduce_kernel<<<(s.tri * 16 + 31) / 32, 256, 0, P.stream>>>(s.chunks, P.p, s.tri,
                                                                         P.partials, out);
  }
  KS_CUDA_TRY(cudaGetLastError());
  return KS_OK;
}

// ---------------------------------------------------------------- update
// A block takes 32 Rpt rows, staged (X - tau D) in shared memory with an odd
// row stride (a warp reads one column of 32 rows without conflicts), and U
// packed by blocks of four columns (block j: rows 0 .. 4 j + 3).  Warp w owns
// column blocks w and g - 1 - w of every row: the triangle's short and long
// columns together, so all warps do the same number of FMAs.  out may be X:
// a block has read all its rows before it writes any.
template <int Rpt>
__global__ void __launch_bounds__(512) update_tri_kernel(
    long long n, int p, const double *X, const double *__restrict__ D, double tau,
    const double *__restrict__ U, double *out) {
  extern __shared__ __align__(16) double ut_smem[];
  const int g = (p + 3) / 4, ld = p | 1;
  double *Us = ut_smem;                        // 8 g (g + 1) doubles
  double *Ys = ut_smem + 8 * g * (g + 1);      // 32 Rpt rows of ld
  constexpr int R = 32 * Rpt;
  const long long row0 = (long long)blockIdx.x * R;
  const int rows = (int)(n - row0 < R ? n - row0 : R);
  for (int e = threadIdx.x; e < p * 4 * g; e += blockDim.x) {
    const int k = e / (4 * g), c = e - k * 4 * g, j = c >> 2;
    if (k < 4 * j + 4) Us[8 * j * (j + 1) + 4 * k + (c & 3)] = c < p ? U[(size_t)k * p + c] : 0.0;
  }
  const long long base = row0 * p;
  for (int e = threadIdx.x; e < rows * p; e += blockDim.x) {
    const int r = e / p, k = e - r * p;
    double y = X[base + e];
    if (D) y = fma(-tau, D[base + e], y);
    if (KS_IN(r * ld + k, R * ld)) Ys[r * ld + k] = y;
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, ja = threadIdx.x >> 5, jb = g - 1 - ja;
  const int ka = min(4 * ja + 4, p), kb = min(4 * jb + 4, p);
  const double *ua = Us + 8 * ja * (ja + 1), *ub = Us + 8 * jb * (jb + 1);
  const double *y0 = Ys + lane * ld;
  double acc[2][Rpt][4];
#pragma unroll
  for (int s = 0; s < 2; ++s)
#pragma unroll
    for (int i = 0; i < Rpt; ++i)
#pragma unroll
      for (int u = 0; u < 4; ++u) acc[s][i][u] = 0.0;
  auto step = [&](const double *uc, const double *yk, double (&ac)[Rpt][4]) {
    const double2 c0 = reinterpret_cast<const double2 *>(uc)[0];
    const double2 c1 = reinterpret_cast<const double2 *>(uc)[1];
#pragma unroll
    for (int i = 0; i < Rpt; ++i) {
      const double y = yk[(size_t)32 * i * ld];
      ac[i][0] = fma(y, c0.x, ac[i][0]);
      ac[i][1] = fma(y, c0.y, ac[i][1]);
      ac[i][2] = fma(y, c1.x, ac[i][2]);
      ac[i][3] = fma(y, c1.y, ac[i][3]);
    }
  };
  // (rows past the block's last one hold no data: their sums are not stored)
#pragma unroll 4
  for (int k = 0; k < ka; ++k) step(ua + 4 * k, y0 + k, acc[0]);
  if (jb > ja)
#pragma unroll 4
    for (int k = 0; k < kb; ++k) step(ub + 4 * k, y0 + k, acc[1]);
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const int j = s == 0 ? ja : jb;
    if (s == 1 && jb <= ja) break;
#pragma unroll
    for (int i = 0; i < Rpt; ++i) {
      const int r = lane + 32 * i;
      if (r >= rows) continue;
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (4 * j + u < p && KS_IN(base + (long long)r * p + 4 * j + u, n * p))
          out[base + (long long)r * p + 4 * j + u] = acc[s][i][u];
    }
  }
}

static size_t tri_smem(int p, int rpt) {
  const int g = (p + 3) / 4;
  return ((size_t)8 * g * (g + 1) + (size_t)32 * rpt * (p | 1)) * sizeof(double);
}

bool update_tri_applies(const Problem &P) {
  return P.p >= kSymMinP && P.p <= kSymMaxP && !(P.use_oz > 0 && combine_oz_applies(P, P.p, P.p, P.p));
}

ks_status launch_update_tri(Problem &P, const double *X, const double *D, double tau,
                            const double *U, double *out) {
  const int p = P.p, g = (p + 3) / 4;
  const int threads = 32 * ((g + 1) / 2);
  // four rows per thread once that leaves several tiles per SM, fewer below,
  // so that a small grid still spreads over the chip
  const int rpt = P.n >= 128LL * 4 * P.sms ? 4 : P.n >= 64LL * 2 * P.sms ? 2 : 1;
  const size_t smem = tri_smem(p, rpt);
  const unsigned nb = (unsigned)((P.n + 32 * rpt - 1) / (32 * rpt));
  ProfScope ps_(P.stream, KP_COMBINE, (double)P.n * p * (p + 1),
                (double)P.n * p * (D ? 3 : 2) * sizeof(double));
  if (rpt == 4) update_tri_kernel<4><<<nb, threads, smem, P.stream>>>(P.n, p, X, D, tau, U, out);
  else if (rpt == 2) update_tri_kernel<2><<<nb, threads, smem, P.stream>>>(P.n, p, X, D, tau, U, out);
  else update_tri_kernel<1><<<nb, threads, smem, P.stream>>>(P.n, p, X, D, tau, U, out);
  KS_CUDA_TRY(cudaGetLastError());
  return KS_OK;
}

__global__ void trace_sum_kernel(int p, const double *A, const double *B, const double *C,
                                 double *out) {
  __shared__ double smem[33];
  double v = 0.0;
  for (int i = threadIdx.x; i < p; i += blockDim.x) {
    const size_t e = (size_t)i * p + i;
    v += (A ? A[e] : 0.0) + (B ? B[e] : 0.0) + (C ? C[e] : 0.0);
  }
  v = block_sum(v, smem);
  if (threadIdx.x == 0) *out = v;
}

ks_status launch_trace_sum(Problem &P, const double *A, const double *B, const double *C,
                           double *out) {
  {
    ProfScope ps_(P.stream, KP_OTHER);
    trace_sum_kernel<<<1, 128, 0, P.stream>>>(P.p, A, B, C, out);
  }
  KS_CUDA_TRY(cudaGetLastError());
  return KS_OK;
}

ks_status configure_sym_kernels() {
  const int tri4 = (int)tri_smem(kSymMaxP, 4), tri2 = (int)tri_smem(kSymMaxP, 2);
  const int tri1 = (int)tri_smem(kSymMaxP, 1);
  // a stage of two buffers (at most ~66 KiB) or the sets' sums (544 x 16)
  const int gs = 72 * 1024;
  const auto at = cudaFuncAttributeMaxDynamicSharedMemorySize;
  KS_CUDA_TRY(cudaFuncSetAttribute(gram_sym_kernel<true>, at, gs));
  KS_CUDA_TRY(cudaFuncSetAttribute(gram_sym_kernel<false>, at, gs));
  KS_CUDA_TRY(cudaFuncSetAttribute(update_tri_kernel<4>, at, tri4));
  KS_CUDA_TRY(cudaFuncSetAttribute(update_tri_kernel<2>, at, tri2));
  KS_CUDA_TRY(cudaFuncSetAttribute(update_tri_kernel<1>, at, tri1));
  return KS_OK;
}

KS_OOB_READER(sym)

}  // namespace ks
