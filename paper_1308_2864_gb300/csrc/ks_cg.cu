// Hartree potential: conjugate gradients for K vH = 4 pi h^3 rho with zero
// Dirichlet values (the discrete L^+ rho of Sec. 2.3 for the Q1 stiffness),
// as one persistent cooperative kernel.
//
// Preconditioned form (the default).  K is diagonal in the orthonormal sine
// basis that diagonalises the 1-D factors K1 and M1,
//   K^{-1} = (Phi x Phi x Phi) Lambda^{-1} (Phi x Phi x Phi),
//   Lambda_abc = k_a m_b m_c + m_a k_b m_c + m_a m_b k_c.
// Applied in FP32 it is P = K^{-1} (1 + O(1e-5)), so close that defect
// correction
//   z = P r,  x += z,  r -= K z   (r and K z in FP64)
// reduces the residual by four to six digits per step, as many as conjugate
// gradients with the same P, without its two inner products: a step is three
// transform phases and one update, four grid barriers (six for CG), and
// the update needs no search direction.  A step that does not reduce the
// residual by half hands the system to the CG loop below (which also serves
// cg_precond = 0).  The sine transforms use the parity of the modes: a sine
// mode is symmetric (k odd) or antisymmetric (k even) about the middle of its
// axis, so folding the input (u_j = v_j + v_{N+1-j}, w_j = v_j - v_{N+1-j})
// leaves two N/2 x N/2 products per axis, half the work of one N x N, and the
// parities split a plane into independent work items.  N <= kFusedMaxN: both
// in-plane axes in one pass, all in shared memory; above, six tiled axis
// passes.  What bounds a solve is the chain of phases: a barrier costs 2.5 to
// 4 us, a transform phase its loads' latency, the update the FP64 pipe.
// Measured, PCG with full transforms -> this form: warm solve at 64^3 172 ->
// 104 us, at 105^3 519 -> 293 us; cold at 24^3 80 -> 63 us (of which packed FMAs in
// the transforms' tiles 2 to 6 us).  Cold at 81^3 463 -> 177 us, with a step fewer
// by the same stopping rule: the second residual is below 1e-10 of ||b|| here (4e-11
// to 7e-11) and was 1.04e-10 there, and the potential's error, which stops where the
// residual does, goes from 3e-14 to 3e-13 .. 8e-13 with it.  Over 44 grids of 20^3 to
// 161^3 and three densities each (relative error of the potential in the 2-norm) it
// is 0.15 times PCG's in the geometric mean, at most 1.6e-11 against 7.4e-11, and
// larger for 26 of 132, those that PCG gave a third step.
// Tiled passes, cold: 129^3 1.99 -> 1.72 ms, 161^3 3.16 -> 2.70 ms, 200^3 6.16 ->
// 5.22 ms.
//
// Each step's reductions are partial sums written per block and summed by
// every block in the same order, so all blocks take identical branch
// decisions and the result is deterministic.
#include "ks_device.cuh"

namespace ks {

struct CgArgs {
  int N;
  long long n;
  StencilCoef c;
  double bscale;              // 4 pi h^3
  const double *rho;
  double *x, *r, *pa, *pb, *q, *z;
  float *r32;                 // FP32 copy of r for the transforms (in pa's storage)
  float *t1, *t2;             // sine-transform work vectors
  const float *phi;           // N x N sine basis
  const float *kap, *mu;      // 1-D eigenvalues of K1 and M1
  double *part;               // 4 * vnb
  GridBarrier *bar;
  int *status;
  double *iters_out;
  double tol;
  int maxit;
  int warm;
  int precond;
  int fused;                  // fused shared-memory preconditioner (N <= kFusedMaxN)
  int incr;                   // warm start with r = b_old - K x still in r
  double *rho_prev;           // density of the last solve (its b / bscale)
  int vb, vnb;                // this block's index among the vnb blocks that solve this system
};

__device__ __forceinline__ bool cg_barrier(const CgArgs &a, unsigned int &epoch) {
  return grid_barrier_n(a.bar, a.status, (unsigned int)a.vnb, epoch);
}

// (K v)_k for v = a + beta * b (b ignored when UseB is false), Dirichlet.
// The Q1 stiffness has zero face coefficients, so only the centre, the 12
// edge and the 8 corner neighbours contribute.
template <bool UseB>
__device__ __forceinline__ double stiff_apply(const double *a, const double *b, double beta,
                                              int N, int ix, int iy, int iz,
                                              const StencilCoef &c, double *centre) {
  double se = 0.0, sc = 0.0, s0 = 0.0;
  const long long NN = (long long)N * N;
#pragma unroll
  for (int dz = -1; dz <= 1; ++dz) {
    const int z = iz + dz;
    if (z < 0 || z >= N) continue;
#pragma unroll
    for (int dy = -1; dy <= 1; ++dy) {
      const int y = iy + dy;
      if (y < 0 || y >= N) continue;
#pragma unroll
      for (int dx = -1; dx <= 1; ++dx) {
        const int x = ix + dx;
        if (x < 0 || x >= N) continue;
        const int nzc = (dx != 0) + (dy != 0) + (dz != 0);
        if (nzc == 1) continue;
        const long long kk = z * NN + (long long)y * N + x;
        double v = ldcg(a + kk);
        if (UseB) v = fma(beta, ldcg(b + kk), v);
        if (nzc == 0) s0 = v;
        else if (nzc == 2) se += v;
        else sc += v;
      }
    }
  }
  *centre = s0;
  return c.k0 * s0 + c.ke * se + c.kc * sc;
}

// Tiled form for N > kFusedMaxN: each axis pass is the product C = Phi X,
// where the columns of X are the grid lines along the axis (element (s, k, c)
// of slab s, axis index k and column c at s*ss + k*sa + c*sc).  A work item
// is a tile of kTJ frequencies x kTC columns; the K dimension is staged in
// chunks of kTK axis points (X chunk and Phi chunk in shared memory), and a
// thread keeps a 4 x 8 block of outputs (rows tj + 16 a, columns tc + 16 b)
// whose FMA chains run over k in ascending order.  Phi is symmetric and
// orthogonal, so the same matrix serves the forward and the inverse passes.
// Mode 1 (after the forward z pass) divides by Lambda of the frequency
// triple; Mode 2 (the last inverse pass) writes FP64 z.
constexpr int kTJ = 64, kTC = 128, kTK = 32, kTCPad = kTC + 1;
static_assert(kCgThreads == 256, "the 16 x 16 thread grid of the tiled sine pass");

template <int Mode>
__device__ void tiled_pass(const CgArgs &a, const float *in, float *out32, double *out64, int axis,
                           float *sh) {
  const int N = a.N;
  const long long NN = (long long)N * N;
  long long sa, sc, ss, C;
  int S;
  if (axis == 0) { sa = 1; sc = N; ss = 0; S = 1; C = NN; }
  else if (axis == 1) { sa = N; sc = 1; ss = NN; S = N; C = N; }
  else { sa = NN; sc = 1; ss = 0; S = 1; C = NN; }
  const long long ctiles = (C + kTC - 1) / kTC;
  const int jblocks = (N + kTJ - 1) / kTJ;
  const long long total = (long long)S * ctiles * jblocks;
  float *Xs = sh, *Ps = sh + kTK * kTCPad;
  const int tid = threadIdx.x, tj = tid >> 4, tc = tid & 15;
  for (long long w = a.vb; w < total; w += a.vnb) {
    const int jb = (int)(w % jblocks) * kTJ;
    const long long w2 = w / jblocks;
    const long long c0 = (w2 % ctiles) * kTC;
    const long long base = (w2 / ctiles) * ss;
    float acc[4][8];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int v = 0; v < 8; ++v) acc[u][v] = 0.f;
    for (int k0 = 0; k0 < N; k0 += kTK) {
      __syncthreads();
      // X chunk (kTK x kTC): consecutive threads take consecutive addresses
      // (along the axis for the x pass, along the columns otherwise)
      for (int t = tid; t < kTK * kTC; t += kCgThreads) {
        const int kk = axis == 0 ? t % kTK : t / kTC;
        const int cc = axis == 0 ? t / kTK : t % kTC;
        const int k = k0 + kk;
        const long long c = c0 + cc;
        float v = 0.f;
        if (k < N && c < C) {
          const long long idx = base + k * sa + c * sc;
          v = __ldcg(in + idx);
        }
        Xs[kk * kTCPad + cc] = v;
      }
      // Phi chunk (kTK x kTJ): Ps[kk][jj] = Phi[k0 + kk][jb + jj]
      for (int t = tid; t < kTK * kTJ; t += kCgThreads) {
        const int jj = t % kTJ, kk = t / kTJ;
        const int k = k0 + kk, j = jb + jj;
        Ps[t] = (k < N && j < N) ? __ldg(a.phi + (long long)k * N + j) : 0.f;
      }
      __syncthreads();
#pragma unroll 4
      for (int kk = 0; kk < kTK; ++kk) {
        float pv[4], xv[8];
#pragma unroll
        for (int u = 0; u < 4; ++u) pv[u] = Ps[kk * kTJ + tj + 16 * u];
#pragma unroll
        for (int v = 0; v < 8; ++v) xv[v] = Xs[kk * kTCPad + tc + 16 * v];
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int v = 0; v < 8; ++v) acc[u][v] = fmaf(pv[u], xv[v], acc[u][v]);
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int j = jb + tj + 16 * u;
      if (j >= N) continue;
#pragma unroll
      for (int v = 0; v < 8; ++v) {
        const long long c = c0 + tc + 16 * v;
        if (c >= C) continue;
        const long long idx = base + j * sa + c * sc;
        float val = acc[u][v];
        if (Mode == 1) {
          const int ix = (int)(idx % N), iy = (int)((idx / N) % N), iz = (int)(idx / NN);
          const float lam = a.kap[ix] * a.mu[iy] * a.mu[iz] + a.mu[ix] * a.kap[iy] * a.mu[iz] +
                            a.mu[ix] * a.mu[iy] * a.kap[iz];
          val = val / lam;
        }
        if (Mode == 2) {
          out64[idx] = (double)val;
        } else {
          out32[idx] = val;
        }
      }
    }
  }
}

constexpr size_t kTiledSmem = (size_t)(kTK * kTCPad + kTK * kTJ) * sizeof(float);

// z = P r (six tiled passes, a grid barrier after each of the first five);
// false when a barrier failed.
__device__ bool apply_precond(const CgArgs &a, unsigned int &epoch) {
  extern __shared__ float dyn[];
  tiled_pass<0>(a, a.r32, a.t1, nullptr, 0, dyn);
  if (!cg_barrier(a, epoch)) return false;
  tiled_pass<0>(a, a.t1, a.t2, nullptr, 1, dyn);
  if (!cg_barrier(a, epoch)) return false;
  tiled_pass<1>(a, a.t2, a.t1, nullptr, 2, dyn);
  if (!cg_barrier(a, epoch)) return false;
  tiled_pass<0>(a, a.t1, a.t2, nullptr, 2, dyn);
  if (!cg_barrier(a, epoch)) return false;
  tiled_pass<0>(a, a.t2, a.t1, nullptr, 1, dyn);
  if (!cg_barrier(a, epoch)) return false;
  tiled_pass<2>(a, a.t1, nullptr, a.z, 0, dyn);
  return true;
}

// ---------------------------------------------------------------- fused form
// Modes of one axis in parity order: the h1 = ceil(N/2) symmetric ones
// (0-based 0, 2, ...), then the h0 = floor(N/2) antisymmetric ones.  Work
// vectors hold the transformed axes in this order.
//   A  item (z, parity of ky, parity of kx): the folded quarter of plane z of
//      r -> its modes (y, then x)
//   B  item (ky, parity of kx): forward along z, Lambda^{-1}, inverse along z
//   C  item (z, half of the y pairs): inverse along y, then x -> z in FP64
// Shared memory, in units of hp x hp floats (hp = h1 rounded up to 4): the
// half bases F_e, F_o (row j, column mode) and their transposes I_e, I_o, and
// four work matrices: 100 KiB at N = 105, two blocks per SM.
constexpr int kFusedMaxN = 128;

__host__ __device__ constexpr int half_pad(int N) { return ((N + 1) / 2 + 3) / 4 * 4; }
// y pairs of pass C's first half
__host__ __device__ constexpr int half_split(int N) { return (((N + 1) / 2 + 1) / 2 + 3) / 4 * 4; }
__host__ __device__ constexpr size_t fused_smem_floats(int N) {
  const size_t m = (size_t)half_pad(N) * half_pad(N);
  const size_t c = 2 * m + (size_t)N * 2 * half_split(N);      // pass C: T and Yt
  return 4 * m + (c > 4 * m ? c : 4 * m);
}

struct FusedDims {
  int N, h1, h0, hp;
  long long NN;
  float *fe, *fo, *ie, *io, *w;
  __device__ FusedDims(int N_, float *sh) : N(N_) {
    h1 = (N + 1) / 2;
    h0 = N / 2;
    hp = half_pad(N);
    NN = (long long)N * N;
    const int m = hp * hp;
    fe = sh;
    fo = sh + m;
    ie = sh + 2 * m;
    io = sh + 3 * m;
    w = sh + 4 * m;
  }
};

// The half bases from the N x N sine matrix (once per kernel).
__device__ __forceinline__ void load_phi(const CgArgs &a, float *sh, bool fwd = true,
                                         bool inv = true) {
  const FusedDims d(a.N, sh);
  for (int e = threadIdx.x; e < d.N * d.h1; e += kCgThreads) {
    const int k = e / d.h1, j = e - k * d.h1, m = k >> 1;    // mode k, node j
    if ((k & 1) && j >= d.h0) continue;
    const float v = __ldg(a.phi + (long long)k * d.N + j);
    if (!KS_IN(j * d.hp + m, d.hp * d.hp) || !KS_IN(m * d.hp + j, d.hp * d.hp)) continue;
    if (fwd) ((k & 1) ? d.fo : d.fe)[j * d.hp + m] = v;
    if (inv) ((k & 1) ? d.io : d.ie)[m * d.hp + j] = v;
  }
}

template <int TT>
__device__ __forceinline__ void ldv(const float *p, float (&v)[TT]) {
  if constexpr (TT == 4) {
    const float4 q = *reinterpret_cast<const float4 *>(p);
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
  } else {
    const float2 q = *reinterpret_cast<const float2 *>(p);
    v[0] = q.x; v[1] = q.y;
  }
}

// acc[u][v] = sum_k A[k][m0 + u] B[k][n0 + v] (row strides lda, ldb); packed
// FMAs over the columns (f2_fma), each a chain over ascending k.
template <int TT>
__device__ __forceinline__ void tile_fma(const float *A, int lda, const float *B, int ldb, int K,
                                         float (&acc)[TT][TT]) {
  f2_t c[TT][TT / 2];
#pragma unroll
  for (int u = 0; u < TT; ++u)
#pragma unroll
    for (int v = 0; v < TT / 2; ++v) c[u][v] = 0ull;
#pragma unroll 4
  for (int k = 0; k < K; ++k) {
    float av[TT];
    f2_t bv[TT / 2];
    ldv<TT>(A + k * lda, av);
    if constexpr (TT == 4) {
      const ulonglong2 q = *reinterpret_cast<const ulonglong2 *>(B + k * ldb);
      bv[0] = q.x;
      bv[1] = q.y;
    } else {
      bv[0] = *reinterpret_cast<const f2_t *>(B + k * ldb);
    }
#pragma unroll
    for (int u = 0; u < TT; ++u) {
      const f2_t a2 = f2_dup(av[u]);
#pragma unroll
      for (int v = 0; v < TT / 2; ++v) c[u][v] = f2_fma(a2, bv[v], c[u][v]);
    }
  }
#pragma unroll
  for (int u = 0; u < TT; ++u)
#pragma unroll
    for (int v = 0; v < TT / 2; ++v) f2_split(c[u][v], acc[u][2 * v], acc[u][2 * v + 1]);
}

// out(m0, n0, acc) for every TT x TT tile of C = A^T B (M x Nn, K terms), both
// operands k-major in shared memory; columns past M or Nn read padding and
// only reach entries that `out` drops.
template <int TT, typename Out>
__device__ __forceinline__ void tile_gemm(int M, int Nn, int K, const float *A, int lda,
                                          const float *B, int ldb, Out out) {
  const int tn = (Nn + TT - 1) / TT, tiles = (M + TT - 1) / TT * tn;
  for (int t = threadIdx.x; t < tiles; t += kCgThreads) {
    const int m0 = t / tn * TT, n0 = t % tn * TT;
    if (!KS_IN(m0 + TT - 1, lda) || !KS_IN(n0 + TT - 1, ldb)) continue;
    float acc[TT][TT];
    tile_fma<TT>(A + m0, lda, B + n0, ldb, K, acc);
    out(m0, n0, acc);
  }
}

// The same for two products of one shape (K1 and K2 terms): out(m0, n0, e, o).
template <int TT, typename Out>
__device__ __forceinline__ void tile_gemm2(int M, int Nn, int K1, const float *A1, const float *B1,
                                           int K2, const float *A2, const float *B2, int lda,
                                           int ldb, Out out) {
  const int tn = (Nn + TT - 1) / TT, tiles = (M + TT - 1) / TT * tn;
  for (int t = threadIdx.x; t < tiles; t += kCgThreads) {
    const int m0 = t / tn * TT, n0 = t % tn * TT;
    if (!KS_IN(m0 + TT - 1, lda) || !KS_IN(n0 + TT - 1, ldb)) continue;
    float e[TT][TT], o[TT][TT];
    tile_fma<TT>(A1 + m0, lda, B1 + n0, ldb, K1, e);
    tile_fma<TT>(A2 + m0, lda, B2 + n0, ldb, K2, o);
    out(m0, n0, e, o);
  }
}

template <int TT>
__device__ __forceinline__ void fused_pass_a(const CgArgs &a, const float *r32, float *out,
                                             float *sh) {
  const FusedDims d(a.N, sh);
  const int N = d.N, hp = d.hp;
  float *Q = d.w, *Wt = d.w + hp * hp;
  for (int item = a.vb; item < 4 * N; item += a.vnb) {
    const int z = item >> 2, py = (item >> 1) & 1, px = item & 1;
    const int hy = py ? d.h0 : d.h1, hx = px ? d.h0 : d.h1;
    const float sy = py ? -1.f : 1.f, sx = px ? -1.f : 1.f;
    const float *P = r32 + z * d.NN;
    __syncthreads();
    // the four mirror images of a folded entry; four entries in flight
    for (int e0 = threadIdx.x; e0 < hy * hx; e0 += 4 * kCgThreads) {
      float v[4][4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int e = e0 + u * kCgThreads;
        const int j = e / hx, i = e - j * hx, j2 = N - 1 - j, i2 = N - 1 - i;
        const bool ok = e < hy * hx && KS_IN(z * d.NN + (long long)j2 * N + i2, a.n);
        v[u][0] = ok ? __ldcg(P + j * N + i) : 0.f;
        v[u][1] = ok && i2 != i ? __ldcg(P + j * N + i2) : 0.f;
        v[u][2] = ok && j2 != j ? __ldcg(P + j2 * N + i) : 0.f;
        v[u][3] = ok && j2 != j && i2 != i ? __ldcg(P + j2 * N + i2) : 0.f;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int e = e0 + u * kCgThreads;
        if (e >= hy * hx) break;
        const int j = e / hx, i = e - j * hx;
        Q[j * hp + i] = fmaf(sy, fmaf(sx, v[u][3], v[u][2]), fmaf(sx, v[u][1], v[u][0]));
      }
    }
    __syncthreads();
    tile_gemm<TT>(hy, hx, hy, py ? d.fo : d.fe, hp, Q, hp,
                  [&](int m0, int n0, float (&c)[TT][TT]) {
#pragma unroll
                    for (int v = 0; v < TT; ++v)
#pragma unroll
                      for (int u = 0; u < TT; ++u) Wt[(n0 + v) * hp + m0 + u] = c[u][v];
                  });
    __syncthreads();
    tile_gemm<TT>(hy, hx, hx, Wt, hp, px ? d.fo : d.fe, hp,
                  [&](int m0, int n0, float (&c)[TT][TT]) {
#pragma unroll
                    for (int u = 0; u < TT; ++u)
#pragma unroll
                      for (int v = 0; v < TT; ++v) {
                        const long long k = z * d.NN + (long long)(py * d.h1 + m0 + u) * N +
                                            px * d.h1 + n0 + v;
                        if (m0 + u < hy && n0 + v < hx && KS_IN(k, a.n)) out[k] = c[u][v];
                      }
                  });
  }
}

template <int TT>
__device__ __forceinline__ void fused_pass_b(const CgArgs &a, const float *in, float *out,
                                             float *sh) {
  const FusedDims d(a.N, sh);
  const int N = d.N, hp = d.hp, m2 = hp * hp;
  float *U = d.w, *V = d.w + m2, *Fe = d.w + 2 * m2, *Fo = d.w + 3 * m2;
  for (int item = a.vb; item < 2 * N; item += a.vnb) {
    const int ky = item >> 1, px = item & 1, hx = px ? d.h0 : d.h1;
    const long long col = (long long)ky * N + px * d.h1;
    __syncthreads();
    for (int e0 = threadIdx.x; e0 < d.h1 * hx; e0 += 8 * kCgThreads) {
      float v[8][2];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int e = e0 + u * kCgThreads, j = e / hx, l = e - j * hx;
        const bool ok = e < d.h1 * hx && KS_IN((N - 1 - j) * d.NN + col + l, a.n);
        v[u][0] = ok ? __ldcg(in + j * d.NN + col + l) : 0.f;
        v[u][1] = ok && j < d.h0 ? __ldcg(in + (N - 1 - j) * d.NN + col + l) : 0.f;
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int e = e0 + u * kCgThreads;
        if (e >= d.h1 * hx) break;
        const int j = e / hx, l = e - j * hx;
        U[j * hp + l] = v[u][0] + v[u][1];
        V[j * hp + l] = v[u][0] - v[u][1];
      }
    }
    __syncthreads();
    const int ty = ky < d.h1 ? 2 * ky : 2 * (ky - d.h1) + 1;
    const float ky_ = __ldg(a.kap + ty), my_ = __ldg(a.mu + ty);
    auto scaled = [&](float *F, int pz, int hz, int m0, int n0, float (&c)[TT][TT]) {
#pragma unroll
      for (int u = 0; u < TT; ++u)
#pragma unroll
        for (int v = 0; v < TT; ++v) {
          const int m = m0 + u, l = n0 + v;
          if (m >= hz || l >= hx) continue;
          const int tz = 2 * m + pz, tx = 2 * l + px;
          const float kz = __ldg(a.kap + tz), mz = __ldg(a.mu + tz);
          const float kx = __ldg(a.kap + tx), mx = __ldg(a.mu + tx);
          F[m * hp + l] = c[u][v] / (kx * my_ * mz + mx * ky_ * mz + mx * my_ * kz);
        }
    };
    tile_gemm<TT>(d.h1, hx, d.h1, d.fe, hp, U, hp, [&](int m0, int n0, float (&c)[TT][TT]) {
      scaled(Fe, 0, d.h1, m0, n0, c);
    });
    tile_gemm<TT>(d.h0, hx, d.h0, d.fo, hp, V, hp, [&](int m0, int n0, float (&c)[TT][TT]) {
      scaled(Fo, 1, d.h0, m0, n0, c);
    });
    __syncthreads();
    tile_gemm2<TT>(d.h1, hx, d.h1, d.ie, Fe, d.h0, d.io, Fo, hp, hp,
                   [&](int m0, int n0, float (&e)[TT][TT], float (&o)[TT][TT]) {
#pragma unroll
                     for (int u = 0; u < TT; ++u)
#pragma unroll
                       for (int v = 0; v < TT; ++v) {
                         const int j = m0 + u, l = n0 + v;
                         if (j >= d.h1 || l >= hx) continue;
                         if (!KS_IN((N - 1 - j) * d.NN + col + l, a.n)) continue;
                         const bool pair = j < d.h0;      // false: the middle node
                         out[j * d.NN + col + l] = pair ? e[u][v] + o[u][v] : e[u][v];
                         if (pair) out[(N - 1 - j) * d.NN + col + l] = e[u][v] - o[u][v];
                       }
                   });
  }
}

template <int TT>
__device__ __forceinline__ void fused_pass_c(const CgArgs &a, const float *in, double *out,
                                             float *sh) {
  const FusedDims d(a.N, sh);
  const int N = d.N, hp = d.hp, m2 = hp * hp;
  const int hj = half_split(N);
  const int ldy = 2 * hj;
  // T: the plane's modes of one kx parity (rows: symmetric, then antisymmetric
  // ky); Yt: N modes kx (symmetric, then antisymmetric) x (rows y = j, then
  // y = N - 1 - j)
  float *T = d.w, *Yt = d.w + 2 * m2;
  for (int item = a.vb; item < 2 * N; item += a.vnb) {
    const int z = item >> 1, jbase = (item & 1) * hj;
    const int nj = min(hj, d.h1 - jbase);
    if (nj <= 0) continue;
    for (int px = 0; px < 2; ++px) {
      const int hx = px ? d.h0 : d.h1;
      __syncthreads();
      const float *src = in + z * d.NN + px * d.h1;
      for (int e0 = threadIdx.x; e0 < N * hx; e0 += 8 * kCgThreads) {
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int e = e0 + u * kCgThreads, m = e / hx, l = e - m * hx;
          v[u] = e < N * hx && KS_IN(z * d.NN + px * d.h1 + (long long)m * N + l, a.n)
                     ? __ldcg(src + (long long)m * N + l)
                     : 0.f;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int e = e0 + u * kCgThreads;
          if (e >= N * hx) break;
          const int m = e / hx, l = e - m * hx;
          T[(m < d.h1 ? m : hp + m - d.h1) * hp + l] = v[u];
        }
      }
      __syncthreads();
      tile_gemm2<TT>(nj, hx, d.h1, d.ie + jbase, T, d.h0, d.io + jbase, T + m2, hp, hp,
                     [&](int m0, int n0, float (&e)[TT][TT], float (&o)[TT][TT]) {
#pragma unroll
                       for (int v = 0; v < TT; ++v) {
                         const int l = n0 + v;
                         if (l >= hx) continue;
                         float *y = Yt + ((px ? d.h1 : 0) + l) * ldy;
#pragma unroll
                         for (int u = 0; u < TT; ++u) {
                           if (m0 + u >= hj) continue;
                           const bool pair = jbase + m0 + u < d.h0;
                           if (!KS_IN(((px ? d.h1 : 0) + l) * ldy + hj + m0 + u, N * ldy)) continue;
                           y[m0 + u] = pair ? e[u][v] + o[u][v] : e[u][v];
                           y[hj + m0 + u] = pair ? e[u][v] - o[u][v] : 0.f;
                         }
                       }
                     });
    }
    __syncthreads();
    // rows y of both kinds, inverse along x
    const int tn = (d.h1 + TT - 1) / TT, tiles = (2 * hj / TT) * tn;
    for (int t = threadIdx.x; t < tiles; t += kCgThreads) {
      const int m0 = t / tn * TT, n0 = t % tn * TT;
      float e[TT][TT], o[TT][TT];
      tile_fma<TT>(Yt + m0, ldy, d.ie + n0, hp, d.h1, e);
      tile_fma<TT>(Yt + d.h1 * ldy + m0, ldy, d.io + n0, hp, d.h0, o);
#pragma unroll
      for (int u = 0; u < TT; ++u) {
        const int row = m0 + u, jj = row < hj ? row : row - hj, j = jbase + jj;
        if (jj >= nj || (row >= hj && j >= d.h0)) continue;
        const int y = row < hj ? j : N - 1 - j;
        double *dst = out + z * d.NN + (long long)y * N;
#pragma unroll
        for (int v = 0; v < TT; ++v) {
          const int i = n0 + v;
          if (i >= d.h1 || !KS_IN(z * d.NN + (long long)y * N + N - 1 - i, a.n)) continue;
          const bool pair = i < d.h0;
          dst[i] = (double)(pair ? e[u][v] + o[u][v] : e[u][v]);
          if (pair) dst[N - 1 - i] = (double)(e[u][v] - o[u][v]);
        }
      }
    }
  }
}

// Tile edge of the transforms: 2 x 2 outputs per thread keep 256 threads busy
// up to hp = 32 (N = 64), 4 x 4 (half the shared-memory reads) above.
__device__ __forceinline__ bool small_tiles(int N) { return half_pad(N) <= 32; }

// z = P r of the fused form: three phases, a barrier after the first two.
__device__ bool apply_precond_fused(const CgArgs &a, unsigned int &epoch) {
  extern __shared__ float dyn[];
  const bool s = small_tiles(a.N);
  if (s) fused_pass_a<2>(a, a.r32, a.t1, dyn); else fused_pass_a<4>(a, a.r32, a.t1, dyn);
  if (!cg_barrier(a, epoch)) return false;
  if (s) fused_pass_b<2>(a, a.t1, a.t2, dyn); else fused_pass_b<4>(a, a.t1, a.t2, dyn);
  if (!cg_barrier(a, epoch)) return false;
  if (s) fused_pass_c<2>(a, a.t2, a.z, dyn); else fused_pass_c<4>(a, a.t2, a.z, dyn);
  return true;
}

// ---------------------------------------------------------------- update
// x += z (x = z when `first`), r -= K z and r32 = r over the nodes of
// this block's share; returns this thread's part of r.r.  A thread takes a
// column of kUpY nodes along y and kUpZ along z at one x (a warp: 32
// consecutive x): with the plane sums s = z(x-1) + z(x+1), f, e of six rows
// shared by its nodes, K z costs 15 FP64 instructions per node instead of 23
// (K A = b0(z) + bn(z-1) + bn(z+1), b0 = (k0/ke) c + e, bn = f + e/2, times ke).
constexpr int kUpY = 4, kUpZ = 2;

__device__ __forceinline__ double defect_update(const CgArgs &a, bool first, double k0r) {
  const int N = a.N;
  const long long NN = (long long)N * N;
  const int uy = (N + kUpY - 1) / kUpY, uz = (N + kUpZ - 1) / kUpZ;
  const long long units = (long long)N * uy * uz;
  double rl = 0.0;
  // warps of the launch in turn over the blocks, so that a grid with fewer
  // units than threads still spreads over the SMs
  const long long w0 = (long long)(threadIdx.x >> 5) * a.vnb + a.vb;
  for (long long w = w0; w * 32 < units; w += (long long)a.vnb * (kCgThreads / 32)) {
    const long long un = w * 32 + (threadIdx.x & 31);
    if (un >= units) continue;
    const int x = (int)(un % N);
    const long long q = un / N;
    const int y0 = (int)(q % uy) * kUpY, z0 = (int)(q / uy) * kUpZ;
    double kz[kUpZ][kUpY], cz[kUpZ][kUpY];
#pragma unroll
    for (int pl = 0; pl < kUpZ + 2; ++pl) {
      const int z = z0 + pl - 1;
      const bool zok = z >= 0 && z < N;
      double c[kUpY + 2], s[kUpY + 2];
#pragma unroll
      for (int y = 0; y < kUpY + 2; ++y) {
        const int gy = y0 + y - 1;
        const bool ok = zok && gy >= 0 && gy < N;
        const double *p = a.z + (ok ? z * NN + (long long)gy * N + x : 0);
        c[y] = ok ? __ldcg(p) : 0.0;
        s[y] = (ok && x > 0 ? __ldcg(p - 1) : 0.0) + (ok && x + 1 < N ? __ldcg(p + 1) : 0.0);
      }
#pragma unroll
      for (int r = 0; r < kUpY; ++r) {
        const double f = s[r + 1] + (c[r] + c[r + 2]);
        const double e = s[r] + s[r + 2];
        const double bn = fma(0.5, e, f);
#pragma unroll
        for (int o = 0; o < kUpZ; ++o) {
          if (pl == o) kz[o][r] = bn;
          else if (pl == o + 1) {
            kz[o][r] += fma(k0r, c[r + 1], e);
            cz[o][r] = c[r + 1];
          } else if (pl == o + 2) {
            kz[o][r] += bn;
          }
        }
      }
    }
#pragma unroll
    for (int o = 0; o < kUpZ; ++o)
#pragma unroll
      for (int r = 0; r < kUpY; ++r) {
        if (z0 + o >= N || y0 + r >= N) continue;
        const long long k = (z0 + o) * NN + (long long)(y0 + r) * N + x;
        if (!KS_IN(k, a.n)) continue;
        a.x[k] = first ? cz[o][r] : a.x[k] + cz[o][r];
        const double rk = fma(-a.c.ke, kz[o][r], a.r[k]);
        a.r[k] = rk;
        a.r32[k] = (float)rk;
        rl = fma(rk, rk, rl);
      }
  }
  return rl;
}

// The whole solve of one system on the blocks a.vb = 0 .. a.vnb - 1 (which
// must be co-resident: a cooperative launch).  A warm start whose residual is
// still in r (a.incr) forms the new one without a stencil, r = r_old + (b -
// b_old), from the right-hand side of the last solve (rho_prev).
__device__ void cg_body(const CgArgs &a) {
  __shared__ double smem[2 * 33];
  const int nb = a.vnb;
  unsigned int epoch = 0;
  double *partA = a.part, *partB = a.part + nb, *partC = a.part + 2 * nb, *partD = a.part + 3 * nb;
  const long long tid = (long long)a.vb * blockDim.x + threadIdx.x;
  const long long stride = (long long)a.vnb * blockDim.x;
  const int N = a.N;
  const long long NN = (long long)N * N;
  if (a.fused && a.precond) {
    extern __shared__ float dyn[];
    load_phi(a, dyn);
  }

  // r = b - K x0 (x0 = 0 for a cold start; r_old + b - b_old when
  // incremental), b.b, and rho_prev = rho for the next solve
  double rr_l = 0.0, bb_l = 0.0;
  for (long long k = tid; k < a.n; k += stride) {
    const double rk_rho = a.rho[k];
    const double b = a.bscale * rk_rho;
    double rk;
    if (a.incr) {
      rk = a.r[k] + a.bscale * (rk_rho - a.rho_prev[k]);
    } else {
      double kx = 0.0, dummy;
      if (a.warm) {
        const int ix = (int)(k % N), iy = (int)((k / N) % N), iz = (int)(k / NN);
        kx = stiff_apply<false>(a.x, nullptr, 0.0, N, ix, iy, iz, a.c, &dummy);
      }
      rk = b - kx;
    }
    a.r[k] = rk;
    if (a.precond) a.r32[k] = (float)rk;
    a.rho_prev[k] = rk_rho;
    rr_l = fma(rk, rk, rr_l);
    bb_l = fma(b, b, bb_l);
  }
  double rb[2] = {rr_l, bb_l};
  block_sum_n<2>(rb, smem);
  if (threadIdx.x == 0) { partB[a.vb] = rb[0]; partD[a.vb] = rb[1]; }
  if (!cg_barrier(a, epoch)) return;
  rb[0] = rb[1] = 0.0;
  for (int i = threadIdx.x; i < nb; i += blockDim.x) {
    rb[0] += ldcg(partB + i);
    rb[1] += ldcg(partD + i);
  }
  block_sum_n<2>(rb, smem);
  double rr = rb[0];
  const double bb = rb[1];
  const double thr = a.tol * a.tol * bb;
  // a non-finite right-hand side or start makes every comparison below false
  bool bad = !isfinite(rr) || !isfinite(bb);
  int it = 0;
  bool done = !(rr > thr);
  bool fresh = !a.warm;                     // x not written yet (a cold start)
  if (a.precond) {
    const double k0r = a.c.k0 / a.c.ke;
    while (!done && it < a.maxit) {
      if (a.fused ? !apply_precond_fused(a, epoch) : !apply_precond(a, epoch)) return;
      if (!cg_barrier(a, epoch)) return;
      const double rl = defect_update(a, fresh, k0r);
      fresh = false;
      const double s = block_sum(rl, smem);
      if (threadIdx.x == 0) partA[a.vb] = s;
      if (!cg_barrier(a, epoch)) return;
      const double rr_new = block_sum_array(partA, nb, smem);
      ++it;
      if (!isfinite(rr_new)) { bad = true; break; }
      const bool slow = rr_new > 0.25 * rr;
      rr = rr_new;
      done = !(rr > thr);
      if (slow) break;
    }
  }
  if (fresh) {
    for (long long k = tid; k < a.n; k += stride) a.x[k] = 0.0;
  }
  if (!done && !bad && it < a.maxit) {
    // conjugate gradients: each iteration applies the stiffness once, q = K p
    // carried as q = K s + beta q_old (K p by linearity, p = s + beta p_old)
    const double *s_vec = a.r;
    double rho_cg = rr, beta = 0.0;
    double *pold = a.pa, *pnew = a.pb;
    for (int j = 0; rr > thr && it < a.maxit; ++j, ++it) {
      // phase 1: p = s + beta p_old and q = K s + beta q_old (own nodes), p.q
      double pq_l = 0.0;
      for (long long k = tid; k < a.n; k += stride) {
        const int ix = (int)(k % N), iy = (int)((k / N) % N), iz = (int)(k / NN);
        double sk;
        const double ks = stiff_apply<false>(s_vec, nullptr, 0.0, N, ix, iy, iz, a.c, &sk);
        const double pk = j == 0 ? sk : fma(beta, pold[k], sk);
        const double qk = j == 0 ? ks : fma(beta, a.q[k], ks);
        pnew[k] = pk;
        a.q[k] = qk;
        pq_l = fma(pk, qk, pq_l);
      }
      {
        const double s = block_sum(pq_l, smem);
        if (threadIdx.x == 0) partC[a.vb] = s;
      }
      if (!cg_barrier(a, epoch)) return;
      const double pq = block_sum_array(partC, nb, smem);
      if (!(pq > 0.0) || !isfinite(pq)) { bad = true; break; }
      const double alpha = rho_cg / pq;
      // phase 2: x += alpha p, r -= alpha q, r.r
      double rl = 0.0;
      for (long long k = tid; k < a.n; k += stride) {
        a.x[k] = fma(alpha, pnew[k], a.x[k]);
        const double rk = fma(-alpha, a.q[k], a.r[k]);
        a.r[k] = rk;
        rl = fma(rk, rk, rl);
      }
      {
        const double s = block_sum(rl, smem);
        if (threadIdx.x == 0) partB[a.vb] = s;
      }
      if (!cg_barrier(a, epoch)) return;
      const double rr_new = block_sum_array(partB, nb, smem);
      if (!isfinite(rr_new)) { bad = true; break; }
      beta = rr_new / rho_cg;
      rho_cg = rr_new;
      rr = rr_new;
      double *tmp = pold; pold = pnew; pnew = tmp;
    }
  }
  if (a.vb == 0 && threadIdx.x == 0) {
    *a.iters_out = (double)it;
    if (bad) atomicCAS(a.status, 0, (int)KS_ENAN);
    else if (rr > thr) atomicCAS(a.status, 0, (int)KS_ENOCONV);
  }
}

__global__ void __launch_bounds__(kCgThreads) cg_kernel(CgArgs a) {
  a.vb = blockIdx.x;
  a.vnb = gridDim.x;
  cg_body(a);
}

// Sine basis Phi_{jk} = sqrt(2/(N+1)) sin(j k pi/(N+1)) (j, k = 1..N) and
// the 1-D eigenvalues kappa_j = (2/h)(1 - cos t_j), mu_j = (h/3)(2 + cos t_j),
// t_j = j pi/(N+1), in single precision for the preconditioner.
__global__ void sine_setup_kernel(int N, double h, float *phi, float *kap, float *mu) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e < N * N) {
    const int j = e / N + 1, k = e % N + 1;
    const long long jk = (long long)j * k % (2 * (N + 1));
    phi[e] = (float)(sqrt(2.0 / (N + 1)) * sinpi((double)jk / (N + 1)));
  }
  if (e < N) {
    const double c = cospi((double)(e + 1) / (N + 1));
    kap[e] = (float)((2.0 / h) * (1.0 - c));
    mu[e] = (float)((h / 3.0) * (2.0 + c));
  }
}

ks_status launch_sine_setup(Problem &P) {
  const int total = P.N * P.N;
  {
    ProfScope ps_(P.stream, KP_SETUP);
    sine_setup_kernel<<<(total + kThreads - 1) / kThreads, kThreads, 0, P.stream>>>(
        P.N, P.h, P.dst_phi, P.dst_kap, P.dst_mu);
  }
  KS_CUDA_TRY(cudaGetLastError());
  return KS_OK;
}

constexpr int kCgIncrMax = 64;

ks_status launch_cg(Problem &P, const double *rho, double *v, double *r, bool warm) {
  CgArgs a;
  a.N = P.N;
  a.n = P.n;
  a.c = q1_coefficients(P.h);
  a.bscale = 4.0 * M_PI * P.h * P.h * P.h;
  a.rho = rho;
  a.x = v;
  a.r = r;
  a.pa = P.cg_pa;
  a.pb = P.cg_pb;
  a.r32 = reinterpret_cast<float *>(P.cg_pa);
  a.q = P.cg_q;
  a.z = P.cg_z;
  a.t1 = P.cg_t1;
  a.t2 = P.cg_t2;
  a.phi = P.dst_phi;
  a.kap = P.dst_kap;
  a.mu = P.dst_mu;
  a.part = P.partials;
  a.bar = P.bar;
  a.status = P.dstatus;
  a.iters_out = P.scal + SC_CG_ITERS;
  a.tol = P.cg_tol_phase > 0.0 ? P.cg_tol_phase : P.cg_tol;
  a.maxit = P.cg_maxit;
  a.warm = warm ? 1 : 0;
  a.precond = P.cg_precond;
  a.fused = P.N <= kFusedMaxN ? 1 : 0;
  // the residual of the last solve is reused while the problem's own vH and
  // r carry it; every kCgIncrMax-th warm start recomputes it from x, so
  // that the rounding of the recurrences cannot build up
  const bool own = v == P.vH && r == P.cg_r;
  a.incr = (warm && own && P.cg_inc_ok && P.cg_inc_count < kCgIncrMax) ? 1 : 0;
  a.rho_prev = P.cg_rho_prev;
  P.cg_inc_count = a.incr ? P.cg_inc_count + 1 : 0;
  P.cg_inc_ok = own;
  const size_t dyn = cg_dynamic_smem(P.N);
  KS_CUDA_TRY(cudaMemsetAsync(P.bar, 0, sizeof(GridBarrier), P.stream));
  void *args[] = {&a};
  {
    ProfScope ps_(P.stream, KP_CG);
    KS_CUDA_TRY(cudaLaunchCooperativeKernel((const void *)cg_kernel, dim3(P.cg_blocks),
                                            dim3(kCgThreads), args, dyn, P.stream));
  }
  return KS_OK;
}

// ---------------------------------------------------------------- batched
// The solve of every job of a batch, one launch per phase over all jobs
// (no grid barrier: a phase's last block of each job finishes that job's
// reductions and scalar updates in device memory).  Phases:
//   init     r = b - K x (x = 0 when cold), r.r, b.b, tolerance
//   A/B/C    the fused sine-basis transforms, one block per (job, plane)
//            resp. (job, ky); C writes z
//   update   x += z, r -= K z, r.r -> convergence, or a step that did not halve
//            the residual: the job is handed to the CG iterations (as in cg_body)
//   it1, it2 a CG iteration, for jobs without the preconditioner and those handed
//            over (launched when there is such a job): p = r + beta p_old,
//            q = K p, p.q -> alpha; x += alpha p, r -= alpha q, r.r
// A job that has converged (or failed) skips every later phase.  The host
// reads the number of jobs still iterating, and of those in CG, once per iteration.
struct CgState {
  double rr, bb, thr, rho, beta, alpha;
  int it, done, maxit, precond;
  int cg_it;                       // CG iterations done
};

// Last block of one job's nb blocks: sums of the nchan partial channels
// part[c * nb + vb] (in block order) into s[]; true in that block only.
__device__ bool job_tail(double *part, int nb, int nchan, unsigned int *counter, double *smem,
                         double *s) {
  __shared__ int s_last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    const unsigned int prev = atomicAdd(counter, 1u);
    s_last = (prev == (unsigned int)nb - 1u);
  }
  __syncthreads();
  if (!s_last) return false;
  __threadfence();
  for (int c = 0; c < nchan; ++c) s[c] = block_sum_array(part + (long long)c * nb, nb, smem);
  if (threadIdx.x == 0) *counter = 0u;
  return true;
}

struct CgBatchView {
  const CgArgs *args;
  CgState *st;
  const int *start;                // block map of the phase
  int J;
  const unsigned char *active;
  const double *tolw;              // per job: tolerance, warm flag
  unsigned int *counters;          // one per job
};

__device__ __forceinline__ bool cg_job(const CgBatchView &v, int &j, int &vb, int &nb) {
  j = batch_job_of(v.start, v.J, blockIdx.x);
  if (!v.active[j] || v.st[j].done) return false;
  vb = blockIdx.x - v.start[j];
  nb = v.start[j + 1] - v.start[j];
  return true;
}

__global__ void __launch_bounds__(kCgThreads) cg_b_init(CgBatchView v) {
  __shared__ double smem[33];
  const int j = batch_job_of(v.start, v.J, blockIdx.x);
  if (!v.active[j]) return;
  const int vb = blockIdx.x - v.start[j], nb = v.start[j + 1] - v.start[j];
  const CgArgs &a = v.args[j];
  const int warm = v.tolw[2 * j + 1] != 0.0;
  const int N = a.N;
  const long long NN = (long long)N * N;
  double rr_l = 0.0, bb_l = 0.0;
  for (long long k = (long long)vb * blockDim.x + threadIdx.x; k < a.n;
       k += (long long)nb * blockDim.x) {
    const double b = a.bscale * a.rho[k];
    double kx = 0.0, dummy;
    if (warm) {
      const int ix = (int)(k % N), iy = (int)((k / N) % N), iz = (int)(k / NN);
      kx = stiff_apply<false>(a.x, nullptr, 0.0, N, ix, iy, iz, a.c, &dummy);
    } else {
      a.x[k] = 0.0;
    }
    const double rk = b - kx;
    a.r[k] = rk;
    if (a.precond) a.r32[k] = (float)rk;
    rr_l = fma(rk, rk, rr_l);
    bb_l = fma(b, b, bb_l);
  }
  const double s1 = block_sum(rr_l, smem), s2 = block_sum(bb_l, smem);
  if (threadIdx.x == 0) {
    a.part[vb] = s1;
    a.part[nb + vb] = s2;
  }
  double s[2];
  if (!job_tail(a.part, nb, 2, v.counters + j, smem, s)) return;
  if (threadIdx.x == 0) {
    CgState &t = v.st[j];
    const double tol = v.tolw[2 * j];
    t.rr = s[0];
    t.bb = s[1];
    t.thr = tol * tol * s[1];
    t.rho = s[0];
    t.beta = 0.0;
    t.it = 0;
    t.cg_it = 0;
    t.maxit = a.maxit;
    t.precond = a.precond;
    t.done = t.rr <= t.thr ? 1 : 0;
    *a.iters_out = 0.0;
  }
}

// Transform phases (fused form; jobs with N > kFusedMaxN are refused at batch
// creation).  Stage 0: r32 -> t1 (in-plane modes); 1: t1 -> t2 (along z); 2:
// t2 -> z.
template <int Stage>
__global__ void __launch_bounds__(kCgThreads) cg_b_precond(CgBatchView v) {
  extern __shared__ float dyn[];
  int j, vb, nb;
  if (!cg_job(v, j, vb, nb)) return;
  CgArgs a = v.args[j];
  if (!v.st[j].precond) return;
  a.vb = vb;
  a.vnb = nb;
  load_phi(a, dyn, Stage <= 1, Stage >= 1);
  const bool s = small_tiles(a.N);
  if (Stage == 0) {
    if (s) fused_pass_a<2>(a, a.r32, a.t1, dyn); else fused_pass_a<4>(a, a.r32, a.t1, dyn);
  } else if (Stage == 1) {
    if (s) fused_pass_b<2>(a, a.t1, a.t2, dyn); else fused_pass_b<4>(a, a.t1, a.t2, dyn);
  } else {
    if (s) fused_pass_c<2>(a, a.t2, a.z, dyn); else fused_pass_c<4>(a, a.t2, a.z, dyn);
  }
}

// One job's residual norm after a step: convergence, limits, failure.
__device__ __forceinline__ void cg_step_done(const CgArgs &a, CgState &u, double rr) {
  ++u.it;
  u.rr = rr;
  *a.iters_out = (double)u.it;
  if (!isfinite(rr)) {
    u.done = 1;
    atomicCAS(a.status, 0, (int)KS_ENAN);
  } else if (rr <= u.thr) {
    u.done = 1;
  } else if (u.it >= u.maxit) {
    u.done = 1;
    atomicCAS(a.status, 0, (int)KS_ENOCONV);
  }
}

__global__ void __launch_bounds__(kCgThreads) cg_b_update(CgBatchView v) {
  __shared__ double smem[33];
  int j, vb, nb;
  if (!cg_job(v, j, vb, nb)) return;
  CgArgs a = v.args[j];
  if (!v.st[j].precond) return;
  a.vb = vb;
  a.vnb = nb;
  const double sum = block_sum(defect_update(a, false, a.c.k0 / a.c.ke), smem);
  if (threadIdx.x == 0) a.part[vb] = sum;
  double s[1];
  if (!job_tail(a.part, nb, 1, v.counters + j, smem, s)) return;
  if (threadIdx.x == 0) {
    CgState &u = v.st[j];
    const bool slow = s[0] > 0.25 * u.rr;
    cg_step_done(a, u, s[0]);
    if (slow && !u.done) {
      u.precond = 0;
      u.rho = s[0];
    }
  }
}

__global__ void __launch_bounds__(kCgThreads) cg_b_it1(CgBatchView v) {
  __shared__ double smem[33];
  int j, vb, nb;
  if (!cg_job(v, j, vb, nb)) return;
  const CgArgs &a = v.args[j];
  const CgState t = v.st[j];
  if (t.precond) return;
  const int N = a.N;
  const long long NN = (long long)N * N;
  const double *s_vec = a.r;
  double *pold = (t.cg_it % 2 == 0) ? a.pb : a.pa, *pnew = (t.cg_it % 2 == 0) ? a.pa : a.pb;
  double pq_l = 0.0;
  for (long long k = (long long)vb * blockDim.x + threadIdx.x; k < a.n;
       k += (long long)nb * blockDim.x) {
    const int ix = (int)(k % N), iy = (int)((k / N) % N), iz = (int)(k / NN);
    double pk;
    const double qk =
        t.cg_it == 0 ? stiff_apply<false>(s_vec, nullptr, 0.0, N, ix, iy, iz, a.c, &pk)
                     : stiff_apply<true>(s_vec, pold, t.beta, N, ix, iy, iz, a.c, &pk);
    pnew[k] = pk;
    a.q[k] = qk;
    pq_l = fma(pk, qk, pq_l);
  }
  const double sum = block_sum(pq_l, smem);
  if (threadIdx.x == 0) a.part[vb] = sum;
  double s[1];
  if (!job_tail(a.part, nb, 1, v.counters + j, smem, s)) return;
  if (threadIdx.x == 0) {
    CgState &u = v.st[j];
    if (!(s[0] > 0.0) || !isfinite(s[0])) {
      u.done = 1;
      atomicCAS(a.status, 0, (int)KS_ENAN);
    } else {
      u.alpha = u.rho / s[0];
    }
  }
}

__global__ void __launch_bounds__(kCgThreads) cg_b_it2(CgBatchView v) {
  __shared__ double smem[33];
  int j, vb, nb;
  if (!cg_job(v, j, vb, nb)) return;
  const CgArgs &a = v.args[j];
  const CgState t = v.st[j];
  if (t.precond) return;
  const double *p = (t.cg_it % 2 == 0) ? a.pa : a.pb;
  double rl = 0.0;
  for (long long k = (long long)vb * blockDim.x + threadIdx.x; k < a.n;
       k += (long long)nb * blockDim.x) {
    a.x[k] = fma(t.alpha, p[k], a.x[k]);
    const double rk = fma(-t.alpha, a.q[k], a.r[k]);
    a.r[k] = rk;
    rl = fma(rk, rk, rl);
  }
  const double sum = block_sum(rl, smem);
  if (threadIdx.x == 0) a.part[vb] = sum;
  double s[1];
  if (!job_tail(a.part, nb, 1, v.counters + j, smem, s)) return;
  if (threadIdx.x == 0) {
    CgState &u = v.st[j];
    cg_step_done(a, u, s[0]);
    ++u.cg_it;
    u.beta = s[0] / u.rho;
    u.rho = s[0];
  }
}

// Active jobs still iterating: out[0] all of them, out[1] those in CG.
__global__ void cg_b_count(const CgState *st, const unsigned char *active, int J, int *out) {
  __shared__ int cnt[2];
  if (threadIdx.x < 2) cnt[threadIdx.x] = 0;
  __syncthreads();
  int c = 0, g = 0;
  for (int j = threadIdx.x; j < J; j += blockDim.x)
    if (active[j] && !st[j].done) {
      ++c;
      g += !st[j].precond;
    }
  atomicAdd(&cnt[0], c);
  atomicAdd(&cnt[1], g);
  __syncthreads();
  if (threadIdx.x < 2) out[threadIdx.x] = cnt[threadIdx.x];
}

ks_status batch_cg_setup(Batch &B) {
  if (B.maxN > kFusedMaxN)
    return set_error(KS_EINVAL, "batch: N above %d (the fused Hartree preconditioner)", kFusedMaxN);
  KS_CUDA_TRY(cudaFuncSetAttribute(cg_b_precond<0>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)cg_dynamic_smem(kFusedMaxN)));
  KS_CUDA_TRY(cudaFuncSetAttribute(cg_b_precond<1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)cg_dynamic_smem(kFusedMaxN)));
  KS_CUDA_TRY(cudaFuncSetAttribute(cg_b_precond<2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)cg_dynamic_smem(kFusedMaxN)));
  std::vector<CgArgs> args(B.J);
  for (int j = 0; j < B.J; ++j) {
    Problem &P = B.probs[j]->P;
    const BJob &b = B.jobs_host[j];
    CgArgs &a = args[j];
    a = CgArgs{};
    a.N = P.N;
    a.n = P.n;
    a.c = q1_coefficients(P.h);
    a.bscale = 4.0 * M_PI * P.h * P.h * P.h;
    a.rho = P.rho;
    a.x = P.vH;
    a.r = P.cg_r;
    a.pa = P.cg_pa;
    a.pb = P.cg_pb;
    a.r32 = reinterpret_cast<float *>(P.cg_pa);
    a.q = P.cg_q;
    a.z = P.cg_z;
    a.t1 = P.cg_t1;
    a.t2 = P.cg_t2;
    a.phi = P.dst_phi;
    a.kap = P.dst_kap;
    a.mu = P.dst_mu;
    a.part = P.partials;
    a.bar = P.bar;
    a.status = b.status;
    a.iters_out = b.scal + SC_CG_ITERS;
    a.tol = P.cg_tol;
    a.maxit = P.cg_maxit;
    a.precond = P.cg_precond;
    a.fused = 1;
  }
  void *mem = nullptr;
  const size_t abytes = ((sizeof(CgArgs) * B.J + 255) / 256) * 256;
  const size_t sbytes = ((sizeof(CgState) * B.J + 255) / 256) * 256;
  const size_t tbytes = sizeof(double) * 2 * B.J, cbytes = sizeof(unsigned int) * (B.J + 1);
  KS_CUDA_TRY(cudaMalloc(&mem, abytes + sbytes + tbytes + cbytes));
  char *m = static_cast<char *>(mem);
  B.cg_args_dev = mem;
  B.cg_state_dev = m + abytes;
  B.cg_tolw_dev = reinterpret_cast<double *>(m + abytes + sbytes);
  B.cg_counters = reinterpret_cast<unsigned int *>(m + abytes + sbytes + tbytes);
  KS_CUDA_TRY(cudaMemsetAsync(B.cg_state_dev, 0, sbytes, B.stream));
  KS_CUDA_TRY(cudaMemsetAsync(B.cg_counters, 0, cbytes, B.stream));
  KS_CUDA_TRY(cudaMemcpyAsync(B.cg_args_dev, args.data(), sizeof(CgArgs) * B.J,
                              cudaMemcpyHostToDevice, B.stream));
  KS_CUDA_TRY(cudaStreamSynchronize(B.stream));
  B.bytes += abytes + sbytes + tbytes + cbytes;
  return KS_OK;
}

// Hartree solve of every active job (warm-started where B.warm says so) to
// relative residual max(tol, the job's cg_tol), in three pieces so that the
// launches can be captured in a CUDA graph:
//   batch_cg_upload   per-job tolerance and warm flag (host -> device)
//   batch_cg_launch   init + `iters` iterations and the
//                     count of jobs still iterating (no host synchronisation)
//   batch_cg_continue more iterations, one host check each, until no job is
//                     left (after a synchronisation that read the count)
static CgBatchView cg_view(Batch &B, int map) {
  return CgBatchView{static_cast<const CgArgs *>(B.cg_args_dev),
                     static_cast<CgState *>(B.cg_state_dev), B.map(map), B.J, B.active_dev,
                     B.cg_tolw_dev, B.cg_counters};
}

void cg_batch_blocks(int N, long long *a, long long *bc, long long *update) {
  *a = 4LL * N;
  *bc = 2LL * N;
  const long long uy = (N + kUpY - 1) / kUpY, uz = (N + kUpZ - 1) / kUpZ;
  *update = (N * uy * uz + kCgThreads - 1) / kCgThreads;
}

static ks_status cg_precond_launch(Batch &B) {
  const CgBatchView va = cg_view(B, BM_CG_A), vbc = cg_view(B, BM_CG_BC);
  const int na = B.total(BM_CG_A), nbc = B.total(BM_CG_BC);
  const size_t dyn = cg_dynamic_smem(B.maxN);
  cg_b_precond<0><<<na, kCgThreads, dyn, B.stream>>>(va);
  cg_b_precond<1><<<nbc, kCgThreads, dyn, B.stream>>>(vbc);
  cg_b_precond<2><<<nbc, kCgThreads, dyn, B.stream>>>(vbc);
  KS_CUDA_TRY(cudaGetLastError());
  return KS_OK;
}

// One step of every job still iterating: correction of the preconditioned
// jobs (pre), CG iteration of the others (plain; none in the usual batch).
static ks_status cg_iteration_launch(Batch &B, bool pre, bool plain) {
  const CgBatchView nodes = cg_view(B, BM_CG_NODES);
  const int nn = B.total(BM_CG_NODES);
  ProfScope ps_(B.stream, KP_CG, 0.0, 0.0, (pre ? 4 : 0) + (plain ? 2 : 0));
  if (pre) {
    KS_TRY(cg_precond_launch(B));
    cg_b_update<<<B.total(BM_CG_UPDATE), kCgThreads, 0, B.stream>>>(cg_view(B, BM_CG_UPDATE));
  }
  if (plain) {
    cg_b_it1<<<nn, kCgThreads, 0, B.stream>>>(nodes);
    cg_b_it2<<<nn, kCgThreads, 0, B.stream>>>(nodes);
  }
  KS_CUDA_TRY(cudaGetLastError());
  return KS_OK;
}

static ks_status cg_count_launch(Batch &B) {
  ProfScope ps_(B.stream, KP_CG);
  cg_b_count<<<1, 256, 0, B.stream>>>(static_cast<const CgState *>(B.cg_state_dev), B.active_dev,
                                      B.J, B.cg_remaining_dev);
  KS_CUDA_TRY(cudaGetLastError());
  return KS_OK;
}

ks_status batch_cg_upload(Batch &B, double tol) {
  for (int j = 0; j < B.J; ++j) {
    const double t = tol > B.probs[j]->P.cg_tol ? tol : B.probs[j]->P.cg_tol;
    B.cg_tolw_host[2 * j] = t;
    B.cg_tolw_host[2 * j + 1] = B.warm[j] ? 1.0 : 0.0;
  }
  KS_CUDA_TRY(cudaMemcpyAsync(B.cg_tolw_dev, B.cg_tolw_host, sizeof(double) * 2 * B.J,
                              cudaMemcpyHostToDevice, B.stream));
  return KS_OK;
}

ks_status batch_cg_launch(Batch &B, int iters) {
  const CgBatchView nodes = cg_view(B, BM_CG_NODES);
  {
    ProfScope ps_(B.stream, KP_CG);
    cg_b_init<<<B.total(BM_CG_NODES), kCgThreads, 0, B.stream>>>(nodes);
    KS_CUDA_TRY(cudaGetLastError());
  }
  // (a job handed over to CG in these steps goes on in batch_cg_continue)
  bool plain = false, pre = false;
  for (int j = 0; j < B.J; ++j) (B.probs[j]->P.cg_precond ? pre : plain) = true;
  for (int it = 0; it < iters; ++it) KS_TRY(cg_iteration_launch(B, pre, plain));
  return cg_count_launch(B);
}

ks_status batch_cg_continue(Batch &B) {
  int maxit = 0;
  for (int j = 0; j < B.J; ++j)
    if (B.active_host[j] && B.probs[j]->P.cg_maxit > maxit) maxit = B.probs[j]->P.cg_maxit;
  for (int it = 0; it < maxit; ++it) {
    KS_CUDA_TRY(cudaMemcpyAsync(B.cg_remaining_host, B.cg_remaining_dev, 2 * sizeof(int),
                                cudaMemcpyDeviceToHost, B.stream));
    KS_CUDA_TRY(cudaStreamSynchronize(B.stream));
    const int left = B.cg_remaining_host[0], plain = B.cg_remaining_host[1];
    if (left == 0) break;
    KS_TRY(cg_iteration_launch(B, left > plain, plain > 0));
    KS_TRY(cg_count_launch(B));
  }
  return KS_OK;
}

ks_status batch_cg(Batch &B, double tol) {
  KS_TRY(batch_cg_upload(B, tol));
  KS_TRY(batch_cg_launch(B, 0));
  return batch_cg_continue(B);
}

size_t cg_dynamic_smem(int N) {
  return N <= kFusedMaxN ? fused_smem_floats(N) * sizeof(float) : kTiledSmem;
}

int cg_grid_blocks(int sms, int n, int N) {
  const size_t dyn = cg_dynamic_smem(N);
  // always opt in to the largest fused size, so that problems of different
  // N (e.g. concurrent server jobs) never lower the limit under each other
  if (cudaFuncSetAttribute(cg_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)cg_dynamic_smem(kFusedMaxN)) != cudaSuccess) {
    cudaGetLastError();
    return -1;
  }
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, cg_kernel, kCgThreads, dyn) !=
      cudaSuccess || per_sm < 1)
    per_sm = 1;
  // a block per item of the transforms' widest phase, or enough blocks for the
  // nodes; more would only make the barriers dearer
  long long want = (n + kCgThreads - 1) / kCgThreads;
  if (N <= kFusedMaxN && want < 4LL * N) want = 4LL * N;
  long long cap = (long long)sms * (per_sm < 2 ? per_sm : 2);
  if (want > cap) want = cap;
  if (want < 1) want = 1;
  return (int)want;
}

KS_OOB_READER(cg)

}  // namespace ks
