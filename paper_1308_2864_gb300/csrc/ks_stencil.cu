// 27-point Q1 stencils over blocks of orbitals (row-major n x p, orbital
// index fastest):
//
//   hamiltonian:  E_X = f K X + 2 f h^3 Diag(V_eff) X   (the derivative of
//                 Eq. EKS discretised, Sec. 2.3's E_X = H(X) X), M X, and
//                 the kinetic energy (f/2) sum X . K X
//   mass:         M X
//   mass_dots:    M D, ||D||_M^2 = sum D . M D and the Barzilai-Borwein
//                 traces of Eq. bb-1 in the M inner product.
//   hamiltonian, increment form (FP32 phase with X = X_b + delta): the
//                 stencil runs on delta and, with the base X_b, its gradient
//                 E_b = f K X_b + 2 f h^3 Diag(V_b) X_b and potential V_b,
//                 gives the change of the gradient from the base,
//                 e = E_X - E_b = f K delta + 2 f h^3 (Diag(V - V_b) X_b
//                 + Diag(V) delta), M delta, and the change of the kinetic
//                 energy, sum delta . (f K X_b + (f/2) K delta) with
//                 f K X_b = E_b - 2 f h^3 V_b X_b, accumulated with
//                 compensation; every rounding scales with delta or V - V_b.
//
// Plane-marching form.  For a plane z' and a node (x, y) let
//   c(z') = X(x, y, z'),  f(z') = sum of the 4 in-plane face neighbours,
//   e(z') = sum of the 4 in-plane corner neighbours.
// The 27-point neighbourhood of (x, y, z) splits into classes
//   centre = c(z), faces = f(z) + c(z-1) + c(z+1),
//   edges = e(z) + f(z-1) + f(z+1), corners = e(z-1) + e(z+1),
// and the Q1 coefficients depend only on the class (the stiffness face
// coefficient is zero).  A block owns a TX x TY tile of nodes and a chunk of
// PC orbitals, marches along z over a segment of planes, stages one plane
// (with a one-node halo) in shared memory per step, and keeps (c, f, e) of
// the last three planes in registers, so each plane sum is formed once and
// used by three output planes.  Consecutive threads take consecutive
// orbitals of one node, so every global access is a contiguous row segment.
//
// Two ways of staging a plane:
//   TMA (default when the row pitch p * sizeof(T) and the base address are
//     multiples of 16 bytes): the (TX+2) x (TY+2) x PC halo box of a plane is
//     one cp.async.bulk.tensor load into a ring of kStStages shared-memory
//     stages, issued kStStages planes ahead by one thread and completed on
//     an mbarrier; the zero Dirichlet halo comes from the copy's
//     out-of-bounds fill.  V_eff of the output plane is staged in the
//     working precision once per node.
//   plain loads (any p): all threads copy the halo box element by element.
#include "ks_async.cuh"
#include "ks_device.cuh"

namespace ks {

enum StencilKind : int { SK_HAM = 0, SK_MASS = 1, SK_MASS_DOT = 2, SK_MASS_BB = 3, SK_HAM_INC = 4 };

constexpr int kStThreads = 256;
constexpr int kStNodesPerThread = 4;

template <int PC>
struct StTile {
  static constexpr int G = kStThreads / PC;                // node groups
  static constexpr int NODES = G * kStNodesPerThread;      // nodes per tile
  static constexpr int TX = PC >= 16 ? 8 : 16;
  static constexpr int TY = NODES / TX;
  static constexpr int HX = TX + 2, HY = TY + 2;
};

// Nodes of a thread.  FP64: consecutive in y, so that the column sums
// u(x-1, y) + u(x+1, y) of six rows serve the four nodes.  FP32: one of each
// quarter of the tile, consecutive groups on consecutive nodes.
template <typename T, int PC>
__device__ __forceinline__ void st_nodes(int grp, int (&lx)[kStNodesPerThread],
                                         int (&ly)[kStNodesPerThread]) {
  using Tl = StTile<PC>;
  static_assert(Tl::G % Tl::TX == 0 && Tl::G / Tl::TX * kStNodesPerThread == Tl::TY,
                "the groups' columns tile the block");
#pragma unroll
  for (int r = 0; r < kStNodesPerThread; ++r) {
    if constexpr (sizeof(T) == 8) {
      lx[r] = grp % Tl::TX;
      ly[r] = grp / Tl::TX * kStNodesPerThread + r;
    } else {
      const int node = grp + r * Tl::G;
      lx[r] = node % Tl::TX;
      ly[r] = node / Tl::TX;
    }
  }
}

struct StArgs {
  int N, p, zseg, tiles_x, tiles_y, chunks;
  StencilCoef c;
  double occ, h3;
  double kfac;                // factor of K X in E_X: occ, or mu occ (TFW kinetic)
  double k0r;                 // k0 / ke
  const void *A;              // input block (X or D)
  void *out1;                 // E_X (SK_HAM) or M A
  void *out2;                 // M X (SK_HAM, optional)
  const double *veff;
  const void *X, *MX, *Xp, *MXp, *Dp, *MDp;   // SK_MASS_BB; SK_HAM_INC: X = X_b, MX = E_b
  const double *veff_b;       // SK_HAM_INC: V_b
  double *part;               // block partials, channel-major
  int nb;                     // number of blocks (partials stride)
  double *red_out;            // reduced channels (scaled by red_scale)
  double red_scale;
  unsigned int *counter;
  int *status;                // device status word (TMA waits that give up)
  float cf[9];                // k0, ke, kc, m0, mf, me, mc, kfac, 2 occ h^3 rounded to FP32 (host)
};

// Coefficients in the working precision (FP32 ones rounded on the host: a
// per-thread conversion would be nine FP64-pipe instructions per thread).
template <typename T>
struct StCoefT {
  T k0, ke, kc, m0, mf, me, mc, kin, vscale;
  T k0r = 0;                  // FP64: k0 / ke
  bool lumped = false;        // FP64: M = m0 I
  __device__ explicit StCoefT(const StArgs &a) {
    if constexpr (sizeof(T) == 4) {
      k0 = a.cf[0]; ke = a.cf[1]; kc = a.cf[2]; m0 = a.cf[3]; mf = a.cf[4];
      me = a.cf[5]; mc = a.cf[6]; kin = a.cf[7]; vscale = a.cf[8];
    } else {
      k0 = a.c.k0; ke = a.c.ke; kc = a.c.kc; m0 = a.c.m0; mf = a.c.mf;
      me = a.c.me; mc = a.c.mc; vscale = 2.0 * a.occ * a.h3;
      kin = a.kfac * ke;      // of K A in units of ke
      k0r = a.k0r;
      lumped = mc == 0.0;
    }
  }
};

// A thread's running plane sums.  With c, f, e the centre, face and corner
// sums of a plane, a node's output plane needs
//   M A = 4 a(z) + a(z-1) + a(z+1),       a = 16 c + 4 f + e   (times mc)
//   K A = b0(z) + bn(z-1) + bn(z+1),      b0 = (k0/ke) c + e, bn = f + e/2 (times ke)
// because the Q1 coefficients are products of 1-D ones (mass 4 : 1 per axis;
// kc = ke/2, no face term in K).  FP64 carries a, b0 and bn from plane to
// plane: 16.5 FP64 instructions per entry of the Hamiltonian with M X, 8 of
// the mass alone, against 22 and 15 for the class sums (faces, edges,
// corners) combined at the output plane.  The FP64 pipe (16 clocks per warp
// instruction) is the bound of the FP64 stencils, so their time follows that
// count.  FP32, which is bound by memory, keeps the class sums.
template <typename T, int Kind>
struct StCols {
  static constexpr int R = kStNodesPerThread;
  static constexpr bool kHam = Kind == SK_HAM || Kind == SK_HAM_INC;
  static constexpr bool kNew = sizeof(T) == 8;
  // c: centre; f: a (FP64) or the face sum; e: bn (FP64) or the corner sum; g: b0
  T c_old[R], c_mid[R], c_new[R], f_old[R], f_mid[R], f_new[R], e_old[R], e_mid[R], e_new[R];
  T g_mid[R], g_new[R];

  // sums of one staged plane; at(r, dx, dy): value at offset (dx, dy) from node r
  template <typename At>
  __device__ __forceinline__ void plane(At at, const StCoefT<T> &cf, bool want_m) {
    if constexpr (!kNew) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        c_new[r] = at(r, 0, 0);
        f_new[r] = (at(r, -1, 0) + at(r, 1, 0)) + (at(r, 0, -1) + at(r, 0, 1));
        e_new[r] = (at(r, -1, -1) + at(r, 1, -1)) + (at(r, -1, 1) + at(r, 1, 1));
      }
      return;
    }
    T c[R + 2], s[R + 2];
#pragma unroll
    for (int y = 0; y < R + 2; ++y) {
      c[y] = at(0, 0, y - 1);
      s[y] = at(0, -1, y - 1) + at(0, 1, y - 1);
    }
    if constexpr (kHam) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const T f = s[r + 1] + (c[r] + c[r + 2]);
        const T e = s[r] + s[r + 2];
        c_new[r] = c[r + 1];
        if (want_m) f_new[r] = fma((T)16, c[r + 1], fma((T)4, f, e));
        e_new[r] = fma((T)0.5, e, f);
        g_new[r] = fma(cf.k0r, c[r + 1], e);
      }
    } else {
#pragma unroll
      for (int y = 0; y < R + 2; ++y) s[y] = fma((T)4, c[y], s[y]);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        c_new[r] = c[r + 1];
        f_new[r] = fma((T)4, s[r + 1], s[r] + s[r + 2]);
      }
    }
  }
  // M A at node r of the middle plane
  __device__ __forceinline__ T mass(int r, const StCoefT<T> &cf) const {
    if constexpr (kNew) {
      if (cf.lumped) return cf.m0 * c_mid[r];
      return cf.mc * fma((T)4, f_mid[r], f_old[r] + f_new[r]);
    } else {
      const T faces = f_mid[r] + (c_old[r] + c_new[r]);
      const T edges = e_mid[r] + (f_old[r] + f_new[r]);
      const T corners = e_old[r] + e_new[r];
      // (the order of the first two products is part of the FP32 result)
      const T mcf = kHam ? fma(cf.m0, c_mid[r], cf.mf * faces) : fma(cf.mf, faces, cf.m0 * c_mid[r]);
      return fma(cf.mc, corners, fma(cf.me, edges, mcf));
    }
  }
  // K A, in units of ke for FP64
  __device__ __forceinline__ T stiff(int r, const StCoefT<T> &cf) const {
    if constexpr (kNew) {
      return g_mid[r] + (e_old[r] + e_new[r]);
    } else {
      const T edges = e_mid[r] + (f_old[r] + f_new[r]);
      const T corners = e_old[r] + e_new[r];
      return fma(cf.kc, corners, fma(cf.k0, c_mid[r], cf.ke * edges));
    }
  }
  __device__ __forceinline__ void shift() {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if constexpr (kNew) {
        c_mid[r] = c_new[r];
        f_old[r] = f_mid[r]; f_mid[r] = f_new[r];
        if constexpr (kHam) {
          e_old[r] = e_mid[r]; e_mid[r] = e_new[r];
          g_mid[r] = g_new[r];
        }
      } else {
        c_old[r] = c_mid[r]; f_old[r] = f_mid[r]; e_old[r] = e_mid[r];
        c_mid[r] = c_new[r]; f_mid[r] = f_new[r]; e_mid[r] = e_new[r];
      }
    }
  }
};

// Plain-load form of one block (vb = the block's index in the system's
// launch geometry); the single-system kernel and the batched kernel of a
// job table both run it.  Latency of the walk bounds it, so everything a plane
// reads from memory is in flight before its sums: the next halo box and the
// node-local inputs, which (left at their use, behind the stores of the node
// before) waited four times per plane.  Measured, FP32 stencils of 24 batched
// jobs (N 20 to 38, p 4 to 32): E_X 48 -> 34 us per launch, M D with the BB traces and
// the mass products 79 -> 53 us; M x of 105^3 x 1 in FP64 51 -> 37 us.
template <typename T, int PC, int Kind>
__device__ __forceinline__ void stencil_plain_body(const StArgs &a, int vb) {
  using Tl = StTile<PC>;
  __shared__ T tile[Tl::HY * Tl::HX * PC];
  __shared__ double smem[Kind == SK_MASS_BB ? 4 * 33 : 33];
  const int N = a.N, p = a.p;
  // block -> (tile x, tile y, orbital chunk, z segment)
  int b = vb;
  const int txi = b % a.tiles_x; b /= a.tiles_x;
  const int tyi = b % a.tiles_y; b /= a.tiles_y;
  const int oc = b % a.chunks; b /= a.chunks;
  const int zs = b;
  const int x0 = txi * Tl::TX, y0 = tyi * Tl::TY;
  const int z0 = zs * a.zseg;
  const int z1 = min(z0 + a.zseg, N);
  const int lane = threadIdx.x % PC, grp = threadIdx.x / PC;
  const int o = oc * PC + lane;
  const bool ovalid = o < p;
  const T *A = (const T *)a.A;

  int lx[kStNodesPerThread], ly[kStNodesPerThread];
  st_nodes<T, PC>(grp, lx, ly);
  const StCoefT<T> cf(a);
  const bool want_m = Kind != SK_HAM || sizeof(T) == 4 || a.out2 != nullptr;
  StCols<T, Kind> sc;

  // the halo box of the next plane travels in registers (pf) while the
  // current plane's outputs are formed; plane() stores it to the shared tile
  // and forms (c, f, e) of this thread's nodes
  constexpr int kBox = Tl::HY * Tl::HX * PC;
  constexpr int kPf = (kBox + kStThreads - 1) / kStThreads;
  T pf[kPf];
  // where each of them lies within a plane (-1: outside the grid), formed once
  // instead of in every plane
  int off[kPf];
#pragma unroll
  for (int i = 0; i < kPf; ++i) {
    const int t = threadIdx.x + i * kStThreads;
    const int l = t % PC, hn = t / PC;
    const int gx = x0 + hn % Tl::HX - 1, gy = y0 + hn / Tl::HX - 1, go = oc * PC + l;
    off[i] = t < kBox && gx >= 0 && gx < N && gy >= 0 && gy < N && go < p
                 ? (gy * N + gx) * p + go : -1;
  }
  auto fetch = [&](int zp) {
    const T *Az = A + (long long)zp * N * N * p;
    const bool zok = zp >= 0 && zp < N;
#pragma unroll
    for (int i = 0; i < kPf; ++i) pf[i] = zok && off[i] >= 0 ? __ldg(Az + off[i]) : (T)0;
  };
  auto plane = [&]() {
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kPf; ++i) {
      const int t = threadIdx.x + i * kStThreads;
      if (t < kBox) tile[t] = pf[i];
    }
    __syncthreads();
    sc.plane(
        [&](int r, int dx, int dy) {
          const int ti = ((ly[r] + 1 + dy) * Tl::HX + lx[r] + 1 + dx) * PC + lane;
          return KS_IN(ti, kBox) ? tile[ti] : (T)0;
        },
        cf, want_m);
  };

  fetch(z0 - 1);
  plane();
  sc.shift();
  fetch(z0);
  plane();
  sc.shift();
  if (z0 < z1) fetch(z0 + 1);

  T acc0 = 0, acc1 = 0, acc2 = 0, acc3 = 0;
  // this thread's entries within a plane (-1: none)
  int ent[kStNodesPerThread];
#pragma unroll
  for (int r = 0; r < kStNodesPerThread; ++r) {
    const int gx = x0 + lx[r], gy = y0 + ly[r];
    ent[r] = ovalid && gx < N && gy < N ? gy * N + gx : -1;
  }

  for (int z = z0; z < z1; ++z) {
    const long long zb = (long long)z * N * N, nodes = (long long)N * N * N;
    // the node-local inputs of plane z, all in flight at once: left at their use
    // they would wait for each other behind the stores of the node before
    double va[kStNodesPerThread];
    T bb[6][kStNodesPerThread];
    auto locals = [&]() {
#pragma unroll
      for (int r = 0; r < kStNodesPerThread; ++r) {
        const long long k = zb + ent[r], idx = k * p + o;
        const bool in = ent[r] >= 0 && KS_IN(k, nodes) && KS_IN(idx, nodes * p);
        if (Kind == SK_HAM || Kind == SK_HAM_INC) va[r] = in ? a.veff[k] : 0.0;
        if (Kind == SK_MASS_BB) {
          bb[0][r] = in ? ((const T *)a.X)[idx] : (T)0;
          bb[1][r] = in ? ((const T *)a.Xp)[idx] : (T)0;
          bb[2][r] = in ? ((const T *)a.MX)[idx] : (T)0;
          bb[3][r] = in ? ((const T *)a.MXp)[idx] : (T)0;
          bb[4][r] = in ? ((const T *)a.Dp)[idx] : (T)0;
          bb[5][r] = in ? ((const T *)a.MDp)[idx] : (T)0;
        }
      }
    };
    constexpr bool kEarly = sizeof(T) == 4;        // FP64: registers
    if (kEarly) locals();
    plane();                                       // plane z + 1
    if (z + 1 < z1) fetch(z + 2);                  // in flight during the outputs of plane z
    if (!kEarly) locals();
#pragma unroll
    for (int r = 0; r < kStNodesPerThread; ++r) {
      const T centre = sc.c_mid[r];
      const long long k = zb + ent[r], idx = k * p + o;
      if (ent[r] >= 0 && KS_IN(k, nodes) && KS_IN(idx, nodes * p)) {
        const T m = want_m ? sc.mass(r, cf) : (T)0;
        if (Kind == SK_HAM) {
          const T kx = sc.stiff(r, cf);
          if (sizeof(T) == 4 || a.out1) ((T *)a.out1)[idx] = fma(cf.kin, kx, cf.vscale * (T)va[r] * centre);
          if (a.out2) ((T *)a.out2)[idx] = m;
          acc0 = fma(centre, kx, acc0);
        } else if (Kind == SK_HAM_INC) {
          const T kx = sc.stiff(r, cf);
          const T xb = ((const T *)a.X)[idx], eb = ((const T *)a.MX)[idx];
          const T v = (T)va[r], vb = (T)a.veff_b[k], dv = (T)(va[r] - a.veff_b[k]);
          ((T *)a.out1)[idx] = cf.kin * kx + cf.vscale * (dv * xb + v * centre);
          if (a.out2) ((T *)a.out2)[idx] = m;
          // compensated sum of delta . (2 f K X_b + f K delta); acc1 holds the
          // running rounding error
          const T fkxb = eb - cf.vscale * vb * xb;
          const T t = centre * ((T)2 * fkxb + cf.kin * kx);
          const T y = t - acc1;
          const T sum = acc0 + y;
          acc1 = (sum - acc0) - y;
          acc0 = sum;
        } else {
          if (Kind != SK_MASS_DOT || sizeof(T) == 4 || a.out1) ((T *)a.out1)[idx] = m;
          if (Kind >= SK_MASS_DOT) acc0 = fma(centre, m, acc0);
          if (Kind == SK_MASS_BB) {
            const T dx = bb[0][r] - bb[1][r];
            const T dmx = bb[2][r] - bb[3][r];
            const T dd = centre - bb[4][r];
            const T dmd = m - bb[5][r];
            acc1 = fma(dx, dmx, acc1);
            acc2 = fma(dx, dmd, acc2);
            acc3 = fma(dd, dmd, acc3);
          }
        }
      }
    }
    sc.shift();
  }
  if (Kind == SK_MASS) return;
  if (Kind == SK_HAM && StCols<T, Kind>::kNew) acc0 *= cf.ke;
  if constexpr (Kind == SK_MASS_BB) {
    double s[4] = {(double)acc0, (double)acc1, (double)acc2, (double)acc3};
    block_sum_n<4>(s, smem);
    if (threadIdx.x == 0)
#pragma unroll
      for (int i = 0; i < 4; ++i) a.part[i * a.nb + vb] = s[i];
  } else {
    const double s0 =
        block_sum(Kind == SK_HAM_INC ? (double)acc0 - (double)acc1 : (double)acc0, smem);
    if (threadIdx.x == 0) a.part[vb] = s0;
  }
  grid_reduce_tail<Kind == SK_MASS_BB ? 4 : 1>(a.part, a.nb, a.red_out, a.red_scale, a.counter,
                                               smem);
}

// Resident blocks that the plain-load kernels are compiled for: the walk over
// the planes is latency, and FP64 at one block per SM (over 128 registers) or
// the short FP32 kinds at two leave the SM idle between a plane's loads and use.
template <typename T, int Kind>
constexpr int st_min_blocks() {
  return sizeof(T) == 4 && (Kind == SK_MASS || Kind == SK_MASS_DOT) ? 3 : 2;
}

template <typename T, int PC, int Kind>
__global__ void __launch_bounds__(kStThreads, (st_min_blocks<T, Kind>())) stencil_kernel(StArgs a) {
  stencil_plain_body<T, PC, Kind>(a, blockIdx.x);
}

constexpr int kStStages = 3;

// Blocks read at the output node only (no halo), staged by TMA with the
// plane: SK_HAM_INC X_b and E_b; SK_MASS_BB X, MX, Xp, MXp, Dp, MDp in FP32
// (in FP64 the six boxes would not leave room for two blocks per SM: the
// kernel loads them from global memory at the output step instead).
template <typename T, int Kind>
constexpr int st_naux() {
  return Kind == SK_HAM_INC ? 2 : (Kind == SK_MASS_BB && sizeof(T) == 4) ? 6 : 0;
}

template <typename T, int PC, int Kind>
struct StRing {
  using Tl = StTile<PC>;
  static constexpr int NAUX = st_naux<T, Kind>();
  static constexpr int BOX = Tl::HY * Tl::HX * PC;                 // elements of one halo box
  static constexpr uint32_t BOX_BYTES = BOX * sizeof(T);
  static constexpr int HALO = ((BOX_BYTES + 127) / 128) * 128 / sizeof(T);   // 128-byte aligned
  static constexpr int AUXB = Tl::TY * Tl::TX * PC;                // elements of one node box
  static constexpr uint32_t AUX_BYTES = AUXB * sizeof(T);
  static constexpr int AUX = ((AUX_BYTES + 127) / 128) * 128 / sizeof(T);
  static constexpr int STAGE = HALO + NAUX * AUX;
  // the stages plus slack to align the ring to 128 bytes at run time
  static constexpr size_t SMEM = (size_t)kStStages * STAGE * sizeof(T) + 128;
};

struct StTmaArgs {
  CUtensorMap map;            // (orbital, x, y, z) view of the input block
  CUtensorMap aux[6];         // the same views of the node-local inputs (st_naux of them)
  StArgs a;
};

template <typename T, int PC, int Kind>
__global__ void __launch_bounds__(kStThreads, 2) stencil_tma_kernel(const __grid_constant__ StTmaArgs ta) {
  using Tl = StTile<PC>;
  using Rg = StRing<T, PC, Kind>;
  constexpr int TXY = Tl::TX * Tl::TY;
  constexpr int NAUX = Rg::NAUX;
  static_assert(TXY <= kStThreads, "one V_eff loader per node");
  extern __shared__ __align__(128) unsigned char st_ring_raw[];
  T *ring = reinterpret_cast<T *>(st_ring_raw + ((128u - (smem_addr(st_ring_raw) & 127u)) & 127u));
  __shared__ __align__(8) uint64_t full[kStStages];
  __shared__ T vs[3][TXY];
  // SK_HAM_INC: V_b and V - V_b (formed in FP64) of the same planes
  __shared__ T vbs[Kind == SK_HAM_INC ? 3 : 1][Kind == SK_HAM_INC ? TXY : 1];
  __shared__ T dvs[Kind == SK_HAM_INC ? 3 : 1][Kind == SK_HAM_INC ? TXY : 1];
  __shared__ double smem[Kind == SK_MASS_BB ? 4 * 33 : 33];
  const StArgs &a = ta.a;
  const int N = a.N, p = a.p;
  int b = blockIdx.x;
  const int txi = b % a.tiles_x; b /= a.tiles_x;
  const int tyi = b % a.tiles_y; b /= a.tiles_y;
  const int oc = b % a.chunks; b /= a.chunks;
  const int zs = b;
  const int x0 = txi * Tl::TX, y0 = tyi * Tl::TY;
  const int z0 = zs * a.zseg;
  const int z1 = min(z0 + a.zseg, N);
  const int nplanes = z1 - z0 + 2;          // planes z0 - 1 .. z1
  const int lane = threadIdx.x % PC, grp = threadIdx.x / PC;
  const int o = oc * PC + lane;
  const bool ovalid = o < p;

  // stage q holds the halo box of plane z0 - 1 + q and, from q = 2 on, the
  // node boxes of the output plane of step q (z0 - 2 + q)
  auto load_stage = [&](int q) {
    T *dst = ring + (q % kStStages) * Rg::STAGE;
    uint64_t *bar = &full[q % kStStages];
    const bool with_aux = NAUX > 0 && q >= 2;
    mbar_arrive_expect_tx(bar, Rg::BOX_BYTES + (with_aux ? NAUX * Rg::AUX_BYTES : 0u));
    tma_load_4d(dst, &ta.map, bar, oc * PC, x0 - 1, y0 - 1, z0 - 1 + q);
    if (with_aux)
#pragma unroll
      for (int i = 0; i < NAUX; ++i)
        tma_load_4d(dst + Rg::HALO + i * Rg::AUX, &ta.aux[i], bar, oc * PC, x0, y0, z0 - 2 + q);
  };
  if (threadIdx.x == 0) {
    prefetch_tensor_map(&ta.map);
#pragma unroll
    for (int i = 0; i < NAUX; ++i) prefetch_tensor_map(&ta.aux[i]);
#pragma unroll
    for (int st = 0; st < kStStages; ++st) mbar_init(&full[st], 1);
    fence_barrier_init();
  }
  __syncthreads();
  if (threadIdx.x == 0)
    for (int q = 0; q < kStStages && q < nplanes; ++q) load_stage(q);

  int lx[kStNodesPerThread], ly[kStNodesPerThread];
  st_nodes<T, PC>(grp, lx, ly);
  // V_eff of plane z0 - 1 + q is read one iteration ahead by the thread that
  // owns the node, converted once and kept in vs[q % 3]
  const int vx = x0 + (int)threadIdx.x % Tl::TX, vy = y0 + (int)threadIdx.x / Tl::TX;
  constexpr bool kHam = Kind == SK_HAM || Kind == SK_HAM_INC;
  // FP64 keeps 2 f h^3 V_eff: one product per node, not per entry
  constexpr bool kScaledV = Kind == SK_HAM && sizeof(T) == 8;
  const bool vown = kHam && (int)threadIdx.x < TXY && vx < N && vy < N;
  double vreg = 0.0, vbreg = 0.0;
  const long long nodes = (long long)N * N * N;
  if (vown && z0 >= 1 && KS_IN(((long long)(z0 - 1) * N + vy) * N + vx, nodes)) {
    vreg = a.veff[((long long)(z0 - 1) * N + vy) * N + vx];
    if (Kind == SK_HAM_INC) vbreg = a.veff_b[((long long)(z0 - 1) * N + vy) * N + vx];
  }

  const StCoefT<T> cf(a);
  T acc0 = 0, acc1 = 0, acc2 = 0, acc3 = 0;
  const bool want_m = Kind != SK_HAM || sizeof(T) == 4 || a.out2 != nullptr;
  StCols<T, Kind> sc;
  int failed_at = -1;
  for (int q = 0; q < nplanes; ++q) {
    const int zp = z0 - 1 + q;
    const int st = q % kStStages;
    if (kHam && (int)threadIdx.x < TXY) {
      vs[q % 3][threadIdx.x] = kScaledV ? cf.vscale * (T)vreg : (T)vreg;
      if (Kind == SK_HAM_INC) {
        vbs[q % 3][threadIdx.x] = (T)vbreg;
        dvs[q % 3][threadIdx.x] = (T)(vreg - vbreg);
      }
      vreg = 0.0;
      vbreg = 0.0;
      if (vown && zp + 1 < N && KS_IN(((long long)(zp + 1) * N + vy) * N + vx, nodes)) {
        vreg = a.veff[((long long)(zp + 1) * N + vy) * N + vx];
        if (Kind == SK_HAM_INC) vbreg = a.veff_b[((long long)(zp + 1) * N + vy) * N + vx];
      }
    }
    const bool got = mbar_wait_parity(&full[st], (uint32_t)((q / kStStages) & 1));
    const T *tile = ring + st * Rg::STAGE;
    sc.plane(
        [&](int r, int dx, int dy) {
          const int ti = ((ly[r] + 1 + dy) * Tl::HX + lx[r] + 1 + dx) * PC + lane;
          return KS_IN(ti, Rg::BOX) ? tile[ti] : (T)0;
        },
        cf, want_m);
    if (q >= 2) {
      const int z = zp - 1;
      const T *vz = vs[(q + 2) % 3];
      T bb[6][kStNodesPerThread];
      if constexpr (NAUX > 0) {
        // the node-local inputs of this output plane, staged with it
#pragma unroll
        for (int i = 0; i < NAUX; ++i)
#pragma unroll
          for (int r = 0; r < kStNodesPerThread; ++r)
          {
            const int ti = (ly[r] * Tl::TX + lx[r]) * PC + lane;
            bb[i][r] = KS_IN(ti, Rg::AUXB) ? tile[Rg::HALO + i * Rg::AUX + ti] : (T)0;
          }
      } else if (Kind == SK_MASS_BB) {
        // all loads of the plane first, so they are in flight together
#pragma unroll
        for (int r = 0; r < kStNodesPerThread; ++r) {
          const int gx = x0 + lx[r], gy = y0 + ly[r];
          if (ovalid && gx < N && gy < N &&
              KS_IN((((long long)z * N + gy) * N + gx) * p + o, nodes * p)) {
            const long long idx = (((long long)z * N + gy) * N + gx) * p + o;
            bb[0][r] = ((const T *)a.X)[idx];
            bb[1][r] = ((const T *)a.MX)[idx];
            bb[2][r] = ((const T *)a.Xp)[idx];
            bb[3][r] = ((const T *)a.MXp)[idx];
            bb[4][r] = ((const T *)a.Dp)[idx];
            bb[5][r] = ((const T *)a.MDp)[idx];
          }
        }
      }
#pragma unroll
      for (int r = 0; r < kStNodesPerThread; ++r) {
        const int gx = x0 + lx[r], gy = y0 + ly[r];
        const T centre = sc.c_mid[r];
        if (ovalid && gx < N && gy < N && KS_IN(((long long)z * N + gy) * N + gx, nodes) &&
            KS_IN((((long long)z * N + gy) * N + gx) * p + o, nodes * p)) {
          const long long k = ((long long)z * N + gy) * N + gx;
          const long long idx = k * p + o;
          const T m = want_m ? sc.mass(r, cf) : (T)0;
          if (Kind == SK_HAM) {
            const T kx = sc.stiff(r, cf);
            if (sizeof(T) == 4 || a.out1) {
              const T v = vz[ly[r] * Tl::TX + lx[r]];
              ((T *)a.out1)[idx] = fma(cf.kin, kx, (kScaledV ? v : cf.vscale * v) * centre);
            }
            if (a.out2) ((T *)a.out2)[idx] = m;
            acc0 = fma(centre, kx, acc0);
          } else if (Kind == SK_HAM_INC) {
            const T kx = sc.stiff(r, cf);
            const T xb = bb[0][r], eb = bb[1][r];
            const int nd = ly[r] * Tl::TX + lx[r];
            const int pl = (q + 2) % 3;
            const T v = vz[nd], vb = vbs[pl][nd], dv = dvs[pl][nd];
            ((T *)a.out1)[idx] = cf.kin * kx + cf.vscale * (dv * xb + v * centre);
            if (a.out2) ((T *)a.out2)[idx] = m;
            const T fkxb = eb - cf.vscale * vb * xb;
            const T t = centre * ((T)2 * fkxb + cf.kin * kx);
            const T y = t - acc1;
            const T sum = acc0 + y;
            acc1 = (sum - acc0) - y;
            acc0 = sum;
          } else {
            if (Kind != SK_MASS_DOT || sizeof(T) == 4 || a.out1) ((T *)a.out1)[idx] = m;
            if (Kind >= SK_MASS_DOT) acc0 = fma(centre, m, acc0);
            if (Kind == SK_MASS_BB) {
              const T dx = bb[0][r] - bb[2][r];
              const T dmx = bb[1][r] - bb[3][r];
              const T dd = centre - bb[4][r];
              const T dmd = m - bb[5][r];
              acc1 = fma(dx, dmx, acc1);
              acc2 = fma(dx, dmd, acc2);
              acc3 = fma(dd, dmd, acc3);
            }
          }
        }
      }
    }
    // every thread is done with this stage: refill it kStStages planes ahead
    if (__syncthreads_or(!got)) {
      failed_at = q;
      break;
    }
    if (threadIdx.x == 0 && q + kStStages < nplanes) load_stage(q + kStStages);
    sc.shift();
  }
  if (failed_at >= 0) {
    // record the timeout, give the copies still in flight a bounded wait,
    // and still take part in the reduction so that its counter re-arms
    if (threadIdx.x == 0) {
      atomicCAS(a.status, 0, (int)KS_ETIMEOUT);
      for (int q = failed_at; q < failed_at + kStStages && q < nplanes; ++q)
        mbar_wait_parity(&full[q % kStStages], (uint32_t)((q / kStStages) & 1));
    }
    acc0 = acc1 = acc2 = acc3 = 0;
  }
  if (Kind == SK_MASS) return;
  if (Kind == SK_HAM && StCols<T, Kind>::kNew) acc0 *= cf.ke;
  if constexpr (Kind == SK_MASS_BB) {
    double s[4] = {(double)acc0, (double)acc1, (double)acc2, (double)acc3};
    block_sum_n<4>(s, smem);
    if (threadIdx.x == 0)
#pragma unroll
      for (int i = 0; i < 4; ++i) a.part[i * a.nb + blockIdx.x] = s[i];
  } else {
    const double s0 =
        block_sum(Kind == SK_HAM_INC ? (double)acc0 - (double)acc1 : (double)acc0, smem);
    if (threadIdx.x == 0) a.part[blockIdx.x] = s0;
  }
  grid_reduce_tail<Kind == SK_MASS_BB ? 4 : 1>(a.part, a.nb, a.red_out, a.red_scale, a.counter,
                                               smem);
}

// ---------------------------------------------------------------- FP32, p >= 32
// The TMA form in FP32 with 32-orbital chunks.  Memory should bound it (three
// to nine blocks of 4 bytes per entry), but one entry at a time cost some 55
// warp instructions per 32 entries and 1.9 loaded halo entries per node, and the
// kernel ran at 3.6 TB/s, bound by issue.  Here a thread owns two adjacent
// orbitals of a column of four nodes: 8-byte shared loads, packed FP32
// arithmetic (add / mul / fma.rn.f32x2, the same roundings as the scalar
// forms), column sums shared by the four nodes, offsets formed once per
// kernel; the 8 x 8 node tile loads 1.6 halo entries per node.  96^3 x 128,
// Hamiltonian with M X: 383 -> 278 us (3.6 -> 4.9 TB/s of 1.37 GB).
struct StF2 {
  static constexpr int TX = 8, TY = 8, PC = 32, HX = TX + 2, HY = TY + 2, R = 4;
  static constexpr int BOX = HX * HY * PC, AUX = TX * TY * PC;       // floats
  static_assert(BOX * 4 % 128 == 0 && AUX * 4 % 128 == 0, "stages stay 128-byte aligned");
  static_assert(kStThreads == PC / 2 * TX * (TY / R), "one thread per orbital pair and column");
};

template <int Kind>
constexpr size_t st_f2_smem() {
  return (size_t)kStStages * (StF2::BOX + st_naux<float, Kind>() * StF2::AUX) * sizeof(float) + 128;
}

template <int Kind>
__global__ void __launch_bounds__(kStThreads, Kind == SK_MASS_BB ? 1 : 2)
    stencil_f32x2_kernel(const __grid_constant__ StTmaArgs ta) {
  using S = StF2;
  constexpr int NAUX = st_naux<float, Kind>(), STAGE = S::BOX + NAUX * S::AUX, TXY = S::TX * S::TY;
  constexpr bool kHam = Kind == SK_HAM || Kind == SK_HAM_INC;
  extern __shared__ __align__(128) unsigned char st_ring_raw[];
  float *ring =
      reinterpret_cast<float *>(st_ring_raw + ((128u - (smem_addr(st_ring_raw) & 127u)) & 127u));
  __shared__ __align__(8) uint64_t full[kStStages];
  // SK_HAM: 2 f h^3 V; SK_HAM_INC: V, V_b and V - V_b (formed in FP64)
  __shared__ float vs[kHam ? 3 : 1][kHam ? TXY : 1];
  __shared__ float vbs[Kind == SK_HAM_INC ? 3 : 1][Kind == SK_HAM_INC ? TXY : 1];
  __shared__ float dvs[Kind == SK_HAM_INC ? 3 : 1][Kind == SK_HAM_INC ? TXY : 1];
  __shared__ double smem[Kind == SK_MASS_BB ? 4 * 33 : 33];
  const StArgs &a = ta.a;
  const int N = a.N, p = a.p;
  int b = blockIdx.x;
  const int x0 = b % a.tiles_x * S::TX; b /= a.tiles_x;
  const int y0 = b % a.tiles_y * S::TY; b /= a.tiles_y;
  const int o0 = b % a.chunks * S::PC; b /= a.chunks;
  const int z0 = b * a.zseg;
  const int z1 = min(z0 + a.zseg, N);
  const int nplanes = z1 - z0 + 2;
  const int pair = threadIdx.x % (S::PC / 2), col = threadIdx.x / (S::PC / 2);
  const int lx = col % S::TX, ly = col / S::TX * S::R;

  auto load_stage = [&](int q) {
    float *dst = ring + (q % kStStages) * STAGE;
    uint64_t *bar = &full[q % kStStages];
    const bool with_aux = NAUX > 0 && q >= 2;
    mbar_arrive_expect_tx(bar, (S::BOX + (with_aux ? NAUX * S::AUX : 0)) * 4u);
    tma_load_4d(dst, &ta.map, bar, o0, x0 - 1, y0 - 1, z0 - 1 + q);
    if (with_aux)
#pragma unroll
      for (int i = 0; i < NAUX; ++i)
        tma_load_4d(dst + S::BOX + i * S::AUX, &ta.aux[i], bar, o0, x0, y0, z0 - 2 + q);
  };
  if (threadIdx.x == 0) {
    prefetch_tensor_map(&ta.map);
#pragma unroll
    for (int i = 0; i < NAUX; ++i) prefetch_tensor_map(&ta.aux[i]);
#pragma unroll
    for (int st = 0; st < kStStages; ++st) mbar_init(&full[st], 1);
    fence_barrier_init();
  }
  __syncthreads();
  if (threadIdx.x == 0)
    for (int q = 0; q < kStStages && q < nplanes; ++q) load_stage(q);

  // V_eff of plane z0 - 1 + q, read one step ahead by the thread that owns the node
  const int vx = x0 + (int)threadIdx.x % S::TX, vy = y0 + (int)threadIdx.x / S::TX;
  const bool vown = kHam && (int)threadIdx.x < TXY && vx < N && vy < N;
  const long long NN = (long long)N * N;
  double vreg = 0.0, vbreg = 0.0;
  if (vown && z0 >= 1) {
    vreg = a.veff[(z0 - 1) * NN + (long long)vy * N + vx];
    if (Kind == SK_HAM_INC) vbreg = a.veff_b[(z0 - 1) * NN + (long long)vy * N + vx];
  }
  // entry offsets of the four nodes in plane z0 (p is a multiple of 4: a pair
  // is inside the row as a whole)
  const int o = o0 + 2 * pair, gx = x0 + lx;
  bool ok[S::R];
  long long at[S::R];
#pragma unroll
  for (int r = 0; r < S::R; ++r) {
    const int gy = y0 + ly + r;
    ok[r] = o < p && gx < N && gy < N &&
            KS_IN((((long long)(z1 - 1) * N + gy) * N + gx) * p + o + 1, NN * N * p);
    at[r] = (((long long)z0 * N + gy) * N + gx) * p + o;
  }
  const long long plane = NN * p;
  const f2_t k0 = f2_dup(a.cf[0]), ke = f2_dup(a.cf[1]), kc = f2_dup(a.cf[2]);
  const f2_t m0 = f2_dup(a.cf[3]), mf = f2_dup(a.cf[4]), me = f2_dup(a.cf[5]), mc = f2_dup(a.cf[6]);
  const f2_t kin = f2_dup(a.cf[7]), vscale = f2_dup(a.cf[8]);
  f2_t acc[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) acc[i] = 0ull;
  f2_t co[S::R], fo[S::R], eo[S::R], cm[S::R], fm[S::R], em[S::R];
#pragma unroll
  for (int r = 0; r < S::R; ++r) co[r] = fo[r] = eo[r] = cm[r] = fm[r] = em[r] = 0ull;
  const int base = (ly * S::HX + lx) * S::PC + 2 * pair;      // row y - 1, column x - 1
  const int nbase = (ly * S::TX + lx) * S::PC + 2 * pair;     // node boxes
  auto ld = [](const float *q) { return *reinterpret_cast<const f2_t *>(q); };
  int failed_at = -1;
  for (int q = 0; q < nplanes; ++q) {
    const int zp = z0 - 1 + q, st = q % kStStages;
    if (kHam && (int)threadIdx.x < TXY) {
      vs[q % 3][threadIdx.x] = Kind == SK_HAM ? a.cf[8] * (float)vreg : (float)vreg;
      if (Kind == SK_HAM_INC) {
        vbs[q % 3][threadIdx.x] = (float)vbreg;
        dvs[q % 3][threadIdx.x] = (float)(vreg - vbreg);
      }
      vreg = 0.0;
      vbreg = 0.0;
      if (vown && zp + 1 < N) {
        vreg = a.veff[(zp + 1) * NN + (long long)vy * N + vx];
        if (Kind == SK_HAM_INC) vbreg = a.veff_b[(zp + 1) * NN + (long long)vy * N + vx];
      }
    }
    const bool got = mbar_wait_parity(&full[st], (uint32_t)((q / kStStages) & 1));
    const float *tile = ring + st * STAGE;
    f2_t cn[S::R], fn[S::R], en[S::R];
    {
      f2_t c[S::R + 2], s[S::R + 2];
#pragma unroll
      for (int y = 0; y < S::R + 2; ++y) {
        const float *row = tile + base + y * S::HX * S::PC;
        c[y] = ld(row + S::PC);
        s[y] = f2_add(ld(row), ld(row + 2 * S::PC));
      }
#pragma unroll
      for (int r = 0; r < S::R; ++r) {
        cn[r] = c[r + 1];
        fn[r] = f2_add(s[r + 1], f2_add(c[r], c[r + 2]));
        en[r] = f2_add(s[r], s[r + 2]);
      }
    }
    if (q >= 2) {
      const long long zo = (long long)(q - 2) * plane;
#pragma unroll
      for (int r = 0; r < S::R; ++r) {
        const f2_t edges = f2_add(em[r], f2_add(fo[r], fn[r]));
        const f2_t corners = f2_add(eo[r], en[r]);
        const f2_t faces = f2_add(fm[r], f2_add(co[r], cn[r]));
        // (the same order of products as the scalar forms, StCols::mass)
        const f2_t mcf =
            kHam ? f2_fma(m0, cm[r], f2_mul(mf, faces)) : f2_fma(mf, faces, f2_mul(m0, cm[r]));
        const f2_t m = f2_fma(mc, corners, f2_fma(me, edges, mcf));
        const int nd = (ly + r) * S::TX + lx, pl = (q + 2) % 3;
        const float *aux = tile + S::BOX + nbase + r * S::TX * S::PC;
        if (kHam) {
          const f2_t kx = f2_fma(kc, corners, f2_fma(k0, cm[r], f2_mul(ke, edges)));
          f2_t ex;
          if (Kind == SK_HAM) {
            ex = f2_fma(kin, kx, f2_mul(f2_dup(vs[pl][nd]), cm[r]));
            if (ok[r]) acc[0] = f2_fma(cm[r], kx, acc[0]);
          } else {
            const f2_t xb = ld(aux), eb = ld(aux + S::AUX);
            const f2_t v = f2_dup(vs[pl][nd]), vb = f2_dup(vbs[pl][nd]), dv = f2_dup(dvs[pl][nd]);
            const f2_t kd = f2_mul(kin, kx);
            ex = f2_fma(vscale, f2_fma(dv, xb, f2_mul(v, cm[r])), kd);
            // compensated sum of delta . (2 f K X_b + f K delta); acc[1] holds the
            // running rounding error
            const f2_t fkxb = f2_sub(eb, f2_mul(f2_mul(vscale, vb), xb));
            const f2_t t = f2_mul(cm[r], f2_fma(f2_dup(2.f), fkxb, kd));
            if (ok[r]) {
              const f2_t y = f2_sub(t, acc[1]);
              const f2_t sum = f2_add(acc[0], y);
              acc[1] = f2_sub(f2_sub(sum, acc[0]), y);
              acc[0] = sum;
            }
          }
          if (ok[r]) {
            *reinterpret_cast<f2_t *>((float *)a.out1 + at[r] + zo) = ex;
            if (a.out2) *reinterpret_cast<f2_t *>((float *)a.out2 + at[r] + zo) = m;
          }
        } else if (ok[r]) {
          *reinterpret_cast<f2_t *>((float *)a.out1 + at[r] + zo) = m;
          if (Kind >= SK_MASS_DOT) acc[0] = f2_fma(cm[r], m, acc[0]);
          if (Kind == SK_MASS_BB) {
            const f2_t dx = f2_sub(ld(aux), ld(aux + 2 * S::AUX));
            const f2_t dmx = f2_sub(ld(aux + S::AUX), ld(aux + 3 * S::AUX));
            const f2_t dd = f2_sub(cm[r], ld(aux + 4 * S::AUX));
            const f2_t dmd = f2_sub(m, ld(aux + 5 * S::AUX));
            acc[1] = f2_fma(dx, dmx, acc[1]);
            acc[2] = f2_fma(dx, dmd, acc[2]);
            acc[3] = f2_fma(dd, dmd, acc[3]);
          }
        }
      }
    }
    // every thread is done with this stage: refill it kStStages planes ahead
    if (__syncthreads_or(!got)) {
      failed_at = q;
      break;
    }
    if (threadIdx.x == 0 && q + kStStages < nplanes) load_stage(q + kStStages);
#pragma unroll
    for (int r = 0; r < S::R; ++r) {
      co[r] = cm[r]; fo[r] = fm[r]; eo[r] = em[r];
      cm[r] = cn[r]; fm[r] = fn[r]; em[r] = en[r];
    }
  }
  if (failed_at >= 0) {
    // record the timeout, give the copies still in flight a bounded wait,
    // and still take part in the reduction so that its counter re-arms
    if (threadIdx.x == 0) {
      atomicCAS(a.status, 0, (int)KS_ETIMEOUT);
      for (int q = failed_at; q < failed_at + kStStages && q < nplanes; ++q)
        mbar_wait_parity(&full[q % kStStages], (uint32_t)((q / kStStages) & 1));
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[i] = 0ull;
  }
  if (Kind == SK_MASS) return;
  if constexpr (Kind == SK_MASS_BB) {
    double s[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) s[i] = f2_sum(acc[i]);
    block_sum_n<4>(s, smem);
    if (threadIdx.x == 0)
#pragma unroll
      for (int i = 0; i < 4; ++i) a.part[i * a.nb + blockIdx.x] = s[i];
  } else {
    const double s0 = block_sum(
        Kind == SK_HAM_INC ? f2_sum(acc[0]) - f2_sum(acc[1]) : f2_sum(acc[0]), smem);
    if (threadIdx.x == 0) a.part[blockIdx.x] = s0;
  }
  grid_reduce_tail<Kind == SK_MASS_BB ? 4 : 1>(a.part, a.nb, a.red_out, a.red_scale, a.counter,
                                               smem);
}

// Geometry of a launch: tiles, orbital chunks and z segments; the number of
// segments is lowered until the block partials (nchan per block) fit.
// `halo` > 0 (one system alone on the device): the segment length with the
// shortest schedule.  The blocks of an SM share its pipes, so an SM with k
// blocks needs k (zseg + halo) plane times, halo being the cost of a block's
// two extra planes; a few blocks too many per SM (a nearly empty last wave)
// cost as much as the shortest segments' halos, and a grid with fewer blocks
// than SMs leaves SMs idle, so both are weighed: 24^3 x 4 runs 96 blocks of
// one plane (12 of 8 before), 64^3 x 64 1024 of 16 planes (7 per SM).
// `halo` = 0 (jobs that share the device): about 8 blocks per SM, segments of
// at least 8 planes, or segments of `planes` planes when given.
static ks_status stencil_geometry_of(const Problem &P, int tx, int ty, int pc, int nchan,
                                     StArgs &a, double halo, int planes) {
  a.N = P.N;
  a.p = P.p;
  a.tiles_x = (P.N + tx - 1) / tx;
  a.tiles_y = (P.N + ty - 1) / ty;
  a.chunks = (P.p + pc - 1) / pc;
  const long long base = (long long)a.tiles_x * a.tiles_y * a.chunks;
  long long segs = (8LL * P.sms + base - 1) / base;
  const long long maxsegs = (P.N + 7) / 8;
  if (segs > maxsegs) segs = maxsegs;
  if (planes > 0) segs = (P.N + planes - 1) / planes;
  if (halo > 0.0) {
    double best = 1e300;
    for (int z = P.N; z >= 1; --z) {
      const long long used = (P.N + z - 1) / z;
      const double cost = (double)((base * used + P.sms - 1) / P.sms) * (z + halo);
      if (cost < best) {
        best = cost;
        segs = used;
      }
    }
  }
  if (segs < 1) segs = 1;
  for (;;) {
    a.zseg = (int)((P.N + segs - 1) / segs);
    const long long used = (P.N + a.zseg - 1) / a.zseg;
    const long long nb = base * used;
    if (nchan == 0 || (size_t)(nb * nchan) <= P.partials_len) {
      if (nb > 0x7fffffffLL) return set_error(KS_EINVAL, "stencil: grid too large");
      a.nb = (int)nb;
      return KS_OK;
    }
    if (used == 1) return set_error(KS_EINVAL, "stencil: partial buffer too small");
    segs = used / 2;
  }
}

template <int PC>
static ks_status stencil_geometry(const Problem &P, int nchan, StArgs &a, double halo,
                                  int planes = 0) {
  using Tl = StTile<PC>;
  return stencil_geometry_of(P, Tl::TX, Tl::TY, PC, nchan, a, halo, planes);
}

// Whether a launch's operands can be described by tensor maps (row pitch and
// bases multiples of 16 bytes).
template <typename T, int Kind>
static bool stencil_tma_ok(const Problem &P, const StArgs &a) {
  const void *aux[6] = {a.X, a.MX, a.Xp, a.MXp, a.Dp, a.MDp};
  if (!P.use_tma || ((size_t)P.p * sizeof(T)) % 16 != 0 ||
      reinterpret_cast<uintptr_t>(a.A) % 16 != 0)
    return false;
  for (int i = 0; i < st_naux<T, Kind>(); ++i)
    if (!aux[i] || reinterpret_cast<uintptr_t>(aux[i]) % 16 != 0) return false;
  return sizeof(T) == 8 || (reinterpret_cast<uintptr_t>(a.out1) % 8 == 0 &&
                            reinterpret_cast<uintptr_t>(a.out2) % 8 == 0);
}

// TMA form of one launch; false (and nothing launched) when the input
// cannot be described by a tensor map (row pitch or base address not a
// multiple of 16 bytes).
// (The packed FP32 kernel also stores pairs: 8-byte aligned outputs.)
template <typename T, int PC, int Kind>
static bool stencil_launch_tma(Problem &P, const StArgs &a, int cls, double flops, double bytes,
                               ks_status *st) {
  constexpr bool kF2 = sizeof(T) == 4 && PC == 32;
  constexpr int TX = kF2 ? StF2::TX : StTile<PC>::TX, TY = kF2 ? StF2::TY : StTile<PC>::TY;
  constexpr int NAUX = st_naux<T, Kind>();
  *st = KS_OK;
  const void *aux[6] = {a.X, a.MX, a.Xp, a.MXp, a.Dp, a.MDp};
  if (!stencil_tma_ok<T, Kind>(P, a)) return false;
  StTmaArgs ta;
  ta.a = a;
  const uint64_t dims[4] = {(uint64_t)P.p, (uint64_t)P.N, (uint64_t)P.N, (uint64_t)P.N};
  const uint32_t box[4] = {(uint32_t)PC, (uint32_t)TX + 2, (uint32_t)TY + 2, 1u};
  const uint32_t nbox[4] = {(uint32_t)PC, (uint32_t)TX, (uint32_t)TY, 1u};
  if (encode_tensor_map_4d(&ta.map, a.A, (int)sizeof(T), dims, box) != KS_OK) return false;
  for (int i = 0; i < NAUX; ++i)
    if (encode_tensor_map_4d(&ta.aux[i], aux[i], (int)sizeof(T), dims, nbox) != KS_OK)
      return false;
  if constexpr (kF2) {
    {
      ProfScope ps_(P.stream, cls, flops, bytes);
      stencil_f32x2_kernel<Kind><<<a.nb, kStThreads, st_f2_smem<Kind>(), P.stream>>>(ta);
    }
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) *st = cuda_error(e, "stencil_f32x2_kernel");
    return true;
  } else {
  using Rg = StRing<T, PC, Kind>;
  {
    ProfScope ps_(P.stream, cls, flops, bytes);
    stencil_tma_kernel<T, PC, Kind><<<a.nb, kStThreads, Rg::SMEM, P.stream>>>(ta);
  }
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) *st = cuda_error(e, "stencil_tma_kernel");
  return true;
  }
}

// The rings' opt-in to their dynamic shared memory, on the current device: a
// function's limit belongs to the device, so it is set when a problem is created
// (like the other kernels') and not once per process.
template <typename T, int PC, int Kind>
static ks_status stencil_opt_in() {
  const auto at = cudaFuncAttributeMaxDynamicSharedMemorySize;
  if constexpr (sizeof(T) == 4 && PC == 32) {
    static_assert(st_f2_smem<Kind>() <= 224 * 1024, "the ring fits an SM");
    KS_CUDA_TRY(cudaFuncSetAttribute(stencil_f32x2_kernel<Kind>, at, (int)st_f2_smem<Kind>()));
  } else {
    using Rg = StRing<T, PC, Kind>;
    // the ring plus the static shared memory (mbarriers, V_eff planes,
    // reduction scratch: up to ~10 KiB) for two blocks per SM
    static_assert(Rg::SMEM + 10 * 1024 <= 113 * 1024, "two blocks of the ring fit an SM");
    // (48 KiB, static memory included, need no opt-in)
    if constexpr (Rg::SMEM + 10 * 1024 > 48 * 1024)
      KS_CUDA_TRY(cudaFuncSetAttribute(stencil_tma_kernel<T, PC, Kind>, at, (int)Rg::SMEM));
  }
  return KS_OK;
}

template <int PC>
static ks_status stencil_opt_in_pc() {
  KS_TRY((stencil_opt_in<double, PC, SK_HAM>()));
  KS_TRY((stencil_opt_in<double, PC, SK_MASS>()));
  KS_TRY((stencil_opt_in<double, PC, SK_MASS_DOT>()));
  KS_TRY((stencil_opt_in<double, PC, SK_MASS_BB>()));
  KS_TRY((stencil_opt_in<float, PC, SK_HAM>()));
  KS_TRY((stencil_opt_in<float, PC, SK_MASS>()));
  KS_TRY((stencil_opt_in<float, PC, SK_MASS_DOT>()));
  KS_TRY((stencil_opt_in<float, PC, SK_MASS_BB>()));
  return stencil_opt_in<float, PC, SK_HAM_INC>();
}

// (of the orbital chunk that stencil_launch takes for p)
ks_status configure_stencil_kernels(int p) {
  if (p >= 32) return stencil_opt_in_pc<32>();
  if (p >= 16) return stencil_opt_in_pc<16>();
  if (p >= 8) return stencil_opt_in_pc<8>();
  return p == 1 ? KS_OK : stencil_opt_in_pc<4>();
}

template <typename T, int PC, int Kind>
static ks_status stencil_launch_pc(Problem &P, StArgs &a, int nchan, double flops, double bytes) {
  // FP64: a halo plane costs its in-plane sums, over half of a plane's
  // instructions, two of them 1.2 planes.  FP32 reads it from L2 and is
  // bound by memory, where more and shorter segments overlap better
  constexpr bool kF2 = sizeof(T) == 4 && PC == 32;
  const bool f2 = kF2 && stencil_tma_ok<T, Kind>(P, a);
  if (f2) KS_TRY(stencil_geometry_of(P, StF2::TX, StF2::TY, StF2::PC, nchan, a, 0.0, 0));
  else KS_TRY(stencil_geometry<PC>(P, nchan, a, sizeof(T) == 8 ? 1.2 : 0.0));
  a.c = q1_coefficients(P.h);
  a.k0r = a.c.k0 / a.c.ke;
  if (P.mass == KS_MASS_LUMPED) {      // row sums of M: h^3 on the centre
    a.c.m0 = P.h * P.h * P.h;
    a.c.mf = a.c.me = a.c.mc = 0.0;
  }
  const double cd[9] = {a.c.k0, a.c.ke, a.c.kc, a.c.m0, a.c.mf, a.c.me, a.c.mc, a.kfac,
                        2.0 * a.occ * a.h3};
  for (int i = 0; i < 9; ++i) a.cf[i] = (float)cd[i];
  a.part = P.partials;
  a.counter = P.red_counter;
  a.status = P.dstatus;
  const int cls = (Kind == SK_HAM || Kind == SK_HAM_INC) ? KP_HAMILTONIAN : KP_MASS;
  ks_status st;
  // one amplitude (PC = 1, p = 1) has an 8-byte row pitch, which no tensor
  // map can describe: plain staging only
  if constexpr (PC >= 4) {
    if (stencil_launch_tma<T, PC, Kind>(P, a, cls, flops, bytes, &st)) return st;
    // plain staging has its own tiles
    if (f2) KS_TRY(stencil_geometry<PC>(P, nchan, a, 0.0));
  }
  {
    ProfScope ps_(P.stream, cls, flops, bytes);
    stencil_kernel<T, PC, Kind><<<a.nb, kStThreads, 0, P.stream>>>(a);
  }
  KS_CUDA_TRY(cudaGetLastError());
  return KS_OK;
}

template <typename T, int Kind>
static ks_status stencil_launch(Problem &P, StArgs &a, int nchan, double flops, double bytes) {
  if (P.p >= 32) return stencil_launch_pc<T, 32, Kind>(P, a, nchan, flops, bytes);
  if (P.p >= 16) return stencil_launch_pc<T, 16, Kind>(P, a, nchan, flops, bytes);
  if (P.p >= 8) return stencil_launch_pc<T, 8, Kind>(P, a, nchan, flops, bytes);
  if (P.p == 1) return stencil_launch_pc<T, 1, Kind>(P, a, nchan, flops, bytes);
  return stencil_launch_pc<T, 4, Kind>(P, a, nchan, flops, bytes);
}

template <typename T>
ks_status launch_hamiltonian(Problem &P, const T *X, const double *veff, T *EX, T *MX,
                             double *ekin_out) {
  StArgs a{};
  a.occ = P.occ;
  a.kfac = P.occ * P.kin_w;
  a.h3 = P.h * P.h * P.h;
  a.A = X;
  a.out1 = EX;
  a.out2 = MX;
  a.veff = veff;
  a.red_out = ekin_out;
  a.red_scale = 0.5 * a.kfac;
  const double total = (double)P.n * P.p;
  return stencil_launch<T, SK_HAM>(P, a, 1, 27.0 * total,
                                   total * sizeof(T) * (1 + (EX ? 1 : 0) + (MX ? 1 : 0)) + 8.0 * P.n);
}

ks_status launch_hamiltonian_inc(Problem &P, const float *d, const double *veff,
                                 const double *veff_b, const float *xb, const float *eb,
                                 float *e, float *Md, double *dkin_out) {
  StArgs a{};
  a.occ = P.occ;
  a.kfac = P.occ * P.kin_w;
  a.h3 = P.h * P.h * P.h;
  a.A = d;
  a.out1 = e;
  a.out2 = Md;
  a.veff = veff;
  a.veff_b = veff_b;
  a.X = xb;
  a.MX = eb;
  a.red_out = dkin_out;
  a.red_scale = 0.5;
  const double total = (double)P.n * P.p;
  return stencil_launch<float, SK_HAM_INC>(P, a, 1, 33.0 * total,
                                           total * sizeof(float) * (Md ? 5 : 4) + 8.0 * P.n);
}

template <typename T>
ks_status launch_mass(Problem &P, const T *X, T *MX) {
  StArgs a{};
  a.A = X;
  a.out1 = MX;
  const double total = (double)P.n * P.p;
  return stencil_launch<T, SK_MASS>(P, a, 0, 21.0 * total, 2.0 * total * sizeof(T));
}

template <typename T>
ks_status launch_mass_dots(Problem &P, const T *D, T *MD, const T *X, const T *MX,
                           const BBPrevT<T> *prev, double *out4) {
  StArgs a{};
  a.A = D;
  a.out1 = MD;
  a.red_out = out4;
  a.red_scale = 1.0;
  const double total = (double)P.n * P.p;
  if (prev) {
    a.X = X;
    a.MX = MX;
    a.Xp = prev->X;
    a.MXp = prev->MX;
    a.Dp = prev->D;
    a.MDp = prev->MD;
    return stencil_launch<T, SK_MASS_BB>(P, a, 4, 31.0 * total, 8.0 * total * sizeof(T));
  }
  return stencil_launch<T, SK_MASS_DOT>(P, a, 1, 23.0 * total,
                                        (MD ? 2.0 : 1.0) * total * sizeof(T));
}

// ---------------------------------------------------------------- batched
// Slots of one batched stencil launch (BJob::blk indices, -1 = none).
struct StSlots {
  int a, o1, o2, x, mx, xp, mxp, dp, mdp;
};

template <typename T, int PC, int Kind>
__global__ void __launch_bounds__(kStThreads, (st_min_blocks<T, Kind>())) stencil_batch_kernel(
    const BJob *__restrict__ jobs, const int *__restrict__ start, int J,
    const unsigned char *__restrict__ active, StSlots sl) {
  const int j = batch_job_of(start, J, blockIdx.x);
  if (!active[j]) return;
  const BJob &b = jobs[j];
  StArgs a;
  a.N = b.N;
  a.p = b.p;
  a.zseg = b.st_zseg;
  a.tiles_x = b.st_tiles_x;
  a.tiles_y = b.st_tiles_y;
  a.chunks = b.st_chunks;
  a.c.k0 = b.qc[0]; a.c.kf = b.qc[1]; a.c.ke = b.qc[2]; a.c.kc = b.qc[3];
  a.c.m0 = b.qc[4]; a.c.mf = b.qc[5]; a.c.me = b.qc[6]; a.c.mc = b.qc[7];
#pragma unroll
  for (int i = 0; i < 9; ++i) a.cf[i] = b.qcf[i];
  a.k0r = a.c.k0 / a.c.ke;
  a.occ = b.occ;
  a.kfac = b.occ;
  a.h3 = b.h3;
  a.A = b.blk[sl.a];
  a.out1 = b.blk[sl.o1];
  a.out2 = sl.o2 >= 0 ? b.blk[sl.o2] : nullptr;
  a.veff = b.veff;
  if (Kind == SK_MASS_BB) {
    a.X = b.blk[sl.x];
    a.MX = b.blk[sl.mx];
    a.Xp = b.blk[sl.xp];
    a.MXp = b.blk[sl.mxp];
    a.Dp = b.blk[sl.dp];
    a.MDp = b.blk[sl.mdp];
  }
  a.part = b.partials;
  a.nb = b.st_nb;
  a.red_out = b.scal + (Kind == SK_HAM ? SC_EKIN : SC_DNORM2);
  a.red_scale = Kind == SK_HAM ? 0.5 * b.occ : 1.0;
  a.counter = b.red_counter;
  a.status = b.status;
  stencil_plain_body<T, PC, Kind>(a, blockIdx.x - start[j]);
}

template <typename T, int Kind>
static ks_status stencil_batch_launch(Batch &B, const StSlots &sl) {
  const int maps[4] = {BM_ST4, BM_ST8, BM_ST16, BM_ST32};
  const int cls = Kind == SK_HAM ? KP_HAMILTONIAN : KP_MASS;
  for (int c = 0; c < 4; ++c) {
    const int nb = B.total(maps[c]);
    if (nb == 0) continue;
    {
      ProfScope ps_(B.stream, cls);
      const int *st = B.map(maps[c]);
      if (c == 0) stencil_batch_kernel<T, 4, Kind><<<nb, kStThreads, 0, B.stream>>>(B.jobs_dev, st, B.J, B.active_dev, sl);
      else if (c == 1) stencil_batch_kernel<T, 8, Kind><<<nb, kStThreads, 0, B.stream>>>(B.jobs_dev, st, B.J, B.active_dev, sl);
      else if (c == 2) stencil_batch_kernel<T, 16, Kind><<<nb, kStThreads, 0, B.stream>>>(B.jobs_dev, st, B.J, B.active_dev, sl);
      else stencil_batch_kernel<T, 32, Kind><<<nb, kStThreads, 0, B.stream>>>(B.jobs_dev, st, B.J, B.active_dev, sl);
    }
    KS_CUDA_TRY(cudaGetLastError());
  }
  return KS_OK;
}

template <typename T>
ks_status batch_hamiltonian(Batch &B, int sX, int sEX, int sMX) {
  const StSlots sl{sX, sEX, sMX, -1, -1, -1, -1, -1, -1};
  return stencil_batch_launch<T, SK_HAM>(B, sl);
}

template <typename T>
ks_status batch_mass(Batch &B, int sX, int sMX) {
  const StSlots sl{sX, sMX, -1, -1, -1, -1, -1, -1, -1};
  return stencil_batch_launch<T, SK_MASS>(B, sl);
}

template <typename T>
ks_status batch_mass_dots(Batch &B, int sD, int sMD, int sX, int sMX, int sXp, int sMXp, int sDp,
                          int sMDp) {
  const StSlots sl{sD, sMD, -1, sX, sMX, sXp, sMXp, sDp, sMDp};
  if (sXp >= 0) return stencil_batch_launch<T, SK_MASS_BB>(B, sl);
  return stencil_batch_launch<T, SK_MASS_DOT>(B, sl);
}

// Per job: PC class of its p and the block geometry of that class (room for
// four reduction channels in its partials).
ks_status batch_stencil_geometry(Batch &B) {
  const int planes = B.tune.st_planes;
  for (int j = 0; j < B.J; ++j) {
    Problem &P = B.probs[j]->P;
    BJob &b = B.jobs_host[j];
    StArgs a{};
    if (P.p >= 32) KS_TRY(stencil_geometry<32>(P, 4, a, 0.0, planes));
    else if (P.p >= 16) KS_TRY(stencil_geometry<16>(P, 4, a, 0.0, planes));
    else if (P.p >= 8) KS_TRY(stencil_geometry<8>(P, 4, a, 0.0, planes));
    else KS_TRY(stencil_geometry<4>(P, 4, a, 0.0, planes));
    b.st_zseg = a.zseg;
    b.st_tiles_x = a.tiles_x;
    b.st_tiles_y = a.tiles_y;
    b.st_chunks = a.chunks;
    b.st_nb = a.nb;
  }
  return KS_OK;
}

#define KS_BINST(T)                                                                        \
  template ks_status batch_hamiltonian<T>(Batch &, int, int, int);                         \
  template ks_status batch_mass<T>(Batch &, int, int);                                     \
  template ks_status batch_mass_dots<T>(Batch &, int, int, int, int, int, int, int, int);
KS_BINST(double)
KS_BINST(float)
#undef KS_BINST

#define KS_INST(T)                                                                        \
  template ks_status launch_hamiltonian<T>(Problem &, const T *, const double *, T *, T *, \
                                           double *);                                    \
  template ks_status launch_mass<T>(Problem &, const T *, T *);                          \
  template ks_status launch_mass_dots<T>(Problem &, const T *, T *, const T *, const T *, \
                                         const BBPrevT<T> *, double *);
KS_INST(double)
KS_INST(float)
#undef KS_INST

KS_OOB_READER(stencil)

}  // namespace ks
