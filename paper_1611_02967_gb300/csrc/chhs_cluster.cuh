// chhs_cluster.cuh -- the coarse levels of a double-precision V-cycle in one
// launch: a cluster of up to 16 blocks holds them in (distributed) shared
// memory.
//
// On a level of 64 x 64 cells or less a colour pass is bound by latency: one
// warp's chain of FP64 instructions (~64 cycles each) plus, as a launch of
// its own, ~1.3 us of launch and drain.  Here every block of the cluster
// owns a slab of rows of each level, the passes exchange the
// slabs' edge rows through distributed shared memory, and a cluster barrier
// (~570 cycles measured at 512 threads) takes the launch's place.
//
// Slabs: level l gives every block R_l = 2 ceil(rows / (2 blocks)) rows, an
// even number starting at an even row, so that the four children of a coarse
// cell lie in one block; small levels leave blocks idle.  A block keeps one
// halo row below and above its slab; a pass stores the updated cells of its
// first and last row into the neighbours' halos as well, so all stencil reads
// are local.  Cells of one colour only read the other colour, so a pass never
// writes a halo cell that the neighbour reads in the same pass.
// The levels from `tail` on (at most chhs_tuning.tail_cells cells: a warp or
// less per colour, where the cluster barrier costs more than the work) are
// held by block 0 whole and run there as in k_tail, the others waiting at the
// barrier.
//
// Measured (GB300, default tuning, both sides in turn): with a launch per pass
// against the cluster with one update per launch-like pass, a 64 x 64 step of
// 6.6 V-cycles, all of it in the cluster, 840 -> 734 us, and a 512 x 512 step,
// where the levels 64 x 64 ... 16 x 16 move here, 2.53 -> 2.48 ms; that against
// the cells of a level in registers (cluster_passes), the outer-flux restriction
// and the asynchronous copies 700 -> 655 us and 2.34 -> 2.29 ms.
#pragma once
#include <cooperative_groups.h>

#include "chhs_kernels.cuh"

namespace chhs_dev {

constexpr int kClusterMax = 16;

// Levels of at most this many cells run in the cluster (shared memory for a
// block's share of 64 x 64, 32 x 32, ... is ~115 KB).
constexpr int kClusterCells = 4096;

struct ClusterPlan {
  int blocks;  // blocks of the cluster
  int tail;    // first level held by block 0 alone (of n)
  int rows[kTailMaxLevels];  // slab rows R_l of each block on level l
};

// Slab rows of a level of nr rows over `blocks` blocks.
__host__ __device__ inline int cluster_rows(int nr, int blocks) { return 2 * ((nr + 2 * blocks - 1) / (2 * blocks)); }

// Cells of a level's arrays in shared memory: the slab and its two halo rows.
__host__ __device__ inline size_t cluster_cells(int rows, int row_cells) { return (size_t)(rows + 2) * row_cells; }

__host__ __device__ inline size_t cluster_smem_bytes(const Tail<double>& tl, const ClusterPlan& P) {
  size_t b = 0;
  for (int l = 0; l < tl.n; ++l)
    b += tail_fields<2, false>() *
         tail_align(sizeof(double) * cluster_cells(P.rows[l], tl.lev[l].nx));
  return b;
}

// What a block needs to know of a level, formed once into shared memory: read
// through the kernel's parameters with a level index that is not known at
// compile time, every visit of a level cost ~1 700 cycles of constant-cache
// misses.
struct SlabInfo {
  double ih2, h2, sih2, e34ih2;
  float rnx, rny, rhw;
  int nx, ny, nz, ncell;
  int off, st;        // bytes: the level's arrays in shared memory, one array
  int S, R, r0, nr, NR;
};

// One block's slab of a level: the Level with its arrays in shared memory,
// indexed from the slab's first row (halo rows at row -1 and row nr).
struct Slab {
  Level<double> L;
  int S;   // cells per row
  int R;   // rows per block
  int r0;  // first row of this block
  int nr;  // rows of this block (0 when idle)
  int NR;  // rows of the level
};

__device__ __forceinline__ SlabInfo cluster_info(const Tail<double>& tl, const ClusterPlan& P, int l, int rank) {
  size_t off = 0;
  for (int q = 0; q < l; ++q)
    off += tail_fields<2, false>() *
           tail_align(sizeof(double) * cluster_cells(P.rows[q], tl.lev[q].nx));
  const Level<double>& G = tl.lev[l];
  SlabInfo B;
  B.ih2 = G.ih2;
  B.h2 = G.h2;
  B.sih2 = G.sih2;
  B.e34ih2 = G.e34ih2;
  B.rnx = G.rnx;
  B.rny = G.rny;
  B.rhw = G.rhw;
  B.nx = G.nx;
  B.ny = G.ny;
  B.nz = G.nz;
  B.ncell = G.ncell;
  B.S = G.nx;
  B.R = P.rows[l];
  B.NR = G.ny;
  B.r0 = rank * B.R;
  B.nr = max(0, min(B.R, B.NR - B.r0));
  B.off = (int)off;
  B.st = (int)tail_align(sizeof(double) * cluster_cells(B.R, B.S));
  return B;
}

__device__ __forceinline__ Slab cluster_slab(const SlabInfo& I, unsigned char* smem) {
  Slab B;
  B.S = I.S;
  B.R = I.R;
  B.r0 = I.r0;
  B.nr = I.nr;
  B.NR = I.NR;
  Level<double>& L = B.L;
  L.nx = I.nx;
  L.ny = I.ny;
  L.nz = I.nz;
  L.ncell = I.ncell;
  L.rnx = I.rnx;
  L.rny = I.rny;
  L.rhw = I.rhw;
  L.ih2 = I.ih2;
  L.h2 = I.h2;
  L.sih2 = I.sih2;
  L.e34ih2 = I.e34ih2;
  int q = 0;
  auto carve = [&]() { return reinterpret_cast<double*>(smem + I.off + (q++) * I.st) + I.S; };
  L.phi = carve(); L.mu = carve(); L.p = carve();
  L.fphi = carve(); L.fmu = carve(); L.fp = carve();
  L.phim = carve(); L.phi0 = carve(); L.mu0 = carve(); L.p0 = carve();
  L.ax = carve(); L.ay = carve(); L.Mx = carve(); L.My = carve();
  L.sM = carve(); L.sa = carve();
  L.cAe = carve(); L.cC = carve(); L.cGn = carve(); L.cHn = carve(); L.cQ = carve(); L.cH = carve();
  L.phis = nullptr;
  level_constants(L);
  return B;
}

__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// The address of this block's shared-memory location x in block `rank`.
__device__ __forceinline__ double* remote(double* x, int rank) {
  return static_cast<double*>(cooperative_groups::this_cluster().map_shared_rank(x, rank));
}

// Stores v into array a at row r (level rows) and cell s of it: in the slab
// of the row's owner and in the halos of the blocks beside it.
__device__ __forceinline__ void cluster_put(const Slab& B, double* a, int r, int s, double v, bool halos) {
  const int o = r / B.R, lr = r - o * B.R;
  remote(a, o)[s + B.S * lr] = v;
  if (!halos) return;
  if (lr == 0 && o > 0) remote(a, o - 1)[s + B.S * B.R] = v;
  if (lr == B.R - 1 && r + 1 < B.NR) remote(a, o + 1)[s - B.S] = v;
}

// One colour pass of a slab with more cells of a colour than cluster_passes
// holds (the split update of k_smooth_split), its edge rows stored to the
// neighbours too; ends with the cluster barrier.
__device__ __forceinline__ void cluster_smooth(const Slab& B, const Coefs<double>& K, int rank, int colour, bool rhs) {
  __shared__ float xch[2][kTailGroups][4 * 32];
  const Level<double>& L = B.L;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = warp / 3, role = warp - 3 * g;
  const int hw = (L.nx + 1) >> 1;
  const int total = hw * B.nr;
  if (g < kTailGroups) {
    const int rounds = (total + 32 * kTailGroups - 1) / (32 * kTailGroups);
    for (int q = 0; q < rounds; ++q) {
      const int t = q * 32 * kTailGroups + g * 32 + lane;
      const int row = small_div(t, L.rhw);
      const int ti = t - row * hw, j = B.r0 + row, i = 2 * ti + ((j + colour) & 1);
      const bool act = t < total && i < L.nx;
      const int c = act ? i + B.S * row : 0;
      cell_update_split<2>(L, K, role, act, c, i, j, 0, rhs, &xch[q & 1][g][lane], [g] {
        asm volatile("bar.sync %0, 96;" ::"r"(g + 1) : "memory");
      });
      if (act && role == 0) {
        if (row == 0 && B.r0 > 0) {
          const int h = i + B.S * B.R;
          remote(L.phi, rank - 1)[h] = L.phi[c];
          remote(L.mu, rank - 1)[h] = L.mu[c];
          remote(L.p, rank - 1)[h] = L.p[c];
        }
        if (row == B.R - 1 && B.r0 + B.R < B.NR) {
          const int h = i - B.S;
          remote(L.phi, rank + 1)[h] = L.phi[c];
          remote(L.mu, rank + 1)[h] = L.mu[c];
          remote(L.p, rank + 1)[h] = L.p[c];
        }
      }
    }
  }
  cluster_barrier();
}

// f += N(R u) on the slab (no pre-smoothing sweep to carry it): the three
// rows on the three warps of a group, as tail_rhs.
__device__ __forceinline__ void cluster_rhs(const Slab& B, const Coefs<double>& K) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = warp / 3, role = warp - 3 * g;
  if (g < kTailGroups)
    for (int t = g * 32 + lane; t < B.S * B.nr; t += 32 * kTailGroups) {
      const int row = small_div(t, B.L.rnx), i = t - row * B.L.nx;
      double u;
      f_row(B.L, role)[t] += n_row<2>(B.L, K, role, B.L.phi0, B.L.mu0, B.L.p0, t, i, B.r0 + row, 0, u);
    }
  __syncthreads();
}

// A cell of a colour as one of the three warps of its group holds it through
// the passes of a level: place, neighbours (the cell itself on a missing face),
// its row's coefficients (zero on missing faces), right-hand side and constants.
struct SplitCell {
  bool act, down, up;  // an active cell; in the slab's first (last) row with a neighbour block
  int c, s;            // index in the slab, cell within its row
  unsigned in;         // interior faces
  int e[4];
  double a[4], M[4];   // a: roles 0 and 1, M: role 0
  double f, s0, s1;    // role 0: sM, sa; 1: sa, n_c; 2: Q, H
  float ae, cC, cGn, cHn;
};

__device__ __forceinline__ void split_cell(SplitCell& x, const Slab& B, int g, int lane, int role, int colour) {
  const Level<double>& L = B.L;
  const int hw = (L.nx + 1) >> 1;
  const int t = g * 32 + lane;
  const int row = small_div(t, L.rhw);
  const int ti = t - row * hw, j = B.r0 + row, i = 2 * ti + ((j + colour) & 1);
  x.act = g < kTailGroups && t < hw * B.nr && i < L.nx;
  x.s = x.act ? i : 0;
  x.c = x.act ? i + B.S * row : 0;
  x.down = x.act && row == 0 && B.r0 > 0;
  x.up = x.act && row == B.R - 1 && B.r0 + B.R < B.NR;
  if (!x.act) return;
  const bool in[4] = {i > 0, i + 1 < L.nx, j > 0, j + 1 < L.ny};
  const int de[4] = {-1, 1, -L.nx, L.nx};
  x.in = 0u;
  int m = 0;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    x.e[q] = in[q] ? x.c + de[q] : x.c;
    const int fe = in[q] ? ((q & 1) ? x.c : x.c + de[q]) : x.c;  // the lower of the two cells holds the face
    const double* af = q < 2 ? L.ax : L.ay;
    const double* Mf = q < 2 ? L.Mx : L.My;
    x.a[q] = in[q] && role < 2 ? af[fe] : 0.0;
    x.M[q] = in[q] && role == 0 ? Mf[fe] : 0.0;
    x.in |= in[q] ? 1u << q : 0u;
    m += in[q] ? 1 : 0;
  }
  x.f = f_row(L, role)[x.c];
  x.s0 = role == 0 ? L.sM[x.c] : role == 1 ? L.sa[x.c] : L.cQ[x.c];
  x.s1 = role == 0 ? L.sa[x.c] : role == 1 ? count_value<double>(m) : L.cH[x.c];
  x.ae = L.kAe[x.c];
  x.cC = L.kC[x.c];
  x.cGn = L.kGn[x.c];
  x.cHn = L.kHn[x.c];
}

// The sums over the cell's faces that its row needs, on the fields (phi, mu, p):
// role 0 sum (M mu_e + a p_e), role 1 sum a mu_e and sum p_e, role 2 sum phi_e.
__device__ __forceinline__ void split_sums(const SplitCell& x, int role, const double* phi, const double* mu,
                                           const double* p, double& A, double& P) {
  A = -0.0;
  P = -0.0;
  if (role == 0) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      A += x.M[q] * mu[x.e[q]];
      A += x.a[q] * p[x.e[q]];
    }
  } else if (role == 1) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const double pe = p[x.e[q]];
      A += x.a[q] * mu[x.e[q]];
      P += (x.in >> q) & 1u ? pe : -0.0;
    }
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const double ph = phi[x.e[q]];
      P += (x.in >> q) & 1u ? ph : -0.0;
    }
  }
}

// npass (even) colour passes of the slab, at most 32 cells of a colour per
// group: as cell_update_split, with the cells of both colours held in
// registers through all passes and each warp finishing its own unknown (warp 0
// phi, 1 p, 2 mu).  rhs: complete the right-hand side in the first two.
// local: the level is this block's alone.
template <bool LOCAL>
__device__ __forceinline__ void cluster_passes(const Slab& B, const Coefs<double>& K, int rank, int npass, bool rhs) {
  __shared__ float xch[kTailGroups + 1][5 * 32];
  const Level<double>& L = B.L;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = warp / 3, role = warp - 3 * g;
  float* const x = &xch[g][lane];
  SplitCell cells[2];
  split_cell(cells[0], B, g, lane, role, 0);
  split_cell(cells[1], B, g, lane, role, 1);
  double* const own = role == 0 ? L.phi : role == 1 ? L.p : L.mu;
  double* const fr = f_row(L, role);
  const int hw = (L.nx + 1) >> 1;
  const bool busy = g < kTailGroups && g * 32 < hw * B.nr;  // the whole group alike
  for (int k = 0; k < npass; k += 2)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      SplitCell& z = cells[h];
      double u = 0.0;
      if (busy) {
        if (z.act) {
          double A, P;
          if (rhs && k == 0) {
            split_sums(z, role, L.phi0, L.mu0, L.p0, A, P);
            if (role == 0)
              z.f += L.phi0[z.c] - L.sih2 * ((A - z.s0 * L.mu0[z.c]) - z.s1 * L.p0[z.c]);
            else if (role == 1)
              z.f += -L.ih2 * ((P - z.s1 * L.p0[z.c]) + K.gamma * (A - z.s0 * L.mu0[z.c]));
            else
              z.f += (L.mu0[z.c] + L.e34ih2 * P) - cubic_P(L.phi0[z.c], z.s1, z.s0);
            fr[z.c] = z.f;
          }
          split_sums(z, role, L.phi, L.mu, L.p, A, P);
          u = own[z.c];
          if (role == 0) {
            const double R1 = (z.f - u) + L.sih2 * ((A - z.s0 * L.mu[z.c]) - z.s1 * L.p[z.c]);
            x[128] = f64_to_f32_rz(R1);
          } else if (role == 1) {
            const double R3 = z.f + L.ih2 * ((P - z.s1 * u) + K.gamma * (A - z.s0 * L.mu[z.c]));
            x[0] = z.cHn * f64_to_f32_rz(R3);
          } else {
            const double v = L.phi[z.c], t = 0.25 * v + z.s1, t2 = t * v + z.s0;
            const double R2 = ((z.f - u) - L.e34ih2 * P) + t2 * v;
            const float vf = f64_to_f32_rz(v), Bn = (0.25f * vf + f64_to_f32_rz(t)) * vf + f64_to_f32_rz(t2);
            x[32] = f64_to_f32_rz(R2);
            x[64] = Bn;
            x[96] = rcp_approx(1.f + z.ae * Bn);
          }
        }
        asm volatile("bar.sync %0, 96;" ::"r"(g + 1) : "memory");
        if (z.act) {
          const float R3n = x[0], R2 = x[32], Bn = x[64], rd = x[96], R1 = x[128];
          const float dphi = ((R1 - z.ae * R2) - z.cC * R3n) * rd;
          const float dmu = R2 + Bn * dphi;
          const float dp = R3n - z.cGn * dmu;
          u += f32_to_f64_exact(role == 0 ? dphi : role == 1 ? dp : dmu);
          own[z.c] = u;
          if (!LOCAL) {
            if (z.down) remote(own, rank - 1)[z.s + B.S * B.R] = u;
            if (z.up) remote(own, rank + 1)[z.s - B.S] = u;
          }
        }
      }
      if (LOCAL) __syncthreads();
      else cluster_barrier();
    }
}

// Whether cluster_passes can hold the slab's cells (every block alike).
__device__ __forceinline__ bool cluster_holds(const Slab& B) {
  return ((B.L.nx + 1) >> 1) * (B.R < B.NR ? B.R : B.NR) <= 32 * kTailGroups;
}

// Residual and restriction of the slab: a coarse cell per lane, its three rows
// on the three warps of a group, only the fluxes of the faces around its
// children (k_residual_restrict64).  Each coarse value goes to its owner's slab
// and to the halos that hold its row.
__device__ __forceinline__ void cluster_restrict(const Slab& F, const Slab& C, const Coefs<double>& K) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = warp / 3, role = warp - 3 * g;
  const Level<double>& L = F.L;
  const int total = C.S * (F.nr >> 1), nx = L.nx;
  if (g < kTailGroups)
    for (int t = g * 32 + lane; t < total; t += 32 * kTailGroups) {
      const int jl = small_div(t, C.L.rnx), I = t - jl * C.L.nx;
      const int c0 = 2 * I + nx * 2 * jl, c1 = c0 + nx;  // the children's rows in the slab
      const int j = F.r0 + 2 * jl;
      // the outer faces: cell, neighbour, face index (the lower cell's), direction
      const bool xm = I > 0, xp = 2 * I + 2 < nx, ym = j > 0, yp = j + 2 < L.ny;
      auto faces = [&](auto fn) {
        fn(xm, c0, c0 - 1, c0 - 1, 0);
        fn(xp, c0 + 1, c0 + 2, c0 + 1, 0);
        fn(xm, c1, c1 - 1, c1 - 1, 0);
        fn(xp, c1 + 1, c1 + 2, c1 + 1, 0);
        fn(ym, c0, c0 - nx, c0 - nx, 1);
        fn(ym, c0 + 1, c0 - nx + 1, c0 - nx + 1, 1);
        fn(yp, c1, c1 + nx, c1, 1);
        fn(yp, c1 + 1, c1 + nx + 1, c1 + 1, 1);
      };
      auto sum4 = [&](const double* a) { return (a[c0] + a[c0 + 1]) + (a[c1] + a[c1 + 1]); };
      const double fs = sum4(f_row(L, role));
      double r, u;
      if (role == 0) {
        double v = 0.0;
        faces([&](bool in, int c, int e, int fe, int d) {
          const int es = in ? e : c, fs_ = in ? fe : c;
          const double a = in ? (d ? L.ay : L.ax)[fs_] : 0.0, M = in ? (d ? L.My : L.Mx)[fs_] : 0.0;
          v = ::fma(M, L.mu[es] - L.mu[c], v);
          v = ::fma(a, L.p[es] - L.p[c], v);
        });
        u = sum4(L.phi);
        r = ::fma(L.sih2, v, fs - u);
      } else if (role == 1) {
        double aw = 0.0, w = 0.0;
        faces([&](bool in, int c, int e, int fe, int d) {
          const int es = in ? e : c, fs_ = in ? fe : c;
          const double a = in ? (d ? L.ay : L.ax)[fs_] : 0.0;
          aw = ::fma(a, L.mu[es] - L.mu[c], aw);
          w += L.p[es] - L.p[c];
        });
        u = sum4(L.p);
        r = ::fma(L.ih2, ::fma(K.gamma, aw, w), fs);
      } else {
        double sd = 0.0, s2 = fs;
        faces([&](bool in, int c, int e, int, int) {
          const double ph = L.phi[in ? e : c];
          sd += in ? ph : -0.0;
        });
        auto cubic = [&](int c) {
          const double v = L.phi[c];
          s2 = ::fma(::fma(::fma(0.25, v, L.cH[c]), v, L.cQ[c]), v, s2);
        };
        cubic(c0);
        cubic(c0 + 1);
        cubic(c1);
        cubic(c1 + 1);
        u = sum4(L.mu);
        r = ::fma(-L.e34ih2, ::fma(2.0, sum4(L.phi), sd), s2 - u);
      }
      const int row = (F.r0 >> 1) + jl;
      cluster_put(C, f_row(C.L, role), row, I, 0.25 * r, false);
      cluster_put(C, role == 0 ? C.L.phi : role == 1 ? C.L.p : C.L.mu, row, I, 0.25 * u, true);
      cluster_put(C, role == 0 ? C.L.phi0 : role == 1 ? C.L.p0 : C.L.mu0, row, I, 0.25 * u, true);
    }
}

// u += P(u_c - u_c^0) on the slab and its halo rows (whose owners do the
// same), the coarse values read from their owners.  Ends with the cluster
// barrier: the next pass stores into the neighbours' halos.
__device__ __forceinline__ void cluster_prolong(const Slab& F, const Slab& C) {
  if (F.nr > 0) {
    const int lo = F.r0 > 0 ? -1 : 0, hi = F.r0 + F.nr < F.NR ? F.nr + 1 : F.nr;
    const int total = F.S * (hi - lo);
    for (int t = threadIdx.x; t < total; t += blockDim.x) {
      const int x = small_div(t, F.L.rnx), i = t - x * F.L.nx;
      const int r = F.r0 + lo + x;
      const int o = (r >> 1) / C.R, q = (i >> 1) + C.S * ((r >> 1) - o * C.R);
      const int c = t + F.S * lo;
      F.L.phi[c] += remote(C.L.phi, o)[q] - remote(C.L.phi0, o)[q];
      F.L.mu[c] += remote(C.L.mu, o)[q] - remote(C.L.mu0, o)[q];
      F.L.p[c] += remote(C.L.p, o)[q] - remote(C.L.p0, o)[q];
    }
  }
  cluster_barrier();
}

// Asynchronous copies of one array element from global to shared memory.
__device__ __forceinline__ void copy_async(double* dst, const double* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src));
}
__device__ __forceinline__ void copy_async(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src));
}

// nu_top: sweeps of the top level (the finest level's counts when the whole
// hierarchy is in the cluster), tl.nu1 / tl.nu2 those of the levels below.
static __global__ void __launch_bounds__(kTailThreads, 1) k_cluster(const __grid_constant__ Tail<double> tl,
                                                                   const __grid_constant__ ClusterPlan P,
                                                                   Coefs<double> K, int nu1_top, int nu2_top) {
  extern __shared__ __align__(16) unsigned char cl_smem[];
  __shared__ SlabInfo info[kTailMaxLevels];
  pdl_enter();
  const int rank = (int)cooperative_groups::this_cluster().block_rank();
  const int n = tl.n;
  if ((int)threadIdx.x < n) info[threadIdx.x] = cluster_info(tl, P, threadIdx.x, rank);
  __syncthreads();
  auto slab = [&](int l) { return cluster_slab(info[l], cl_smem); };
  // copy in: the coefficients of every level and the top level's fields, all in
  // flight together
  for (int l = 0; l < n; ++l) {
    const Slab B = slab(l);
    if (B.nr == 0) continue;
    const Level<double>& G = tl.lev[l];
    const Level<double>& S = B.L;
    const int base = B.S * B.r0;
    for (int t = threadIdx.x; t < B.S * B.nr; t += blockDim.x) {
      const int c = base + t;
      copy_async(S.ax + t, G.ax + c);
      copy_async(S.ay + t, G.ay + c);
      copy_async(S.Mx + t, G.Mx + c);
      copy_async(S.My + t, G.My + c);
      copy_async(S.sM + t, G.sM + c);
      copy_async(S.sa + t, G.sa + c);
      copy_async(S.cQ + t, G.cQ + c);
      copy_async(S.cH + t, G.cH + c);
      copy_async(S.kAe + t, G.kAe + c);
      copy_async(S.kC + t, G.kC + c);
      copy_async(S.kGn + t, G.kGn + c);
      copy_async(S.kHn + t, G.kHn + c);
      if (l == 0) {
        copy_async(S.fphi + t, G.fphi + c);
        copy_async(S.fmu + t, G.fmu + c);
        copy_async(S.fp + t, G.fp + c);
      }
    }
    // the halo below: its +y face coefficients belong to this slab's first row
    if (B.r0 > 0)
      for (int t = threadIdx.x; t < B.S; t += blockDim.x) {
        copy_async(S.ay + t - B.S, G.ay + base - B.S + t);
        copy_async(S.My + t - B.S, G.My + base - B.S + t);
      }
    if (l == 0) {  // the top level's state, halos included
      const int lo = B.r0 > 0 ? -B.S : 0, hi = B.S * (B.r0 + B.nr < B.NR ? B.nr + 1 : B.nr);
      for (int t = lo + (int)threadIdx.x; t < hi; t += blockDim.x) {
        const int c = base + t;
        copy_async(S.phi + t, G.phi + c);
        copy_async(S.mu + t, G.mu + c);
        copy_async(S.p + t, G.p + c);
        if (tl.top_rhs) {
          copy_async(S.phi0 + t, G.phi0 + c);
          copy_async(S.mu0 + t, G.mu0 + c);
          copy_async(S.p0 + t, G.p0 + c);
        }
      }
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  cluster_barrier();

  for (int l = 0; l < P.tail; ++l) {
    const Slab B = slab(l);
    bool rhs = l > 0 || tl.top_rhs;
    const int nu1 = l == 0 ? nu1_top : tl.nu1;
    if (rhs && nu1 == 0) {
      cluster_rhs(B, K);
      rhs = false;
    }
    if (cluster_holds(B)) {
      cluster_passes<false>(B, K, rank, 2 * nu1, rhs);
    } else {
      for (int it = 0; it < nu1; ++it)
        for (int colour = 0; colour < 2; ++colour) cluster_smooth(B, K, rank, colour, rhs && it == 0);
    }
    cluster_restrict(B, slab(l + 1), K);
    cluster_barrier();
  }
  if (rank == 0) {  // the bottom levels, whole in this block
    for (int l = P.tail; l + 1 < n; ++l) {
      const Slab B = slab(l);
      if (tl.nu1 == 0) tail_rhs<double, 2, false>(B.L, K);
      if (cluster_holds(B)) {
        cluster_passes<true>(B, K, 0, 2 * tl.nu1, true);
      } else {
        for (int it = 0; it < tl.nu1; ++it)
          for (int colour = 0; colour < 2; ++colour) tail_smooth<double, 2, false>(B.L, K, colour, it == 0);
      }
      cluster_restrict(B, slab(l + 1), K);
      __syncthreads();
    }
    {
      const Level<double> Lc = slab(n - 1).L;
      tail_rhs<double, 2, false>(Lc, K);
      coarsest_solve<double, 2, false>(Lc, K);
    }
    for (int l = n - 2; l >= P.tail; --l) {
      const Slab B = slab(l);
      tail_prolong<double, 2>(B.L, slab(l + 1).L);
      if (cluster_holds(B)) {
        cluster_passes<true>(B, K, 0, 2 * tl.nu2, false);
      } else {
        for (int it = 0; it < tl.nu2; ++it)
          for (int colour = 0; colour < 2; ++colour) tail_smooth<double, 2, false>(B.L, K, colour, false);
      }
    }
  }
  cluster_barrier();
  for (int l = P.tail - 1; l >= 0; --l) {
    const Slab B = slab(l);
    cluster_prolong(B, slab(l + 1));
    const int nu2 = l == 0 ? nu2_top : tl.nu2;
    if (cluster_holds(B)) {
      cluster_passes<false>(B, K, rank, 2 * nu2, false);
    } else {
      for (int it = 0; it < nu2; ++it)
        for (int colour = 0; colour < 2; ++colour) cluster_smooth(B, K, rank, colour, false);
    }
  }
  // every block is past its last read of another block's shared memory here
  // (the barrier that ends the last pass)
  const Level<double>& G = tl.lev[0];
  const Slab B = slab(0);
  for (int t = threadIdx.x; t < B.S * B.nr; t += blockDim.x) {
    G.phi[B.S * B.r0 + t] = B.L.phi[t];
    G.mu[B.S * B.r0 + t] = B.L.mu[t];
    G.p[B.S * B.r0 + t] = B.L.p[t];
  }
}

}  // namespace chhs_dev
