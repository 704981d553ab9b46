// chhs_cluster.cuh -- the coarse levels of a double-precision V-cycle in one
// launch: a cluster of up to 16 blocks holds them in (distributed) shared
// memory.
//
// On a level of 64 x 64 cells or less a colour pass is bound by latency: one
// warp's chain of FP64 instructions (~64 cycles each) plus, as a launch of
// its own, ~1.3 us of launch and drain.  Here every block of the cluster
// owns a slab of rows (planes in 3D) of each level, the passes exchange the
// slabs' edge rows through distributed shared memory, and a cluster barrier
// (~570 cycles measured at 512 threads) takes the launch's place.
//
// Slabs: level l gives every block R_l = 2 ceil(rows / (2 blocks)) rows, an
// even number starting at an even row, so that the 2^d children of a coarse
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
// Measured (GB300, default tuning): a 64 x 64 step of 6.6 V-cycles, all of it
// in the cluster, 847 us with a launch per pass -> 735 us; 512 x 512, where the
// levels 64 x 64 ... 16 x 16 move here, 2.55 -> 2.48 ms.
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

template <int DIM>
__host__ __device__ inline int cluster_row_cells(int nx, int ny) { return DIM == 3 ? nx * ny : nx; }

template <int DIM>
__host__ __device__ inline size_t cluster_smem_bytes(const Tail<double>& tl, const ClusterPlan& P) {
  size_t b = 0;
  for (int l = 0; l < tl.n; ++l)
    b += tail_fields<DIM, false>() *
         tail_align(sizeof(double) * cluster_cells(P.rows[l], cluster_row_cells<DIM>(tl.lev[l].nx, tl.lev[l].ny)));
  return b;
}

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

template <int DIM>
__device__ __forceinline__ Slab cluster_slab(const Tail<double>& tl, const ClusterPlan& P, int l, int rank,
                                             unsigned char* smem) {
  size_t off = 0;
  for (int q = 0; q < l; ++q)
    off += tail_fields<DIM, false>() *
           tail_align(sizeof(double) * cluster_cells(P.rows[q], cluster_row_cells<DIM>(tl.lev[q].nx, tl.lev[q].ny)));
  Slab B;
  B.L = tl.lev[l];
  Level<double>& L = B.L;
  B.S = cluster_row_cells<DIM>(L.nx, L.ny);
  B.R = P.rows[l];
  B.NR = DIM == 3 ? L.nz : L.ny;
  B.r0 = rank * B.R;
  B.nr = max(0, min(B.R, B.NR - B.r0));
  const size_t st = tail_align(sizeof(double) * cluster_cells(B.R, B.S));
  int q = 0;
  auto carve = [&]() { return reinterpret_cast<double*>(smem + off + (q++) * st) + B.S; };
  L.phi = carve(); L.mu = carve(); L.p = carve();
  L.fphi = carve(); L.fmu = carve(); L.fp = carve();
  L.phim = carve(); L.phi0 = carve(); L.mu0 = carve(); L.p0 = carve();
  L.ax = carve(); L.ay = carve(); L.Mx = carve(); L.My = carve();
  L.sM = carve(); L.sa = carve();
  L.cAe = carve(); L.cC = carve(); L.cGn = carve(); L.cHn = carve(); L.cQ = carve(); L.cH = carve();
  if (DIM == 3) { L.az = carve(); L.Mz = carve(); }
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

// (i, j, k) of slab cell t of nx x (ny x) nr cells; the row (plane) index is
// level-wide.
template <int DIM>
__device__ __forceinline__ void slab_ijk(const Slab& B, int t, int& i, int& j, int& k) {
  const int r = small_div(t, B.L.rnx);
  i = t - r * B.L.nx;
  if (DIM == 3) {
    const int kl = small_div(r, B.L.rny);
    j = r - kl * B.L.ny;
    k = B.r0 + kl;
  } else {
    j = B.r0 + r;
    k = 0;
  }
}

// One colour pass on the block's slab (the split update of k_smooth_split),
// its edge rows stored to the neighbours too; ends with the cluster barrier.
template <int DIM>
__device__ __forceinline__ void cluster_smooth(const Slab& B, const Coefs<double>& K, int rank, int colour, bool rhs) {
  __shared__ float xch[2][kTailGroups][4 * 32];
  const Level<double>& L = B.L;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = warp / 3, role = warp - 3 * g;
  const int hw = (L.nx + 1) >> 1;
  const int total = hw * (DIM == 3 ? L.ny : 1) * B.nr;
  if (g < kTailGroups) {
    const int rounds = (total + 32 * kTailGroups - 1) / (32 * kTailGroups);
    for (int q = 0; q < rounds; ++q) {
      const int t = q * 32 * kTailGroups + g * 32 + lane;
      const int row = small_div(t, L.rhw);
      const int ti = t - row * hw;
      int j, k, lr;
      if (DIM == 3) {
        lr = small_div(row, L.rny);
        j = row - lr * L.ny;
        k = B.r0 + lr;
      } else {
        lr = row;
        j = B.r0 + row;
        k = 0;
      }
      const int i = 2 * ti + ((j + k + colour) & 1);
      const bool act = t < total && i < L.nx;
      const int s = i + (DIM == 3 ? L.nx * j : 0);  // cell within its row (plane)
      const int c = act ? s + B.S * lr : 0;
      cell_update_split<DIM>(L, K, role, act, c, i, j, k, rhs, &xch[q & 1][g][lane], [g] {
        asm volatile("bar.sync %0, 96;" ::"r"(g + 1) : "memory");
      });
      if (act && role == 0) {
        if (lr == 0 && B.r0 > 0) {
          const int h = s + B.S * B.R;
          remote(L.phi, rank - 1)[h] = L.phi[c];
          remote(L.mu, rank - 1)[h] = L.mu[c];
          remote(L.p, rank - 1)[h] = L.p[c];
        }
        if (lr == B.R - 1 && B.r0 + B.R < B.NR) {
          const int h = s - B.S;
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
template <int DIM>
__device__ __forceinline__ void cluster_rhs(const Slab& B, const Coefs<double>& K) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = warp / 3, role = warp - 3 * g;
  if (g < kTailGroups)
    for (int t = g * 32 + lane; t < B.S * B.nr; t += 32 * kTailGroups) {
      int i, j, k;
      slab_ijk<DIM>(B, t, i, j, k);
      double u;
      f_row(B.L, role)[t] += n_row<DIM>(B.L, K, role, B.L.phi0, B.L.mu0, B.L.p0, t, i, j, k, u);
    }
  __syncthreads();
}

// Residual and restriction of the slab (tail_restrict's split form): each
// coarse value goes to its owner's slab and to the halos that hold its row.
template <int DIM>
__device__ __forceinline__ void cluster_restrict(const Slab& F, const Slab& C, const Coefs<double>& K) {
  constexpr int NCH = DIM == 3 ? 8 : 4;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = warp / 3, role = warp - 3 * g;
  if (g < kTailGroups) {
    const double w = DIM == 3 ? 0.125 : 0.25;
    const int ncoarse = C.S * (F.nr >> 1), total = ncoarse * NCH;
    const int rounds = (total + 32 * kTailGroups - 1) / (32 * kTailGroups);
    for (int q = 0; q < rounds; ++q) {
      const int t = q * 32 * kTailGroups + g * 32 + lane;
      const bool act = t < total;
      const int m = t / NCH, d = t % NCH;
      double rr = 0.0, u = 0.0;
      int s = 0, row = 0;
      if (act) {
        const int lrow = small_div(m, C.L.rnx);  // row of the coarse slab (x-row in 3D)
        const int I = m - lrow * C.L.nx;
        int J, KK;
        if (DIM == 3) {
          const int kl = small_div(lrow, C.L.rny);
          J = lrow - kl * C.L.ny;
          KK = (F.r0 >> 1) + kl;
          s = I + C.L.nx * J;
          row = KK;
        } else {
          J = (F.r0 >> 1) + lrow;
          KK = 0;
          s = I;
          row = J;
        }
        const int i = 2 * I + (d & 1), j = 2 * J + ((d >> 1) & 1), k = 2 * KK + (d >> 2);
        const int c = DIM == 3 ? i + F.L.nx * (j + F.L.ny * (k - F.r0)) : i + F.L.nx * (j - F.r0);
        const double n = n_row<DIM>(F.L, K, role, F.L.phi, F.L.mu, F.L.p, c, i, j, k, u);
        rr = f_row(F.L, role)[c] - n;
      }
#pragma unroll
      for (int o = 1; o < NCH; o <<= 1) {
        rr += __shfl_xor_sync(0xffffffffu, rr, o);
        u += __shfl_xor_sync(0xffffffffu, u, o);
      }
      if (act && d < 3) {  // three lanes of the 2^d share the stores of f, u and u^0
        double* a = d == 0 ? f_row(C.L, role)
                    : d == 1 ? (role == 0 ? C.L.phi : role == 1 ? C.L.p : C.L.mu)
                             : (role == 0 ? C.L.phi0 : role == 1 ? C.L.p0 : C.L.mu0);
        cluster_put(C, a, row, s, w * (d == 0 ? rr : u), d != 0);
      }
    }
  }
  cluster_barrier();
}

// u += P(u_c - u_c^0) on the slab and its halo rows (whose owners do the
// same), the coarse values read from their owners.  Ends with the cluster
// barrier: the next pass stores into the neighbours' halos.
template <int DIM>
__device__ __forceinline__ void cluster_prolong(const Slab& F, const Slab& C) {
  if (F.nr > 0) {
    const int lo = F.r0 > 0 ? -1 : 0, hi = F.r0 + F.nr < F.NR ? F.nr + 1 : F.nr;
    const int total = F.S * (hi - lo);
    for (int t = threadIdx.x; t < total; t += blockDim.x) {
      const int x = small_div(t, F.L.rnx);
      const int i = t - x * F.L.nx;
      int r, s;
      if (DIM == 3) {
        const int kl = small_div(x, F.L.rny), j = x - kl * F.L.ny;
        r = F.r0 + lo + kl;
        s = (i >> 1) + C.L.nx * (j >> 1);
      } else {
        r = F.r0 + lo + x;
        s = i >> 1;
      }
      const int o = (r >> 1) / C.R, q = s + C.S * ((r >> 1) - o * C.R);
      const int c = t + F.S * lo;
      F.L.phi[c] += remote(C.L.phi, o)[q] - remote(C.L.phi0, o)[q];
      F.L.mu[c] += remote(C.L.mu, o)[q] - remote(C.L.mu0, o)[q];
      F.L.p[c] += remote(C.L.p, o)[q] - remote(C.L.p0, o)[q];
    }
  }
  cluster_barrier();
}

// nu_top: sweeps of the top level (the finest level's counts when the whole
// hierarchy is in the cluster), tl.nu1 / tl.nu2 those of the levels below.
template <int DIM>
__global__ void __launch_bounds__(kTailThreads, 1) k_cluster(const __grid_constant__ Tail<double> tl,
                                                             const __grid_constant__ ClusterPlan P, Coefs<double> K,
                                                             int nu1_top, int nu2_top) {
  extern __shared__ __align__(16) unsigned char cl_smem[];
  pdl_enter();
  const int rank = (int)cooperative_groups::this_cluster().block_rank();
  const int n = tl.n;
  for (int l = 0; l < n; ++l) {
    const Level<double>& G = tl.lev[l];
    const Slab B = cluster_slab<DIM>(tl, P, l, rank, cl_smem);
    const Level<double>& S = B.L;
    const int base = B.S * B.r0;
    for (int t = threadIdx.x; t < B.S * B.nr; t += blockDim.x) {
      const int c = base + t;
      double v[15];
      v[0] = G.phim[c]; v[1] = G.ax[c]; v[2] = G.ay[c]; v[3] = G.Mx[c]; v[4] = G.My[c];
      v[5] = G.sM[c]; v[6] = G.sa[c]; v[11] = G.cQ[c]; v[14] = G.cH[c];
      const float k0 = G.kAe[c], k1 = G.kC[c], k2 = G.kGn[c], k3 = G.kHn[c];
      if (DIM == 3) { v[12] = G.az[c]; v[13] = G.Mz[c]; }
      S.phim[t] = v[0]; S.ax[t] = v[1]; S.ay[t] = v[2]; S.Mx[t] = v[3]; S.My[t] = v[4];
      S.sM[t] = v[5]; S.sa[t] = v[6]; S.cQ[t] = v[11]; S.cH[t] = v[14];
      S.kAe[t] = k0; S.kC[t] = k1; S.kGn[t] = k2; S.kHn[t] = k3;
      if (DIM == 3) { S.az[t] = v[12]; S.Mz[t] = v[13]; }
      if (l == 0) {
        S.fphi[t] = G.fphi[c]; S.fmu[t] = G.fmu[c]; S.fp[t] = G.fp[c];
      }
    }
    if (B.nr > 0) {
      // the halo below: its +y (+z) face coefficients belong to this slab's first row
      if (B.r0 > 0) {
        const double* a = DIM == 3 ? G.az : G.ay;
        const double* M = DIM == 3 ? G.Mz : G.My;
        for (int t = threadIdx.x; t < B.S; t += blockDim.x) {
          (DIM == 3 ? S.az : S.ay)[t - B.S] = a[base - B.S + t];
          (DIM == 3 ? S.Mz : S.My)[t - B.S] = M[base - B.S + t];
        }
      }
      if (l == 0) {  // the top level's state, halos included
        const int lo = B.r0 > 0 ? -B.S : 0, hi = B.S * (B.r0 + B.nr < B.NR ? B.nr + 1 : B.nr);
        for (int t = lo + (int)threadIdx.x; t < hi; t += blockDim.x) {
          const int c = base + t;
          double u[6];
          u[0] = G.phi[c]; u[1] = G.mu[c]; u[2] = G.p[c];
          if (tl.top_rhs) { u[3] = G.phi0[c]; u[4] = G.mu0[c]; u[5] = G.p0[c]; }
          S.phi[t] = u[0]; S.mu[t] = u[1]; S.p[t] = u[2];
          if (tl.top_rhs) { S.phi0[t] = u[3]; S.mu0[t] = u[4]; S.p0[t] = u[5]; }
        }
      }
    }
  }
  cluster_barrier();

  for (int l = 0; l < P.tail; ++l) {
    const Slab B = cluster_slab<DIM>(tl, P, l, rank, cl_smem);
    bool rhs = l > 0 || tl.top_rhs;
    const int nu1 = l == 0 ? nu1_top : tl.nu1;
    if (rhs && nu1 == 0) {
      cluster_rhs<DIM>(B, K);
      rhs = false;
    }
    for (int it = 0; it < nu1; ++it)
      for (int colour = 0; colour < 2; ++colour) cluster_smooth<DIM>(B, K, rank, colour, rhs && it == 0);
    cluster_restrict<DIM>(B, cluster_slab<DIM>(tl, P, l + 1, rank, cl_smem), K);
  }
  if (rank == 0) {  // the bottom levels, whole in this block
    for (int l = P.tail; l + 1 < n; ++l) {
      const Level<double> L = cluster_slab<DIM>(tl, P, l, 0, cl_smem).L;
      if (tl.nu1 == 0) tail_rhs<double, DIM, false>(L, K);
      for (int it = 0; it < tl.nu1; ++it)
        for (int colour = 0; colour < 2; ++colour) tail_smooth<double, DIM, false>(L, K, colour, it == 0);
      tail_restrict<double, DIM, false>(L, cluster_slab<DIM>(tl, P, l + 1, 0, cl_smem).L, K);
    }
    {
      const Level<double> Lc = cluster_slab<DIM>(tl, P, n - 1, 0, cl_smem).L;
      tail_rhs<double, DIM, false>(Lc, K);
      coarsest_solve<double, DIM, false>(Lc, K);
    }
    for (int l = n - 2; l >= P.tail; --l) {
      const Level<double> L = cluster_slab<DIM>(tl, P, l, 0, cl_smem).L;
      tail_prolong<double, DIM>(L, cluster_slab<DIM>(tl, P, l + 1, 0, cl_smem).L);
      for (int it = 0; it < tl.nu2; ++it)
        for (int colour = 0; colour < 2; ++colour) tail_smooth<double, DIM, false>(L, K, colour, false);
    }
  }
  cluster_barrier();
  for (int l = P.tail - 1; l >= 0; --l) {
    const Slab B = cluster_slab<DIM>(tl, P, l, rank, cl_smem);
    cluster_prolong<DIM>(B, cluster_slab<DIM>(tl, P, l + 1, rank, cl_smem));
    const int nu2 = l == 0 ? nu2_top : tl.nu2;
    for (int it = 0; it < nu2; ++it)
      for (int colour = 0; colour < 2; ++colour) cluster_smooth<DIM>(B, K, rank, colour, false);
  }
  // every block is past its last read of another block's shared memory here
  // (the barrier that ends the last pass)
  const Level<double>& G = tl.lev[0];
  const Slab B = cluster_slab<DIM>(tl, P, 0, rank, cl_smem);
  for (int t = threadIdx.x; t < B.S * B.nr; t += blockDim.x) {
    G.phi[B.S * B.r0 + t] = B.L.phi[t];
    G.mu[B.S * B.r0 + t] = B.L.mu[t];
    G.p[B.S * B.r0 + t] = B.L.p[t];
  }
}

}  // namespace chhs_dev
