// chhs_tail3.cuh -- the one-block coarse tail of the 3D single-precision
// (correction-form) V-cycles, a thread per two cells of a row.
//
// The levels of the tail (at most 1024 cells, down to the coarsest) are
// latency.  A thread keeps a red and a black cell, neighbours in x, in
// registers through all passes of a level -- state, right-hand sides, face
// values, constants; a pass updates its cell of the colour from the other and
// from five neighbour cells in shared memory, and stores it.  Four consecutive
// lanes hold the 2 x 2 x 2 cells of a coarse cell, whose residuals they add by
// shuffles.  Levels of at most 8 such groups are one warp's (warp barriers),
// and a coarsest grid of at most 32 cells is a cell per lane with shuffles,
// a larger one a cell per thread.  The double-precision coarsest solve runs on
// the general tail's code.
//
// The arithmetic is chhs_corr3.cuh's, cell by cell in the same order, so a
// level gives the same bits here and in the grid-wide passes.
// Measured: three steps of 128^3 9.86 -> 9.54 ms (tail 27 -> 20 us kernel by
// kernel), of 96 x 80 x 48, whose coarsest grid has 90 cells, 3.92 -> 3.60 ms.
// (Tried and slower: a cluster of 16 blocks that takes 16^3 or 32^3 as well,
// with the next planes read through distributed shared memory.  Its passes
// took 1 700-4 600 cycles, as much as the grid-wide launches in the step graph.)
#pragma once
#include "chhs_corr3.cuh"
#include "chhs_tail2.cuh"

namespace chhs_dev {

constexpr int kTail3Threads = 512;  // most threads of a CUDA block: 4 per group of 2 x 2 x 2 cells
// Shared memory of a level of nb groups of 2 x 2 x 2 cells above the coarsest,
// per cell: (phi, mu, p), R u, right-hand sides, phi*, phi^m, phi_b.
__host__ __device__ inline size_t tail3_level_bytes(int nb) { return (size_t)nb * 8 * (4 + 3 + 3 + 3) * sizeof(float); }

__host__ __device__ inline size_t tail3_smem_bytes(const int* ncell, int n, int coarsest_f64) {
  size_t b = 0;
  for (int l = 0; l + 1 < n; ++l) b += tail3_level_bytes(ncell[l] >> 3);
  b += tail_fields<3, true>() * tail_align(sizeof(float) * ncell[n - 1]);
  if (coarsest_f64) b += tail_fields<3, true>() * tail_align(sizeof(double) * ncell[n - 1]);
  return b;
}

// A level's scalars in shared memory (as Tail2Scalars).
struct Tail3Scalars {
  float ih2, h2, sih2, e34ih2, rhx, rhy;
  int hx, hy, hz, nb, off;
};

// A level in shared memory: cell x (0, 1) of thread e's pair at x n + e.
struct Tail3Level {
  float4* s0;
  float *u, *fs, *pss, *pms, *pbs;
  int n;  // threads: 4 per group
  __device__ __forceinline__ float4* s(int x, int e) const { return s0 + x * n + e; }
  __device__ __forceinline__ float* u0(int k, int x, int e) const { return u + (2 * k + x) * n + e; }
  __device__ __forceinline__ float* f(int k, int x, int e) const { return fs + (2 * k + x) * n + e; }
  __device__ __forceinline__ float* ps(int x, int e) const { return pss + x * n + e; }
  __device__ __forceinline__ float* pm(int x, int e) const { return pms + x * n + e; }
  __device__ __forceinline__ float* pb(int x, int e) const { return pbs + x * n + e; }
};

__device__ __forceinline__ Tail3Level tail3_level(const Tail3Scalars& L, unsigned char* smem) {
  float* a = reinterpret_cast<float*>(smem + L.off);
  Tail3Level T;
  T.n = 4 * L.nb;
  T.s0 = reinterpret_cast<float4*>(a);
  T.u = a + 8 * T.n;
  T.fs = a + 14 * T.n;
  T.pss = a + 20 * T.n;
  T.pms = a + 22 * T.n;
  T.pbs = a + 24 * T.n;
  return T;
}

__device__ __forceinline__ Val3 tail3_get(const float4* p) {
  const float4 v = *p;
  return Val3{v.x, v.y, v.z};
}

// The barrier between passes of a level: the block's, or its first warp's.
__device__ __forceinline__ void tail3_sync(bool warp) {
  if (warp) __syncwarp();
  else __syncthreads();
}

// A thread's place in a level: group (I, J, K) of 2 x 2 x 2 cells, row (jy, kz)
// of its four.
struct Tail3Place {
  int I, J, K, jy, kz;
};
__device__ __forceinline__ Tail3Place tail3_place(const Tail3Scalars& L, int g) {  // g: the thread
  const int q = g >> 2, r = small_div(q, L.rhx);
  Tail3Place p;
  p.I = q - r * L.hx;
  p.K = small_div(r, L.rhy);
  p.J = r - p.K * L.hy;
  p.jy = g & 1;
  p.kz = (g >> 1) & 1;
  return p;
}

// The pair of cells of a thread: [0] the red one (an even number of odd
// coordinates), at x = xr, [1] the black one.
struct Tail3Pair {
  Val3 c[2];
  float f[2][3];
  Chi3 ch[2];
  Newton3 nw[2];
  float ai, ao[2], a[2][4];  // x face inside, the other x face of each cell, faces y-, y+, z-, z+
  int xr;
  // neighbours in shared memory: the cell beyond each cell's outer x face, and
  // beyond y-, y+, z-, z+; a missing face has the cell itself
  const float4 *nx[2], *nd[2][4];
};

__device__ __forceinline__ void tail3_faces(const Tail3Pair& b, int h, float (&a)[6]) {
  const bool x1 = (b.xr ^ h) != 0;  // the cell is the right one of the pair
  a[0] = x1 ? b.ai : b.ao[h];
  a[1] = x1 ? b.ao[h] : b.ai;
#pragma unroll
  for (int d = 0; d < 4; ++d) a[2 + d] = b.a[h][d];
}

__device__ __forceinline__ void tail3_stencil(const Tail3Pair& b, int h, Val3 (&nb)[6], float (&a)[6]) {
  const bool x1 = (b.xr ^ h) != 0;
  const Val3 out = tail3_get(b.nx[h]);
  const Val3& in = b.c[1 - h];
  nb[0] = x1 ? in : out;
  nb[1] = x1 ? out : in;
#pragma unroll
  for (int d = 0; d < 4; ++d) nb[2 + d] = tail3_get(b.nd[h][d]);
  tail3_faces(b, h, a);
}

// Thread e's pair of a level: neighbours, face values, constants, state and
// right-hand side from shared memory.
__device__ __forceinline__ void tail3_setup(Tail3Pair& b, const Tail3Level& T, const Tail3Scalars& L, int e,
                                            const Coefs<float>& K) {
  const Tail3Place p = tail3_place(L, e);
  const int gy = 4 * L.hx, gz = gy * L.hy;  // threads from a group to the next in y, z
  b.xr = p.jy ^ p.kz;
  const bool inx[2] = {p.I > 0, p.I + 1 < L.hx};  // x-, x+ of the pair
  const bool in[4] = {p.jy || p.J > 0, !p.jy || p.J + 1 < L.hy, p.kz || p.K > 0, !p.kz || p.K + 1 < L.hz};
  // the threads beyond y-, y+, z-, z+: the group's other row, or the next group's
  const int en[4] = {in[0] ? (p.jy ? e - 1 : e - gy + 1) : e, in[1] ? (p.jy ? e + gy - 1 : e + 1) : e,
                     in[2] ? (p.kz ? e - 2 : e - gz + 2) : e, in[3] ? (p.kz ? e + gz - 2 : e + 2) : e};
  const float ps[2] = {*T.ps(0, e), *T.ps(1, e)};
  b.ai = 0.5f * (ps[0] + ps[1]);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int x = b.xr ^ h;  // the cell's place in the pair
    const bool inside = x ? inx[1] : inx[0];
    // beyond x- of the left cell lies the right cell of the pair before, and the other way
    const int ex = inside ? (x ? e + 4 : e - 4) : e, cx = inside ? 1 - x : x;
    b.nx[h] = T.s(cx, ex);
    const float pc = x ? ps[1] : ps[0];
    b.ao[h] = inside ? 0.5f * (pc + *T.ps(cx, ex)) : 0.f;
    int m = 1 + (inside ? 1 : 0);
#pragma unroll
    for (int d = 0; d < 4; ++d) {
      b.nd[h][d] = T.s(x, en[d]);
      b.a[h][d] = in[d] ? 0.5f * (pc + *T.ps(x, en[d])) : 0.f;
      m += in[d] ? 1 : 0;
    }
    float a[6];
    tail3_faces(b, h, a);
    b.nw[h] = newton3<3>(L, K.gamma, a, m);
    b.ch[h] = chi3_of(*T.pm(x, e), *T.pb(x, e));
    b.c[h] = tail3_get(T.s(x, e));
#pragma unroll
    for (int k = 0; k < 3; ++k) b.f[h][k] = *T.f(k, x, e);
  }
}

// npass (even) colour passes.
__device__ __forceinline__ void tail3_passes(Tail3Pair& b, const Tail3Level& T, int t, bool act, bool warp, int npass,
                                             const Tail3Scalars& L, const Coefs<float>& K) {
  for (int k = 0; k < npass; k += 2)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (act) {
        Val3 nb[6];
        float a[6];
        tail3_stencil(b, h, nb, a);
        const Val3 v = update3<3>(L, K, b.c[h], nb, a, b.f[h][0], b.f[h][1], b.f[h][2], b.ch[h], b.nw[h]);
        b.c[h] = v;
        *T.s(b.xr ^ h, t) = make_float4(v.phi, v.mu, v.p, 0.f);
      }
      tail3_sync(warp);
    }
}

// A coarse cell after restriction.
struct Tail3Coarse {
  Val3 u;
  float f1, f2, f3, pb;
};

// The mean residual, state and phi_b of the group, added in the order of
// k_residual_restrict_c (x in the thread, y and z by shuffles); every lane of
// the warp calls it.
__device__ __forceinline__ Tail3Coarse tail3_restrict(const Tail3Pair& b, const Tail3Level& T, int e, bool act,
                                                      const Tail3Scalars& L, const Coefs<float>& K) {
  float v[7] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  if (act) {
    float r[2][3];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      Val3 nb[6];
      float a[6];
      tail3_stencil(b, h, nb, a);
      const Val3 n = n_corr<3>(L, sums3<3>(b.c[h], nb, a, K.gamma), b.c[h], b.ch[h]);
      r[h][0] = b.f[h][0] - n.phi;
      r[h][1] = b.f[h][1] - n.mu;
      r[h][2] = b.f[h][2] - n.p;
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) v[k] = r[0][k] + r[1][k];
    v[3] = b.c[0].phi + b.c[1].phi;
    v[4] = b.c[0].mu + b.c[1].mu;
    v[5] = b.c[0].p + b.c[1].p;
    v[6] = *T.pb(0, e) + *T.pb(1, e);
  }
#pragma unroll
  for (int k = 0; k < 7; ++k) {
    v[k] += __shfl_xor_sync(0xffffffffu, v[k], 1);
    v[k] += __shfl_xor_sync(0xffffffffu, v[k], 2);
    v[k] *= 0.125f;
  }
  return Tail3Coarse{Val3{v[3], v[4], v[5]}, v[0], v[1], v[2], v[6]};
}

// The coarsest grid of at most 32 cells, cell c on lane c (coarsest_solve's
// sweeps and stopping rule); returns the correction u - R u.
__device__ __forceinline__ Val3 tail3_coarsest(const Level<float>& L, const Coefs<float>& K, const Tail3Coarse& q,
                                               float ps, float pm, int lane) {
  const unsigned all = 0xffffffffu;
  const bool act = lane < L.ncell;
  const int r = small_div(lane, L.rnx), i = lane - r * L.nx, k = small_div(r, L.rny), j = r - k * L.ny;
  const int sy = L.nx, sz = L.nx * L.ny;
  const bool in[6] = {i > 0, i + 1 < L.nx, j > 0, j + 1 < L.ny, k > 0, k + 1 < L.nz};
  const int off[6] = {-1, 1, -sy, sy, -sz, sz};
  int src[6], m = 0;
  float a[6];
#pragma unroll
  for (int d = 0; d < 6; ++d) {
    const bool on = act && in[d];
    src[d] = on ? lane + off[d] : lane;
    const float af = 0.5f * (ps + __shfl_sync(all, ps, src[d]));
    a[d] = on ? af : 0.f;
    m += on ? 1 : 0;
  }
  const Newton3 nw = newton3<3>(L, K.gamma, a, max(m, 1));
  const Chi3 ch = chi3_of(pm, q.pb);
  Val3 u = q.u;
  auto stencil = [&](Val3 (&nb)[6]) {
#pragma unroll
    for (int d = 0; d < 6; ++d)
      nb[d] = Val3{__shfl_sync(all, u.phi, src[d]), __shfl_sync(all, u.mu, src[d]), __shfl_sync(all, u.p, src[d])};
  };
  Val3 nb[6];
  stencil(nb);
  const Val3 n0 = n_corr<3>(L, sums3<3>(u, nb, a, K.gamma), u, ch);
  const float f1 = q.f1 + n0.phi, f2 = q.f2 + n0.mu, f3 = q.f3 + n0.p;
  float acc0 = -1.f, prev = 0.f;
  for (int it = 0; it <= kCoarsestMaxSweeps; ++it) {
    stencil(nb);
    const Val3 n = n_corr<3>(L, sums3<3>(u, nb, a, K.gamma), u, ch);
    const float r1 = f1 - n.phi, r2 = f2 - n.mu, r3 = K.s * (f3 - n.p);
    float tot = act ? r1 * r1 + r2 * r2 + r3 * r3 : 0.f;
    for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(all, tot, o);
    if (acc0 < 0.f) acc0 = tot;
    if (!(tot > kCoarsestTarget2 * acc0) || tot < 1e-37f) break;
    if (it >= 8 && tot >= prev) break;
    prev = tot;
    for (int colour = 0; colour < 2; ++colour) {
      stencil(nb);
      const Val3 v = update3<3>(L, K, u, nb, a, f1, f2, f3, ch, nw);
      if (((i + j + k + colour) & 1) == 0) u = v;
    }
  }
  return Val3{u.phi - q.u.phi, u.mu - q.u.mu, u.p - q.u.p};
}

// The same for more cells, at most one per thread: cell t on thread t, exchanged
// through buf, the block's sums through red (a float per warp).  Every thread
// of the block calls it.
__device__ __forceinline__ Val3 tail3_coarsest_block(const Level<float>& L, const Coefs<float>& K,
                                                     const Tail3Coarse& q, float ps, float pm, int t, float4* buf,
                                                     float* red) {
  const bool act = t < L.ncell;
  const int r = small_div(t, L.rnx), i = t - r * L.nx, k = small_div(r, L.rny), j = r - k * L.ny;
  const int sy = L.nx, sz = L.nx * L.ny;
  const bool in[6] = {i > 0, i + 1 < L.nx, j > 0, j + 1 < L.ny, k > 0, k + 1 < L.nz};
  const int off[6] = {-1, 1, -sy, sy, -sz, sz};
  Val3 u = q.u;
  if (act) buf[t] = make_float4(u.phi, u.mu, u.p, ps);
  __syncthreads();
  int src[6], m = 0;
  float a[6];
#pragma unroll
  for (int d = 0; d < 6; ++d) {
    const bool on = act && in[d];
    src[d] = on ? t + off[d] : (act ? t : 0);
    const float af = 0.5f * (ps + buf[src[d]].w);
    a[d] = on ? af : 0.f;
    m += on ? 1 : 0;
  }
  const Newton3 nw = newton3<3>(L, K.gamma, a, max(m, 1));
  const Chi3 ch = chi3_of(pm, q.pb);
  auto stencil = [&](Val3 (&nb)[6]) {
#pragma unroll
    for (int d = 0; d < 6; ++d) nb[d] = tail3_get(buf + src[d]);
  };
  Val3 nb[6];
  stencil(nb);
  const Val3 n0 = n_corr<3>(L, sums3<3>(u, nb, a, K.gamma), u, ch);
  const float f1 = q.f1 + n0.phi, f2 = q.f2 + n0.mu, f3 = q.f3 + n0.p;
  float acc0 = -1.f, prev = 0.f;
  for (int it = 0; it <= kCoarsestMaxSweeps; ++it) {
    stencil(nb);
    const Val3 n = n_corr<3>(L, sums3<3>(u, nb, a, K.gamma), u, ch);
    const float r1 = f1 - n.phi, r2 = f2 - n.mu, r3 = K.s * (f3 - n.p);
    const float part = warp_sum(act ? r1 * r1 + r2 * r2 + r3 * r3 : 0.f);
    if ((t & 31) == 0) red[t >> 5] = part;
    __syncthreads();
    float tot = 0.f;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += red[w];
    if (acc0 < 0.f) acc0 = tot;
    if (!(tot > kCoarsestTarget2 * acc0) || tot < 1e-37f) break;
    if (it >= 8 && tot >= prev) break;
    prev = tot;
    for (int colour = 0; colour < 2; ++colour) {
      if (act && ((i + j + k + colour) & 1) == 0) {
        stencil(nb);
        u = update3<3>(L, K, u, nb, a, f1, f2, f3, ch, nw);
        buf[t] = make_float4(u.phi, u.mu, u.p, ps);
      }
      __syncthreads();
    }
  }
  return Val3{u.phi - q.u.phi, u.mu - q.u.mu, u.p - q.u.p};
}

// The tail's levels tl.lev[0 .. n-1], n >= 2, level 0 of at most blockDim.x pairs.
__device__ __forceinline__ void tail3_body(const Tail<float>& tl, const Coefs<float>& K, unsigned char* smem) {
  __shared__ Tail3Scalars sc[kTailMaxLevels];  // of the levels above the coarsest; [n - 1].off: their end
  __shared__ float red[kTail3Threads / 32];
  const int n = tl.n, t = threadIdx.x, lane = t & 31;
  const Level<float>& Gc = tl.lev[n - 1];
  const bool general = tl.coarsest_f64 != 0;           // the coarsest solve on the general code
  const bool lanes = Gc.ncell <= 32 && !general;
  if (t < n) {
    const Level<float>& G = tl.lev[t];
    size_t off = 0;
    for (int q = 0; q < t; ++q) off += tail3_level_bytes(tl.lev[q].ncell >> 3);
    const int hx = max(G.nx >> 1, 1), hy = max(G.ny >> 1, 1), nb = max(G.ncell >> 3, 1);
    sc[t] = Tail3Scalars{G.ih2, G.h2, G.sih2, G.e34ih2, __frcp_rn((float)hx), __frcp_rn((float)hy),
                         hx, hy, G.nz >> 1, nb, (int)off};
  }
  __syncthreads();
  const int coff = sc[n - 1].off;
  // the coarsest cells handed over (u, f, phi_b) and their corrections back, and
  // tail3_coarsest_block's exchange behind them
  float* const cc = reinterpret_cast<float*>(smem + coff);
  const int nc = Gc.ncell;
  float4* const cbuf = reinterpret_cast<float4*>(cc + 8 * nc);
  // this thread's pair of level l, if it has one
  auto mine = [&](const Tail3Scalars& L) { return t < 4 * L.nb; };
  auto first_cell = [&](const Tail3Scalars& L, const Level<float>& G) {
    const Tail3Place p = tail3_place(L, t);
    return 2 * p.I + G.nx * (2 * p.J + p.jy + G.ny * (2 * p.K + p.kz));
  };
  // copy in: phi* and phi^m of every level, the top level's fields
  for (int l = 0; l + 1 < n; ++l) {
    const Level<float>& G = tl.lev[l];
    const Tail3Scalars S = sc[l];
    if (!mine(S)) continue;
    const Tail3Level T = tail3_level(S, smem);
    const int c = first_cell(S, G);
    auto ld = [&](const float* a) { return *reinterpret_cast<const float2*>(a + c); };
    const float2 ps = ld(G.phis), pm = ld(G.phim);
    if (l == 0) {
      const float2 u = ld(G.phi), v = ld(G.mu), w = ld(G.p), f1 = ld(G.fphi), f2 = ld(G.fmu), f3 = ld(G.fp),
                   pb = ld(G.phib);
      *T.s(0, t) = make_float4(u.x, v.x, w.x, 0.f);
      *T.s(1, t) = make_float4(u.y, v.y, w.y, 0.f);
      *T.f(0, 0, t) = f1.x;
      *T.f(0, 1, t) = f1.y;
      *T.f(1, 0, t) = f2.x;
      *T.f(1, 1, t) = f2.y;
      *T.f(2, 0, t) = f3.x;
      *T.f(2, 1, t) = f3.y;
      *T.pb(0, t) = pb.x;
      *T.pb(1, t) = pb.y;
    }
    *T.ps(0, t) = ps.x;
    *T.ps(1, t) = ps.y;
    *T.pm(0, t) = pm.x;
    *T.pm(1, t) = pm.y;
  }
  float cps = 0.f, cpm = 0.f;
  {
    if (!general) {
      if (t < Gc.ncell) {
        cps = Gc.phis[t];
        cpm = Gc.phim[t];
      }
    } else {
      const Level<float> S = tail_carve<float, 3, true>(Gc, smem + coff);
      for (int c = t; c < Gc.ncell; c += blockDim.x) {
        S.phim[c] = Gc.phim[c]; S.ax[c] = Gc.ax[c]; S.ay[c] = Gc.ay[c]; S.Mx[c] = Gc.Mx[c]; S.My[c] = Gc.My[c];
        S.sM[c] = Gc.sM[c]; S.sa[c] = Gc.sa[c]; S.cAe[c] = Gc.cAe[c]; S.cC[c] = Gc.cC[c]; S.cGn[c] = Gc.cGn[c];
        S.cHn[c] = Gc.cHn[c]; S.cQ[c] = Gc.cQ[c]; S.cH[c] = Gc.cH[c]; S.az[c] = Gc.az[c]; S.Mz[c] = Gc.Mz[c];
      }
    }
  }
  __syncthreads();

  Tail3Pair b;
  Val3 corr{0.f, 0.f, 0.f};
  // the coarse cell of this thread's group: thread and x of it on the next level
  auto coarse_at = [&](const Tail3Scalars& L, const Tail3Scalars& C, int& e, int& x) {
    const Tail3Place p = tail3_place(L, t);
    e = 4 * ((p.I >> 1) + C.hx * ((p.J >> 1) + C.hy * (p.K >> 1))) + (p.J & 1) + 2 * (p.K & 1);
    x = p.I & 1;
  };
  auto down = [&](int l, bool warp) {
    const Tail3Scalars L = sc[l];
    const Tail3Level T = tail3_level(L, smem);
    const bool act = mine(L);
    const bool rhs = l > 0 || tl.top_rhs;
    if (act) {
      tail3_setup(b, T, L, t, K);
      if (rhs) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          Val3 nb[6];
          float a[6];
          tail3_stencil(b, h, nb, a);
          const Val3 v = n_corr<3>(L, sums3<3>(b.c[h], nb, a, K.gamma), b.c[h], b.ch[h]);
          b.f[h][0] += v.phi;
          b.f[h][1] += v.mu;
          b.f[h][2] += v.p;
#pragma unroll
          for (int k = 0; k < 3; ++k) *T.f(k, b.xr ^ h, t) = b.f[h][k];
        }
      }
    }
    if (rhs) tail3_sync(warp);
    tail3_passes(b, T, t, act, warp, 2 * tl.nu1, L, K);
    const Tail3Coarse q = tail3_restrict(b, T, t, act, L, K);
    if (act && (t & 3) == 0) {
      if (l + 2 < n) {
        const Tail3Scalars LC = sc[l + 1];
        const Tail3Level C = tail3_level(LC, smem);
        int e, x;
        coarse_at(L, LC, e, x);
        *C.s(x, e) = make_float4(q.u.phi, q.u.mu, q.u.p, 0.f);
        *C.u0(0, x, e) = q.u.phi;
        *C.u0(1, x, e) = q.u.mu;
        *C.u0(2, x, e) = q.u.p;
        *C.f(0, x, e) = q.f1;
        *C.f(1, x, e) = q.f2;
        *C.f(2, x, e) = q.f3;
        *C.pb(x, e) = q.pb;
      } else if (!general) {
        const int c = t >> 2;
        cc[0 * nc + c] = q.u.phi;
        cc[1 * nc + c] = q.u.mu;
        cc[2 * nc + c] = q.u.p;
        cc[3 * nc + c] = q.f1;
        cc[4 * nc + c] = q.f2;
        cc[5 * nc + c] = q.f3;
        cc[6 * nc + c] = q.pb;
      } else {
        // group t / 4 sits on that coarse cell
        const Level<float> S = tail_carve<float, 3, true>(Gc, smem + coff);
        const int c = t >> 2;
        S.phi[c] = S.phi0[c] = q.u.phi;
        S.mu[c] = S.mu0[c] = q.u.mu;
        S.p[c] = S.p0[c] = q.u.p;
        S.fphi[c] = q.f1;
        S.fmu[c] = q.f2;
        S.fp[c] = q.f3;
        S.phib[c] = q.pb;
      }
    }
    tail3_sync(warp);
    if (l + 2 == n && lanes) {
      if (t < 32) {
        const int c = min(lane, nc - 1);
        const Tail3Coarse z{Val3{cc[c], cc[nc + c], cc[2 * nc + c]}, cc[3 * nc + c], cc[4 * nc + c], cc[5 * nc + c],
                            cc[6 * nc + c]};
        const Val3 d = tail3_coarsest(Gc, K, z, cps, cpm, lane);
        if (lane < nc) {
          cc[lane] = d.phi;
          cc[nc + lane] = d.mu;
          cc[2 * nc + lane] = d.p;
        }
      }
      tail3_sync(warp);
      if (act) corr = Val3{cc[t >> 2], cc[nc + (t >> 2)], cc[2 * nc + (t >> 2)]};
    }
  };
  auto up = [&](int l, bool warp) {
    const Tail3Scalars L = sc[l];
    const Tail3Level T = tail3_level(L, smem);
    const bool act = mine(L);
    if (act) {
      Val3 d = corr;
      if (l + 2 < n) {
        const Tail3Scalars LC = sc[l + 1];
        const Tail3Level C = tail3_level(LC, smem);
        int e, x;
        coarse_at(L, LC, e, x);
        const Val3 v = tail3_get(C.s(x, e));
        d = Val3{v.phi - *C.u0(0, x, e), v.mu - *C.u0(1, x, e), v.p - *C.u0(2, x, e)};
      }
      tail3_setup(b, T, L, t, K);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        b.c[h].phi += d.phi;
        b.c[h].mu += d.mu;
        b.c[h].p += d.p;
        *T.s(b.xr ^ h, t) = make_float4(b.c[h].phi, b.c[h].mu, b.c[h].p, 0.f);
      }
    }
    tail3_sync(warp);
    tail3_passes(b, T, t, act, warp, 2 * tl.nu2, L, K);
  };
  // levels of more than 8 groups on the whole block, the smaller ones on warp 0
  int small = 0;
  while (small + 1 < n && sc[small].nb > 8) ++small;
  for (int l = 0; l + 1 < n && (l < small || t < 32); ++l) down(l, l >= small);
  if (!lanes && !general) {  // the level above has more than 8 groups: every thread is here
    const int c = min(t, nc - 1);
    const Tail3Coarse z{Val3{cc[c], cc[nc + c], cc[2 * nc + c]}, cc[3 * nc + c], cc[4 * nc + c], cc[5 * nc + c],
                        cc[6 * nc + c]};
    const Val3 d = tail3_coarsest_block(Gc, K, z, cps, cpm, t, cbuf, red);
    if (t < nc) {
      cc[t] = d.phi;
      cc[nc + t] = d.mu;
      cc[2 * nc + t] = d.p;
    }
    __syncthreads();
    if ((t >> 2) < nc) corr = Val3{cc[t >> 2], cc[nc + (t >> 2)], cc[2 * nc + (t >> 2)]};
  } else if (!lanes) {
    __syncthreads();
    const Level<float> S = tail_carve<float, 3, true>(Gc, smem + coff);
    tail_rhs<float, 3, true>(S, K);
    coarsest_solve_f64<3>(S, K, smem + coff + tail_fields<3, true>() * tail_align(sizeof(float) * Gc.ncell));
    const int c = t >> 2;
    if (c < Gc.ncell) corr = Val3{S.phi[c] - S.phi0[c], S.mu[c] - S.mu0[c], S.p[c] - S.p0[c]};
    __syncthreads();
  }
  for (int l = n - 2; l >= 0; --l) {
    if (l >= small) {
      if (t >= 32) continue;
    } else if (l == small - 1) {
      __syncthreads();  // warp 0's levels are done
    }
    up(l, l >= small);
  }
  const Tail3Scalars S = sc[0];
  if (mine(S)) {
    const Level<float>& G = tl.lev[0];
    const Tail3Level T = tail3_level(S, smem);
    const int c = first_cell(S, G);
    const float4 x = *T.s(0, t), y = *T.s(1, t);
    *reinterpret_cast<float2*>(G.phi + c) = make_float2(x.x, y.x);
    *reinterpret_cast<float2*>(G.mu + c) = make_float2(x.y, y.y);
    *reinterpret_cast<float2*>(G.p + c) = make_float2(x.z, y.z);
  }
}

static __global__ void __launch_bounds__(kTail3Threads, 1) k_tail3(const __grid_constant__ Tail<float> tl,
                                                                  Coefs<float> K) {
  extern __shared__ __align__(16) unsigned char tail3_smem[];
  pdl_enter();
  tail3_body(tl, K, tail3_smem);
}

}  // namespace chhs_dev
