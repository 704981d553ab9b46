// chhs_tail2.cuh -- the one-block coarse tail of the 2D single-precision
// (correction-form) V-cycles, a thread per 2 x 2 cells.
//
// The levels of the tail (at most 32 x 32 cells by default, down to the
// coarsest) are latency: a colour pass of the general tail (tail_smooth) took
// 700-1000 cycles, most of it index arithmetic, the loads of 25 stored fields
// and a chain through them.  Here a thread keeps the 2 x 2 cells of a level in
// registers through all its passes as in chhs_tile.cuh (the same arithmetic):
// a pass reads four neighbour cells, updates two and stores them.  Levels of
// at most 32 threads (16 x 16 cells has 64, 8 x 8 has 16) are one warp's, with
// a warp barrier between passes; the coarsest grid of at most 32 cells is a
// cell per lane, its neighbours by shuffles, a larger one a cell per thread.
// The double-precision coarsest solve (coarsest_f64) runs on the general tail's
// code.
// Measured: the tail of a 512^2 step 33 -> 16 us (32 thousand cycles, a pass of
// one warp 320-350), the step 690 -> 588 us; 640 x 384 930 -> 765 us.
#pragma once
#include "chhs_tile.cuh"

namespace chhs_dev {

// Shared memory of a level above the coarsest, nb blocks of 2 x 2 cells:
// per cell position (phi, mu, p), the restricted iterate R u, the right-hand
// sides, phi^m, phi_b and q0, q1 of TileConst, and per block the constants that
// do not depend on the V-cycle (the 12 face values, Ae, x, hn, em per cell).
constexpr int kTail2Consts = 28;
struct Tail2Level {
  float4* s0;  // (mu, p, phi): position m (of 4) of block q at m nb + q
  float *u, *fs, *pms, *pbs, *qs, *cs;  // field k, position m of block q at (4 k + m) nb + q
  int hx, hy, nb;                       // blocks per row, rows, blocks
  __device__ __forceinline__ float4* s(int m, int q) const { return s0 + m * nb + q; }
  __device__ __forceinline__ float& u0(int k, int m, int q) const { return u[(4 * k + m) * nb + q]; }
  __device__ __forceinline__ float& f(int k, int m, int q) const { return fs[(4 * k + m) * nb + q]; }
  __device__ __forceinline__ float& pm(int m, int q) const { return pms[m * nb + q]; }
  __device__ __forceinline__ float& pb(int m, int q) const { return pbs[m * nb + q]; }
  __device__ __forceinline__ float& q01(int k, int m, int q) const { return qs[(4 * k + m) * nb + q]; }
  __device__ __forceinline__ float& con(int k, int q) const { return cs[k * nb + q]; }
};

__host__ __device__ inline size_t tail2_level_bytes(int nb) {
  return tail_align((size_t)nb * (16 + 12 + 12 + 4 + 4 + 8 + kTail2Consts) * sizeof(float));
}

// A level's scalars, copied to shared memory once: read with a level index
// that is not known at compile time, the kernel's parameters come through
// constant-cache misses (~1 500 cycles per level visit, measured).
struct Tail2Scalars {
  float ih2, h2, sih2, e34ih2, rhx;
  int hx, hy, nb, off;
};

// What the block shares beside the levels, at the start of the dynamic shared
// memory: as static memory it would also be taken from the largest one-level
// grids of k_tail, which need all of a block's.
struct Tail2Shared {
  Tail2Scalars sc[kTailMaxLevels];  // of the levels above the coarsest; [n - 1].off: their end
  float red[kTailThreads / 32];
};
constexpr size_t kTail2Head = (sizeof(Tail2Shared) + 15) / 16 * 16;

// Shared memory of tail2_body: its levels take 84 bytes a cell where the general
// code's take 92, so that only tails of less than 64 cells above the coarsest
// need more than tail_smem_bytes.
__host__ __device__ inline size_t tail2_smem_bytes(const int* ncell, int n, int coarsest_f64) {
  size_t b = kTail2Head;
  for (int l = 0; l + 1 < n; ++l) b += tail2_level_bytes(ncell[l] >> 2);
  if (!coarsest_f64) return b + (ncell[n - 1] > 32 ? sizeof(float4) * ncell[n - 1] : 0);
  return b + tail_smem_bytes<float, 2, true>(ncell + n - 1, 1, 1);
}
// A level of more than 2 x 2 cells per thread would not fit beside the coarsest
// in a block's 227 KB: no check of its own is needed.
static_assert((size_t)(227 * 1024) / (5 * tail_fields<2, true>()) <= 4 * kTailThreads,
              "a two-level tail that fits in shared memory has a thread per 2 x 2 cells");

__device__ __forceinline__ Tail2Level tail2_level(const Tail2Scalars& L, unsigned char* smem) {
  Tail2Level T;
  T.hx = L.hx;
  T.hy = L.hy;
  T.nb = L.nb;
  float* a = reinterpret_cast<float*>(smem + L.off);
  T.s0 = reinterpret_cast<float4*>(a);
  T.u = a + 16 * T.nb;
  T.fs = a + 28 * T.nb;
  T.pms = a + 40 * T.nb;
  T.pbs = a + 44 * T.nb;
  T.qs = a + 48 * T.nb;
  T.cs = a + 56 * T.nb;
  return T;
}

// One thread's 2 x 2 cells of a level: registers and the neighbour cells'
// places (a cell's own on a boundary face, so its differences vanish).
struct Tail2Block {
  TileCell c[4];
  float f1[4], f2[4], f3[4];
  TileConst k[4];
  float a01, a23, a02, a13;                          // faces inside
  float aw0, aw2, ae1, ae3, as0, as1, an2, an3;      // faces outside, zero on the boundary
  const float4 *w0, *w2, *e1, *e3, *s0, *s1, *n2, *n3;
};

__device__ __forceinline__ TileCell tail2_get(const float4* p) {
  const float4 v = *p;
  return TileCell{v.z, v.x, v.y};
}
__device__ __forceinline__ void tail2_put(float4* p, const TileCell& c) { *p = make_float4(c.mu, c.p, c.phi, 0.f); }

// The constants of block q of level L (global phi*, phi^m) into shared memory.
__device__ __forceinline__ void tail2_constants(const Tail2Level& T, int q, const Level<float>& L,
                                                const Tail2Scalars& S, const Coefs<float>& K) {
  const int J = small_div(q, S.rhx), I = q - J * T.hx;
  const bool eW = I == 0, eE = I == T.hx - 1, eS = J == 0, eN = J == T.hy - 1;
  const int nx = L.nx, c = 2 * I + nx * 2 * J;
  const float p0 = L.phis[c], p1 = L.phis[c + 1], p2 = L.phis[c + nx], p3 = L.phis[c + nx + 1];
  const float w0 = L.phis[eW ? c : c - 1], w2 = L.phis[eW ? c : c + nx - 1];
  const float e1 = L.phis[eE ? c : c + 2], e3 = L.phis[eE ? c : c + nx + 2];
  const float s0 = L.phis[eS ? c : c - nx], s1 = L.phis[eS ? c : c - nx + 1];
  const float n2 = L.phis[eN ? c : c + 2 * nx], n3 = L.phis[eN ? c : c + 2 * nx + 1];
  const float m0 = L.phim[c], m1 = L.phim[c + 1], m2 = L.phim[c + nx], m3 = L.phim[c + nx + 1];
  auto avg = [](float x, float y) { return 0.5f * (x + y); };
  const float a01 = avg(p0, p1), a23 = avg(p2, p3), a02 = avg(p0, p2), a13 = avg(p1, p3);
  const float aw0 = eW ? 0.f : avg(p0, w0), aw2 = eW ? 0.f : avg(p2, w2);
  const float ae1 = eE ? 0.f : avg(p1, e1), ae3 = eE ? 0.f : avg(p3, e3);
  const float as0 = eS ? 0.f : avg(p0, s0), as1 = eS ? 0.f : avg(p1, s1);
  const float an2 = eN ? 0.f : avg(p2, n2), an3 = eN ? 0.f : avg(p3, n3);
  const float a[12] = {a01, a23, a02, a13, aw0, aw2, ae1, ae3, as0, as1, an2, an3};
#pragma unroll
  for (int k = 0; k < 12; ++k) T.con(k, q) = a[k];
  const int w = eW ? 0 : 1, e = eE ? 0 : 1, s = eS ? 0 : 1, n = eN ? 0 : 1;
  auto put = [&](int m, const TileConst& k) {
    T.con(12 + m, q) = k.Ae;
    T.con(16 + m, q) = k.x;
    T.con(20 + m, q) = k.hn;
    T.con(24 + m, q) = k.em;
  };
  put(0, tile_constants(S, K, 0.f, 0.f, a01, a02, aw0, as0, 2 + w + s));
  put(1, tile_constants(S, K, 0.f, 0.f, a01, a13, ae1, as1, 2 + e + s));
  put(2, tile_constants(S, K, 0.f, 0.f, a23, a02, aw2, an2, 2 + w + n));
  put(3, tile_constants(S, K, 0.f, 0.f, a23, a13, ae3, an3, 2 + e + n));
  T.pm(0, q) = m0;
  T.pm(1, q) = m1;
  T.pm(2, q) = m2;
  T.pm(3, q) = m3;
}

// Thread t's block into registers: the neighbour cells' places, the constants,
// the state and the right-hand side.  On the way down (first) q0 and q1 are
// formed from phi_b and kept for the way up.
__device__ __forceinline__ void tail2_setup(Tail2Block& b, const Tail2Level& T, int t, float rhx, bool first) {
  const int J = small_div(t, rhx), I = t - J * T.hx;
  const bool eW = I == 0, eE = I == T.hx - 1, eS = J == 0, eN = J == T.hy - 1;
  b.w0 = eW ? T.s(0, t) : T.s(1, t) - 1;
  b.w2 = eW ? T.s(2, t) : T.s(3, t) - 1;
  b.e1 = eE ? T.s(1, t) : T.s(0, t) + 1;
  b.e3 = eE ? T.s(3, t) : T.s(2, t) + 1;
  b.s0 = eS ? T.s(0, t) : T.s(2, t) - T.hx;
  b.s1 = eS ? T.s(1, t) : T.s(3, t) - T.hx;
  b.n2 = eN ? T.s(2, t) : T.s(0, t) + T.hx;
  b.n3 = eN ? T.s(3, t) : T.s(1, t) + T.hx;
  float* const a[12] = {&b.a01, &b.a23, &b.a02, &b.a13, &b.aw0, &b.aw2, &b.ae1, &b.ae3, &b.as0, &b.as1, &b.an2, &b.an3};
#pragma unroll
  for (int k = 0; k < 12; ++k) *a[k] = T.con(k, t);
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    b.k[m].Ae = T.con(12 + m, t);
    b.k[m].x = T.con(16 + m, t);
    b.k[m].hn = T.con(20 + m, t);
    b.k[m].em = T.con(24 + m, t);
    b.c[m] = tail2_get(T.s(m, t));
    b.f1[m] = T.f(0, m, t);
    b.f2[m] = T.f(1, m, t);
    b.f3[m] = T.f(2, m, t);
    if (first) {
      tile_quad(b.k[m], T.pm(m, t), T.pb(m, t));
      T.q01(0, m, t) = b.k[m].q0;
      T.q01(1, m, t) = b.k[m].q1;
    } else {
      b.k[m].q0 = T.q01(0, m, t);
      b.k[m].q1 = T.q01(1, m, t);
    }
  }
}

// The barrier between passes: the block's, or warp 0's on a level of one warp.
__device__ __forceinline__ void tail2_sync(bool warp) {
  if (warp) __syncwarp();
  else __syncthreads();
}

// npass colour passes (even) of a level; every thread of the block (or of
// warp 0) calls it, act says whether it holds a block.
__device__ __forceinline__ void tail2_passes(Tail2Block& b, const Tail2Level& T, int t, bool act, bool warp, int npass,
                                             const Tail2Scalars& L, const Coefs<float>& K) {
  for (int k = 0; k < npass; k += 2) {
    if (act) {
      tile_update(b.c[0], b.c[1], b.c[2], tail2_get(b.w0), tail2_get(b.s0), b.a01, b.a02, b.aw0, b.as0, b.f1[0],
                  b.f2[0], b.f3[0], b.k[0], L, K);
      tile_update(b.c[3], b.c[2], b.c[1], tail2_get(b.e3), tail2_get(b.n3), b.a23, b.a13, b.ae3, b.an3, b.f1[3],
                  b.f2[3], b.f3[3], b.k[3], L, K);
      tail2_put(T.s(0, t), b.c[0]);
      tail2_put(T.s(3, t), b.c[3]);
    }
    tail2_sync(warp);
    if (act) {
      tile_update(b.c[1], b.c[0], b.c[3], tail2_get(b.e1), tail2_get(b.s1), b.a01, b.a13, b.ae1, b.as1, b.f1[1],
                  b.f2[1], b.f3[1], b.k[1], L, K);
      tile_update(b.c[2], b.c[3], b.c[0], tail2_get(b.w2), tail2_get(b.n2), b.a23, b.a02, b.aw2, b.an2, b.f1[2],
                  b.f2[2], b.f3[2], b.k[2], L, K);
      tail2_put(T.s(1, t), b.c[1]);
      tail2_put(T.s(2, t), b.c[2]);
    }
    tail2_sync(warp);
  }
}

// f += N(R u) of the block's cells (the state is still R u).
__device__ __forceinline__ void tail2_rhs(Tail2Block& b, const Tail2Scalars& L, const Coefs<float>& K) {
  tile_add_N(b.f1[0], b.f2[0], b.f3[0], b.c[0], b.c[1], b.c[2], tail2_get(b.w0), tail2_get(b.s0), b.a01, b.a02, b.aw0,
             b.as0, b.k[0], L, K);
  tile_add_N(b.f1[1], b.f2[1], b.f3[1], b.c[1], b.c[0], b.c[3], tail2_get(b.e1), tail2_get(b.s1), b.a01, b.a13, b.ae1,
             b.as1, b.k[1], L, K);
  tile_add_N(b.f1[2], b.f2[2], b.f3[2], b.c[2], b.c[3], b.c[0], tail2_get(b.w2), tail2_get(b.n2), b.a23, b.a02, b.aw2,
             b.an2, b.k[2], L, K);
  tile_add_N(b.f1[3], b.f2[3], b.f3[3], b.c[3], b.c[2], b.c[1], tail2_get(b.e3), tail2_get(b.n3), b.a23, b.a13, b.ae3,
             b.an3, b.k[3], L, K);
}

// The coarse cell of the block: its restricted residual, state and phi_b.
struct Tail2Coarse {
  TileCell u;
  float f1, f2, f3, pb;
};

__device__ __forceinline__ Tail2Coarse tail2_restrict(const Tail2Block& b, const Tail2Level& T, int t,
                                                      const Tail2Scalars& L, const Coefs<float>& K) {
  const TileOuter o{tail2_get(b.w0), tail2_get(b.w2), tail2_get(b.e1), tail2_get(b.e3),
                    tail2_get(b.s0), tail2_get(b.s1), tail2_get(b.n2), tail2_get(b.n3)};
  Tail2Coarse q;
  tile_block_residual(b.c[0], b.c[1], b.c[2], b.c[3], o, b.aw0, b.aw2, b.ae1, b.ae3, b.as0, b.as1, b.an2, b.an3, b.f1,
                      b.f2, b.f3, b.k[0], b.k[1], b.k[2], b.k[3], L, K, q.f1, q.f2, q.f3);
  q.u = TileCell{0.25f * ((b.c[0].phi + b.c[1].phi) + (b.c[2].phi + b.c[3].phi)),
                 0.25f * ((b.c[0].mu + b.c[1].mu) + (b.c[2].mu + b.c[3].mu)),
                 0.25f * ((b.c[0].p + b.c[1].p) + (b.c[2].p + b.c[3].p))};
  q.pb = 0.25f * ((T.pb(0, t) + T.pb(1, t)) + (T.pb(2, t) + T.pb(3, t)));
  return q;
}

// The coarsest grid of at most 32 cells: cell c on lane c, the sweeps and the
// stopping rule of coarsest_solve.  q: the lane's cell after restriction;
// returns the correction u - R u.
__device__ __forceinline__ TileCell tail2_coarsest(const Level<float>& L, const Coefs<float>& K, const Tail2Coarse& q,
                                                   float ps, float pm, int lane) {
  const unsigned all = 0xffffffffu;
  const bool act = lane < L.ncell;
  const int j = small_div(lane, L.rnx), i = lane - j * L.nx;
  const bool in0 = act && i > 0, in1 = act && i + 1 < L.nx, in2 = act && j > 0, in3 = act && j + 1 < L.ny;
  const int l0 = in0 ? lane - 1 : lane, l1 = in1 ? lane + 1 : lane, l2 = in2 ? lane - L.nx : lane,
            l3 = in3 ? lane + L.nx : lane;
  const float p0 = __shfl_sync(all, ps, l0), p1 = __shfl_sync(all, ps, l1), p2 = __shfl_sync(all, ps, l2),
              p3 = __shfl_sync(all, ps, l3);
  const float a0 = in0 ? 0.5f * (ps + p0) : 0.f, a1 = in1 ? 0.5f * (ps + p1) : 0.f, a2 = in2 ? 0.5f * (ps + p2) : 0.f,
              a3 = in3 ? 0.5f * (ps + p3) : 0.f;
  const int faces = max(1, (int)in0 + (int)in1 + (int)in2 + (int)in3);
  const TileConst k = tile_constants(L, K, pm, q.pb, a0, a1, a2, a3, faces);
  TileCell u = q.u;
  float f1 = q.f1, f2 = q.f2, f3 = q.f3;
  auto from = [&](int l) {
    return TileCell{__shfl_sync(all, u.phi, l), __shfl_sync(all, u.mu, l), __shfl_sync(all, u.p, l)};
  };
  {
    const TileCell n0 = from(l0), n1 = from(l1), n2 = from(l2), n3 = from(l3);
    tile_add_N(f1, f2, f3, u, n0, n1, n2, n3, a0, a1, a2, a3, k, L, K);
  }
  float acc0 = -1.f, prev = 0.f;
  for (int it = 0; it <= kCoarsestMaxSweeps; ++it) {
    float tot = 0.f;
    {
      const TileCell n0 = from(l0), n1 = from(l1), n2 = from(l2), n3 = from(l3);
      float r1 = 0.f, r2 = 0.f, r3 = 0.f;
      tile_add_N(r1, r2, r3, u, n0, n1, n2, n3, a0, a1, a2, a3, k, L, K);
      r1 = f1 - r1;
      r2 = f2 - r2;
      r3 = K.s * (f3 - r3);
      tot = act ? r1 * r1 + r2 * r2 + r3 * r3 : 0.f;
    }
    for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(all, tot, o);
    if (acc0 < 0.f) acc0 = tot;
    if (!(tot > kCoarsestTarget2 * acc0) || tot < 1e-37f) break;
    if (it >= 8 && tot >= prev) break;
    prev = tot;
    for (int colour = 0; colour < 2; ++colour) {
      const TileCell n0 = from(l0), n1 = from(l1), n2 = from(l2), n3 = from(l3);
      TileCell v = u;
      tile_update(v, n0, n1, n2, n3, a0, a1, a2, a3, f1, f2, f3, k, L, K);
      if (((i + j + colour) & 1) == 0) u = v;
    }
  }
  return TileCell{u.phi - q.u.phi, u.mu - q.u.mu, u.p - q.u.p};
}

// The same for more cells, at most one per thread: cell t on thread t, exchanged
// through buf, the block's sums through red (a float per warp).  Every thread
// of the block calls it.
__device__ __forceinline__ TileCell tail2_coarsest_block(const Level<float>& L, const Coefs<float>& K,
                                                         const Tail2Coarse& q, float ps, float pm, int t, float4* buf,
                                                         float* red) {
  const bool act = t < L.ncell;
  const int j = small_div(t, L.rnx), i = t - j * L.nx;
  TileCell u = q.u;
  if (act) buf[t] = make_float4(u.mu, u.p, u.phi, ps);
  __syncthreads();
  const bool in0 = act && i > 0, in1 = act && i + 1 < L.nx, in2 = act && j > 0, in3 = act && j + 1 < L.ny;
  const int own = act ? t : 0;
  const float4 *b0 = buf + (in0 ? t - 1 : own), *b1 = buf + (in1 ? t + 1 : own), *b2 = buf + (in2 ? t - L.nx : own),
               *b3 = buf + (in3 ? t + L.nx : own);
  const float a0 = in0 ? 0.5f * (ps + b0->w) : 0.f, a1 = in1 ? 0.5f * (ps + b1->w) : 0.f,
              a2 = in2 ? 0.5f * (ps + b2->w) : 0.f, a3 = in3 ? 0.5f * (ps + b3->w) : 0.f;
  const int faces = max(1, (int)in0 + (int)in1 + (int)in2 + (int)in3);
  const TileConst k = tile_constants(L, K, pm, q.pb, a0, a1, a2, a3, faces);
  float f1 = q.f1, f2 = q.f2, f3 = q.f3;
  tile_add_N(f1, f2, f3, u, tail2_get(b0), tail2_get(b1), tail2_get(b2), tail2_get(b3), a0, a1, a2, a3, k, L, K);
  float acc0 = -1.f, prev = 0.f;
  for (int it = 0; it <= kCoarsestMaxSweeps; ++it) {
    float r1 = 0.f, r2 = 0.f, r3 = 0.f;
    tile_add_N(r1, r2, r3, u, tail2_get(b0), tail2_get(b1), tail2_get(b2), tail2_get(b3), a0, a1, a2, a3, k, L, K);
    r1 = f1 - r1;
    r2 = f2 - r2;
    r3 = K.s * (f3 - r3);
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
      if (act && ((i + j + colour) & 1) == 0) {
        tile_update(u, tail2_get(b0), tail2_get(b1), tail2_get(b2), tail2_get(b3), a0, a1, a2, a3, f1, f2, f3, k, L, K);
        buf[t] = make_float4(u.mu, u.p, u.phi, ps);
      }
      __syncthreads();
    }
  }
  return TileCell{u.phi - q.u.phi, u.mu - q.u.mu, u.p - q.u.p};
}

// The tail's levels tl.lev[0 .. n-1], n >= 2: those above the coarsest have
// even extents and level 0 at most blockDim.x blocks of 2 x 2 cells.
__device__ __forceinline__ void tail2_body(const Tail<float>& tl, const Coefs<float>& K, unsigned char* smem) {
  const int n = tl.n, t = threadIdx.x, lane = t & 31;
  const Level<float>& Gc = tl.lev[n - 1];
  const bool general = tl.coarsest_f64 != 0;              // the coarsest solve on the general code
  const bool lanes = Gc.ncell <= 32 && !general;          // the coarsest grid on the lanes of warp 0
  Tail2Shared& shared = *reinterpret_cast<Tail2Shared*>(smem);
  float* const red = shared.red;
  Tail2Scalars* const sc = shared.sc;
  if (t < n) {
    const Level<float>& G = tl.lev[t];
    size_t off = kTail2Head;
    for (int q = 0; q < t; ++q) off += tail2_level_bytes(tl.lev[q].ncell >> 2);
    const int hx = G.nx >> 1;
    sc[t] = Tail2Scalars{G.ih2, G.h2, G.sih2, G.e34ih2, __frcp_rn((float)max(hx, 1)), hx, G.ny >> 1, G.ncell >> 2, (int)off};
  }
  __syncthreads();
  const int coff = sc[n - 1].off;  // the general code's coarsest level
  // the top level's state, right-hand sides and phi_b (the loads come first;
  // the constants of all levels are formed while they are on the way)
  const Level<float>& G0 = tl.lev[0];
  const Tail2Level T0 = tail2_level(sc[0], smem);
  float u[4], v[4], w[4], g1[4], g2[4], g3[4], pb[4];
  if (t < T0.nb) {
    const int J = small_div(t, sc[0].rhx), I = t - J * T0.hx;
    const int c0 = 2 * I + G0.nx * 2 * J, c1 = c0 + G0.nx;
    auto ld = [&](const float* a, float (&x)[4]) {
      const float2 lo = *reinterpret_cast<const float2*>(a + c0), hi = *reinterpret_cast<const float2*>(a + c1);
      x[0] = lo.x;
      x[1] = lo.y;
      x[2] = hi.x;
      x[3] = hi.y;
    };
    ld(G0.phi, u);
    ld(G0.mu, v);
    ld(G0.p, w);
    ld(G0.fphi, g1);
    ld(G0.fmu, g2);
    ld(G0.fp, g3);
    ld(G0.phib, pb);
  }
  float cps = 0.f, cpm = 0.f;
  if (!general) {
    if (t < Gc.ncell) {
      cps = Gc.phis[t];
      cpm = Gc.phim[t];
    }
  } else {
    const Level<float> S = tail_carve<float, 2, true>(Gc, smem + coff);
    for (int c = t; c < Gc.ncell; c += blockDim.x) {
      S.phim[c] = Gc.phim[c]; S.ax[c] = Gc.ax[c]; S.ay[c] = Gc.ay[c]; S.Mx[c] = Gc.Mx[c]; S.My[c] = Gc.My[c];
      S.sM[c] = Gc.sM[c]; S.sa[c] = Gc.sa[c]; S.cAe[c] = Gc.cAe[c]; S.cC[c] = Gc.cC[c]; S.cGn[c] = Gc.cGn[c];
      S.cHn[c] = Gc.cHn[c]; S.cQ[c] = Gc.cQ[c]; S.cH[c] = Gc.cH[c];
    }
  }
  // every level's blocks in one sequence over the threads, so that the small
  // levels' are other warps' work
  int total = 0;
  for (int l = 0; l + 1 < n; ++l) total += sc[l].nb;
  for (int e = t; e < total; e += blockDim.x) {
    int l = 0, q = e;
    while (q >= sc[l].nb) q -= sc[l++].nb;
    tail2_constants(tail2_level(sc[l], smem), q, tl.lev[l], sc[l], K);
  }
  if (t < T0.nb) {
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      *T0.s(m, t) = make_float4(v[m], w[m], u[m], 0.f);
      T0.f(0, m, t) = g1[m];
      T0.f(1, m, t) = g2[m];
      T0.f(2, m, t) = g3[m];
      T0.pb(m, t) = pb[m];
    }
  }
  __syncthreads();

  Tail2Block b;
  Tail2Coarse z{};               // the coarsest cell t (the level above's block t sits on it)
  TileCell corr{0.f, 0.f, 0.f};  // the next coarser level's correction at the block's coarse cell
  auto down = [&](int l, bool warp) {
    const Tail2Scalars L = sc[l];
    const Tail2Level T = tail2_level(L, smem);
    const bool act = t < T.nb;
    const bool rhs = l > 0 || tl.top_rhs;
    if (act) {
      tail2_setup(b, T, t, L.rhx, true);
      if (rhs) {
        tail2_rhs(b, L, K);
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          T.f(0, m, t) = b.f1[m];
          T.f(1, m, t) = b.f2[m];
          T.f(2, m, t) = b.f3[m];
        }
      }
    }
    tail2_sync(warp);
    tail2_passes(b, T, t, act, warp, 2 * tl.nu1, L, K);
    Tail2Coarse q{};
    if (act) q = tail2_restrict(b, T, t, L, K);
    if (l + 2 < n) {
      if (act) {
        const Tail2Level C = tail2_level(sc[l + 1], smem);
        const int J = small_div(t, L.rhx), I = t - J * T.hx;
        const int m = (I & 1) + 2 * (J & 1), x = (I >> 1) + C.hx * (J >> 1);
        tail2_put(C.s(m, x), q.u);
        C.u0(0, m, x) = q.u.phi;
        C.u0(1, m, x) = q.u.mu;
        C.u0(2, m, x) = q.u.p;
        C.f(0, m, x) = q.f1;
        C.f(1, m, x) = q.f2;
        C.f(2, m, x) = q.f3;
        C.pb(m, x) = q.pb;
      }
    } else if (lanes) {
      corr = tail2_coarsest(Gc, K, q, cps, cpm, lane);  // warp 0 only: this level has at most 32 blocks
    } else if (!general) {
      z = q;
    } else if (act) {
      const Level<float> S = tail_carve<float, 2, true>(Gc, smem + coff);
      S.phi[t] = S.phi0[t] = q.u.phi;
      S.mu[t] = S.mu0[t] = q.u.mu;
      S.p[t] = S.p0[t] = q.u.p;
      S.fphi[t] = q.f1;
      S.fmu[t] = q.f2;
      S.fp[t] = q.f3;
      S.phib[t] = q.pb;
    }
  };
  auto up = [&](int l, bool warp) {
    const Tail2Scalars L = sc[l];
    const Tail2Level T = tail2_level(L, smem);
    const bool act = t < T.nb;
    if (act) {
      TileCell d = corr;
      if (l + 2 < n) {
        const Tail2Level C = tail2_level(sc[l + 1], smem);
        const int J = small_div(t, L.rhx), I = t - J * T.hx;
        const int m = (I & 1) + 2 * (J & 1), x = (I >> 1) + C.hx * (J >> 1);
        const TileCell v = tail2_get(C.s(m, x));
        d = TileCell{v.phi - C.u0(0, m, x), v.mu - C.u0(1, m, x), v.p - C.u0(2, m, x)};
      }
      tail2_setup(b, T, t, L.rhx, false);
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        b.c[m].phi += d.phi;
        b.c[m].mu += d.mu;
        b.c[m].p += d.p;
        tail2_put(T.s(m, t), b.c[m]);
      }
    }
    tail2_sync(warp);
    tail2_passes(b, T, t, act, warp, 2 * tl.nu2, L, K);
  };
  // the levels of more than 32 blocks on the whole block, the smaller ones on warp 0
  int small = 0;
  while (small + 1 < n && sc[small].nb > 32) ++small;
  // (one call each way: a copy per barrier kind would double the code, and the
  // instructions of a level's first visit come through cache misses)
  for (int l = 0; l + 1 < n && (l < small || t < 32); ++l) {
    down(l, l >= small);
    tail2_sync(l >= small);
  }
  if (!lanes && !general) {  // the level above has more than 32 blocks: every thread is here
    corr = tail2_coarsest_block(Gc, K, z, cps, cpm, t, reinterpret_cast<float4*>(smem + coff), red);
    __syncthreads();
  } else if (!lanes) {
    __syncthreads();
    const Level<float> S = tail_carve<float, 2, true>(Gc, smem + coff);
    tail_rhs<float, 2, true>(S, K);
    coarsest_solve_f64<2>(S, K, smem + coff + tail_fields<2, true>() * tail_align(sizeof(float) * Gc.ncell));
    // level n - 2's block t sits on coarse cell t
    if (t < Gc.ncell) corr = TileCell{S.phi[t] - S.phi0[t], S.mu[t] - S.mu0[t], S.p[t] - S.p0[t]};
    __syncthreads();
  }
  for (int l = n - 2; l >= 0; --l) {
    if (l >= small) {
      if (t >= 32) continue;
    } else if (l == small - 1) {
      __syncthreads();  // warp 0's levels are done
    }
    up(l, l >= small);
    tail2_sync(l >= small);
  }
  {
    const Tail2Level T = T0;
    if (t < T.nb) {
      const int J = small_div(t, sc[0].rhx), I = t - J * T.hx;
      const int c0 = 2 * I + G0.nx * 2 * J, c1 = c0 + G0.nx;
      auto st = [&](float* a, float x0, float x1, float x2, float x3) {
        *reinterpret_cast<float2*>(a + c0) = make_float2(x0, x1);
        *reinterpret_cast<float2*>(a + c1) = make_float2(x2, x3);
      };
      const TileCell A = tail2_get(T.s(0, t)), B = tail2_get(T.s(1, t)), C = tail2_get(T.s(2, t)),
                     D = tail2_get(T.s(3, t));
      st(G0.phi, A.phi, B.phi, C.phi, D.phi);
      st(G0.mu, A.mu, B.mu, C.mu, D.mu);
      st(G0.p, A.p, B.p, C.p, D.p);
    }
  }
}

// The tail as every launch runs it: 2D single-precision levels as above, unless
// the coarsest grid is all there is.
template <typename T, int DIM, bool CORR>
__device__ __forceinline__ void tail_run(const Tail<T>& tl, const Coefs<T>& K) {
  if constexpr (DIM == 2 && sizeof(T) == 4 && CORR) {
    if (tl.n >= 2) {
      extern __shared__ __align__(16) unsigned char tail_smem[];
      tail2_body(tl, K, tail_smem);
      return;
    }
  }
  tail_body<T, DIM, CORR>(tl, K);
}

template <typename T, int DIM, bool CORR>
__global__ void __launch_bounds__(kTailThreads, 1) k_tail(const __grid_constant__ Tail<T> tl, Coefs<T> K) {
  pdl_enter();
  tail_run<T, DIM, CORR>(tl, K);
}

}  // namespace chhs_dev
