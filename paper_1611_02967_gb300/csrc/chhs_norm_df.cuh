// chhs_norm_df.cuh -- the mixed-precision form's defect-correction residual
// f - N(u) of the double-precision iterate, evaluated in double-single
// arithmetic (chhs_df64.cuh) on the single-precision pipes.
//
// Outputs: the stopping norm and the pointwise residual (the loop decision of
// the step graph), the mean of p, and the next inner solve's right-hand side
// (r rounded to single precision, e = 0, phi_b = phi cut to single
// precision).  The residual is formed from the fluxes of the faces between
// two cells c and e, with a = (phi*_c + phi*_e)/2 and d the difference e - c,
//   w = dp + gamma a dmu,          v = dmu + a w  ( = M dmu + a dp ),
//   N1 = phi - s/h^2 sum_f v,      N3 = -1/h^2 sum_f w,
//   N2 = mu + (3/4) eps^2/h^2 sum_f dphi - phi (phi^2 + phi phi^m + (phi^m)^2)/4
// (N2 and f_mu carry the same constant shift (phi^m)^3/4 as the
// double-precision kernels, see cubic_P; f_phi = phi^m and f_p = 0 on the
// finest level), with every double input split into hi + lo and every
// operation a double-single one (chhs_ndf.cuh, with the error measured against
// 64 bits): exact to ~2^-44 of the largest term, far below the 1e-10 stopping
// tolerance.
//
// What bounds it: issue slots (a double-single addition is 8 instructions),
// so the work per cell is kept small.  In 3D a block takes a column of 32 x 8
// cells and marches through up to 16 planes: every double is split once (the
// tile's one-cell ring adds 31 %), every face's flux is formed once and given
// to both of its cells (x and y through shared memory, z in registers), and
// the coefficients come from phi* (w above needs no stored M).  In 2D a warp
// marches up a strip of 32 cells, x neighbours by shuffles, without shared
// memory or block barriers.
//
// Measured per launch (GB300, kernel by kernel with events), against a kernel
// of one plane per block that read the stored a and M, formed each flux on
// both sides and ran three of eight tiles on the FP64 pipe (~1 460
// instructions per cell): 256^3 1056 -> 510 us, 128^3 159 -> 85 us,
// 2048^2 231 -> 133 us.
#pragma once
#include <type_traits>

#include "chhs_ndf.cuh"
#include "chhs_kernels.cuh"

namespace chhs_dev {

constexpr int kNdfTX = 32, kNdfTY = 8;  // 256 threads, one cell of the plane each
constexpr int kNdfSW = kNdfTX + 2, kNdfSH = kNdfTY + 2, kNdfSN = kNdfSW * kNdfSH;
constexpr int kNdfRing = 2 * (kNdfTX + kNdfTY);  // ring cells without the corners

// Planes a block marches through, and the blocks of an nx x ny x nz grid.
__host__ __device__ inline int ndf_blocks_x(int nx) { return (nx + kNdfTX - 1) / kNdfTX; }
__host__ __device__ inline int ndf_blocks_y(int ny) { return (ny + kNdfTY - 1) / kNdfTY; }
__host__ __device__ inline int ndf_planes(int nx, int ny, int nz) {
  const long long columns = (long long)ndf_blocks_x(nx) * ndf_blocks_y(ny);
  int planes = 16;
  while (planes > 2 && columns * ((nz + planes - 1) / planes) < 900) planes >>= 1;
  return planes;
}
// Rows a warp marches through in 2D; a block's eight warps take eight such
// runs of rows of one strip.
__host__ __device__ inline int ndf_rows(int nx, int ny) {
  int rows = 16;
  while (rows > 1 && (long long)ndf_blocks_x(nx) * ((ny + 8 * rows - 1) / (8 * rows)) < 300) rows >>= 1;
  return rows;
}
template <int DIM>
__host__ __device__ inline long long ndf_blocks(int nx, int ny, int nz) {
  if (DIM == 2) {
    const int run = 8 * ndf_rows(nx, ny);
    return (long long)ndf_blocks_x(nx) * ((ny + run - 1) / run);
  }
  const int planes = ndf_planes(nx, ny, nz);
  return (long long)ndf_blocks_x(nx) * ndf_blocks_y(ny) * ((nz + planes - 1) / planes);
}

// The level's scalar coefficients as double-single numbers (host-split).
struct DfCoefs {
  df64 sih2, ih2, e34ih2, gamma;
  float s;
};

// The residual's arithmetic (A): double-single (NdfSingle), or double precision
// for blocks that run on the FP64 pipe.  Both are 8 bytes a value.
//
// Which blocks (chhs_tuning.norm_f64_per8, chhs_opts.f64_residual): from 4 on, so
// many of every 8, as asked; below 4 none.  So few of them were a matter of
// speed, the FP64 pipe working beside the others: 3 of 8 had paid while the
// double-single blocks spent twice the instructions; now the FP64 pipe takes
// longer over them than all blocks take without it (4 of 8 against none: 256^3
// 991 us and 510, 128^3 179 and 85, 2048^2 289 and 133, 512^2 41 and 23), and the
// double-single error is below that of such a mix (chhs_ndf.cuh).  With
// f64_residual the sums are in double precision too.
enum NdfMode { kNdfSingle = 0, kNdfShare = 1, kNdfF64 = 2 };
__host__ __device__ inline NdfMode ndf_mode(int f64_per8, int f64_residual) {
  return f64_residual ? kNdfF64 : f64_per8 >= 4 ? kNdfShare : kNdfSingle;
}

struct NdfDouble {
  using V = double;
  static __device__ __forceinline__ V from(double x) { return x; }
  static __device__ __forceinline__ V add(V a, V b) { return a + b; }
  static __device__ __forceinline__ V sub(V a, V b) { return a - b; }
  static __device__ __forceinline__ V diff(V a, V b) { return a - b; }
  static __device__ __forceinline__ V mul(V a, V b) { return a * b; }
  static __device__ __forceinline__ V mul_wide(V a, V b) { return a * b; }
  static __device__ __forceinline__ V fma(V a, V b, V c) { return ::fma(a, b, c); }
  static __device__ __forceinline__ V fma_wide(V a, V b, V c) { return ::fma(a, b, c); }
  static __device__ __forceinline__ V half(V a) { return 0.5 * a; }
  static __device__ __forceinline__ V zero() { return 0.0; }
  static __device__ __forceinline__ float cut(V a) { return f64_to_f32_rz(a); }
  static __device__ __forceinline__ float base(V a) { return f64_to_f32_rz(a); }
};

// Block sums: thread 0 returns the sum of squares (single precision within a
// warp), the double-single sum of p and the maximum.  (An overflow stays an
// infinity: the error term of an infinite sum is not a number.)
__device__ __forceinline__ void ndf_block_reduce(df64& sq, df64& ps, float& mx) {
  __shared__ float s_sq[kNdfTX * kNdfTY / 32], s_mx[kNdfTX * kNdfTY / 32];
  __shared__ df64 s_ps[kNdfTX * kNdfTY / 32];
  float plain = isfinite(sq.hi) ? sq.hi + sq.lo : sq.hi;
  for (int o = 16; o > 0; o >>= 1) {
    plain += __shfl_down_sync(0xffffffffu, plain, o);
    mx = fmaxf(mx, __shfl_down_sync(0xffffffffu, mx, o));
    const df64 other{__shfl_down_sync(0xffffffffu, ps.hi, o), __shfl_down_sync(0xffffffffu, ps.lo, o)};
    ps = df_add(ps, other);
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) {
    s_sq[wid] = plain;
    s_mx[wid] = mx;
    s_ps[wid] = ps;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    sq = df64{plain, 0.f};
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) {
      plain += s_sq[w];
      sq = df_add(sq, df64{s_sq[w], 0.f});
      mx = fmaxf(mx, s_mx[w]);
      ps = df_add(ps, s_ps[w]);
    }
    if (!isfinite(plain)) sq = df64{plain, 0.f};
  }
  __syncthreads();
}

// Sums of a block's cells: double-single over a thread's beside the
// double-single residual (up to 16 cells; in single precision the squares lost
// more than in the 256-cell blocks before), in double precision with
// f64_residual.
struct NdfSums32 {
  float mx = 0.f;
  df64 sq{0.f, 0.f}, ps{0.f, 0.f};
  __device__ __forceinline__ void add(float r1, float r2, float r3s) {
    const df64 s = df_two_sum(sq.hi, r1 * r1 + r2 * r2 + r3s * r3s);
    sq = df64{s.hi, sq.lo + s.lo};
    mx = fmaxf(mx, fmaxf(fmaxf(fabsf(r1), fabsf(r2)), fabsf(r3s)));
  }
  __device__ __forceinline__ void finish(double (&out)[3]) {
    ndf_block_reduce(sq, ps, mx);
    out[0] = df_to_double(sq);
    out[1] = df_to_double(ps);
    out[2] = (double)mx;
  }
};
struct NdfSums64 {
  double acc[2] = {0.0, 0.0}, mx = 0.0;
  __device__ __forceinline__ void add(double r1, double r2, double r3s) {
    acc[0] = ::fma(r1, r1, acc[0]);
    acc[0] = ::fma(r2, r2, acc[0]);
    acc[0] = ::fma(r3s, r3s, acc[0]);
    mx = max_pos(mx, row_max(r1, r2, r3s));
  }
  __device__ __forceinline__ void finish(double (&out)[3]) {
    block_sum<2>(acc);
    out[0] = acc[0];
    out[1] = acc[1];
    out[2] = block_max(mx);
  }
};

struct NdfShared {
  df64 cell[4][kNdfSN];                      // phi, mu, p, phi* of the tile and its ring
  df64 fx[3][kNdfTY * (kNdfTX + 1)];         // v, w, d of the x faces
  df64 fy[3][(kNdfTY + 1) * kNdfTX];         // ... and of the y faces
};

// A cell's residual from its summed fluxes (sv, sw, sd), and what the next
// inner solve reads; c: its index.
template <class A, class SUMS>
struct NdfOut {
  using V = typename A::V;
  const Level<float>& G;
  V sih2, ih2, e34ih2;
  float s32;
  double s64;
  SUMS& sums;
  __device__ __forceinline__ void cell(int c, const NdfCell<A>& u, V sv, V sw, V sd, double pm64, double fmu64) {
    V r1, r2, r3;
    ndf_residual<A>(u, sv, sw, sd, A::from(pm64), A::from(fmu64), sih2, ih2, e34ih2, r1, r2, r3);
    const float r1f = A::cut(r1), r2f = A::cut(r2), r3f = A::cut(r3);
    if constexpr (std::is_same<SUMS, NdfSums64>::value) {
      sums.add(r1, r2, s64 * r3);
      sums.acc[1] += u.p;
    } else {
      sums.add(r1f, r2f, s32 * r3f);
      if constexpr (std::is_same<A, NdfSingle>::value) sums.ps = df_add(sums.ps, u.p);
      else sums.ps = df_add(sums.ps, df_split(u.p));
    }
    G.fphi[c] = r1f;
    G.fmu[c] = r2f;
    G.fp[c] = r3f;
    G.phi[c] = 0.f;
    G.mu[c] = 0.f;
    G.p[c] = 0.f;
    G.phib[c] = A::base(u.phi);  // phi with its significand cut to 24 bits
  }
};

__device__ __forceinline__ df64 ndf_shfl_up(df64 v) {
  return df64{__shfl_up_sync(0xffffffffu, v.hi, 1), __shfl_up_sync(0xffffffffu, v.lo, 1)};
}
__device__ __forceinline__ double ndf_shfl_up(double v) { return __shfl_up_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ df64 ndf_shfl_down(df64 v) {
  return df64{__shfl_down_sync(0xffffffffu, v.hi, 1), __shfl_down_sync(0xffffffffu, v.lo, 1)};
}
__device__ __forceinline__ double ndf_shfl_down(double v) { return __shfl_down_sync(0xffffffffu, v, 1); }

// 2D: one warp's strip, the cells x0 .. x0+31 of the rows j0 .. j1-1.
template <class A, class SUMS>
__device__ __forceinline__ void ndf_strip(int x0, int j0, int j1, const Level<double>& L, typename A::V gamma,
                                          NdfOut<A, SUMS>& out) {
  using V = typename A::V;
  using Cell = NdfCell<A>;
  using Flux = NdfFlux<A>;
  const Flux none{A::zero(), A::zero(), A::zero()};
  const Cell empty{A::zero(), A::zero(), A::zero(), A::zero()};
  const int nx = L.nx, lane = threadIdx.x & 31, i = x0 + lane;
  const bool in = i < nx;
  const int col = in ? i : 0;
  auto load = [&](int c) { return Cell{A::from(L.phi[c]), A::from(L.mu[c]), A::from(L.p[c]), A::from(L.phis[c])}; };
  // the cells beside the strip, held by its first and last lane
  const int rcol = lane == 0 ? x0 - 1 : x0 + 32;
  const bool ring = (lane == 0 && x0 > 0) || (lane == 31 && x0 + 32 < nx);
  Cell cur = empty;
  Flux below = none;
  if (j0 < j1 && in) {
    cur = load(col + nx * j0);
    if (j0 > 0) below = ndf_face<A>(load(col + nx * (j0 - 1)), cur, gamma);
  }
  for (int j = j0; j < j1; ++j) {
    const int c = col + nx * j;
    const bool up = in && j + 1 < L.ny;
    double nxt[4], pm64 = 0.0, fmu64 = 0.0;
    if (up) {
      nxt[0] = L.phi[c + nx];
      nxt[1] = L.mu[c + nx];
      nxt[2] = L.p[c + nx];
      nxt[3] = L.phis[c + nx];
    }
    if (in) {
      pm64 = L.phim[c];
      fmu64 = L.fmu[c];
    }
    const Cell side = ring ? load(rcol + nx * j) : empty;
    Cell left{ndf_shfl_up(cur.phi), ndf_shfl_up(cur.mu), ndf_shfl_up(cur.p), ndf_shfl_up(cur.ps)};
    if (lane == 0) left = side;
    const Flux W = in && i > 0 ? ndf_face<A>(left, cur, gamma) : none;
    Flux E{ndf_shfl_down(W.v), ndf_shfl_down(W.w), ndf_shfl_down(W.d)};
    if (lane == 31) E = ring ? ndf_face<A>(cur, side, gamma) : none;
    Cell above = empty;
    Flux N = none;
    if (up) {
      above = Cell{A::from(nxt[0]), A::from(nxt[1]), A::from(nxt[2]), A::from(nxt[3])};
      N = ndf_face<A>(cur, above, gamma);
    }
    if (in)
      out.cell(c, cur, A::add(A::sub(E.v, W.v), A::sub(N.v, below.v)), A::add(A::sub(E.w, W.w), A::sub(N.w, below.w)),
               A::add(A::sub(E.d, W.d), A::sub(N.d, below.d)), pm64, fmu64);
    cur = above;
    below = N;
  }
}

// 3D: one block's column, the cells of its tile on the planes k0 .. k1-1.
template <class A, class SUMS>
__device__ __forceinline__ void ndf_column(NdfShared& sh, int x0, int y0, int k0, int k1, const Level<double>& L,
                                           typename A::V gamma, NdfOut<A, SUMS>& out) {
  using V = typename A::V;
  using Cell = NdfCell<A>;
  using Flux = NdfFlux<A>;
  V* const cP = reinterpret_cast<V*>(sh.cell[0]);
  V* const cU = reinterpret_cast<V*>(sh.cell[1]);
  V* const cQ = reinterpret_cast<V*>(sh.cell[2]);
  V* const cS = reinterpret_cast<V*>(sh.cell[3]);
  auto put = [](df64 (&f)[3][kNdfTY * (kNdfTX + 1)], int q, const Flux& F) {
    reinterpret_cast<V*>(f[0])[q] = F.v;
    reinterpret_cast<V*>(f[1])[q] = F.w;
    reinterpret_cast<V*>(f[2])[q] = F.d;
  };
  auto puty = [](df64 (&f)[3][(kNdfTY + 1) * kNdfTX], int q, const Flux& F) {
    reinterpret_cast<V*>(f[0])[q] = F.v;
    reinterpret_cast<V*>(f[1])[q] = F.w;
    reinterpret_cast<V*>(f[2])[q] = F.d;
  };
  auto cell_at = [&](int q) { return Cell{cP[q], cU[q], cQ[q], cS[q]}; };
  auto store_cell = [&](int q, const Cell& c) {
    cP[q] = c.phi;
    cU[q] = c.mu;
    cQ[q] = c.p;
    cS[q] = c.ps;
  };
  const Flux none{A::zero(), A::zero(), A::zero()};
  const int nx = L.nx, ny = L.ny, nz = L.nz, sz = nx * ny;
  const int tx = threadIdx.x % kNdfTX, ty = threadIdx.x / kNdfTX;
  const int i = x0 + tx, j = y0 + ty, q = (tx + 1) + kNdfSW * (ty + 1);
  const bool in = i < nx && j < ny;
  const int c2 = in ? i + nx * j : 0;  // the cell in its plane
  auto load = [&](int c) { return Cell{A::from(L.phi[c]), A::from(L.mu[c]), A::from(L.p[c]), A::from(L.phis[c])}; };
  // ring cells: the columns left and right of the tile, the rows below and above
  const int t = threadIdx.x;
  const int rx = t < kNdfTY ? -1 : t < 2 * kNdfTY ? kNdfTX : (t - 2 * kNdfTY) % kNdfTX;
  const int ry = t < 2 * kNdfTY ? t % kNdfTY : t < 2 * kNdfTY + kNdfTX ? -1 : kNdfTY;
  const bool ring = t < kNdfRing && x0 + rx >= 0 && x0 + rx < nx && y0 + ry >= 0 && y0 + ry < ny;
  const int rq = (rx + 1) + kNdfSW * (ry + 1), rc = ring ? (x0 + rx) + nx * (y0 + ry) : 0;
  // the faces right of the tile's last column and above its last row
  const bool extra = t < kNdfTX + kNdfTY;
  const int ex = t < kNdfTX ? t : kNdfTX - 1, ey = t < kNdfTX ? kNdfTY - 1 : t - kNdfTX;
  const int eq = (ex + 1) + kNdfSW * (ey + 1);
  const bool ein = extra && (t < kNdfTX ? x0 + ex < nx && y0 + kNdfTY < ny : x0 + kNdfTX < nx && y0 + ey < ny);

  Cell cur{A::zero(), A::zero(), A::zero(), A::zero()};
  Flux zlow = none;
  if (in) {
    cur = load(c2 + sz * k0);
    if (k0 > 0) zlow = ndf_face<A>(load(c2 + sz * (k0 - 1)), cur, gamma);
    store_cell(q, cur);
  }
  if (ring) store_cell(rq, load(rc + sz * k0));
  for (int k = k0; k < k1; ++k) {
    __syncthreads();
    const int c = c2 + sz * k;
    double nxt[4], rng[4], pm64 = 0.0, fmu64 = 0.0;  // the next plane's cells, loaded before they are needed
    const bool up = k + 1 < nz;
    if (in) {
      pm64 = L.phim[c];
      fmu64 = L.fmu[c];
      if (up) {
        nxt[0] = L.phi[c + sz];
        nxt[1] = L.mu[c + sz];
        nxt[2] = L.p[c + sz];
        nxt[3] = L.phis[c + sz];
      }
    }
    const bool more = k + 1 < k1;
    if (ring && more) {
      const int r = rc + sz * (k + 1);
      rng[0] = L.phi[r];
      rng[1] = L.mu[r];
      rng[2] = L.p[r];
      rng[3] = L.phis[r];
    }
    const Flux W = in && i > 0 ? ndf_face<A>(cell_at(q - 1), cur, gamma) : none;
    const Flux S = in && j > 0 ? ndf_face<A>(cell_at(q - kNdfSW), cur, gamma) : none;
    put(sh.fx, tx + (kNdfTX + 1) * ty, W);
    puty(sh.fy, tx + kNdfTX * ty, S);
    if (extra) {
      const Flux E = ein ? ndf_face<A>(cell_at(eq), cell_at(t < kNdfTX ? eq + kNdfSW : eq + 1), gamma) : none;
      if (t < kNdfTX) puty(sh.fy, t + kNdfTX * kNdfTY, E);
      else put(sh.fx, kNdfTX + (kNdfTX + 1) * ey, E);
    }
    Cell above{A::zero(), A::zero(), A::zero(), A::zero()};
    Flux zup = none;
    if (in && up) {
      above = Cell{A::from(nxt[0]), A::from(nxt[1]), A::from(nxt[2]), A::from(nxt[3])};
      zup = ndf_face<A>(cur, above, gamma);
    }
    __syncthreads();
    if (in) {
      auto fx = [&](int m) { return reinterpret_cast<const V*>(sh.fx[m])[tx + 1 + (kNdfTX + 1) * ty]; };
      auto fy = [&](int m) { return reinterpret_cast<const V*>(sh.fy[m])[tx + kNdfTX * (ty + 1)]; };
      V sv = A::add(A::sub(fx(0), W.v), A::sub(fy(0), S.v));
      V sw = A::add(A::sub(fx(1), W.w), A::sub(fy(1), S.w));
      V sd = A::add(A::sub(fx(2), W.d), A::sub(fy(2), S.d));
      sv = A::add(sv, A::sub(zup.v, zlow.v));
      sw = A::add(sw, A::sub(zup.w, zlow.w));
      sd = A::add(sd, A::sub(zup.d, zlow.d));
      out.cell(c, cur, sv, sw, sd, pm64, fmu64);
    }
    if (more) {
      if (in) store_cell(q, above);
      if (ring) store_cell(rq, Cell{A::from(rng[0]), A::from(rng[1]), A::from(rng[2]), A::from(rng[3])});
      cur = above;
      zlow = zup;
    }
  }
}

// bx: the block's index among the run's nbx blocks (x-tiles fastest, then
// y-tiles, then the chunks of planes; in 2D strips, then runs of rows).  Returns
// true in the run's last block (which took the loop decision).
template <int DIM, int MODE>
__device__ __forceinline__ bool norm_mixed_df_body(int bx, int nbx, const Level<double>& L, const DfCoefs& K,
                                                   const Coefs<double>& K64, int f64_per8, const Level<float>& G,
                                                   double* partials, DevState* st, cudaGraphConditionalHandle cond,
                                                   int mode, int use_cond) {
  __shared__ __align__(16) unsigned char raw[DIM == 3 ? sizeof(NdfShared) : 16];
  __shared__ bool last;
  const int gx = ndf_blocks_x(L.nx);
  const int rest = bx / gx, x0 = (bx - rest * gx) * kNdfTX;
  auto residual = [&](auto arith, auto& sums, auto sih2, auto ih2, auto e34ih2, auto gamma) {
    using A = decltype(arith);
    NdfOut<A, std::remove_reference_t<decltype(sums)>> out{G, sih2, ih2, e34ih2, K.s, K64.s, sums};
    if constexpr (DIM == 2) {
      const int rows = ndf_rows(L.nx, L.ny), j0 = (rest * (kNdfTX * kNdfTY / 32) + (threadIdx.x >> 5)) * rows;
      ndf_strip<A>(x0, j0, min(j0 + rows, L.ny), L, gamma, out);
    } else {
      const int gy = ndf_blocks_y(L.ny), chunk = rest / gy;
      const int planes = ndf_planes(L.nx, L.ny, L.nz), k0 = chunk * planes;
      ndf_column<A>(reinterpret_cast<NdfShared&>(raw), x0, (rest - chunk * gy) * kNdfTY, k0, min(k0 + planes, L.nz), L, gamma, out);
    }
  };
  double out[3];
  if constexpr (MODE == kNdfF64) {
    NdfSums64 sums;
    residual(NdfDouble{}, sums, L.sih2, L.ih2, L.e34ih2, K64.gamma);
    sums.finish(out);
  } else {
    NdfSums32 sums;
    if (MODE == kNdfShare && (bx & 7) < f64_per8)
      residual(NdfDouble{}, sums, L.sih2, L.ih2, L.e34ih2, K64.gamma);
    else
      residual(NdfSingle{}, sums, K.sih2, K.ih2, K.e34ih2, K.gamma);
    sums.finish(out);
  }
  if (threadIdx.x == 0) {
    partials[3 * bx] = out[0];
    partials[3 * bx + 1] = out[1];
    partials[3 * bx + 2] = out[2];
    __threadfence();
    last = atomicAdd(&st->ticket, 1u) == nbx - 1;
  }
  __syncthreads();
  if (!last) return false;
  __threadfence();
  norm_finish(partials, nbx, L.ncell, st, cond, mode, use_cond);
  return true;
}

template <int DIM, int MODE>
__global__ void __launch_bounds__(kNdfTX * kNdfTY, DIM == 3 ? 3 : 4) k_norm_mixed_df(const __grid_constant__ Level<double> L,
                                                                 DfCoefs K, Coefs<double> K64, int f64_per8,
                                                                 const __grid_constant__ Level<float> G,
                                                                 double* partials, DevState* st,
                                                                 cudaGraphConditionalHandle cond, int mode,
                                                                 int use_cond) {
  pdl_enter();
  norm_mixed_df_body<DIM, MODE>(blockIdx.x, gridDim.x, L, K, K64, f64_per8, G, partials, st, cond, mode, use_cond);
}

}  // namespace chhs_dev
