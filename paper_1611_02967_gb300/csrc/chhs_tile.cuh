// chhs_tile.cuh -- several smoothing passes fused per tile (2D, single
// precision, correction form), a thread per 2 x 2 cells.
//
// One block takes a tile of a level and a halo around it, a thread holds 2 x 2
// cells of it in registers -- state, right-hand sides, the face values a_f of
// phi*, the smoother's constants -- and runs npass red-black colour passes.
// Only (phi, mu, p) of the cells passes through shared memory, so that a pass
// is: read the four neighbour cells that other threads own, update the two
// cells of the colour (they only couple to the thread's other two and to those
// four), store them, block barrier.  Pass k (k = 1 .. npass) leaves the cells
// within halo - k of the tile exactly as npass grid-wide colour passes would
// (cells of a colour are updated from the other colour's previous values either
// way); the cells further out are given up.  The price is the recomputed halo.
//
// Optional steps fused around the passes:
//   prolong  -- on load, u += P(u_c - u_c^0) (the FAS correction from the
//               next coarser level, piecewise constant: one value per thread);
//   rhs      -- before the first pass, f += N(u), completing the FAS
//               right-hand side R r + N_c(R u) (the tile's u still equals R u);
//   restrict -- after the passes (one more cell of halo), the residual summed
//               over the thread's 2 x 2 cells and its mean: u_c = u_c^0 = R u,
//               f_c = R r, phi_b,c = R phi_b.  The fluxes of the faces inside
//               the 2 x 2 cells cancel in that sum and are not formed.
//
// N is evaluated from face differences (d = neighbour - cell): with w = dp +
// gamma a dmu and v = dmu + a w (= M dmu + a dp),
//   N1 = phi - s/h^2 sum v,  N3 = -1/h^2 sum w,  N2 = mu - chi + (3/4) eps^2/h^2 sum dphi.
// A face on the boundary has the cell itself as its neighbour (a mirrored copy
// in the shared-memory slot outside the domain), so all its differences vanish.
//
// What bounds it: latency -- on small levels the load, the passes' block
// barriers and the update's dependent chain, on large ones too: 127 registers
// leave one block of 16 warps per SM, which issues 44 % of the time (ncu,
// 2048^2, with seven instructions per face: 67 M warp instructions, global loads
// the largest stall; five per face since, tile_face).  Two blocks
// at 64 or three at 85 registers spill or cut smaller tiles and are slower
// (2048^2 step 4.77 ms, 5.88 and 5.58).  Blocks that stay and copy the next
// tile's fields asynchronously during the passes sit at the register limit and
// gave 0.86 to 1.03 times that speed as the compiler scheduled them (512^2
// 0.99); L2 prefetches of a tile a wave ahead 0.95.
// One cell per thread with all fields in shared memory and the coefficients
// recomputed in every pass took twice the instructions; its 512^2 step 835 us
// against 683, 640 x 384 1.12 -> 0.94 ms, batch of 24 15.4 -> 14.2 ms.
//
// A tile reads its halo from global memory while other tiles of the same
// launch write their results, so a launch never writes the arrays it reads:
// the pre-smoothing launch reads (phi, mu, p) and f and writes the second
// copy (phi2, mu2, p2) and the completed right-hand side (fc); the
// post-smoothing launch reads those and writes (phi, mu, p).  (Blocks of a
// launch are not all resident at once when other work shares the GPU.)
#pragma once
#include "chhs_kernels.cuh"

namespace chhs_dev {

constexpr int kTileW = 32, kTileH = 16;  // tile of the batched launches
constexpr int kTileThreads = 512;        // most threads of a block (2 x 2 cells each, halo included)
constexpr int kTileMaxPasses = 8;        // more colour passes are split over several launches

// Shared memory of the limit on sweep counts (chhs_create): a tile of tw x th
// with its halo in nine shared fields, the size up to which sweep counts are
// accepted.
__host__ __device__ inline size_t tile_limit_bytes(int halo, int tw, int th) {
  return (size_t)(tw + 2 * halo) * (th + 2 * halo) * 9 * sizeof(float);
}

// A tile launch's shape: interior tw x th (even), halo in 2 x 2 blocks hb,
// threads bx by by (one per 2 x 2 cells) rounded up to whole warps.
struct TileShape {
  int tw, th, hb;
  __host__ __device__ int bx() const { return tw / 2 + 2 * hb; }
  __host__ __device__ int by() const { return th / 2 + 2 * hb; }
  __host__ __device__ int threads() const { return (bx() * by() + 31) / 32 * 32; }
  __host__ __device__ size_t smem() const { return (size_t)bx() * by() * 4 * sizeof(float4); }
};

// The shape for npass passes (and the residual, restrict_out): the asked
// interior, at least 16 x 16 (512^2 step with 16 x 16 tiles below the finest
// level 669 us, 16 x 8 683, 8 x 8 698), its longer side halved until the block
// has room for the halo.  Shapes cut the passes into blocks and change no
// result.  On the finest level 32 x 32 is best (2048^2: 147 us a launch, 32 x
// 16 165, 16 x 16 178): its halo makes 1.9 threads per 2 x 2 cells of it
// against 2.4 and 3.1.
__host__ __device__ inline TileShape tile_shape(int tw, int th, int npass, int restrict_out) {
  TileShape s{tw > 16 ? tw : 16, th > 16 ? th : 16, (npass + (restrict_out ? 1 : 0) + 1) / 2};
  while (s.threads() > kTileThreads && (s.tw > 2 || s.th > 2)) {
    if (s.tw >= s.th) s.tw = s.tw / 4 * 2 > 2 ? s.tw / 4 * 2 : 2;
    else s.th = s.th / 4 * 2 > 2 ? s.th / 4 * 2 : 2;
  }
  return s;
}

// Where a tile launch writes its interior: (phi, mu, p) and, with rhs, the
// completed right-hand side.  On the finest level of the mixed form the
// post-smoothing launch instead adds the finished correction to the
// double-precision iterate (phi64, mu64, p64 non-null): u <- u + e.
struct TileOut {
  float *phi, *mu, *p, *f1, *f2, *f3;
  double *phi64, *mu64, *p64;
};

struct TileCell {
  float phi, mu, p;
};

// (mu, p) of a cell and (sum v, sum w) of its faces as pairs: one instruction
// subtracts or adds both, rounding each as the plain one does (8 of a cell
// update's ~75 instructions fewer; 512^2 step 587 -> 580 us, 640 x 384
// -1.2 %, 2048^2 -0.7 %, the same bits).
using TilePair = unsigned long long;
__device__ __forceinline__ TilePair tile_pack(float x, float y) {
  TilePair r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ float2 tile_unpack(TilePair a) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a));
  return r;
}
__device__ __forceinline__ TilePair tile_sub2(TilePair a, TilePair b) {
  TilePair r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ TilePair tile_add2(TilePair a, TilePair b) {
  TilePair r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// Adds the fluxes of the face to neighbour n (coefficient a) of cell c to s = (sum v, sum w).
__device__ __forceinline__ void tile_face(const TileCell& c, const TileCell& n, float a, float gamma, TilePair& s) {
  const float2 d = tile_unpack(tile_sub2(tile_pack(n.mu, n.p), tile_pack(c.mu, c.p)));
  const float w = fmaf(gamma, __fmul_rn(a, d.x), d.y);
  s = tile_add2(s, tile_pack(fmaf(a, w, d.x), w));
}

// (LV: a Level<float>, or another struct with its scalars ih2, h2, sih2, e34ih2.)
//
// A cell's constants: chi(phi_b + e, phi^m) - chi(phi_b, phi^m) = e (q0 + e (q1 + e/4));
// x = sum a / n_c, hn = h^2 / n_c, em = (3/4) eps^2 n_c / h^2.
struct TileConst {
  float q0, q1, Ae, x, hn, em;
};

__device__ __forceinline__ float tile_chi(float e, const TileConst& k) {
  return __fmul_rn(e, fmaf(e, fmaf(0.25f, e, k.q1), k.q0));
}

// One Newton step of cell c (the update of cell_update: the pressure row
// eliminated) with neighbours n0..n3 across faces a0..a3.
template <class LV>
__device__ __forceinline__ void tile_update(TileCell& c, const TileCell& n0, const TileCell& n1, const TileCell& n2,
                                            const TileCell& n3, float a0, float a1, float a2, float a3, float f1,
                                            float f2, float f3, const TileConst& k, const LV& L,
                                            const Coefs<float>& K) {
  TilePair sums = 0;
  tile_face(c, n0, a0, K.gamma, sums);
  tile_face(c, n1, a1, K.gamma, sums);
  tile_face(c, n2, a2, K.gamma, sums);
  tile_face(c, n3, a3, K.gamma, sums);
  const float sv = tile_unpack(sums).x, sw = tile_unpack(sums).y;
  const float sd = fmaf(-4.f, c.phi, (n0.phi + n1.phi) + (n2.phi + n3.phi));
  const float R1 = fmaf(L.sih2, sv, f1 - c.phi);
  const float R2 = fmaf(-L.e34ih2, sd, (f2 - c.mu) + tile_chi(c.phi, k));
  const float R3 = fmaf(L.ih2, sw, f3);
  const float B = fmaf(c.phi, fmaf(0.75f, c.phi, k.q1 + k.q1), k.q0 + k.em);
  const float num = fmaf(-__fmul_rn(K.s, k.x), R3, fmaf(-k.Ae, R2, R1));
  const float dphi = __fmul_rn(num, rcp_approx(fmaf(k.Ae, B, 1.f)));
  const float dmu = fmaf(B, dphi, R2);
  c.phi += dphi;
  c.mu += dmu;
  c.p += fmaf(-__fmul_rn(K.gamma, k.x), dmu, __fmul_rn(k.hn, R3));
}

__device__ __forceinline__ void tile_quad(TileConst& k, float pm, float pb) {
  k.q0 = __fmul_rn(0.25f, fmaf(pm, pm, __fmul_rn(pb, fmaf(3.f, pb, pm + pm))));
  k.q1 = __fmul_rn(0.25f, fmaf(3.f, pb, pm));
}

// The constants of a cell from phi^m, phi_b, its face values and its number of
// interior faces.
template <class LV>
__device__ __forceinline__ TileConst tile_constants(const LV& L, const Coefs<float>& K, float pm, float pb,
                                                    float a0, float a1, float a2, float a3, int faces) {
  TileConst k;
  const float n = (float)faces, im = rcp_approx(n), sa = (a0 + a1) + (a2 + a3);
  const float sM = fmaf(K.gamma, fmaf(a0, a0, fmaf(a1, a1, fmaf(a2, a2, __fmul_rn(a3, a3)))), n);
  k.x = __fmul_rn(sa, im);
  k.Ae = __fmul_rn(L.sih2, fmaf(-__fmul_rn(K.gamma, sa), k.x, sM));
  k.hn = __fmul_rn(L.h2, im);
  k.em = __fmul_rn(L.e34ih2, n);
  tile_quad(k, pm, pb);
  return k;
}

// f += N at cell c with neighbours n0..n3.
template <class LV>
__device__ __forceinline__ void tile_add_N(float& f1, float& f2, float& f3, const TileCell& c, const TileCell& n0,
                                           const TileCell& n1, const TileCell& n2, const TileCell& n3, float a0,
                                           float a1, float a2, float a3, const TileConst& k, const LV& L,
                                           const Coefs<float>& K) {
  TilePair sums = 0;
  tile_face(c, n0, a0, K.gamma, sums);
  tile_face(c, n1, a1, K.gamma, sums);
  tile_face(c, n2, a2, K.gamma, sums);
  tile_face(c, n3, a3, K.gamma, sums);
  const float sv = tile_unpack(sums).x, sw = tile_unpack(sums).y;
  const float sd = fmaf(-4.f, c.phi, (n0.phi + n1.phi) + (n2.phi + n3.phi));
  f1 += fmaf(-L.sih2, sv, c.phi);
  f2 += fmaf(L.e34ih2, sd, c.mu - tile_chi(c.phi, k));
  f3 = fmaf(-L.ih2, sw, f3);
}

// The neighbours outside a block of 2 x 2 cells A, B (row below), C, D.
struct TileOuter {
  TileCell w0, w2, e1, e3, s0, s1, n2, n3;
};

// The mean residual of the block: the fluxes of the faces inside it cancel.
template <class LV>
__device__ __forceinline__ void tile_block_residual(const TileCell& A, const TileCell& B, const TileCell& C,
                                                    const TileCell& D, const TileOuter& o, float aw0, float aw2,
                                                    float ae1, float ae3, float as0, float as1, float an2, float an3,
                                                    const float (&f1)[4], const float (&f2)[4], const float (&f3)[4],
                                                    const TileConst& kA, const TileConst& kB, const TileConst& kC,
                                                    const TileConst& kD, const LV& L,
                                                    const Coefs<float>& K, float& r1, float& r2, float& r3) {
  TilePair sums = 0;
  tile_face(A, o.w0, aw0, K.gamma, sums);
  tile_face(C, o.w2, aw2, K.gamma, sums);
  tile_face(B, o.e1, ae1, K.gamma, sums);
  tile_face(D, o.e3, ae3, K.gamma, sums);
  tile_face(A, o.s0, as0, K.gamma, sums);
  tile_face(B, o.s1, as1, K.gamma, sums);
  tile_face(C, o.n2, an2, K.gamma, sums);
  tile_face(D, o.n3, an3, K.gamma, sums);
  const float sv = tile_unpack(sums).x, sw = tile_unpack(sums).y;
  const float sd = ((o.w0.phi - A.phi) + (o.w2.phi - C.phi)) + ((o.e1.phi - B.phi) + (o.e3.phi - D.phi)) +
                   (((o.s0.phi - A.phi) + (o.s1.phi - B.phi)) + ((o.n2.phi - C.phi) + (o.n3.phi - D.phi)));
  const float m1 = ((f1[0] - A.phi) + (f1[1] - B.phi)) + ((f1[2] - C.phi) + (f1[3] - D.phi));
  const float m2 = (((f2[0] - A.mu) + tile_chi(A.phi, kA)) + ((f2[1] - B.mu) + tile_chi(B.phi, kB))) +
                   (((f2[2] - C.mu) + tile_chi(C.phi, kC)) + ((f2[3] - D.mu) + tile_chi(D.phi, kD)));
  r1 = 0.25f * fmaf(L.sih2, sv, m1);
  r2 = 0.25f * fmaf(-L.e34ih2, sd, m2);
  r3 = 0.25f * fmaf(L.ih2, sw, (f3[0] + f3[1]) + (f3[2] + f3[3]));
}

__device__ __forceinline__ void tile_body(int bx, int by, const Level<float>& L, const Level<float>& Cl,
                                          const Coefs<float>& K, int npass, int rhs, int prolong, int restrict_out,
                                          const TileOut& out, const TileShape& T) {
  extern __shared__ __align__(16) unsigned char tile_smem[];
  const int BX = T.bx(), NB = BX * T.by(), t = threadIdx.x;
  float4* const sA = reinterpret_cast<float4*>(tile_smem);  // cells (0,0) of the 2 x 2 blocks: mu, p, phi, phi*
  float4* const sB = sA + NB;                               // (1,0)
  float4* const sC = sB + NB;                               // (0,1)
  float4* const sD = sC + NB;                               // (1,1)
  const int ty = small_div(t, __frcp_rn((float)BX)), tx = t - ty * BX;
  const int hx = L.nx >> 1, hy = L.ny >> 1;                       // 2 x 2 blocks of the level
  const int I = bx * (T.tw >> 1) - T.hb + tx, J = by * (T.th >> 1) - T.hb + ty;
  const bool in = t < NB && I >= 0 && J >= 0 && I < hx && J < hy;
  // distance of the block from the tile, in blocks
  const int ddx = max(T.hb - tx, tx - (BX - 1 - T.hb)), ddy = max(T.hb - ty, ty - (T.by() - 1 - T.hb));
  const int dist = max(max(ddx, ddy), 0);
  const bool inner = in && dist == 0;
  // neighbour slots (the thread's own at the region's rim, whose cells are given up)
  const int iW = tx > 0 ? t - 1 : t, iE = tx < BX - 1 ? t + 1 : t;
  const int iS = ty > 0 ? t - BX : t, iN = ty < T.by() - 1 ? t + BX : t;
  // boundary faces whose mirrored cell lives in a slot outside the domain
  const bool eW = in && I == 0, eE = in && I == hx - 1, eS = in && J == 0, eN = in && J == hy - 1;
  const bool gW = eW && iW != t, gE = eE && iE != t, gS = eS && iS != t, gN = eN && iN != t;
  const bool ghosts = gW || gE || gS || gN;
  const int c0 = in ? 2 * I + L.nx * 2 * J : 0, c1 = c0 + L.nx;

  TileCell A{0.f, 0.f, 0.f}, B = A, C = A, D = A;
  float f1[4], f2[4], f3[4], pm[4], pb[4], ps[4];  // of A, B, C, D
  auto ld = [&](const float* a, float (&v)[4]) {
    const float2 lo = *reinterpret_cast<const float2*>(a + c0), hi = *reinterpret_cast<const float2*>(a + c1);
    v[0] = lo.x;
    v[1] = lo.y;
    v[2] = hi.x;
    v[3] = hi.y;
  };
  if (in) {
    float u[4], v[4], w[4];
    ld(L.phi, u);
    ld(L.mu, v);
    ld(L.p, w);
    ld(L.phis, ps);
    ld(L.fphi, f1);
    ld(L.fmu, f2);
    ld(L.fp, f3);
    ld(L.phim, pm);
    ld(L.phib, pb);
    if (prolong) {
      const int q = I + Cl.nx * J;
      const float dphi = Cl.phi[q] - Cl.phi0[q], dmu = Cl.mu[q] - Cl.mu0[q], dp = Cl.p[q] - Cl.p0[q];
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        u[m] += dphi;
        v[m] += dmu;
        w[m] += dp;
      }
    }
    A = TileCell{u[0], v[0], w[0]};
    B = TileCell{u[1], v[1], w[1]};
    C = TileCell{u[2], v[2], w[2]};
    D = TileCell{u[3], v[3], w[3]};
  }
  auto put = [](float4* s, int q, const TileCell& c) {
    s[q].x = c.mu;
    s[q].y = c.p;
    s[q].z = c.phi;
  };
  auto get = [](const float4* s, int q) {
    const float4 v = s[q];
    return TileCell{v.z, v.x, v.y};
  };
  // the mirrored copies of the red (A, D) or black (B, C) cells
  auto mirror_red = [&]() {
    if (gW) put(sB, iW, A);
    if (gS) put(sC, iS, A);
    if (gE) put(sC, iE, D);
    if (gN) put(sB, iN, D);
  };
  auto mirror_black = [&]() {
    if (gE) put(sA, iE, B);
    if (gS) put(sD, iS, B);
    if (gW) put(sD, iW, C);
    if (gN) put(sA, iN, C);
  };
  if (in) {
    sA[t] = make_float4(A.mu, A.p, A.phi, ps[0]);
    sB[t] = make_float4(B.mu, B.p, B.phi, ps[1]);
    sC[t] = make_float4(C.mu, C.p, C.phi, ps[2]);
    sD[t] = make_float4(D.mu, D.p, D.phi, ps[3]);
    if (ghosts) {
      mirror_red();
      mirror_black();
    }
  }
  __syncthreads();
  // face values a_f: inside the block AB, CD, AC, BD; outside AW, CW, BE, DE, AS, BS, CN, DN
  float aAB = 0.f, aCD = 0.f, aAC = 0.f, aBD = 0.f, aAW = 0.f, aCW = 0.f, aBE = 0.f, aDE = 0.f, aAS = 0.f, aBS = 0.f,
        aCN = 0.f, aDN = 0.f;
  TileConst kA{}, kB{}, kC{}, kD{};
  if (in) {
    auto avg = [](float x, float y) { return 0.5f * (x + y); };
    aAB = avg(ps[0], ps[1]);
    aCD = avg(ps[2], ps[3]);
    aAC = avg(ps[0], ps[2]);
    aBD = avg(ps[1], ps[3]);
    // zero on boundary faces
    aAW = eW ? 0.f : avg(ps[0], sB[iW].w);
    aCW = eW ? 0.f : avg(ps[2], sD[iW].w);
    aBE = eE ? 0.f : avg(ps[1], sA[iE].w);
    aDE = eE ? 0.f : avg(ps[3], sC[iE].w);
    aAS = eS ? 0.f : avg(ps[0], sC[iS].w);
    aBS = eS ? 0.f : avg(ps[1], sD[iS].w);
    aCN = eN ? 0.f : avg(ps[2], sA[iN].w);
    aDN = eN ? 0.f : avg(ps[3], sB[iN].w);
    const int w = eW ? 0 : 1, e = eE ? 0 : 1, s = eS ? 0 : 1, n = eN ? 0 : 1;
    kA = tile_constants(L, K, pm[0], pb[0], aAB, aAC, aAW, aAS, 2 + w + s);
    kB = tile_constants(L, K, pm[1], pb[1], aAB, aBD, aBE, aBS, 2 + e + s);
    kC = tile_constants(L, K, pm[2], pb[2], aCD, aAC, aCW, aCN, 2 + w + n);
    kD = tile_constants(L, K, pm[3], pb[3], aCD, aBD, aDE, aDN, 2 + e + n);
  }

  if (rhs && in) {  // f += N(R u)
    const TileCell AW = get(sB, iW), CW = get(sD, iW), BE = get(sA, iE), DE = get(sC, iE);
    const TileCell AS = get(sC, iS), BS = get(sD, iS), CN = get(sA, iN), DN = get(sB, iN);
    tile_add_N(f1[0], f2[0], f3[0], A, B, C, AW, AS, aAB, aAC, aAW, aAS, kA, L, K);
    tile_add_N(f1[1], f2[1], f3[1], B, A, D, BE, BS, aAB, aBD, aBE, aBS, kB, L, K);
    tile_add_N(f1[2], f2[2], f3[2], C, D, A, CW, CN, aCD, aAC, aCW, aCN, kC, L, K);
    tile_add_N(f1[3], f2[3], f3[3], D, C, B, DE, DN, aCD, aBD, aDE, aDN, kD, L, K);
  }
  // the pass writes what the right-hand side's threads may still read
  if (rhs) __syncthreads();

  for (int k = 1; k <= npass; k += 2) {
    // a block takes part while a cell of it is still needed (within npass - k
    // of the tile, one more for the residual)
    const int need = npass - k + (restrict_out ? 1 : 0);
    if (in && 2 * dist - 1 <= need) {
      tile_update(A, B, C, get(sB, iW), get(sC, iS), aAB, aAC, aAW, aAS, f1[0], f2[0], f3[0], kA, L, K);
      tile_update(D, C, B, get(sC, iE), get(sB, iN), aCD, aBD, aDE, aDN, f1[3], f2[3], f3[3], kD, L, K);
      put(sA, t, A);
      put(sD, t, D);
      if (ghosts) mirror_red();
    }
    __syncthreads();
    if (k == npass) break;
    if (in && 2 * dist - 1 <= need - 1) {
      tile_update(B, A, D, get(sA, iE), get(sD, iS), aAB, aBD, aBE, aBS, f1[1], f2[1], f3[1], kB, L, K);
      tile_update(C, D, A, get(sD, iW), get(sA, iN), aCD, aAC, aCW, aCN, f1[2], f2[2], f3[2], kC, L, K);
      put(sB, t, B);
      put(sC, t, C);
      if (ghosts) mirror_black();
    }
    __syncthreads();
  }

  if (!inner) return;
  auto st = [&](float* a, float x0, float x1, float x2, float x3) {
    *reinterpret_cast<float2*>(a + c0) = make_float2(x0, x1);
    *reinterpret_cast<float2*>(a + c1) = make_float2(x2, x3);
  };
  if (out.phi64) {
    auto upd = [&](double* a, float x0, float x1, float x2, float x3) {
      double2* lo = reinterpret_cast<double2*>(a + c0);
      double2* hi = reinterpret_cast<double2*>(a + c1);
      double2 l = *lo, h = *hi;
      l.x += (double)x0;
      l.y += (double)x1;
      h.x += (double)x2;
      h.y += (double)x3;
      *lo = l;
      *hi = h;
    };
    upd(out.phi64, A.phi, B.phi, C.phi, D.phi);
    upd(out.mu64, A.mu, B.mu, C.mu, D.mu);
    upd(out.p64, A.p, B.p, C.p, D.p);
  } else {
    st(out.phi, A.phi, B.phi, C.phi, D.phi);
    st(out.mu, A.mu, B.mu, C.mu, D.mu);
    st(out.p, A.p, B.p, C.p, D.p);
  }
  if (rhs) {
    st(out.f1, f1[0], f1[1], f1[2], f1[3]);
    st(out.f2, f2[0], f2[1], f2[2], f2[3]);
    st(out.f3, f3[0], f3[1], f3[2], f3[3]);
  }
  if (restrict_out) {
    const TileOuter o{get(sB, iW), get(sD, iW), get(sA, iE), get(sC, iE), get(sC, iS), get(sD, iS), get(sA, iN), get(sB, iN)};
    float r1, r2, r3;
    tile_block_residual(A, B, C, D, o, aAW, aCW, aBE, aDE, aAS, aBS, aCN, aDN, f1, f2, f3, kA, kB, kC, kD, L, K, r1, r2,
                        r3);
    const float uphi = (A.phi + B.phi) + (C.phi + D.phi), umu = (A.mu + B.mu) + (C.mu + D.mu);
    const float up = (A.p + B.p) + (C.p + D.p);
    const int q = I + Cl.nx * J;
    Cl.fphi[q] = r1;
    Cl.fmu[q] = r2;
    Cl.fp[q] = r3;
    Cl.phi[q] = Cl.phi0[q] = 0.25f * uphi;
    Cl.mu[q] = Cl.mu0[q] = 0.25f * umu;
    Cl.p[q] = Cl.p0[q] = 0.25f * up;
    Cl.phib[q] = 0.25f * ((pb[0] + pb[1]) + (pb[2] + pb[3]));
  }
}

// gate (nullable): the run's loop flag; the launch does nothing once the
// run has stopped iterating (a run of a batch that has converged).
static __global__ void __launch_bounds__(kTileThreads) k_tile(const __grid_constant__ Level<float> L,
                                                             const __grid_constant__ Level<float> Cl, Coefs<float> K,
                                                             int npass, int rhs, int prolong, int restrict_out,
                                                             const __grid_constant__ TileOut out, const int* gate,
                                                             TileShape T) {
  pdl_enter();
  if (gate && *(volatile const int*)gate == 0) return;
  tile_body(blockIdx.x, blockIdx.y, L, Cl, K, npass, rhs, prolong, restrict_out, out, T);
}

}  // namespace chhs_dev
