// Energy sub-step of the split step, one warp per strip (Hu & Liu, arXiv
// 1812.10375, Eqs. 17-19, 22-27): one RK4 sub-step (Eq. 18, dt = 1/N) of the energy
// equation with finite-volume harmonic face conductivities, on rho^n and u^n
// held over the sub-steps.
//
// A warp owns a strip of 56 output columns (64 frame columns, two neighbouring
// ones per lane, a 4-column halo on either side recomputed by the neighbouring
// strips) and a segment of L output rows, and walks up the rows once.  At walk
// step r it takes row r, forms the coefficients of Eq. (17) and RK4 stage 1 at
// row r - 1, stage 2 at r - 2, stage 3 at r - 3 and stage 4 (the new temperature)
// at r - 4.  A stage at row y needs the previous stage at rows y - 1 .. y + 1;
// the row y + 1 value was produced earlier in the same walk step.
//
// The arithmetic of a cell is that of the tiled and the two-warp kernels
// (hlb_split.cuh, hlb_energy_walk.cuh), operation by operation and, for a lattice by
// itself, rounding by rounding: both columns of a packed instruction round on their
// own, so its new temperature is the same bit for bit.  A batch sums two
// conductivities with one rounding less in half of its rows (pair_step), so its
// cells agree with a lattice by itself to FP32 rounding only.
//
// Why this shape: the update is bound by instruction issue and by the latency of a
// row's dependent stages, not by memory (20 B per cell).  Two columns per lane make
// most arithmetic instructions packed ones, the neighbouring columns come from two
// shuffles per row and field, shared memory holds the prefetched input rows only,
// and no barrier is needed.  One warp per CTA keeps everything that selects a branch
// or a row uniform, out of the vector registers (384-thread CTAs spilled 1 KB).  The
// loop is unrolled by three, not four: the rings' indices become constants and its
// instructions still fit the cache nearest to a scheduler (four rows: 0.7 warps per
// issue waited for instructions).  Segments of up to 12 rows take the one-row form
// (pair_short in hlb.cu).  Twelve warps per SM instead of eight (168 registers)
// spilled and were slower on one lattice and no faster on the sweep.
// Against the two-warp walk with one column per thread, the kernel alone: 32-domain
// sweep (4.9 M cells, 1,142 segments of 86 rows) 0.066 against 0.079 ms; 14 lattices
// of 400 x 600 0.052 against 0.059; 400 x 400 about 0.009 against 0.052, mostly by its
// shorter segments (walk_rows in hlb.cu).
#pragma once
#include "hlb_pair.cuh"
#include "hlb_split.cuh"

namespace hlb {

constexpr int EPW = 64;      // frame columns of a warp
constexpr int EP_OUT = 56;   // output columns of a strip
constexpr int EP_H = 4;      // x halo
constexpr int EP_U = 3;      // rows per pass of the throughput form's loop
constexpr int EP_TS = 16;    // slots of the rings of input rows (rows t - 4 .. t + 8)
constexpr int EP_PF = 6;     // rows fetched ahead
constexpr int EP_CTAS = 8;   // resident one-warp CTAs per SM (two per scheduler, at most 255 registers)

struct PairShared {
  float T[EP_TS][EPW], rho[EP_TS][EPW], ux[EP_TS][EPW], uy[EP_TS][EPW];
  float2 qf[4][32];    // face conductivity of a wall-flux row
  float2 flux[3][32];  // (hi, lo) of q_bottom, q_interface, q_top per lane
};

// Coefficients of the right-hand side at a row (C_AE .. C_BS of hlb_split.cuh).
struct PairCoef {
  float2 aE, aW, aN, aS, p, q, A, B;
};

// The rows of a field that a stage still needs, by row mod 3: the lane's pair and
// the columns next to it; and what row y's right-hand side has so far.
struct PairWin {
  float2 T[3];
  float w[3], e[3];
  float2 G;  // T(y) - T(y-1), y the newest row
  float2 k;  // the east and west faces of the newest row
  float2 X;  // its latent-heat source
};

// Rings indexed by row mod 3; the loop is unrolled by three so that every index is
// a compile-time constant.
struct PairState {
  PairWin w[4];         // T^n, T1, T2, T3
  PairCoef cf[3];
  float2 acc[3];        // K1 + 2 K2 + 2 K3 of rows r - 1, r - 2, r - 3
  float2 lam, ux, uy;   // row r - 1
  float2 lamS, qS;      // lambda of row r - 2, 1 / (lambda + lambda) of the face above it
  float2 dux[3], suy[3], uyS;  // E - W of u_x and E + W of u_y, u_y of row r - 2
  float2 eh, el;
};

struct PairCtx {
  const float* src0;  // 16-byte pieces of this lane in row 0 (planes 0/1 and 2/3)
  const float* src1;
  const float* T_in;
  const float* rho_n;
  const float* ux_n;
  const float* uy_n;
  float* T_out;
  int lane, gx0, gx1, ys, ye;
  bool own0, own1, last;
};

// Start the copies of rows t .. t + U - 1 (rows above the lattice repeat row
// ny - 1; rows below it are not read) into their slots, as one group.
template <int U, bool VEC>
__device__ __forceinline__ void pair_fetch(const StepArgs& A, const PairCtx& C, PairShared& sm, int t) {
#pragma unroll
  for (int k = 0; k < U; ++k) {
    const int row = t + k;
    if (row < 0) continue;
    const int o = min(row, A.ny - 1) * A.nx, st = row & (EP_TS - 1);
    if constexpr (VEC) {
      const int col = 4 * (C.lane & 15);
      cp_async16(C.lane < 16 ? &sm.T[st][col] : &sm.rho[st][col], C.src0 + o);
      cp_async16(C.lane < 16 ? &sm.ux[st][col] : &sm.uy[st][col], C.src1 + o);
    } else {
      const int i = 2 * C.lane;
      cp_async4(&sm.T[st][i], C.T_in + o + C.gx0);
      cp_async4(&sm.T[st][i + 1], C.T_in + o + C.gx1);
      cp_async4(&sm.rho[st][i], C.rho_n + o + C.gx0);
      cp_async4(&sm.rho[st][i + 1], C.rho_n + o + C.gx1);
      cp_async4(&sm.ux[st][i], C.ux_n + o + C.gx0);
      cp_async4(&sm.ux[st][i + 1], C.ux_n + o + C.gx1);
      cp_async4(&sm.uy[st][i], C.uy_n + o + C.gx0);
      cp_async4(&sm.uy[st][i + 1], C.uy_n + o + C.gx1);
    }
  }
  cp_async_commit();
}

__device__ __forceinline__ float2& pair_slot(float (&ring)[EP_TS][EPW], int row, int lane) {
  return *reinterpret_cast<float2*>(&ring[row & (EP_TS - 1)][2 * lane]);
}

// Latent-heat source As T + Bs s (1 + kappa - kappa s), s = sqrt(T / Tc).
__device__ __forceinline__ float2 pair_source(const StepArgs& A, const PairCoef& c, float2 T) {
  const float2 s = make_float2(sqrt_approx(__fmul_rn(fmaxf(T.x, 0.f), A.invTc)),
                               sqrt_approx(__fmul_rn(fmaxf(T.y, 0.f), A.invTc)));
  return fma2(c.A, T, mul2(mul2(c.B, s), cfma2(s, -A.kappa, __fadd_rn(1.f, A.kappa))));
}

// East and west face terms of a row T with edge columns w, e.
__device__ __forceinline__ float2 pair_ew(const PairCoef& c, float2 T, float w, float e) {
  const float2 dE = make_float2(__fsub_rn(T.y, T.x), __fsub_rn(e, T.y));
  const float2 dW = make_float2(__fsub_rn(w, T.x), __fsub_rn(T.x, T.y));
  return fma2(c.aW, dW, mul2(c.aE, dE));
}

// The newest row v (edges we, ee; ring place N) of field w completes the right-hand
// side of the row below it (place Y, coefficients bN .. bq; place S: the row below
// that).  Gs, Gn: the differences below and above row y.
template <int N, int Y, int S>
__device__ __forceinline__ float2 pair_finish(float2 bN, float2 bS, float2 bp, float2 bq, PairWin& w, float2 k, float2 X,
                                              float2 v, float we, float ee, float2& Gs, float2& Gn) {
  Gs = w.G;
  Gn = sub2(v, w.T[Y]);
  k = fma2(bN, Gn, k);
  k = nfma2(bS, Gs, k);  // T_S - T = -Gs
  k = nfma2(bp, make_float2(__fsub_rn(v.y, w.w[S]), __fsub_rn(ee, w.T[S].x)), k);  // T_NE - T_SW
  k = nfma2(bq, make_float2(__fsub_rn(w.T[S].y, we), __fsub_rn(w.e[S], v.x)), k);  // T_SE - T_NW
  w.G = Gn;
  w.T[N] = v;
  w.w[N] = we;
  w.e[N] = ee;
  return sub2(k, X);
}

// The same for a stage value's newest row v, whose own right-hand side (coefficients
// c) starts here.
template <int N, int Y, int S>
__device__ __forceinline__ float2 pair_advance(const StepArgs& A, float2 bN, float2 bS, float2 bp, float2 bq,
                                               const PairCoef& c, PairWin& w, float2 v, float2& Gs, float2& Gn) {
  float we, ee;
  pair_edges(v, we, ee);
  const float2 k = pair_finish<N, Y, S>(bN, bS, bp, bq, w, w.k, w.X, v, we, ee, Gs, Gn);
  w.X = pair_source(A, c, v);
  w.k = pair_ew(c, v, we, ee);
  return k;
}

// One walk step at row r, the P-th of its group.  BND: some row of the step is
// below the lattice, Dirichlet, a wall-flux row, a top wall or a ghost row
// (pair_bnd).  Every phase runs on every row: rows outside the segment (and the
// first steps' rows) get values that nothing valid reads, and only the store is
// guarded.
template <int P, bool BND, bool VEC, bool BATCH>
__device__ __forceinline__ void pair_step(const StepArgs& A, const PairCtx& C, PairState& S, PairShared& sm, int r) {
  constexpr int I0 = P, I1 = (P + 2) % 3, I2 = (P + 1) % 3;  // ring places of rows r, r - 1, r - 2
  const Geo g = make_geo(A);
  const int ny = A.ny, W = A.W, lane = C.lane;

  float2 T = pair_slot(sm.T, r, lane), lam = cmul2(pair_slot(sm.rho, r, lane), A.cvk);
  float2 ux = pair_slot(sm.ux, r, lane), uy = pair_slot(sm.uy, r, lane);
  if (!BND && r < W) {
    lam = bc2(A.lambda_w);
    ux = uy = bc2(0.f);
  }
  if (BND) {
    const int gr = r < ny ? r : ny - 1;
    if (r < 0 || g.dirichlet_row(gr)) {
      T = bc2(r < 0 ? 0.f : (gr == 0 ? A.T_bottom : A.T_top));
      pair_slot(sm.T, r, lane) = T;
    }
    if (r < 0 || g.solid_row(gr)) {
      lam = bc2(r >= 0 && g.top_wall && gr == ny - 1 ? A.lambda_top : A.lambda_w);
      ux = uy = bc2(0.f);
    }
  }
  // ---- neighbouring columns of row r
  float we, ee;
  pair_edges(ux, we, ee);
  const float2 dux = make_float2(__fsub_rn(ux.y, we), __fsub_rn(ee, ux.x));
  pair_edges(uy, we, ee);
  const float2 suy = make_float2(__fadd_rn(uy.y, we), __fadd_rn(ee, uy.x));

  // ---- coefficients of row y = r - 1 (the ring place of row r - 4, whose aN, p and
  // q the last stage still needs)
  PairCoef& c1 = S.cf[I1];
  const PairCoef &c2 = S.cf[I2], &c3 = S.cf[I0];
  const float2 oN = c1.aN, oS = c1.aS, op = c1.p, oq = c1.q;
  {
    const int y = r - 1;
    const float2 l = S.lam, rho1 = pair_slot(sm.rho, y, lane);
    const bool ysolid = BND ? y < 0 || g.solid_row(y) : y < W;
    // lambda_f / (rho cv) = 2 kd lambda_nb / (lambda + lambda_nb), kd = lambda / (rho cv) of the row
    float kd = A.kd;
    if (ysolid) kd = __fmul_rn(l.x, A.inv_rcv_w);  // a solid row's lambda is uniform
    const float kd2 = __fmul_rn(2.f, kd);
    float lw, le;
    pair_edges(l, lw, le);
    const float2 qN = rcp2(add2(l, lam));
    float2 cE, cW, cN, cS;
    if constexpr (BATCH) {
      // Sums of the row's lambda with a neighbour's: rows 4k and 4k + 1 add the
      // product rho (cv k) unrounded (one multiply-add), the others its rounded
      // value.  The two-warp walk's batch form rounds so (as the compiler contracted
      // its groups of four interior rows, 64 rows to a segment), and a batch here
      // follows it but for single roundings next to those segments' edges: 1 of 4.9 M
      // temperatures of the 32-domain sweep after three steps, 4e-7 of the largest
      // value after 100.  It costs five reciprocals a row, which the other form shares
      // between the columns and rows.
      const int tq = y & ~3;
      const bool fused = !(y & 2) && (tq & 63) && tq >= W + 7 && tq <= ny - 7;
      const float2 sa = fused ? rho1 : l;
      const float sb = fused ? A.cvk : 1.f;
      cE = make_float2(__fmul_rn(__fmul_rn(kd2, l.y), rcp_approx(__fmaf_rn(sa.x, sb, l.y))),
                       __fmul_rn(__fmul_rn(kd2, le), rcp_approx(__fmaf_rn(sa.y, sb, le))));
      cW = make_float2(__fmul_rn(__fmul_rn(kd2, lw), rcp_approx(__fmaf_rn(sa.x, sb, lw))),
                       __fmul_rn(__fmul_rn(kd2, l.x), rcp_approx(__fmaf_rn(sa.y, sb, l.x))));
      cN = mul2(cmul2(lam, kd2), rcp2(cfma2(sa, sb, lam)));
      cS = mul2(cmul2(S.lamS, kd2), rcp2(cfma2(sa, sb, S.lamS)));
    } else {
      const float qm = rcp_approx(__fadd_rn(l.x, l.y));
      cE = make_float2(__fmul_rn(__fmul_rn(kd2, l.y), qm),
                       __fmul_rn(__fmul_rn(kd2, le), rcp_approx(__fadd_rn(l.y, le))));
      cW = make_float2(__fmul_rn(__fmul_rn(kd2, lw), rcp_approx(__fadd_rn(l.x, lw))),
                       __fmul_rn(__fmul_rn(kd2, l.x), qm));
      cN = mul2(cmul2(lam, kd2), qN);
      cS = mul2(cmul2(S.lamS, kd2), S.qS);
    }
    c1.aE = cfma2(S.ux, -1.f / 3.f, cE);
    c1.aW = cfma2(S.ux, 1.f / 3.f, cW);
    c1.aN = cfma2(S.uy, -1.f / 3.f, cN);
    c1.aS = cfma2(S.uy, 1.f / 3.f, cS);
    c1.p = cmul2(add2(S.ux, S.uy), 1.f / 12.f);
    c1.q = cmul2(sub2(S.ux, S.uy), 1.f / 12.f);
    // div u (Eq. 19)
    float2 dv = cmul2(add2(dux, S.dux[I2]), 1.f / 12.f);
    dv = cfma2(S.dux[I1], 1.f / 3.f, dv);
    dv = cfma2(sub2(uy, S.uyS), 1.f / 3.f, dv);
    dv = cfma2(sub2(suy, S.suy[I2]), 1.f / 12.f, dv);
    float2 rh = rho1;
    if (ysolid) dv = rh = bc2(0.f);  // no latent heat in the heater
    const float2 br = cmul2(rh, A.b);
    const float2 om = make_float2(__fsub_rn(1.f, br.x), __fsub_rn(1.f, br.y));
    const float2 tm = make_float2(__fsub_rn(2.f, br.x), __fsub_rn(2.f, br.y));
    const float2 den = make_float2(__fmaf_rn(br.x, tm.x, 1.f), __fmaf_rn(br.y, tm.y, 1.f));
    c1.A = mul2(cmul2(dv, __fdividef(A.R, A.cv)), rcp2(om));
    c1.B = mul2(mul2(cmul2(dv, __fdividef(__fmul_rn(A.a, A.kappa), A.cv)), rh), rcp2(den));
    if (BND) {
      if (g.dirichlet_row(y)) c1.aE = c1.aW = c1.aN = c1.aS = bc2(0.f);  // T held: K = 0
      // row 0 under an imposed flux: no conductive flux through its bottom face
      if (y == 0) c1.aS = bc2(0.f);
      if (y == 1 || y == W || (g.top_wall && y == ny - 2)) {
        // conductivity of the wall-flux face: below the row, or above it under a top wall
        const bool top = g.top_wall && y == ny - 2;
        sm.qf[y & 3][lane] = mul2(mul2(cmul2(l, 2.f), top ? lam : S.lamS), top ? qN : S.qS);
      }
    }
    S.lamS = l;
    S.qS = qN;
    S.uyS = S.uy;
    S.lam = lam;
    S.ux = ux;
    S.uy = uy;
    S.dux[I0] = dux;
    S.suy[I0] = suy;
  }

  // q_bottom (face 0|1), q_interface (face W-1|W) and q_top (face ny-2|ny-1 under
  // a top wall) accumulate the RK-weighted conductive flux of every stage
  auto special = [&](int y, float wk, float2 Gs, float2 Gn, float2& k) {
    if (!BND) return;
    if (y == 0 && g.bottom_flux) k = add2(k, bc2(__fmul_rn(A.q_in, A.inv_rcv_w)));
    if (y >= C.ys && y < C.ye && (y == 1 || y == W || (g.top_wall && y == ny - 2))) {
      const float2 qf = sm.qf[y & 3][lane];
      auto add = [&](int slot, float2 G) {
        float2 a = sm.flux[slot][lane];
        if (C.own0) ff_add(a.x, a.y, __fmul_rn(__fmul_rn(-wk, qf.x), G.x));
        if (C.own1) ff_add(a.x, a.y, __fmul_rn(__fmul_rn(-wk, qf.y), G.y));
        sm.flux[slot][lane] = a;
      };
      if (y == 1) add(0, Gs);
      if (y == W) add(1, Gs);
      if (g.top_wall && y == ny - 2) add(2, Gn);
    }
  };
  const float dt = A.dt, hdt = __fmul_rn(0.5f, dt);
  float2 Gs, Gn, k, v;
  const float2 acc1 = S.acc[0], acc2 = S.acc[1], acc3 = S.acc[2];

  // ---- row r of T^n; stage 1 at y = r - 1
  {
    PairWin& w = S.w[0];
    pair_edges(T, we, ee);
    const float2 Tc = w.T[I1];
    k = pair_finish<I0, I1, I2>(c1.aN, c1.aS, c1.p, c1.q, w, pair_ew(c1, Tc, w.w[I1], w.e[I1]), pair_source(A, c1, Tc),
                                T, we, ee, Gs, Gn);
    special(r - 1, dt * (1.f / 6.f), Gs, Gn, k);
    S.acc[0] = k;
    v = cfma2(k, hdt, Tc);
    if (BND && r - 1 >= ny) v = S.w[1].T[I2];  // zero-gradient ghost above an open top: row ny - 1
  }
  // ---- stage 2 at y = r - 2 (newest row r - 1 of T1)
  k = pair_advance<I1, I2, I0>(A, c2.aN, c2.aS, c2.p, c2.q, c1, S.w[1], v, Gs, Gn);
  special(r - 2, dt * (2.f / 6.f), Gs, Gn, k);
  S.acc[1] = cfma2(k, 2.f, acc1);
  v = cfma2(k, hdt, S.w[0].T[I2]);
  if (BND && r - 2 >= ny) v = S.w[2].T[I0];
  // ---- stage 3 at y = r - 3 (newest row r - 2 of T2)
  k = pair_advance<I2, I0, I1>(A, c3.aN, c3.aS, c3.p, c3.q, c2, S.w[2], v, Gs, Gn);
  special(r - 3, dt * (2.f / 6.f), Gs, Gn, k);
  S.acc[2] = cfma2(k, 2.f, acc2);
  v = cfma2(k, dt, pair_slot(sm.T, r - 3, lane));
  if (BND && r - 3 >= ny) v = S.w[3].T[I1];
  // ---- stage 4 at y = r - 4 (newest row r - 3 of T3): the new temperature
  k = pair_advance<I0, I1, I2>(A, oN, oS, op, oq, c3, S.w[3], v, Gs, Gn);
  const int y = r - 4;
  special(y, dt * (1.f / 6.f), Gs, Gn, k);
  const float2 Tn = cfma2(add2(acc3, k), __fmul_rn(dt, 1.f / 6.f), pair_slot(sm.T, y, lane));
  if (C.own0 && y >= C.ys && y < C.ye) {
    float* out = C.T_out + y * A.nx + C.gx0;
    const bool both = VEC || C.own1;
    if (VEC) {
      *reinterpret_cast<float2*>(out) = Tn;  // nx even: the pair is 8-byte aligned and whole
    } else {
      out[0] = Tn.x;
      if (both) out[1] = Tn.y;
    }
    // sensible energy; a non-finite T stays non-finite in the sum
    const bool solid = BND ? g.solid_row(y) : y < W;
    const float2 rcv = solid ? bc2(A.rcv_w) : cmul2(pair_slot(sm.rho, y, lane), A.cv);
    float2 e = mul2(Tn, rcv);
    if (!both) e.y = 0.f;
    ff_add2(S.eh, S.el, e);
  }
}

// Whether steps t .. t + U - 1 need the boundary rows' tests.
template <int U>
__device__ __forceinline__ bool pair_bnd(const StepArgs& A, int t) {
  const int e = t + U - 1;
  return t <= 5 || (e >= A.W + 1 && t <= A.W + 4) || e > (A.top_bc == TOP_WALL ? A.ny - 2 : A.ny);
}

// U steps from row t on; U = 1 turns the rings by a row afterwards.
template <int U, bool BND, bool VEC, bool BATCH>
__device__ __forceinline__ void pair_group(const StepArgs& A, const PairCtx& C, PairState& S, PairShared& sm, int t) {
  pair_step<0, BND, VEC, BATCH>(A, C, S, sm, t);
  if constexpr (U == 3) {
    pair_step<1, BND, VEC, BATCH>(A, C, S, sm, t + 1);
    pair_step<2, BND, VEC, BATCH>(A, C, S, sm, t + 2);
  } else {
    static_assert(U == 1, "rings of three rows");
    auto turn = [](auto* ring) {  // row r moves to the place of row r - 1, that one to r - 2's, that one to r - 3's
      const auto t = ring[0];
      ring[0] = ring[1];
      ring[1] = ring[2];
      ring[2] = t;
    };
    turn(S.cf);
    turn(S.dux);
    turn(S.suy);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      turn(S.w[q].T);
      turn(S.w[q].w);
      turn(S.w[q].e);
    }
  }
}

// Walk of strip sx, segment sg (rows [sg L, sg L + L)) of one domain by one warp.
// U: rows per pass of the loop.  U = 1 runs every row through the one general
// body: five times less code, and a third more instructions (the rings move).
template <int U, bool VEC, bool BATCH>
__device__ __forceinline__ void energy_pair(const StepArgs& A, PairShared& sm, int L, int sx, int sg, int part, int s,
                                            int nsub) {
  PairCtx C;
  const int NC = A.nx * A.ny;
  C.lane = threadIdx.x & 31;
  C.T_in = s == 1 ? A.T_in : substep_buffer(A, s - 1, nsub);
  C.T_out = substep_buffer(A, s, nsub);
  C.rho_n = A.mom;
  C.ux_n = A.mom + NC;
  C.uy_n = A.mom + 2 * NC;
  const int gxu = sx * EP_OUT - EP_H + 2 * C.lane;
  C.gx0 = wrapx(gxu, A.nx);
  C.gx1 = wrapx(gxu + 1, A.nx);
  const bool inner = C.lane >= EP_H / 2 && C.lane < (EP_H + EP_OUT) / 2;
  C.own0 = inner && gxu < A.nx;
  C.own1 = inner && gxu + 1 < A.nx;
  C.ys = sg * L;
  C.ye = C.ys + L < A.ny ? C.ys + L : A.ny;
  C.last = s == nsub;
  if constexpr (VEC) {
    // nx a multiple of 4: a 4-column piece never straddles the periodic edge
    const int col = wrapx(sx * EP_OUT - EP_H + 4 * (C.lane & 15), A.nx);
    C.src0 = (C.lane < 16 ? C.T_in : C.rho_n) + col;
    C.src1 = (C.lane < 16 ? C.ux_n : C.uy_n) + col;
  }
  PairState S;
  const float2 z = bc2(0.f);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    PairWin& w = S.w[q];
    w.G = w.k = w.X = w.T[0] = w.T[1] = w.T[2] = z;
    w.w[0] = w.w[1] = w.w[2] = w.e[0] = w.e[1] = w.e[2] = 0.f;
  }
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    S.acc[q] = S.dux[q] = S.suy[q] = z;
    S.cf[q].aE = S.cf[q].aW = S.cf[q].aN = S.cf[q].aS = S.cf[q].p = S.cf[q].q = S.cf[q].A = S.cf[q].B = z;
    sm.flux[q][C.lane] = z;
  }
  S.lam = S.lamS = bc2(1.f);  // (rows t0 - 1 and t0 - 2 are not loaded; their faces are not used)
  S.ux = S.uy = S.uyS = S.qS = S.eh = S.el = z;
  const int t0 = C.ys - 4;
#pragma unroll
  for (int n = 0; n < EP_PF / U; ++n) pair_fetch<U, VEC>(A, C, sm, t0 + n * U);
  for (int t = t0; t < C.ye + 4; t += U) {
    // this group's rows (every lane's copies) are complete; the fetched group's slots
    // hold rows that nothing reads any more
    cp_async_wait<EP_PF / U - 1>();
    __syncwarp();
    pair_fetch<U, VEC>(A, C, sm, t + EP_PF);
    if (U == 1 || pair_bnd<U>(A, t))
      pair_group<U, true, VEC, BATCH>(A, C, S, sm, t);
    else
      pair_group<U, false, VEC, BATCH>(A, C, S, sm, t);
  }
  cp_async_wait<0>();  // none left in flight at exit
  // the warp's partials: q_bottom, q_top, q_interface, sensible energy
  const bool bad = C.last && (nonfinite(S.eh.x) || nonfinite(S.eh.y));
  float eh = C.last ? S.eh.x : 0.f, el = C.last ? S.el.x : 0.f;
  if (C.last) ff_merge(eh, el, S.eh.y, S.el.y);
  const float2 fb = sm.flux[0][C.lane], fi = sm.flux[1][C.lane], ft = sm.flux[2][C.lane];
  float hi[NEPART] = {fb.x, ft.x, fi.x, eh}, lo[NEPART] = {fb.y, ft.y, fi.y, el};
#pragma unroll
  for (int q = 0; q < NEPART; ++q) {
    if (__any_sync(0xffffffffu, hi[q] != 0.f || lo[q] != 0.f)) ff_warp_sum(hi[q], lo[q]);
    if (C.lane == 0) {
      double* out = A.epart + (long long)part * NEPART + q;
      const double v = (double)hi[q] + (double)lo[q];
      *out = s > 1 ? *out + v : v;
    }
  }
  if (bad) atomicOr(&A.state->error_flags, ERR_NONFINITE);
}

// One warp per CTA: everything that selects a branch or a row is then uniform
// by construction and stays out of the vector registers.
template <int U>
__global__ void __launch_bounds__(32, EP_CTAS) k_energy_pair(const __grid_constant__ StepArgs A, int L, int s, int nsub) {
  __shared__ __align__(16) PairShared sm;
  // 16-byte prefetch pieces and 8-byte stores where the rows allow them
  if ((A.nx & 3) == 0)
    energy_pair<U, true, false>(A, sm, L, blockIdx.x, blockIdx.y, blockIdx.y * gridDim.x + blockIdx.x, s, nsub);
  else
    energy_pair<U, false, false>(A, sm, L, blockIdx.x, blockIdx.y, blockIdx.y * gridDim.x + blockIdx.x, s, nsub);
}

template <int U>
__global__ void __launch_bounds__(32, EP_CTAS) k_energy_pair_batch(const __grid_constant__ StepArgs P,
                                                                   const DomArgs* __restrict__ desc,
                                                                   const int2* __restrict__ blk,
                                                                   const int* __restrict__ active, int L, int s,
                                                                   int nsub) {
  __shared__ __align__(16) PairShared sm;
  const int2 bl = blk[blockIdx.x];
  if (!active[bl.x]) return;
  StepArgs A = P;
  apply_dom(A, desc[bl.x]);
  const int local = bl.y;
  const int strips = (A.nx + EP_OUT - 1) / EP_OUT;
  if ((A.nx & 3) == 0)
    energy_pair<U, true, true>(A, sm, L, local % strips, local / strips, local, s, nsub);
  else
    energy_pair<U, false, true>(A, sm, L, local % strips, local / strips, local, s, nsub);
}

}  // namespace hlb
