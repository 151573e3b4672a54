// Cell functions of the V-cycle in correction form (float-float arithmetic), shared by the
// single-instance and the batched kernels.
//
// The FAS V-cycle of App. B improves u by solving N(u) = S level by level.  Written for
// the change d = u - u0 from the state u0 in which a level is entered, with rho = S - N(u0)
// its residual there, the same iteration reads
//   r1 = rho1 - d_phi + c Delta_h d_mu
//   r2 = rho2 - d_mu + (g(p0 + d_phi) - g(p0)) + (gam + W) d_phi + Delta_h d_kappa
//   r3 = rho3 - d_kappa + theta Delta_h d_phi
// with p0 the level's phi at entry; the smoother adds omega A^-1 r to d as it did to u, the
// restriction passes p0 = R(p0 + d_phi), d = 0 and rho = R r to the coarse level (there
// S_c - N_c(R u) = R r by the definition of the tau correction, so N_c is never formed),
// and the prolongation adds P d_c (which is P(u_c - R u)).  Iterates agree with the u form
// in exact arithmetic; only differences of u enter, so 48 bits of them carry the same
// information as 64-bit values of u, and only the finest level's u and its residual are
// FP64 (k_df_defect, once per V-cycle).  An operation rounds by 2^-46 of its operands, the cell
// solve's reciprocal by 2^-44.  Against extended precision the iterate after one V-cycle was 2e-13
// (h = 0.05), 2e-12 (h = 0.5, s = 50) to 5e-12 (h = 1e-3) off, 10 to 120 times an FP64
// V-cycle's; the next cycles' residuals see it, and converged steps are not less exact (6e-17 to
// 6e-16 rms, FP64 V-cycles' 6e-17 to 2e-15).
//
// Planes are split by colour: the red cells ((i + j) even) of a plane in an n x m/2 array,
// then the black ones, cell (i, j) at column i >> 1.  A half sweep reads one colour's
// neighbours and the other's own values, so every load of a warp is contiguous (the
// interleaved layout touches twice the sectors).
#pragma once

#include "df_math.cuh"

namespace mpfc {

struct DLev {
  int m, n, nyn;
  float2 *d[3];      // correction (d_phi, d_mu, d_kappa)
  float2 *r[3];      // rho, the residual the level was entered with
  float2 *pb;        // p0, phi the level was entered with
  float2 *pk;        // phi^k (scheme 2)
  const double* W;   // pinning weight (row-major), nullptr: none
};

// Coefficients as float-float; nb-dependent ones for four neighbours or for a Neumann row.
struct DCoef {
  float2 cmu, ih2, th2, gam, omega;
  float2 a, b, b3, Q0, D0w;
  float2 aq;   // determinant / omega = D0w + aq q', q' = p^2 (scheme 1: aq = 3 a / omega) or g' (+ W) (a / omega)
};

struct DPar {
  DLev L;
  DCoef k, kb;
};

__device__ __forceinline__ size_t dplane(const DLev& L) { return (size_t)(L.m >> 1) * L.n; }
// (i, j) -> offset in a colour-split plane
__device__ __forceinline__ size_t dindex(const DLev& L, int i, int j) {
  return (((i + j) & 1) ? dplane(L) : 0) + (size_t)j * (L.m >> 1) + (i >> 1);
}

struct DCell {
  df p, m, k;        // correction at the cell (0 where not yet formed)
  df rho1, rho2, rho3;
  df pb, pk;
  df gw;             // gam + W
  df W;
};

// (g(p) - g(p0)) / d for p = p0 + d
template <int SCH>
__device__ __forceinline__ df gquot(df p, df pb, df pk) {
  if (SCH == 1) return sum3u(sqr(p), mulu(p, pb), sqr(pb));                 // p^2 + p p0 + p0^2
  const df t = mulu(add(p, pb), add(p, pk));                               // ((p + p0)(p + pk) + p0^2 + pk^2) / 4
  return scale2(sum3u(t, sqr(pb), sqr(pk)), 0.25f);
}

__device__ __forceinline__ df mul3(df a) {
  const float h = fmul(3.0f, a.h);
  return df{h, __fmaf_rn(3.0f, a.l, __fmaf_rn(3.0f, a.h, -h))};
}
// g'(p): 3 p^2, or (3 p^2 + 2 p pk + pk^2) / 4 summed as (2 p^2 + (p + pk)^2) / 4
template <int SCH>
__device__ __forceinline__ df df_dg(df p, df pk) {
  if (SCH == 1) return mul3(sqr(p));
  return scale2(addu(scale2(sqr(p), 2.0f), sqr(add(p, pk))), 0.25f);
}

// How much of d is still zero in a level's first sweep: kGen nothing, kOwn the cell's own
// value (first black half sweep), kAll everything (first red half sweep).
constexpr int kGen = 0, kOwn = 1, kAll = 2;

// The cell update: Lp, Lm, Lk are sum_nb - 4 (own) of d_phi, d_mu, d_kappa (unused for
// kAll); the corrections in c are updated.
template <int SCH, int MODE>
__device__ __forceinline__ void df_update(const DCoef& K, df Lp, df Lm, df Lk, DCell& c) {
  df r1, r2, r3, p;
  if (MODE == kAll) {
    r1 = c.rho1;
    r2 = c.rho2;
    r3 = c.rho3;
    p = c.pb;
  } else if (MODE == kOwn) {
    r1 = add(c.rho1, mulu(mk(K.cmu), Lm));
    r2 = add(c.rho2, mulu(mk(K.ih2), Lk));
    r3 = add(c.rho3, mulu(mk(K.th2), Lp));
    p = norm(c.pb);   // with this, the bits of kGen on a zero correction
  } else {
    p = add(c.pb, c.p);
    r1 = norm(sum3u(c.rho1, mulu(mk(K.cmu), Lm), neg(c.p)));
    r3 = norm(sum3u(c.rho3, mulu(mk(K.th2), Lp), neg(c.k)));
    const df G = norm(addu(gquot<SCH>(p, c.pb, c.pk), c.gw));
    r2 = norm(sum4u(c.rho2, mulu(mk(K.ih2), Lk), neg(c.m), mulu(G, c.p)));
  }
  // determinant / omega and the Cramer numerator of mu, Q0 + g'
  df q, Qq;
  if (SCH == 1) {
    q = sqr(p);
    Qq = add(mk(K.Q0), mul3(q));
  } else {
    q = add(df_dg<2>(p, c.pk), c.W);
    Qq = add(mk(K.Q0), q);
  }
  const df wr = rcp(add(mk(K.D0w), mulu(mk(K.aq), q)));
  const df t = norm(addu(mulu(mk(K.b), r3), neg(r2)));
  const df dp = mul(norm(addu(r1, mulu(mk(K.a), t))), wr);
  const df dm = mulu(norm(addu(mulu(Qq, r1), neg(t))), wr);
  const df dk = addu(mulu(mk(K.omega), r3), neg(mulu(mk(K.b3), dp)));
  if (MODE == kGen) {
    c.p = add(c.p, dp);
    c.m = add(c.m, dm);
    c.k = add(c.k, dk);
  } else {
    c.p = dp;
    c.m = norm(dm);
    c.k = norm(dk);
  }
}

// Loads: L1-cached plain loads (the tail kernel's planes may be in shared memory).
__device__ __forceinline__ df ldd(const float2* p) { return mk(*p); }

// Neighbour offsets of cell (x, j) of colour `color` in the other colour's half plane: the
// cell at the same column index always, and the one left or right of it by the row's parity.
struct DNb {
  size_t c0, cx, s, n;   // offsets in a full plane; c0, cx: west and east in some order
};
template <bool NY>
__device__ __forceinline__ DNb df_nb(const DLev& L, int color, int x, int j, size_t own) {
  const int half = L.m >> 1;
  const size_t ob = color ? 0 : dplane(L);   // the other colour
  const size_t row = ob + (size_t)j * half;
  DNb o;
  o.c0 = row + x;
  int xx = ((j + color) & 1) ? x + 1 : x - 1;
  xx = xx < 0 ? half - 1 : (xx == half ? 0 : xx);
  o.cx = row + xx;
  if (NY && L.nyn) {   // a ghost row reads as the boundary row: the cell itself
    o.s = j == 0 ? own : row - half + x;
    o.n = j == L.n - 1 ? own : row + half + x;
  } else {
    o.s = (j == 0 ? ob + (size_t)(L.n - 1) * half : row - half) + x;
    o.n = (j == L.n - 1 ? ob : row + half) + x;
  }
  return o;
}

template <int SCH>
__device__ __forceinline__ void df_load_static(const DLev& L, const DCoef& K, size_t own, int i, int j, DCell& c) {
  c.rho1 = ldd(L.r[0] + own);
  c.rho2 = ldd(L.r[1] + own);
  c.rho3 = ldd(L.r[2] + own);
  c.pb = ldd(L.pb + own);
  c.gw = mk(K.gam);
  c.W = df{0.f, 0.f};
  c.pk = df{0.f, 0.f};
  if (SCH == 2) {
    c.pk = ldd(L.pk + own);
    if (L.W) {
      c.W = df_of(L.W[(size_t)j * L.m + i]);
      c.gw = add(c.gw, c.W);
    }
  }
}

// Half sweep of colour `color` at column x of row j.  NY: the level may have Neumann rows.
// u (FINAL): the finest level's FP64 planes, to which the finished correction is added.
template <int SCH, int MODE, bool NY, bool FINAL>
__device__ __forceinline__ void df_smooth_cell(const DPar& P, int color, int x, int j, double* const* u = nullptr) {
  const DLev& L = P.L;
  const size_t own = (color ? dplane(L) : 0) + (size_t)j * (L.m >> 1) + x;
  const int i = 2 * x + ((j + color) & 1);
  auto body = [&](const DCoef& K) {
    DCell c;
    df_load_static<SCH>(L, K, own, i, j, c);
    df Lp{0.f, 0.f}, Lm{0.f, 0.f}, Lk{0.f, 0.f};
    c.p = c.m = c.k = df{0.f, 0.f};
    if (MODE != kAll) {
      const DNb o = df_nb<NY>(L, color, x, j, own);
      if (MODE == kGen) {
        c.p = ldd(L.d[0] + own);
        c.m = ldd(L.d[1] + own);
        c.k = ldd(L.d[2] + own);
      }
      // kOwn: the cell's own value is zero, also where a ghost row reads it
      auto at = [&](const float2* f, size_t q) {
        if (MODE == kOwn && NY && q == own) return df{0.f, 0.f};
        return ldd(f + q);
      };
      Lp = lap5(ldd(L.d[0] + o.c0), ldd(L.d[0] + o.cx), at(L.d[0], o.s), at(L.d[0], o.n), c.p);
      Lm = lap5(ldd(L.d[1] + o.c0), ldd(L.d[1] + o.cx), at(L.d[1], o.s), at(L.d[1], o.n), c.m);
      Lk = lap5(ldd(L.d[2] + o.c0), ldd(L.d[2] + o.cx), at(L.d[2], o.s), at(L.d[2], o.n), c.k);
    }
    df_update<SCH, MODE>(K, Lp, Lm, Lk, c);
    L.d[0][own] = f2(c.p);
    L.d[1][own] = f2(c.m);
    L.d[2][own] = f2(c.k);
    if (FINAL) {
      const size_t id = (size_t)j * L.m + i;
      u[0][id] += df_to_f64(c.p);
      u[1][id] += df_to_f64(c.m);
      u[2][id] += df_to_f64(c.k);
    }
  };
  if (NY && L.nyn && (j == 0 || j == L.n - 1)) body(P.kb);
  else body(P.k);
}

// 2x2 block sums: of the block's four cells and of the eight cells around it.
struct DBlk {
  size_t in[4], out[8];
};
__device__ __forceinline__ DBlk df_block(const DLev& F, int I, int J) {
  const int half = F.m >> 1, n = F.n, j0 = 2 * J, j1 = j0 + 1;
  const size_t pl = dplane(F);
  const int js = j0 > 0 ? j0 - 1 : (F.nyn ? 0 : n - 1), jn = j1 < n - 1 ? j1 + 1 : (F.nyn ? n - 1 : 0);
  const int w = I > 0 ? I - 1 : half - 1, e = I < half - 1 ? I + 1 : 0;
  const size_t r0 = (size_t)j0 * half, r1 = (size_t)j1 * half, rs = (size_t)js * half, rn = (size_t)jn * half;
  DBlk b;
  b.in[0] = r0 + I;            // (2I, j0) red
  b.in[1] = pl + r0 + I;       // (2I+1, j0) black
  b.in[2] = pl + r1 + I;       // (2I, j1) black
  b.in[3] = r1 + I;            // (2I+1, j1) red
  b.out[0] = pl + r0 + w;      // (2I-1, j0): odd column, even row: black
  b.out[1] = r1 + w;           // (2I-1, j1): red
  b.out[2] = r0 + e;           // (2I+2, j0): red
  b.out[3] = pl + r1 + e;      // (2I+2, j1): black
  const bool so = js & 1, no = jn & 1;   // a ghost row is the boundary row, of the other parity
  b.out[4] = (so ? pl : 0) + rs + I;     // (2I, js)
  b.out[5] = (so ? 0 : pl) + rs + I;     // (2I+1, js)
  b.out[6] = (no ? pl : 0) + rn + I;
  b.out[7] = (no ? 0 : pl) + rn + I;
  return b;
}
__device__ __forceinline__ df df_sum_in(const float2* f, const DBlk& b) {
  return norm(sum4u(ldd(f + b.in[0]), ldd(f + b.in[1]), ldd(f + b.in[2]), ldd(f + b.in[3])));
}
__device__ __forceinline__ df df_sum_out(const float2* f, const DBlk& b) {
  return norm(addu(sum4u(ldd(f + b.out[0]), ldd(f + b.out[1]), ldd(f + b.out[2]), ldd(f + b.out[3])),
                   sum4u(ldd(f + b.out[4]), ldd(f + b.out[5]), ldd(f + b.out[6]), ldd(f + b.out[7]))));
}

// Restriction at coarse cell (I, J): rho_c = R r and p0_c = R(p0 + d_phi).  The block sum of
// the five-point Laplacian is (sum of the 8 bordering cells - 2 sum of the block) / h^2, as in
// the FP64 form.  FIRST: also the first red half sweep of the coarse level (d_c = 0 before
// it), on the values in registers; BASE: p0_c here (else by df_base_cell).  (cI, cJ): the
// coarse cell in PC, where PF is a staged part of the fine level and (I, J) counts from its origin.
template <int SCH, bool FIRST, bool BASE>
__device__ __forceinline__ void df_restrict_cell(const DPar& PF, const DPar& PC, int I, int J, int zero, int cI, int cJ) {
  const DLev& F = PF.L;
  const DLev& C = PC.L;
  const DCoef& K = PF.k;
  const DBlk b = df_block(F, I, J);
  const df sp = df_sum_in(F.d[0], b), sm = df_sum_in(F.d[1], b), sk = df_sum_in(F.d[2], b);
  const df op = df_sum_out(F.d[0], b), om = df_sum_out(F.d[1], b), ok = df_sum_out(F.d[2], b);
  df gs{0.f, 0.f}, sb{0.f, 0.f};
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const df d = ldd(F.d[0] + b.in[q]), p0 = ldd(F.pb + b.in[q]);
    const df pk = (SCH == 2) ? ldd(F.pk + b.in[q]) : df{0.f, 0.f};
    df G = norm(addu(gquot<SCH>(add(p0, d), p0, pk), mk(K.gam)));
    if (SCH == 2 && F.W) G = add(G, df_of(F.W[(size_t)(2 * J + (q >> 1)) * F.m + 2 * I + (q & 1)]));
    gs = add(gs, mulu(G, d));
    sb = add(sb, p0);
  }
  const df rho1 = df_sum_in(F.r[0], b), rho2 = df_sum_in(F.r[1], b), rho3 = df_sum_in(F.r[2], b);
  const df lm = norm(addu(om, scale2(sm, -2.0f))), lk = norm(addu(ok, scale2(sk, -2.0f)));
  const df lp = norm(addu(op, scale2(sp, -2.0f)));
  const df c1 = scale2(norm(sum3u(rho1, mulu(mk(K.cmu), lm), neg(sp))), 0.25f);
  const df c2 = scale2(norm(sum4u(rho2, mulu(mk(K.ih2), lk), neg(sm), gs)), 0.25f);
  const df c3 = scale2(norm(sum3u(rho3, mulu(mk(K.th2), lp), neg(sk))), 0.25f);
  const size_t cid = dindex(C, cI, cJ);
  C.r[0][cid] = f2(c1);
  C.r[1][cid] = f2(c2);
  C.r[2][cid] = f2(c3);
  const df pbc = scale2(add(sb, sp), 0.25f);
  if (BASE) C.pb[cid] = f2(pbc);
  if (zero) {   // no pre-smoothing on the coarse level: its correction starts at zero
    const float2 z = make_float2(0.f, 0.f);
    C.d[0][cid] = z;
    C.d[1][cid] = z;
    C.d[2][cid] = z;
  } else if (FIRST && !((cI + cJ) & 1)) {
    DCell c;
    c.rho1 = c1;
    c.rho2 = c2;
    c.rho3 = c3;
    c.pb = pbc;
    c.pk = (SCH == 2) ? ldd(C.pk + cid) : df{0.f, 0.f};
    c.W = df{0.f, 0.f};
    if (SCH == 2 && C.W) c.W = df_of(C.W[(size_t)cJ * C.m + cI]);
    const df z{0.f, 0.f};
    if (C.nyn && (cJ == 0 || cJ == C.n - 1)) df_update<SCH, kAll>(PC.kb, z, z, z, c);
    else df_update<SCH, kAll>(PC.k, z, z, z, c);
    C.d[0][cid] = f2(c.p);
    C.d[1][cid] = f2(c.m);
    C.d[2][cid] = f2(c.k);
  }
}

template <int SCH, bool FIRST, bool BASE>
__device__ __forceinline__ void df_restrict_cell(const DPar& PF, const DPar& PC, int I, int J, int zero) {
  df_restrict_cell<SCH, FIRST, BASE>(PF, PC, I, J, zero, I, J);
}

// p0_c = R(p0 + d_phi) alone, with the operations of df_restrict_cell.
__device__ __forceinline__ void df_base_cell(const DLev& F, const DLev& C, int I, int J) {
  const DBlk b = df_block(F, I, J);
  const df sp = df_sum_in(F.d[0], b);
  df sb{0.f, 0.f};
#pragma unroll
  for (int q = 0; q < 4; ++q) sb = add(sb, ldd(F.pb + b.in[q]));
  C.pb[dindex(C, I, J)] = f2(scale2(add(sb, sp), 0.25f));
}

// The prolonged correction at a fine cell: weights (9, 3, 3, 1)/16 of the coarse cell that holds
// it, its neighbours in x and y on the fine cell's side, and the diagonal one (9 e = 8 e + e and
// 3 e = 2 e + e, both with exact power-of-two terms).  c9 = 9/16 e.
__device__ __forceinline__ df df_nine(df e) { return add(scale2(e, 0.5f), scale2(e, 0.0625f)); }
__device__ __forceinline__ df df_bilinear(df c9, df x, df y, df xy) {
  const df s = add(x, y);
  return norm(sum4u(c9, scale2(s, 0.125f), scale2(s, 0.0625f), scale2(xy, 0.0625f)));
}
__device__ __forceinline__ df df_prolonged(df e, df x, df y, df xy) { return df_bilinear(df_nine(e), x, y, xy); }

// Prolongation into the four children of coarse cell (I, J): d_f += P d_c.
__device__ __forceinline__ void df_prolong_plane(const DLev& C, const DLev& F, int c, int I, int J) {
  const float2* e = C.d[c];
  const int Iw = I > 0 ? I - 1 : C.m - 1, Ie = I < C.m - 1 ? I + 1 : 0;
  const int Js = J > 0 ? J - 1 : (C.nyn ? 0 : C.n - 1), Jn = J < C.n - 1 ? J + 1 : (C.nyn ? C.n - 1 : 0);
  const df e00 = ldd(e + dindex(C, I, J));
  const df eW = ldd(e + dindex(C, Iw, J)), eE = ldd(e + dindex(C, Ie, J));
  const df eS = ldd(e + dindex(C, I, Js)), eN = ldd(e + dindex(C, I, Jn));
  const df c9 = df_nine(e00);
  const DBlk b = [&] {
    DBlk q;
    const int half = F.m >> 1;
    const size_t pl = dplane(F), r0 = (size_t)(2 * J) * half + I, r1 = r0 + half;
    q.in[0] = r0;
    q.in[1] = pl + r0;
    q.in[2] = pl + r1;
    q.in[3] = r1;
    return q;
  }();
  auto put = [&](int q, df x, df y, df xy) {
    F.d[c][b.in[q]] = f2(add(ldd(F.d[c] + b.in[q]), df_bilinear(c9, x, y, xy)));
  };
  put(0, eW, eS, ldd(e + dindex(C, Iw, Js)));
  put(1, eE, eS, ldd(e + dindex(C, Ie, Js)));
  put(2, eW, eN, ldd(e + dindex(C, Iw, Jn)));
  put(3, eE, eN, ldd(e + dindex(C, Ie, Jn)));
}

}  // namespace mpfc
