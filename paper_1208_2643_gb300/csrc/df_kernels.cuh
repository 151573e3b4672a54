// Pieces of the V-cycle in correction form that the single-instance and the batched kernels
// share beyond the cell functions: the FP64 residual at a cell, the coarsest solve and the
// coarse tail.
#pragma once

#include "df_cells.cuh"
#include "fp64_kernels.cuh"

namespace mpfc {

// Residual norms below this (and still above the tolerance) leave the low parts' range.
constexpr double kDfMinResidual = 0x1p-56;

__device__ __forceinline__ bool df_out_of_range(double x, int e) {
  return (((unsigned)__double2hiint(x) >> 20) & 0x7FFu) >= 1023u + e;
}

// A thread's sum of squared residuals: FP64 (after the guess, where no norm is known to scale
// by), or float-float of values scaled by a power of two near the inverse of the last norm (a
// norm cannot fall by 2^60 or grow by 2^50 in one cycle).  The float-float form spares three
// FP64 multiply-adds a cell and the FP64 additions of the warp's reduction.
struct DSum {
  double d;
  df f;
};
// Norms for which the scaled squares of the next residual keep their low parts in binary32: from
// kDfMinResidual up to far below what a residual value may be (df_of keeps 48 bits to 2^99).
// Zero, infinities and NaN are not among them.
__device__ __forceinline__ bool df_norm_in_range(double res) {
  return f64_exp(res) - (1023u - 56u) <= 56u + 60u;
}
__device__ __forceinline__ float df_norm_scale(double res) {
  const unsigned e = f64_exp(res);
  return (e < 1023u - 100u || e > 1023u + 100u) ? 1.0f : __uint_as_float((127u + 1023u - e) << 23);
}
__device__ __forceinline__ df df_squares(df a, df b, df c, float scale) {
  return norm(sum3u(sqr(scale2(a, scale)), sqr(scale2(b, scale)), sqr(scale2(c, scale))));
}
// One thread's sum in FP64.
template <bool FP64>
__device__ __forceinline__ double df_thread_sum(const DSum& s, float scale) {
  if (FP64) return s.d;
  const double inv = (double)__uint_as_float((254u << 23) - __float_as_uint(scale));   // 1 / scale
  return df_to_f64(s.f) * inv * inv;
}
// The warp's total, valid in lane 0 (blocks 32 threads wide).
template <bool FP64>
__device__ __forceinline__ double df_warp_sum(const DSum& s, float scale) {
  if (FP64) {
    double v = s.d;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
  }
  df f = s.f;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    f = add(f, df{__shfl_down_sync(0xffffffffu, f.h, o), __shfl_down_sync(0xffffffffu, f.l, o)});
  return df_thread_sum<false>(DSum{0.0, f}, scale);
}

// FP64 residual of the iterate at the cells (2x, j) and (2x + 1, j): rho as float-float planes,
// p0 = phi; adds the squares to `sum` and sets `bad` where a value is outside the range the form
// covers.  MODE0, right after the guess: rows 2 and 3 hold by construction (k_guess_kappa,
// k_guess_mu), so rho2 = rho3 = 0; phi^k is split too (scheme 2).  FIRST: the first red half
// sweep on the values in registers (one of the two cells is red, so every lane has one); zero: no
// pre-smoothing, the correction starts at zero.
template <int SCH, bool MODE0, bool FIRST>
__device__ __forceinline__ void df_defect_pair(const Lev& L, const Coef& k, const DPar& P, int x, int j, int zero,
                                               float scale, DSum& sum, bool& bad) {
  const DLev& D = P.L;
  PairResid R;
  resid_pair<SCH, MODE0>(L, k, x, j, R);
  if (SCH == 2 && MODE0) {
    const double2 pk = ld2(L.pk + (size_t)j * L.m + 2 * x);
    R.pk[0] = pk.x;
    R.pk[1] = pk.y;
  }
  const size_t red = (size_t)j * (D.m >> 1) + x, black = red + dplane(D);
  const int qr = j & 1;   // which of the two is red
#pragma unroll
  for (int c = 0; c < 2; ++c) {   // the red cell, the black cell
    const bool second = c == 0 ? qr != 0 : qr == 0;
    const double a = second ? R.a[1] : R.a[0], p = second ? R.p[1] : R.p[0];
    bad |= df_out_of_range(p, 20) | df_out_of_range(a, 40);
    DCell q;
    q.rho1 = df_of(a);
    q.rho2 = q.rho3 = q.pk = q.W = df{0.f, 0.f};
    q.pb = df_of(p);
    if (MODE0) {
      sum.d = fma(a, a, sum.d);
    } else {
      const double b = second ? R.b[1] : R.b[0], d = second ? R.c[1] : R.c[0];
      bad |= df_out_of_range(b, 40) | df_out_of_range(d, 40);
      q.rho2 = df_of(b);
      q.rho3 = df_of(d);
      sum.f = add(sum.f, df_squares(q.rho1, q.rho2, q.rho3, scale));
    }
    const size_t id = c == 0 ? red : black;
    D.r[0][id] = f2(q.rho1);
    D.r[1][id] = f2(q.rho2);
    D.r[2][id] = f2(q.rho3);
    D.pb[id] = f2(q.pb);
    if (SCH == 2 && (MODE0 || (FIRST && c == 0))) {
      q.pk = df_of(second ? R.pk[1] : R.pk[0]);
      if (MODE0) D.pk[id] = f2(q.pk);
    }
    if (zero) {
      const float2 z = make_float2(0.f, 0.f);
      D.d[0][id] = z;
      D.d[1][id] = z;
      D.d[2][id] = z;
    } else if (FIRST && c == 0) {
      if (SCH == 2 && D.W) q.W = df_of(D.W[(size_t)j * D.m + 2 * x + qr]);
      const df z{0.f, 0.f};
      if (D.nyn && (j == 0 || j == D.n - 1)) df_update<SCH, kAll>(P.kb, z, z, z, q);
      else df_update<SCH, kAll>(P.k, z, z, z, q);
      D.d[0][id] = f2(q.p);
      D.d[1][id] = f2(q.m);
      D.d[2][id] = f2(q.k);
    }
  }
}

// ---------------------------------------------------------------------------
// Coarsest grid: Newton on the equation for d_phi with rows 2 and 3 eliminated,
//   F(d) = d - c L (rho2 + g(p0 + d) - g(p0) + (gam + W) d + L (rho3 + theta L d)) - rho1 = 0,
// J = K3 - c L diag(gam + W + g'(p0 + d)): the FP64 form's equation (coarse_newton), with
// F in float-float and FP32 linear solves.  The applied update is below 1e-15 (1 + |p0 + d|_inf),
// as there, or below 1e-14 |d|_inf, the arithmetic's resolution, or was predicted to be on
// the next pass.
// ---------------------------------------------------------------------------
constexpr int kDfTailMax = 10;
constexpr int kDfTailThreads = 512;

__device__ __forceinline__ df nblap_df(const float2* f, int m, int n, int t, int nyn) {
  const int i = t % m, j = t / m;
  return lap5(ldd(f + j * m + wrapm(i - 1, m)), ldd(f + j * m + wrapm(i + 1, m)), ldd(f + ywrap(j - 1, n, nyn) * m + i),
              ldd(f + ywrap(j + 1, n, nyn) * m + i), ldd(f + t));
}

__host__ __device__ constexpr size_t coarse_df_smem(int G) { return sizeof(float2) * 7 * (size_t)G + sizeof(float) * ((size_t)G * (G + 1) + (size_t)G); }

__device__ __forceinline__ float df_dg32(int scheme, float p, float q) {
  return scheme == 1 ? 3.f * p * p : 0.25f * (3.f * p * p + 2.f * p * q + q * q);
}

// One warp, a pivoted elimination in shared memory (gauss_shared) for every update: what
// coarse_chord_df falls back to.  sm: coarse_df_smem.
template <int SCH>
__device__ __noinline__ void coarse_newton_df(const DPar& P, const float* __restrict__ K3f, float2* sm) {
  const DLev& C = P.L;
  const DCoef& K = P.k;
  const int m = C.m, n = C.n, G = m * n, W = G + 1;
  float2* ph = sm;
  float2* s1 = ph + G;
  float2* s2 = s1 + G;
  float2* s3 = s2 + G;
  float2* pk = s3 + G;
  float2* pb = pk + G;
  float2* kap = pb + G;
  float2* muv = s2;   // row 2's value replaces rho2 for an iteration (rho2 stays in the level's plane)
  float* Jm = reinterpret_cast<float*>(kap + G);   // G x (G+1), last column = right-hand side
  float* d = Jm + G * W;
  const int lane = threadIdx.x & 31;
  const unsigned FULL = 0xffffffffu;
  const float2 z2 = make_float2(0.f, 0.f);
  for (int t = lane; t < G; t += 32) {
    const size_t id = dindex(C, t % m, t / m);
    ph[t] = z2;
    s1[t] = C.r[0][id];
    s3[t] = C.r[2][id];
    pb[t] = C.pb[id];
    pk[t] = (SCH == 2) ? C.pk[id] : z2;
  }
  __syncwarp();
  const float* cLf = K3f + G * G;
  auto wt = [&](int t) { return C.W ? df_of(C.W[t]) : df{0.f, 0.f}; };
  auto kappa_at = [&](int t) { return add(mk(s3[t]), mulu(mk(K.th2), nblap_df(ph, m, n, t, C.nyn))); };
  auto mu_at = [&](int t) {
    const df dd = mk(ph[t]), p0 = mk(pb[t]);
    df Q = norm(addu(gquot<SCH>(add(p0, dd), p0, mk(pk[t])), mk(K.gam)));
    if (SCH == 2 && C.W) Q = add(Q, wt(t));
    return norm(sum3u(ldd(C.r[1] + dindex(C, t % m, t / m)), mulu(Q, dd), mulu(mk(K.ih2), nblap_df(kap, m, n, t, C.nyn))));
  };
  for (int it = 0; it < 40; ++it) {
    for (int t = lane; t < G; t += 32) kap[t] = f2(kappa_at(t));
    __syncwarp();
    for (int t = lane; t < G; t += 32) muv[t] = f2(mu_at(t));
    __syncwarp();
    for (int t = lane; t < G; t += 32) {
      const df f = sum3u(mk(s1[t]), neg(mk(ph[t])), mulu(mk(K.cmu), nblap_df(muv, m, n, t, C.nyn)));
      Jm[t * W + G] = fadd(f.h, f.l);
      d[t] = K.gam.x + (SCH == 2 && C.W ? wt(t).h : 0.f) + df_dg32(SCH, fadd(pb[t].x, ph[t].x), pk[t].x);
    }
    __syncwarp();
    for (int idx = lane; idx < G * G; idx += 32) {
      const int r = idx / G, col = idx % G;
      Jm[r * W + col] = K3f[idx] - cLf[idx] * d[col];
    }
    __syncwarp();
    gauss_shared(Jm, d, G);
    float dmax = 0.f, umax = 0.f, emax = 0.f;
    for (int t = lane; t < G; t += 32) {
      const df pn = add(mk(ph[t]), df{d[t], 0.f});
      ph[t] = f2(pn);
      dmax = fmaxf(dmax, fabsf(d[t]));
      emax = fmaxf(emax, fabsf(pn.h));
      umax = fmaxf(umax, fabsf(pn.h + pb[t].x));
    }
    for (int o = 16; o > 0; o >>= 1) {
      dmax = fmaxf(dmax, __shfl_xor_sync(FULL, dmax, o));
      emax = fmaxf(emax, __shfl_xor_sync(FULL, emax, o));
      umax = fmaxf(umax, __shfl_xor_sync(FULL, umax, o));
    }
    __syncwarp();
    if (!(dmax == dmax) || dmax <= fmaxf(1e-15f * (1.f + umax), 1e-14f * emax)) break;
  }
  for (int t = lane; t < G; t += 32) kap[t] = f2(kappa_at(t));
  __syncwarp();
  for (int t = lane; t < G; t += 32) {
    const size_t id = dindex(C, t % m, t / m);
    C.d[0][id] = ph[t];
    C.d[2][id] = kap[t];
    C.d[1][id] = f2(mu_at(t));
  }
}

// Inverse of the G x G matrix entry(row, column) by Gauss-Jordan elimination without pivoting in
// the registers of a CTA of NT threads: CW columns (CW >= G), thread t holds column t % CW of rows
// t / CW + NG i.  Before each step the owners publish the pivot row and column in shared
// memory, double buffered: one barrier a step, of the threads that hold rows.  The elimination
// is a chain of G steps, so a step's instructions count: the column's entries are read four at
// a time, and a thread of the pivot column needs no select (its entry is the published one,
// C - C (1 + 1/piv) = -C / piv).  X gets the inverse column by column.  Returns false (the same
// in every thread that holds rows) where a pivot is small.
template <int NT, int CW, typename Entry>
__device__ __forceinline__ bool gj_invert_block(float* X, int G, Entry entry) {
  constexpr int NG = NT / CW < CW ? NT / CW : CW, NR = CW / NG;   // powers of two
  __shared__ __align__(16) float prow[2][CW], pcol[2][CW];        // pcol: a[i] of group g at NR g + i
  const int q = threadIdx.x % CW, g = threadIdx.x / CW;
  if (g >= NG) return true;
  auto sync = [] { asm volatile("bar.sync 1, %0;" ::"n"(NG * CW) : "memory"); };
  float a[NR];
#pragma unroll
  for (int i = 0; i < NR; ++i) {
    const int r = g + NG * i;
    a[i] = r < G && q < G ? entry(r, q) : 0.f;
    if (q == 0) pcol[0][NR * g + i] = a[i];
  }
  if (g == 0) prow[0][q] = a[0];
  sync();
  bool ok = true;
  for (int c = 0; c < G; ++c) {
    const float* R = prow[c & 1];
    const float* C = pcol[c & 1] + NR * g;
    const float piv = R[c], rq = R[q];
    float f[NR];
    if (NR >= 4) {
#pragma unroll
      for (int i = 0; i < NR; i += 4) {
        const float4 v = *reinterpret_cast<const float4*>(C + i);
        f[i] = v.x; f[i + 1] = v.y; f[i + 2] = v.z; f[i + 3] = v.w;
      }
    } else {
#pragma unroll
      for (int i = 0; i < NR; ++i) f[i] = C[i];
    }
    float rp;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rp) : "f"(piv));
    ok = ok && fabsf(piv) > 0.05f;
    const float pq = q == c ? 1.f + rp : rq * rp;
#pragma unroll
    for (int i = 0; i < NR; ++i) a[i] = fmaf(-f[i], pq, a[i]);
    if ((c & (NG - 1)) == g) a[0] = q == c ? rp : pq;
    const int nx = c + 1;
    if ((nx & (NG - 1)) == 0) {   // the next rows' register comes first (a register array has no index)
      const float t = a[0];
#pragma unroll
      for (int i = 1; i < NR; ++i) a[i - 1] = a[i];
      a[NR - 1] = t;
    }
    if ((nx & (NG - 1)) == g) prow[nx & 1][q] = a[0];
    if (q == nx)
#pragma unroll
      for (int i = 0; i < NR; ++i) pcol[nx & 1][NR * g + i] = a[i];
    sync();
  }
#pragma unroll
  for (int i = 0; i < NR; ++i) {
    const int r = g + NG * ((i + G / NG) & (NR - 1));
    if (r < G && q < G) X[q * G + r] = a[i];
  }
  return ok;
}

// The chord iteration of warp 0 with the inverse X of a lagged Jacobian, NC cells a lane.
// Returns false where the updates stop shrinking by 100x.
template <int SCH, int NC>
__device__ __forceinline__ bool coarse_chord_pass(const DPar& P, const float* X, float2* ph, float2* kap, float2* muv,
                                                  float* rh, int& it, float& dprev) {
  const DLev& C = P.L;
  const DCoef& K = P.k;
  const int m = C.m, n = C.n, G = m * n, lane = threadIdx.x;
  int w[NC], e[NC], s[NC], u[NC], t[NC];
  size_t id[NC];
  df s1[NC], s2[NC], s3[NC], pb[NC], pk[NC], gw[NC], v[NC], kp[NC], mv[NC];
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    t[c] = min(lane + 32 * c, G - 1);   // a lane without a cell repeats the last one, and does not store
    const int j = t[c] / m, i = t[c] - j * m;
    w[c] = j * m + wrapm(i - 1, m);
    e[c] = j * m + wrapm(i + 1, m);
    s[c] = ywrap(j - 1, n, C.nyn) * m + i;
    u[c] = ywrap(j + 1, n, C.nyn) * m + i;
    id[c] = dindex(C, i, j);
    s1[c] = ldd(C.r[0] + id[c]);
    s2[c] = ldd(C.r[1] + id[c]);
    s3[c] = ldd(C.r[2] + id[c]);
    pb[c] = ldd(C.pb + id[c]);
    pk[c] = SCH == 2 ? ldd(C.pk + id[c]) : df{0.f, 0.f};
    gw[c] = SCH == 2 && C.W ? add(mk(K.gam), df_of(C.W[t[c]])) : mk(K.gam);
    v[c] = ldd(ph + t[c]);
  }
  auto has = [&](int c) { return lane + 32 * c < G; };
  auto lap = [&](const float2* f, int c, df own) { return lap5(ldd(f + w[c]), ldd(f + e[c]), ldd(f + s[c]), ldd(f + u[c]), own); };
  auto rows23 = [&] {   // kappa and mu of the current d_phi
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      kp[c] = add(s3[c], mulu(mk(K.th2), lap(ph, c, v[c])));
      if (has(c)) kap[t[c]] = f2(kp[c]);
    }
    __syncwarp();
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const df Q = norm(addu(gquot<SCH>(add(pb[c], v[c]), pb[c], pk[c]), gw[c]));
      mv[c] = norm(sum3u(s2[c], mulu(Q, v[c]), mulu(mk(K.ih2), lap(kap, c, kp[c]))));
    }
  };
  bool done = false;
#pragma unroll 1
  for (; it < 40;) {
    rows23();
#pragma unroll
    for (int c = 0; c < NC; ++c)
      if (has(c)) muv[t[c]] = f2(mv[c]);
    __syncwarp();
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const df f = sum3u(s1[c], neg(v[c]), mulu(mk(K.cmu), lap(muv, c, mv[c])));
      if (has(c)) rh[t[c]] = fadd(f.h, f.l);
    }
    __syncwarp();
    float acc[NC][2] = {};
#pragma unroll 4
    for (int q = 0; q < G; q += 2)   // every level has an even m
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        acc[c][0] = fmaf(X[q * G + t[c]], rh[q], acc[c][0]);
        acc[c][1] = fmaf(X[(q + 1) * G + t[c]], rh[q + 1], acc[c][1]);
      }
    float dm = 0.f, em = 0.f, um = 0.f;
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const float delta = acc[c][0] + acc[c][1];
      v[c] = add(v[c], df{delta, 0.f});
      if (has(c)) ph[t[c]] = f2(v[c]);
      dm = fmaxf(dm, fabsf(delta));
      if (!(delta == delta)) dm = INFINITY;
      em = fmaxf(em, fabsf(v[c].h));
      um = fmaxf(um, fabsf(v[c].h + pb[c].h));
    }
    // non-negative floats order as their bits
    const unsigned FULL = 0xffffffffu;
    const float dmax = __uint_as_float(__reduce_max_sync(FULL, __float_as_uint(dm)));
    const float emax = __uint_as_float(__reduce_max_sync(FULL, __float_as_uint(em)));
    const float umax = __uint_as_float(__reduce_max_sync(FULL, __float_as_uint(um)));
    const float tol = fmaxf(1e-15f * (1.f + umax), 1e-14f * emax);
    __syncwarp();
    done = dmax <= tol || (it > 0 && dmax * (dmax / dprev) <= tol) || !(dmax < INFINITY);
    const bool slow = it > 0 && !(dmax <= 0.01f * dprev);
    dprev = dmax;
    ++it;
    if (done) break;
    if (slow && it < 40) return false;
  }
  rows23();
#pragma unroll
  for (int c = 0; c < NC; ++c)
    if (has(c)) {
      C.d[0][id[c]] = f2(v[c]);
      C.d[1][id[c]] = f2(mv[c]);
      C.d[2][id[c]] = f2(kp[c]);
    }
  return true;
}

// The coarsest solve of a CTA of kDfTailThreads threads: J^-1 of the Jacobian at d = 0 by all of them
// (gj_invert_block), updates J^-1 F by warp 0, J^-1 again where they shrink slowly; the
// pivoting solve where a pivot is small (|.| <= 0.05: J = I + (-c L)(diag(q) + theta L^2) has a
// positive diagonal unless q < 0 dominates) or four inverses were not enough.  sm: coarse_df_smem.
// Bound by the serial chain of the eliminations' steps and of the updates: an elimination by one
// warp for every update on 8 x 6 cells, the coarse tail of 512 x 384, made that kernel 151 us, now
// 44; on 4 x 4 cells (1024^2) a warp's Gauss-Jordan elimination and a tail of three copies of the
// sweep's code 40, now 28.
template <int SCH>
__device__ __forceinline__ void coarse_df_block(const DPar& P, const float* __restrict__ K3f, float2* sm) {
  __shared__ int s_state;   // 0: solved, 1: a new inverse
  const DLev& C = P.L;
  const int G = C.m * C.n;
  float2* ph = sm;
  float2* kap = ph + G;
  float2* muv = kap + G;
  float* diag = reinterpret_cast<float*>(muv + G);
  float* rh = diag + G;
  float* X = rh + G;
  const float* cLf = K3f + G * G;
  const int tid = threadIdx.x;
  if (tid < G) ph[tid] = make_float2(0.f, 0.f);
  int it = 0;
  float dprev = 0.f;
  for (int f = 0;; ++f) {
    if (tid < G) {   // gam + W + g'(p), the Jacobian's FP32 column factor
      const size_t id = dindex(C, tid % C.m, tid / C.m);
      diag[tid] = P.k.gam.x + (SCH == 2 && C.W ? df_of(C.W[tid]).h : 0.f) +
                  df_dg32(SCH, fadd(C.pb[id].x, ph[tid].x), SCH == 2 ? C.pk[id].x : 0.f);
    }
    __syncthreads();
    auto entry = [&](int r, int q) { return fmaf(-cLf[r * G + q], diag[q], K3f[r * G + q]); };
    bool ok = f < 4;
    if (ok) {
      if (G <= 16) ok = gj_invert_block<kDfTailThreads, 16>(X, G, entry);
      else if (G <= 32) ok = gj_invert_block<kDfTailThreads, 32>(X, G, entry);
      else ok = gj_invert_block<kDfTailThreads, 64>(X, G, entry);
    }
    __syncthreads();
    if (tid < 32) {   // warp 0 holds rows: its ok is every such thread's
      if (!ok) {
        coarse_newton_df<SCH>(P, K3f, sm);
        if (tid == 0) s_state = 0;
      } else {
        const bool done = G <= 32 ? coarse_chord_pass<SCH, 1>(P, X, ph, kap, muv, rh, it, dprev)
                                  : coarse_chord_pass<SCH, 2>(P, X, ph, kap, muv, rh, it, dprev);
        if (tid == 0) s_state = done ? 0 : 1;
      }
    }
    __syncthreads();
    if (s_state == 0) return;
  }
}

// ---------------------------------------------------------------------------
// The coarse end of the V-cycle in one CTA: levels lt .. L-1 with __syncthreads between the
// phases and the per-level kernels' cell functions (the same bits).  Levels whose planes fit
// in shared memory live there: level lt's rho, p0 and red first sweep are read at the start
// and its correction is written back at the end; coarser levels exist in shared memory only
// (their phi^k excepted).  Levels that do not fit stay in global memory.
// ---------------------------------------------------------------------------
constexpr size_t kDfTailSmem = 160 * 1024;

struct DTailDim {
  int nlev, nu1, nu2, staged;   // levels 0 .. staged-1 of the tail stay in global memory
};

// lv: the levels' parameters; ready(): called once before any data another kernel wrote is read.
template <int SCH, bool NY, typename Ready>
__device__ __forceinline__ void df_tail_body(const DTailDim& A, const DPar* lv, const float* __restrict__ K3f, float2* tsm,
                                             DPar* sl, Ready ready) {
  const int tid = threadIdx.x, nt = blockDim.x;
  const DLev& Cg = lv[A.nlev - 1].L;
  const int gc = Cg.m * Cg.n;
  // K3 and c L of the coarsest grid, written once at creation: before the wait
  float* k3s = reinterpret_cast<float*>(tsm);
  for (int t = tid; t < 2 * gc * gc; t += nt) k3s[t] = K3f[t];
  float2* scratch = tsm + gc * gc;
  {
    // per-level parameters to shared memory, word by word
    const int words = (int)(sizeof(DPar) / 4) * A.nlev;
    const uint32_t* src = reinterpret_cast<const uint32_t*>(lv);
    uint32_t* dst = reinterpret_cast<uint32_t*>(sl);
    for (int t = tid; t < words; t += nt) dst[t] = src[t];
  }
  __syncthreads();
  if (tid == 0) {
    float2* p = scratch + (coarse_df_smem(gc) + 7) / 8;
    for (int l = A.staged; l < A.nlev; ++l) {
      DLev& v = sl[l].L;
      const int G = v.m * v.n;
      for (int c = 0; c < 3; ++c) {
        v.d[c] = p + c * G;
        v.r[c] = p + (3 + c) * G;
      }
      v.pb = p + 6 * G;
      p += 7 * G;
    }
  }
  __syncthreads();
  // the black half of d is zero before a level's first sweep (whose red half sweep the
  // restriction did): in global memory after the wait, in shared memory before it
  auto zero_black = [&](int l) {
    const DLev& v = sl[l].L;
    const int h = (v.m >> 1) * v.n;
    for (int t = tid; t < h; t += nt)
#pragma unroll
      for (int c = 0; c < 3; ++c) v.d[c][h + t] = make_float2(0.f, 0.f);
  };
  for (int l = A.staged; l < A.nlev; ++l) zero_black(l);
  ready();
  if (A.nu1 > 0)
    for (int l = 0; l < A.staged; ++l) zero_black(l);
  __syncthreads();
  if (A.staged == 0) {   // the tail's first level comes in from global memory
    const DLev& g = lv[0].L;
    const DLev& v = sl[0].L;
    const int G = g.m * g.n;
    for (int t = tid; t < G; t += nt) {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        v.r[c][t] = g.r[c][t];
        if (A.nu1 == 0 || t < (G >> 1)) v.d[c][t] = g.d[c][t];
      }
      v.pb[t] = g.pb[t];
    }
    __syncthreads();
  }
  // down and up as one loop, with one copy of the sweep's code: what a copy costs on its first
  // use (2 to 10 k clocks of instruction fetch) is several warm half sweeps (1.3 k)
  const int down = A.nlev - 1;
  for (int leg = 0; leg < 2 * down; ++leg) {
    const bool up = leg >= down;
    const int l = up ? 2 * down - 1 - leg : leg;
    const DPar& F = sl[l];
    const DPar& C = sl[l + 1];
    const int half = F.L.m >> 1, cells = half * F.L.n, cc = C.L.m * C.L.n;
    if (up) {
      for (int t = tid; t < 3 * cc; t += nt) {
        const int c = t / cc, q = t - c * cc;
        df_prolong_plane(C.L, F.L, c, q % C.L.m, q / C.L.m);
      }
      __syncthreads();
    }
    for (int hs = up ? 0 : 1; hs < 2 * (up ? A.nu2 : A.nu1); ++hs) {
      for (int t = tid; t < cells; t += nt) {
        const int j = t / half;
        df_smooth_cell<SCH, kGen, NY, false>(F, hs & 1, t - j * half, j);
      }
      __syncthreads();
    }
    if (!up) {
      const int zero = A.nu1 == 0 || l + 1 == down;
      for (int t = tid; t < cc; t += nt) df_restrict_cell<SCH, true, true>(F, C, t % C.L.m, t / C.L.m, zero);
      __syncthreads();
      if (l + 1 == down) {
        coarse_df_block<SCH>(sl[down], k3s, scratch);
        __syncthreads();
      }
    }
  }
  if (A.staged == 0) {
    const DLev& g = lv[0].L;
    const DLev& v = sl[0].L;
    const int G = g.m * g.n;
    for (int t = tid; t < G; t += nt)
#pragma unroll
      for (int c = 0; c < 3; ++c) g.d[c][t] = v.d[c][t];
  }
}

// Host side: coefficients in float-float.
inline float2 df_split(double x) {
  const float h = (float)x;
  return make_float2(h, (float)(x - (double)h));
}

// Whether every coefficient of the level is far inside the binary32 range.
inline bool df_coef_ok(const Coef& k) {
  const double v[] = {k.cmu, k.a, k.ih2, k.b, k.b3, k.th2, k.D0w, k.Q0, k.aw, k.a3w};
  for (double x : v)
    if (!(fabs(x) < 0x1p60 && fabs(x) > 0x1p-60)) return false;
  return fabs(k.gam) < 0x1p20;
}

inline DCoef df_coef_of(const Coef& k, int scheme, const Coef& k4) {
  DCoef d;
  d.cmu = df_split(k4.cmu);
  d.ih2 = df_split(k4.ih2);
  d.th2 = df_split(k4.th2);
  d.gam = df_split(k.gam);
  d.omega = df_split(k.omega);
  d.a = df_split(k.a);
  d.b = df_split(k.b);
  d.b3 = df_split(k.b3);
  d.Q0 = df_split(k.Q0);
  d.D0w = df_split(k.D0w);
  d.aq = df_split(scheme == 1 ? k.a3w : k.aw);
  return d;
}

}  // namespace mpfc
