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
// F in float-float and the same FP32 linear solves.  Stops once the applied update is below
// 1e-15 (1 + |p0 + d|_inf), as there, or below 1e-14 |d|_inf, the arithmetic's resolution.
// One warp; sm: 6 G float2 and the FP32 part.
// ---------------------------------------------------------------------------
__device__ __forceinline__ df nblap_df(const float2* f, int m, int n, int t, int nyn) {
  const int i = t % m, j = t / m;
  return lap5(ldd(f + j * m + wrapm(i - 1, m)), ldd(f + j * m + wrapm(i + 1, m)), ldd(f + ywrap(j - 1, n, nyn) * m + i),
              ldd(f + ywrap(j + 1, n, nyn) * m + i), ldd(f + t));
}

__host__ __device__ constexpr size_t coarse_df_smem(int G) { return sizeof(float2) * 7 * (size_t)G + sizeof(float) * ((size_t)G * (G + 1) + (size_t)G); }

template <int SCH, int R>
__device__ void coarse_newton_df(const DPar& P, const float* __restrict__ K3f, float2* sm) {
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
  float2* muv = s2;   // row 2's value replaces rho2 for an iteration (rho2 stays in global memory)
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
  constexpr int RR = R > 0 ? R : 1;
  float k3c[RR], lcc[RR];
  const float* cLf = K3f + G * G;
  if (R > 0) {
#pragma unroll
    for (int r = 0; r < RR; ++r) {
      k3c[r] = (lane < G && r < G) ? K3f[r * G + lane] : 0.f;
      lcc[r] = (lane < G && r < G) ? cLf[r * G + lane] : 0.f;
    }
  }
  auto wt = [&](int t) { return C.W ? df_of(C.W[t]) : df{0.f, 0.f}; };
  auto kappa_at = [&](int t) { return add(mk(s3[t]), mulu(mk(K.th2), nblap_df(ph, m, n, t, C.nyn))); };
  auto mu_at = [&](int t) {
    const df dd = mk(ph[t]), p0 = mk(pb[t]);
    df Q = norm(addu(gquot<SCH>(add(p0, dd), p0, mk(pk[t])), mk(K.gam)));
    if (SCH == 2 && C.W) Q = add(Q, wt(t));
    return norm(sum3u(ldd(C.r[1] + dindex(C, t % m, t / m)), mulu(Q, dd), mulu(mk(K.ih2), nblap_df(kap, m, n, t, C.nyn))));
  };
  auto rhs_at = [&](int t) {
    const df f = sum3u(mk(s1[t]), neg(mk(ph[t])), mulu(mk(K.cmu), nblap_df(muv, m, n, t, C.nyn)));
    return fadd(f.h, f.l);
  };
  auto diag_at = [&](int t) {   // gam + W + g'(p), the Jacobian's FP32 column factor
    const float p = fadd(pb[t].x, ph[t].x), q = pk[t].x;
    const float g = SCH == 1 ? 3.f * p * p : 0.25f * (3.f * p * p + 2.f * p * q + q * q);
    return K.gam.x + (SCH == 2 && C.W ? wt(t).h : 0.f) + g;
  };
  bool refactor = true;
  float dprev = 0.f;
  for (int it = 0; it < 40; ++it) {
    for (int t = lane; t < G; t += 32) kap[t] = f2(kappa_at(t));
    __syncwarp();
    for (int t = lane; t < G; t += 32) muv[t] = f2(mu_at(t));
    __syncwarp();
    float dmax = 0.f, umax = 0.f, emax = 0.f;
    if (R == 16) {
      // chord iteration with J^-1 of a lagged Jacobian, as in coarse_newton
      float* Xs = Jm;
      float* rh = Jm + G * G;
      int* pivs = reinterpret_cast<int*>(d);
      for (int t = lane; t < G; t += 32) rh[t] = rhs_at(t);
      if (refactor) {
        for (int t = lane; t < G; t += 32) d[t] = diag_at(t);
        __syncwarp();
        float a[16];
        const float dc = lane < G ? d[lane] : 0.f;
#pragma unroll
        for (int r = 0; r < 16; ++r)
          a[r] = lane < G ? fmaf(-lcc[r], dc, k3c[r]) : ((lane < 2 * G && lane - G == r) ? 1.f : 0.f);
        __syncwarp();   // d is free from here: pivot indices
        gj_eliminate<16>(a, G, pivs);
        if (lane >= G && lane < 2 * G)
#pragma unroll
          for (int r = 0; r < 16; ++r)
            if (r < G) Xs[r * G + (lane - G)] = a[r];
      }
      __syncwarp();
      float delta = 0.f;
      if (lane < G) {
        const float* xrow = Xs + pivs[lane] * G;
        for (int q = 0; q < G; ++q) delta = fmaf(xrow[q], rh[q], delta);
        const df pn = add(mk(ph[lane]), df{delta, 0.f});
        ph[lane] = f2(pn);
        dmax = fabsf(delta);
        emax = fabsf(pn.h);
        umax = fabsf(pn.h + pb[lane].x);
      }
    } else {
      for (int t = lane; t < G; t += 32) Jm[t * W + G] = rhs_at(t);
      for (int t = lane; t < G; t += 32) d[t] = diag_at(t);
      __syncwarp();
      if (R > 0) {
        float a[RR];
        const float dc = lane < G ? d[lane] : 0.f;
#pragma unroll
        for (int r = 0; r < RR; ++r) {
          const float rhs = (lane == G && r < G) ? Jm[r * W + G] : 0.f;
          a[r] = lane < G ? fmaf(-lcc[r], dc, k3c[r]) : rhs;
        }
        __syncwarp();   // Jm is free from here: pivot scratch
        gauss_jordan_cols<RR>(a, G, d, Jm + G, reinterpret_cast<int*>(Jm));
      } else {
        for (int idx = lane; idx < G * G; idx += 32) {
          const int r = idx / G, col = idx % G;
          Jm[r * W + col] = K3f[idx] - cLf[idx] * d[col];
        }
        __syncwarp();
        gauss_shared(Jm, d, G);
      }
      for (int t = lane; t < G; t += 32) {
        const df pn = add(mk(ph[t]), df{d[t], 0.f});
        ph[t] = f2(pn);
        dmax = fmaxf(dmax, fabsf(d[t]));
        emax = fmaxf(emax, fabsf(pn.h));
        umax = fmaxf(umax, fabsf(pn.h + pb[t].x));
      }
    }
    for (int o = 16; o > 0; o >>= 1) {
      dmax = fmaxf(dmax, __shfl_xor_sync(FULL, dmax, o));
      emax = fmaxf(emax, __shfl_xor_sync(FULL, emax, o));
      umax = fmaxf(umax, __shfl_xor_sync(FULL, umax, o));
    }
    __syncwarp();
    if (!(dmax == dmax) || dmax <= fmaxf(1e-15f * (1.f + umax), 1e-14f * emax)) break;
    refactor = it > 0 && !(dmax <= 0.01f * dprev);
    dprev = dmax;
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

template <int SCH>
__device__ void coarse_df_warp(const DPar& P, const float* __restrict__ K3f, float2* sm) {
  const int G = P.L.m * P.L.n;
  if (G <= 16) coarse_newton_df<SCH, 16>(P, K3f, sm);
  else if (G <= 31) coarse_newton_df<SCH, 32>(P, K3f, sm);
  else coarse_newton_df<SCH, 0>(P, K3f, sm);
}

// ---------------------------------------------------------------------------
// The coarse end of the V-cycle in one CTA: levels lt .. L-1 with __syncthreads between the
// phases and the per-level kernels' cell functions (the same bits).  Levels whose planes fit
// in shared memory live there: level lt's rho, p0 and red first sweep are read at the start
// and its correction is written back at the end; coarser levels exist in shared memory only
// (their phi^k excepted).  Levels that do not fit stay in global memory.
// ---------------------------------------------------------------------------
constexpr int kDfTailMax = 10;
constexpr int kDfTailThreads = 512;
constexpr size_t kDfTailSmem = 160 * 1024;

struct DTailDim {
  int nlev, nu1, nu2, staged;   // levels 0 .. staged-1 of the tail stay in global memory
};

template <int SCH, int MODE, bool NY>
__device__ __forceinline__ void df_tail_half(const DPar& P, int color) {
  const int half = P.L.m >> 1, cells = half * P.L.n;
  for (int t = threadIdx.x; t < cells; t += blockDim.x) {
    const int j = t / half;
    df_smooth_cell<SCH, MODE, NY, false>(P, color, t - j * half, j);
  }
  __syncthreads();
}

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
  ready();
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
  for (int l = 0; l < A.nlev - 1; ++l) {
    const DPar& F = sl[l];
    const DPar& C = sl[l + 1];
    if (A.nu1 > 0) {
      df_tail_half<SCH, kOwn, NY>(F, 1);
      for (int sw = 1; sw < A.nu1; ++sw)
        for (int color = 0; color < 2; ++color) df_tail_half<SCH, kGen, NY>(F, color);
    }
    const int cc = C.L.m * C.L.n;
    const int zero = A.nu1 == 0 || l + 1 == A.nlev - 1;
    for (int t = tid; t < cc; t += nt) df_restrict_cell<SCH, true, true>(F, C, t % C.L.m, t / C.L.m, zero);
    __syncthreads();
  }
  if (tid < 32) coarse_df_warp<SCH>(sl[A.nlev - 1], k3s, scratch);
  __syncthreads();
  for (int l = A.nlev - 2; l >= 0; --l) {
    const DPar& F = sl[l];
    const DPar& C = sl[l + 1];
    const int cc = C.L.m * C.L.n;
    for (int t = tid; t < 3 * cc; t += nt) {
      const int c = t / cc, q = t - c * cc;
      df_prolong_plane(C.L, F.L, c, q % C.L.m, q / C.L.m);
    }
    __syncthreads();
    for (int sw = 0; sw < A.nu2; ++sw)
      for (int color = 0; color < 2; ++color) df_tail_half<SCH, kGen, NY>(F, color);
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
