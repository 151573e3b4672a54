// The FP64 handles' V-cycle in correction form (df_cells.cuh): kernels and launches.
//
// One V-cycle: k_df_defect has left rho = S - N(u) of the finest level (from an FP64
// evaluation at the FP64 iterate u) and the first red half sweep; the levels are swept,
// restricted and prolonged in float-float arithmetic; the finest level's last red and black
// half sweeps add the finished correction to u in FP64; and the next k_df_defect evaluates
// the residual again and decides whether to go on.
#include <math.h>
#include <string.h>

#include <vector>

#include "df_cells.cuh"
#include "fp64_kernels.cuh"
#include "mpfc_internal.h"

using namespace mpfc;

namespace {

// ---------------------------------------------------------------------------
// FP64 residual of the iterate: rho as float-float planes, p0 = phi, the scaled norm and
// the loop decision.  mode 0, right after the guess: rows 2 and 3 hold by construction
// (k_guess_kappa, k_guess_mu), so rho2 = rho3 = 0; phi^k is split too (scheme 2).
// FIRST: the first red half sweep on the values in registers.
// A value outside the range the float-float form covers (|phi| < 2^20, |rho| < 2^40: far
// inside binary32, the cubic included) sets ctl->range; the loop then goes on with the
// FP64 V-cycle.
// ---------------------------------------------------------------------------
struct DefectArgs {
  Lev L;
  Coef k;
  DPar P;
  Ctl* ctl;
  double* partials;
  cudaGraphConditionalHandle hnd, hnd64;   // the loop in correction form, the FP64 loop
  int mode, set_cond, zero;
};

__device__ __forceinline__ bool df_out_of_range(double x, int e) {
  return (((unsigned)__double2hiint(x) >> 20) & 0x7FFu) >= 1023u + e;
}

template <int SCH, bool MODE0, bool FIRST>
__global__ void __launch_bounds__(256) k_df_defect(const __grid_constant__ DefectArgs A) {
  pdl_enter();
  const Lev& L = A.L;
  const DLev& D = A.P.L;
  double v[1] = {0.0};
  bool bad = false;
  const int G = L.m * L.n;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < G; t += gridDim.x * blockDim.x) {
    const int i = t % L.m, j = t / L.m;
    double a, b = 0.0, c = 0.0;
    if (MODE0) {
      a = resid1_at(L, A.k, i, j);
      v[0] = fma(a, a, v[0]);
    } else {
      resid_at<SCH>(L, A.k, i, j, a, b, c);
      v[0] = fma(a, a, fma(b, b, fma(c, c, v[0])));
    }
    const double p = L.phi[t];
    bad |= df_out_of_range(p, 20) | df_out_of_range(a, 40) | df_out_of_range(b, 40) | df_out_of_range(c, 40);
    DCell q;
    q.rho1 = df_of(a);
    q.rho2 = MODE0 ? df{0.f, 0.f} : df_of(b);
    q.rho3 = MODE0 ? df{0.f, 0.f} : df_of(c);
    q.pb = df_of(p);
    q.pk = q.W = df{0.f, 0.f};
    const size_t id = dindex(D, i, j);
    D.r[0][id] = f2(q.rho1);
    D.r[1][id] = f2(q.rho2);
    D.r[2][id] = f2(q.rho3);
    D.pb[id] = f2(q.pb);
    if (SCH == 2 && MODE0) {
      q.pk = df_of(L.pk[t]);
      D.pk[id] = f2(q.pk);
    }
    if (A.zero) {
      const float2 z = make_float2(0.f, 0.f);
      D.d[0][id] = z;
      D.d[1][id] = z;
      D.d[2][id] = z;
    } else if (FIRST && !((i + j) & 1)) {
      if (SCH == 2 && !MODE0) q.pk = ldd(D.pk + id);
      if (SCH == 2 && D.W) q.W = df_of(D.W[t]);
      const df z{0.f, 0.f};
      if (D.nyn && (j == 0 || j == D.n - 1)) df_update<SCH, kAll>(A.P.kb, z, z, z, q);
      else df_update<SCH, kAll>(A.P.k, z, z, z, q);
      D.d[0][id] = f2(q.p);
      D.d[1][id] = f2(q.m);
      D.d[2][id] = f2(q.k);
    }
  }
  if (bad) atomicOr(&A.ctl->range, 1);
  if (!grid_sum<1>(v, A.partials, &A.ctl->counter)) return;
  Ctl* ctl = A.ctl;
  const double res = sqrt(v[0] / (3.0 * (double)G));
  const bool go = resnorm_next(ctl, res, A.mode);
  // residuals this small would lose the low parts' range
  const int range = *(volatile int*)&ctl->range | (go && res < 0x1p-56);
  ctl->range = range;
  if (A.set_cond) {
    cudaGraphSetConditional(A.hnd, go && !range ? 1u : 0u);
    cudaGraphSetConditional(A.hnd64, go && range ? 1u : 0u);
  }
}

// ---------------------------------------------------------------------------
// Per-level kernels
// ---------------------------------------------------------------------------
struct UPlanes {
  double* u[3];
};

// Bound by FP32 issue (about 350 instructions per cell) on the levels that stay in L2 and by
// the memory traffic (52 B per cell and half sweep) on larger ones.
template <int SCH, int MODE, bool NY, bool FINAL>
__global__ void __launch_bounds__(256) k_df_smooth(const __grid_constant__ DPar P, int color,
                                                   const __grid_constant__ UPlanes U) {
  pdl_enter();
  const int x = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y;
  if (x >= (P.L.m >> 1) || j >= P.L.n) return;
  df_smooth_cell<SCH, MODE, NY, FINAL>(P, color, x, j, U.u);
}

template <int SCH, bool FIRST, bool BASE>
__global__ void __launch_bounds__(256) k_df_restrict(const __grid_constant__ DPar F, const __grid_constant__ DPar C,
                                                     int zero) {
  pdl_enter();
  const int I = blockIdx.x * blockDim.x + threadIdx.x, J = blockIdx.y * blockDim.y + threadIdx.y;
  if (I >= C.L.m || J >= C.L.n) return;
  df_restrict_cell<SCH, FIRST, BASE>(F, C, I, J, zero);
}

__global__ void __launch_bounds__(256) k_df_base(const __grid_constant__ DPar F, const __grid_constant__ DPar C) {
  pdl_enter();
  const int I = blockIdx.x * blockDim.x + threadIdx.x, J = blockIdx.y * blockDim.y + threadIdx.y;
  if (I >= C.L.m || J >= C.L.n) return;
  df_base_cell(F.L, C.L, I, J);
}

__global__ void __launch_bounds__(256) k_df_prolong(const __grid_constant__ DPar C, const __grid_constant__ DPar F) {
  pdl_enter();
  const int I = blockIdx.x * blockDim.x + threadIdx.x, J = blockIdx.y * blockDim.y + threadIdx.y;
  if (I >= C.L.m || J >= C.L.n) return;
#pragma unroll
  for (int c = 0; c < 3; ++c) df_prolong_plane(C.L, F.L, c, I, J);
}

// u += d over the whole finest level, for V-cycles whose last half sweeps do not.
__global__ void __launch_bounds__(256) k_df_apply(const __grid_constant__ DPar P, const __grid_constant__ UPlanes U) {
  pdl_enter();
  const int G = P.L.m * P.L.n;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < G; t += gridDim.x * blockDim.x) {
    const size_t id = dindex(P.L, t % P.L.m, t / P.L.m);
#pragma unroll
    for (int c = 0; c < 3; ++c) U.u[c][t] += df_to_f64(ldd(P.L.d[c] + id));
  }
}

// phi^k onto a coarse level, FP64 (for the FP64 V-cycle) and float-float.
__global__ void k_df_restrict_pk(const double* __restrict__ f, double* __restrict__ c, const __grid_constant__ DPar C) {
  pdl_enter();
  const int I = blockIdx.x * blockDim.x + threadIdx.x, J = blockIdx.y * blockDim.y + threadIdx.y;
  if (I >= C.L.m || J >= C.L.n) return;
  const int mf = 2 * C.L.m;
  const size_t a = (size_t)(2 * J) * mf + 2 * I, b = a + mf;
  const double v = 0.25 * ((f[a] + f[a + 1]) + (f[b] + f[b + 1]));
  c[(size_t)J * C.L.m + I] = v;
  C.L.pk[dindex(C.L, I, J)] = f2(df_of(v));
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

template <int SCH>
__global__ void __launch_bounds__(32) k_df_coarse(const __grid_constant__ DPar P, const float* __restrict__ K3f) {
  extern __shared__ float2 csm[];
  pdl_enter();
  coarse_df_warp<SCH>(P, K3f, csm);
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

struct DTailArgs {
  int nlev, nu1, nu2, staged;   // levels 0 .. staged-1 of the tail stay in global memory
  const float* K3f;
  DPar lv[kDfTailMax];
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

template <int SCH, bool NY>
__global__ void __launch_bounds__(kDfTailThreads, 1) k_df_tail(const __grid_constant__ DTailArgs A) {
  extern __shared__ float2 tsm[];
  __shared__ DPar sl[kDfTailMax];
  const int tid = threadIdx.x, nt = blockDim.x;
  const DLev& Cg = A.lv[A.nlev - 1].L;
  const int gc = Cg.m * Cg.n;
  // K3 and c L of the coarsest grid, written once at creation: before the wait
  float* k3s = reinterpret_cast<float*>(tsm);
  for (int t = tid; t < 2 * gc * gc; t += nt) k3s[t] = A.K3f[t];
  float2* scratch = tsm + gc * gc;
  {
    // per-level parameters to shared memory, word by word
    const int words = (int)(sizeof(DPar) / 4) * A.nlev;
    const uint32_t* src = reinterpret_cast<const uint32_t*>(A.lv);
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
  pdl_enter();
  if (A.staged == 0) {   // the tail's first level comes in from global memory
    const DLev& g = A.lv[0].L;
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
    const DLev& g = A.lv[0].L;
    const DLev& v = sl[0].L;
    const int G = g.m * g.n;
    for (int t = tid; t < G; t += nt)
#pragma unroll
      for (int c = 0; c < 3; ++c) g.d[c][t] = v.d[c][t];
  }
}

float2 split(double x) {
  const float h = (float)x;
  return make_float2(h, (float)(x - (double)h));
}

// Whether every coefficient of the level is far inside the binary32 range.
bool coef_ok(const Coef& k) {
  const double v[] = {k.cmu, k.a, k.ih2, k.b, k.b3, k.th2, k.D0w, k.Q0, k.aw, k.a3w};
  for (double x : v)
    if (!(fabs(x) < 0x1p60 && fabs(x) > 0x1p-60)) return false;
  return fabs(k.gam) < 0x1p20;
}

DCoef dcoef_of(const Coef& k, int scheme, const Coef& k4) {
  DCoef d;
  d.cmu = split(k4.cmu);
  d.ih2 = split(k4.ih2);
  d.th2 = split(k4.th2);
  d.gam = split(k.gam);
  d.omega = split(k.omega);
  d.a = split(k.a);
  d.b = split(k.b);
  d.b3 = split(k.b3);
  d.Q0 = split(k.Q0);
  d.D0w = split(k.D0w);
  d.aq = split(scheme == 1 ? k.a3w : k.aw);
  return d;
}

DPar dpar(const mpfc_s* H, int scheme, int l) {
  DPar P;
  P.L = H->dlev[l];
  P.L.W = H->lev[l].W;
  P.k = dcoef_of(H->coef[scheme - 1][l], scheme, H->coef[scheme - 1][l]);
  P.kb = dcoef_of(H->coefb[scheme - 1][l], scheme, H->coef[scheme - 1][l]);
  return P;
}

UPlanes uplanes(const mpfc_s* H) {
  UPlanes U;
  U.u[0] = H->lev[0].phi;
  U.u[1] = H->lev[0].mu;
  U.u[2] = H->lev[0].ka;
  return U;
}

// Handles of at most 64^2 cells run the producers' extra work as launches of its own.
bool df_unfused(const mpfc_s* H) { return (long long)H->p.m * H->p.n <= 64 * 64; }

template <int SCH, int MODE, bool FINAL>
void launch_half(const mpfc_s* H, const DPar& P, int color, cudaStream_t s) {
  const mpfc_launch_shape& sh = H->shape;
  const dim3 g = mpfc_grid_of(sh, P.L.m / 2, P.L.n), b = mpfc_blk_for(sh, P.L.m / 2, P.L.n);
  if (P.L.nyn) mpfc_launch(sh, k_df_smooth<SCH, MODE, true, FINAL>, g, b, 0, s, P, color, uplanes(H));
  else mpfc_launch(sh, k_df_smooth<SCH, MODE, false, FINAL>, g, b, 0, s, P, color, uplanes(H));
}

size_t tail_smem(const mpfc_s* H, int lt, int from) {
  const int L = H->nlev;
  const size_t gc = (size_t)H->lev[L - 1].m * H->lev[L - 1].n;
  size_t cells = 0;
  for (int l = lt + from; l < L; ++l) cells += (size_t)H->lev[l].m * H->lev[l].n;
  return sizeof(float2) * (gc * gc + (coarse_df_smem((int)gc) + 7) / 8 + 7 * cells);
}

template <int SCH>
void launch_df_tail(mpfc_s* H, int lt, cudaStream_t s) {
  DTailArgs A;
  memset(&A, 0, sizeof(A));
  A.nlev = H->nlev - lt;
  A.nu1 = H->p.nu1;
  A.nu2 = H->p.nu2;
  A.K3f = H->K3[SCH - 1];
  for (int i = 0; i < A.nlev; ++i) A.lv[i] = dpar(H, SCH, lt + i);
  while (A.staged < A.nlev && tail_smem(H, lt, A.staged) > kDfTailSmem) ++A.staged;
  const size_t smem = tail_smem(H, lt, A.staged);
  if (H->dlev[0].nyn) mpfc_launch(H->shape, k_df_tail<SCH, true>, dim3(1), dim3(kDfTailThreads), smem, s, A);
  else mpfc_launch(H->shape, k_df_tail<SCH, false>, dim3(1), dim3(kDfTailThreads), smem, s, A);
}

int df_tail_first(const mpfc_s* H) {
  int lt = mpfc_tail_first_level(H);
  if (lt < H->nlev && H->nlev - lt > kDfTailMax) lt = H->nlev - kDfTailMax;
  return lt;
}

template <int SCH>
void vcycle(mpfc_s* H, cudaStream_t s) {
  const mpfc_params& p = H->p;
  const mpfc_launch_shape& sh = H->shape;
  const int L = H->nlev, lt = df_tail_first(H), down = lt < L ? lt : L - 1;
  const bool unfused = df_unfused(H);
  for (int l = 0; l < down; ++l) {
    MpfcRange range(mpfc_level_name(l));
    const DPar F = dpar(H, SCH, l), C = dpar(H, SCH, l + 1);
    if (p.nu1 > 0) {
      if (unfused) launch_half<SCH, kAll, false>(H, F, 0, s);
      launch_half<SCH, kOwn, false>(H, F, 1, s);
      for (int sw = 1; sw < p.nu1; ++sw)
        for (int color = 0; color < 2; ++color) launch_half<SCH, kGen, false>(H, F, color, s);
    }
    // the coarse level's correction starts at zero where no pre-smoothing forms it (the
    // coarsest solve writes all of it)
    const int zero = p.nu1 == 0 && l + 1 < L - 1;
    const bool first = !unfused || l + 1 == lt;   // the tail expects its first red sweep done
    const dim3 g = mpfc_grid_of(sh, C.L.m, C.L.n), b = mpfc_blk_for(sh, C.L.m, C.L.n);
    if (unfused) {
      mpfc_launch(sh, k_df_base, g, b, 0, s, F, C);
      if (first) mpfc_launch(sh, k_df_restrict<SCH, true, false>, g, b, 0, s, F, C, zero);
      else mpfc_launch(sh, k_df_restrict<SCH, false, false>, g, b, 0, s, F, C, zero);
    } else {
      mpfc_launch(sh, k_df_restrict<SCH, true, true>, g, b, 0, s, F, C, zero);
    }
  }
  {
    MpfcRange range(lt < L ? "coarse tail" : "coarsest solve");
    if (lt < L) {
      launch_df_tail<SCH>(H, lt, s);
    } else {
      const int G = H->lev[L - 1].m * H->lev[L - 1].n;
      mpfc_launch(sh, k_df_coarse<SCH>, dim3(1), dim3(32), coarse_df_smem(G), s, dpar(H, SCH, L - 1),
                  (const float*)H->K3[SCH - 1]);
    }
  }
  for (int l = down - 1; l >= 0; --l) {
    MpfcRange range(mpfc_level_name(l));
    const DPar F = dpar(H, SCH, l), C = dpar(H, SCH, l + 1);
    mpfc_launch(sh, k_df_prolong, mpfc_grid_of(sh, C.L.m, C.L.n), mpfc_blk_for(sh, C.L.m, C.L.n), 0, s, C, F);
    for (int sw = 0; sw < p.nu2; ++sw)
      for (int color = 0; color < 2; ++color) {
        if (l == 0 && sw == p.nu2 - 1) launch_half<SCH, kGen, true>(H, F, color, s);
        else launch_half<SCH, kGen, false>(H, F, color, s);
      }
  }
  if (down == 0 || p.nu2 == 0)
    mpfc_launch(sh, k_df_apply, dim3(mpfc_reduce_blocks((size_t)p.m * p.n)), dim3(256), 0, s, dpar(H, SCH, 0), uplanes(H));
}

template <int SCH>
void defect(mpfc_s* H, int mode, cudaGraphConditionalHandle hnd, int set_cond, cudaStream_t s) {
  DefectArgs A;
  memset(&A, 0, sizeof(A));
  A.L = H->lev[0];
  A.k = H->coef[SCH - 1][0];
  A.P = dpar(H, SCH, 0);
  A.ctl = H->ctl;
  A.partials = H->partials;
  A.hnd = hnd;
  A.hnd64 = H->cur_handle64;
  A.mode = mode;
  A.set_cond = set_cond;
  A.zero = H->p.nu1 == 0;
  const dim3 g(mpfc_reduce_blocks((size_t)H->p.m * H->p.n)), b(256);
  // the tail expects its first red sweep done, also where the finest level is in it
  const bool first = !df_unfused(H) || df_tail_first(H) == 0;
  if (mode == 0) {
    if (first) mpfc_launch(H->shape, k_df_defect<SCH, true, true>, g, b, 0, s, A);
    else mpfc_launch(H->shape, k_df_defect<SCH, true, false>, g, b, 0, s, A);
  } else {
    if (first) mpfc_launch(H->shape, k_df_defect<SCH, false, true>, g, b, 0, s, A);
    else mpfc_launch(H->shape, k_df_defect<SCH, false, false>, g, b, 0, s, A);
  }
}

}  // namespace

// The correction form runs on FP64 handles with at least two levels and coefficients far
// inside the binary32 range (h = 1e-6 gives (4/h^2)(4 theta/h^2) = 1e25; the FP64 V-cycle
// keeps such handles).
bool mpfc_df_usable(const mpfc_s* H) {
  if (H->p.precision != MPFC_FP64 || H->nlev < 2) return false;
  for (int s = 0; s < 2; ++s)
    for (int l = 0; l < H->nlev; ++l)
      if (!coef_ok(H->coef[s][l]) || !coef_ok(H->coefb[s][l])) return false;
  return true;
}

// Planes of the correction form.  Level 0: corrections and rho in memory of their own, p0
// and phi^k in the Poisson planes (used only by mpfc_energy); coarser levels in the FP64
// V-cycle's planes, which it writes before it reads them.
size_t mpfc_df_carve(mpfc_s* H, const mpfc_params* p, size_t* off, char* base, const Lev* lev, double* const* px,
                     double* const* pf, int nlev) {
  if (p->precision != MPFC_FP64 || nlev < 2) return 0;
  const size_t start = *off;
  auto take = [&](size_t cells) -> float2* {
    float2* q = base ? reinterpret_cast<float2*>(base + *off) : nullptr;
    *off = (*off + cells * sizeof(float2) + 255) & ~(size_t)255;
    return q;
  };
  for (int l = 0; l < nlev; ++l) {
    DLev v;
    v.m = lev[l].m;
    v.n = lev[l].n;
    v.nyn = lev[l].nyn;
    v.W = nullptr;
    const size_t G = (size_t)v.m * v.n;
    if (l == 0) {
      for (int c = 0; c < 3; ++c) v.d[c] = take(G);
      for (int c = 0; c < 3; ++c) v.r[c] = take(G);
      v.pb = reinterpret_cast<float2*>(px[0]);
      v.pk = reinterpret_cast<float2*>(pf[0]);
    } else {
      double* const d[3] = {lev[l].phi, lev[l].mu, lev[l].ka};
      double* const r[3] = {lev[l].S1, lev[l].S2, lev[l].S3};
      for (int c = 0; c < 3; ++c) {
        v.d[c] = reinterpret_cast<float2*>(d[c]);
        v.r[c] = reinterpret_cast<float2*>(r[c]);
      }
      v.pb = reinterpret_cast<float2*>(lev[l].b1);
      v.pk = reinterpret_cast<float2*>(lev[l].b2);
    }
    if (H && base) H->dlev[l] = v;
  }
  return *off - start;
}

int mpfc_df_init(mpfc_s* H) {
  if (!mpfc_df_usable(H)) return MPFC_OK;
  cudaError_t e = cudaSuccess;
  auto raise = [&](auto* k) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDfTailSmem);
  };
  raise(k_df_tail<1, false>);
  raise(k_df_tail<1, true>);
  raise(k_df_tail<2, false>);
  raise(k_df_tail<2, true>);
  if (e != cudaSuccess) {
    mpfc_set_cuda_error(e, "shared memory of the coarse tail", __FILE__, __LINE__);
    return MPFC_ERR_CUDA;
  }
  return MPFC_OK;
}

void mpfc_df_restrict_pk(mpfc_s* H, int l, cudaStream_t s) {
  const DPar C = dpar(H, 2, l);
  mpfc_launch(H->shape, k_df_restrict_pk, mpfc_grid_of(H->shape, C.L.m, C.L.n), mpfc_blk_for(H->shape, C.L.m, C.L.n), 0, s,
              (const double*)H->lev[l - 1].pk, H->lev[l].pk, C);
}

void mpfc_df_vcycle(mpfc_s* H, int scheme, cudaStream_t s) {
  if (scheme == 1) vcycle<1>(H, s);
  else vcycle<2>(H, s);
}

void mpfc_df_defect(mpfc_s* H, int scheme, int mode, cudaGraphConditionalHandle hnd, int set_cond, cudaStream_t s) {
  if (scheme == 1) defect<1>(H, mode, hnd, set_cond, s);
  else defect<2>(H, mode, hnd, set_cond, s);
}

int mpfc_df_launches_per_cycle(const mpfc_s* H) {
  const int L = H->nlev, lt = df_tail_first(H), down = lt < L ? lt : L - 1;
  const bool unfused = df_unfused(H);
  const int nu1 = H->p.nu1, nu2 = H->p.nu2;
  int per = 2 + 2 * nu2;                                           // restriction, prolongation, post-sweeps
  if (nu1 > 0) per += 2 * nu1 - 1 + (unfused ? 1 : 0);             // the first red half sweep is the producer's
  if (unfused) per += 1;                                           // p0 on its own
  return down * per + 2 + ((down == 0 || nu2 == 0) ? 1 : 0);      // + tail or coarsest solve, + residual, (+ u += d)
}
