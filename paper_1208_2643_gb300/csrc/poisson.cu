// The -1 norm's Poisson problem -Delta_h x = f, f mean-zero (App. A, (A.16)-(A.18)): V(2,2)
// red-black cycles until ||f + Delta_h x|| <= 1e-13 ||f|| (at most 60), as one CUDA graph.
//
// Like the time step's V-cycle it iterates on the change of the finest level's FP64 x from
// its FP64 residual, in float-float arithmetic on colour-split planes (df_cells.cuh), with
// every equation multiplied by h^2: a cell's update is d = (sum_nb d + F) / 4, and the coarse
// right-hand side h_c^2 R(rho) is the plain sum of the four fine h^2 rho.  The levels of at
// most 64^2 cells run in one CTA in shared memory; the coarsest grid is solved with the
// Laplacian's pseudo-inverse (FP32, refined twice against the float-float residual).
//
// One launch per half sweep and level in FP64 with a host-side loop test, and 200 sweeps on
// the coarsest grid (163 us), took 6.35 ms for mpfc_energy at 1024^2 (10 cycles); this
// takes 1.73 ms, of which the energy sums are 0.09.
#include <math.h>
#include <string.h>

#include <vector>

#include "df_cells.cuh"
#include "fp64_kernels.cuh"
#include "mpfc_internal.h"

using namespace mpfc;

namespace {

constexpr int kPoisTailCells = 64 * 64;
constexpr int kPoisTailMax = 12;
constexpr int kPoisThreads = 1024;

__device__ __forceinline__ df third() { return df{0.333333343f, -9.934108e-09f}; }

// A cell's update, d <- (sum of its real neighbours + F) / (their number).
__device__ __forceinline__ void pois_cell(const DLev& L, int color, int x, int j, double* u = nullptr,
                                          const double* scale = nullptr) {
  const size_t own = (color ? dplane(L) : 0) + (size_t)j * (L.m >> 1) + x;
  const bool edge = L.nyn && (j == 0 || j == L.n - 1);
  const DNb o = df_nb<true>(L, color, x, j, own);
  auto at = [&](size_t q) { return q == own ? df{0.f, 0.f} : ldd(L.d[0] + q); };   // a ghost is the cell itself
  const df s = addu(norm(sum4u(ldd(L.d[0] + o.c0), ldd(L.d[0] + o.cx), at(o.s), at(o.n))), ldd(L.r[0] + own));
  const df d = edge ? mul(norm(s), third()) : scale2(norm(s), 0.25f);
  L.d[0][own] = f2(d);
  if (u) u[(size_t)j * L.m + 2 * x + ((j + color) & 1)] += df_to_f64(d) * *scale;   // a power of two: exact
}

__global__ void __launch_bounds__(256) k_pois_half(const __grid_constant__ DLev L, int color, double* u, const double* scale) {
  pdl_enter();
  const int x = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y;
  if (x >= (L.m >> 1) || j >= L.n) return;
  pois_cell(L, color, x, j, u, scale);
}

// F_c = sum over the block of F + sum_nb d - 4 d, and the coarse level's first red half sweep.
__device__ __forceinline__ void pois_restrict_cell(const DLev& Fl, const DLev& C, int I, int J) {
  const DBlk b = df_block(Fl, I, J);
  const df lap = norm(addu(df_sum_out(Fl.d[0], b), scale2(df_sum_in(Fl.d[0], b), -2.0f)));
  const df v = add(df_sum_in(Fl.r[0], b), lap);
  const size_t id = dindex(C, I, J);
  C.r[0][id] = f2(v);
  if (!((I + J) & 1)) {
    C.d[0][id] = f2(C.nyn && (J == 0 || J == C.n - 1) ? mul(v, third()) : scale2(v, 0.25f));
  }
}

__global__ void __launch_bounds__(256) k_pois_restrict(const __grid_constant__ DLev F, const __grid_constant__ DLev C) {
  pdl_enter();
  const int I = blockIdx.x * blockDim.x + threadIdx.x, J = blockIdx.y * blockDim.y + threadIdx.y;
  if (I >= C.m || J >= C.n) return;
  pois_restrict_cell(F, C, I, J);
}

__global__ void __launch_bounds__(256) k_pois_prolong(const __grid_constant__ DLev C, const __grid_constant__ DLev F) {
  pdl_enter();
  const int I = blockIdx.x * blockDim.x + threadIdx.x, J = blockIdx.y * blockDim.y + threadIdx.y;
  if (I >= C.m || J >= C.n) return;
  df_prolong_plane(C, F, 0, I, J);
}

// d = P F on the coarsest grid with two refinements; the whole block.  sm: 2 G float2, G float.
__device__ void pois_coarse(const DLev& C, const float* __restrict__ P, float2* sm) {
  const int G = C.m * C.n;
  float2* x = sm;
  float2* F = sm + G;
  float* r = reinterpret_cast<float*>(F + G);
  const int t = threadIdx.x;
  const size_t id = t < G ? dindex(C, t % C.m, t / C.m) : 0;
  if (t < G) {
    F[t] = C.r[0][id];
    x[t] = make_float2(0.f, 0.f);
  }
  __syncthreads();
  for (int it = 0; it < 3; ++it) {
    if (t < G) {
      const int i = t % C.m, j = t / C.m;
      const df lap = lap5(ldd(x + j * C.m + wrapm(i - 1, C.m)), ldd(x + j * C.m + wrapm(i + 1, C.m)),
                          ldd(x + ywrap(j - 1, C.n, C.nyn) * C.m + i), ldd(x + ywrap(j + 1, C.n, C.nyn) * C.m + i), ldd(x + t));
      const df q = addu(mk(F[t]), lap);
      r[t] = fadd(q.h, q.l);
    }
    __syncthreads();
    if (t < G) {
      float v = 0.f;
      for (int q = 0; q < G; ++q) v = fmaf(P[(size_t)t * G + q], r[q], v);
      x[t] = f2(add(mk(x[t]), df{v, 0.f}));
    }
    __syncthreads();
  }
  if (t < G) C.d[0][id] = x[t];
}

struct PoisTail {
  int nlev;
  const float* P;
  DLev lv[kPoisTailMax];
};

__device__ __forceinline__ void pois_tail_half(const DLev& L, int color) {
  const int half = L.m >> 1, cells = half * L.n;
  for (int t = threadIdx.x; t < cells; t += blockDim.x) pois_cell(L, color, t % half, t / half);
  __syncthreads();
}

// The levels of at most kPoisTailCells cells in shared memory; the first one's F and red
// half sweep come in from global memory and its d goes back.
__global__ void __launch_bounds__(kPoisThreads) k_pois_tail(const __grid_constant__ PoisTail A) {
  extern __shared__ float2 psm[];
  __shared__ DLev sl[kPoisTailMax];
  const int tid = threadIdx.x, nt = blockDim.x;
  const int gc = A.lv[A.nlev - 1].m * A.lv[A.nlev - 1].n;
  if (tid == 0) {
    float2* p = psm + 3 * gc;
    for (int l = 0; l < A.nlev; ++l) {
      DLev v = A.lv[l];
      v.d[0] = p;
      v.r[0] = p + v.m * v.n;
      p += 2 * v.m * v.n;
      sl[l] = v;
    }
  }
  __syncthreads();
  pdl_enter();
  const DLev& g = A.lv[0];
  const int G = g.m * g.n;
  for (int t = tid; t < G; t += nt) {
    sl[0].r[0][t] = g.r[0][t];
    if (t < (G >> 1)) sl[0].d[0][t] = g.d[0][t];
  }
  __syncthreads();
  for (int l = 0; l < A.nlev - 1; ++l) {
    const DLev& F = sl[l];
    const DLev& C = sl[l + 1];
    pois_tail_half(F, 1);
    pois_tail_half(F, 0);
    pois_tail_half(F, 1);
    const int cc = C.m * C.n;
    for (int t = tid; t < cc; t += nt) pois_restrict_cell(F, C, t % C.m, t / C.m);
    __syncthreads();
  }
  pois_coarse(sl[A.nlev - 1], A.P, psm);
  __syncthreads();
  for (int l = A.nlev - 2; l >= 0; --l) {
    const DLev& F = sl[l];
    const DLev& C = sl[l + 1];
    const int cc = C.m * C.n;
    for (int t = tid; t < cc; t += nt) df_prolong_plane(C, F, 0, t % C.m, t / C.m);
    __syncthreads();
    for (int sw = 0; sw < 2; ++sw)
      for (int color = 0; color < 2; ++color) pois_tail_half(F, color);
  }
  for (int t = tid; t < G; t += nt) g.d[0][t] = sl[0].d[0][t];
}

// x += d over the whole level (a hierarchy that is all tail).
__global__ void __launch_bounds__(256) k_pois_apply(const __grid_constant__ DLev L, double* u, const double* scale) {
  pdl_enter();
  const int G = L.m * L.n;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < G; t += gridDim.x * blockDim.x)
    u[t] += df_to_f64(ldd(L.d[0] + dindex(L, t % L.m, t / L.m))) * *scale;
}

// x = 0, f = rhs - mean; sums: 1 sum f^2, 2 cycles (0), 3 the power of two nearest below
// 1 / rms(h^2 f), by which F is scaled into the middle of the binary32 range, and 4 its inverse.
__global__ void __launch_bounds__(256) k_pois_start(const double* __restrict__ rhs, double* __restrict__ f,
                                                    double* __restrict__ x, int G, double h2, Ctl* ctl,
                                                    double* partials) {
  pdl_enter();
  const double mean = ctl->sums[0] / (double)G;
  double v[1] = {0.0};
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < G; t += gridDim.x * blockDim.x) {
    const double r = rhs[t] - mean;
    f[t] = r;
    x[t] = 0.0;
    v[0] = fma(r, r, v[0]);
  }
  if (!grid_sum<1>(v, partials, &ctl->counter)) return;
  const double rms = h2 * sqrt(v[0] / (double)G);
  const int e = rms > 0.0 && !isinf(rms) ? min(max(ilogb(rms), -1000), 1000) : 0;
  ctl->sums[0] = v[0];
  ctl->sums[1] = v[0];
  ctl->sums[2] = 0.0;
  ctl->sums[3] = scalbn(1.0, -e);
  ctl->sums[4] = scalbn(1.0, e);
}

// F = h^2 (f + Delta_h x) in FP64, scaled and split; the first red half sweep; the sum of
// squared residuals (sums[0]) and the loop decision.  FIRST: before the first cycle (x = 0).
template <bool FIRST>
__global__ void __launch_bounds__(256) k_pois_resid(const double* __restrict__ x, const double* __restrict__ f,
                                                    const __grid_constant__ DLev L, double h2, double ih2, Ctl* ctl,
                                                    double* partials, cudaGraphConditionalHandle hnd) {
  pdl_enter();
  const double scale = ctl->sums[3];
  double v[1] = {0.0};
  const int m = L.m, n = L.n, G = m * n;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < G; t += gridDim.x * blockDim.x) {
    const int i = t % m, j = t / m;
    double F = h2 * f[t];
    if (!FIRST) {
      const int im = wrapm(i - 1, m), ip = wrapm(i + 1, m), jm = ywrap(j - 1, n, L.nyn), jp = ywrap(j + 1, n, L.nyn);
      const double s = (x[(size_t)j * m + im] + x[(size_t)j * m + ip]) + (x[(size_t)jm * m + i] + x[(size_t)jp * m + i]);
      F = fma(h2, f[t], fma(-4.0, x[t], s));
      const double r = F * ih2;
      v[0] = fma(r, r, v[0]);
    }
    const df q = df_of(F * scale);
    const size_t id = dindex(L, i, j);
    L.r[0][id] = f2(q);
    if (!((i + j) & 1)) L.d[0][id] = f2(L.nyn && (j == 0 || j == n - 1) ? mul(q, third()) : scale2(q, 0.25f));
  }
  if (FIRST) {
    // a zero or non-finite right-hand side: x = 0
    if (blockIdx.x == 0 && threadIdx.x == 0) cudaGraphSetConditional(hnd, ctl->sums[1] > 0.0 && !isinf(ctl->sums[1]) ? 1u : 0u);
    return;
  }
  if (!grid_sum<1>(v, partials, &ctl->counter)) return;
  ctl->sums[0] = v[0];
  ctl->sums[2] += 1.0;
  const bool go = v[0] > 1e-26 * ctl->sums[1] && ctl->sums[2] < 60.0;   // a NaN ends the loop
  cudaGraphSetConditional(hnd, go ? 1u : 0u);
}

// The levels' planes: corrections and right-hand sides in the levels' Poisson planes, on the
// finest level (whose x and f are FP64 there) in mu's and kappa's, which every step writes
// before it reads them.
DLev plev(const mpfc_s* H, int l) {
  DLev v;
  memset(&v, 0, sizeof(v));
  v.m = H->lev[l].m;
  v.n = H->lev[l].n;
  v.nyn = H->lev[l].nyn;
  v.d[0] = reinterpret_cast<float2*>(l ? H->px[l] : H->lev[0].mu);
  v.r[0] = reinterpret_cast<float2*>(l ? H->pf[l] : H->lev[0].ka);
  return v;
}

int pois_tail_first(const mpfc_s* H) {
  int lt = H->nlev - 1;
  while (lt > 0 && H->nlev - lt < kPoisTailMax && (long long)H->lev[lt - 1].m * H->lev[lt - 1].n <= kPoisTailCells) --lt;
  return lt;
}

size_t pois_tail_smem(const mpfc_s* H, int lt) {
  size_t cells = 0;
  for (int l = lt; l < H->nlev; ++l) cells += (size_t)H->lev[l].m * H->lev[l].n;
  const size_t gc = (size_t)H->lev[H->nlev - 1].m * H->lev[H->nlev - 1].n;
  return sizeof(float2) * (3 * gc + 2 * cells);
}

void pois_half(const mpfc_s* H, const DLev& L, int color, double* u, cudaStream_t s) {
  const mpfc_launch_shape& sh = H->pshape;
  mpfc_launch(sh, k_pois_half, mpfc_grid_of(sh, L.m / 2, L.n), mpfc_blk_for(sh, L.m / 2, L.n), 0, s, L, color, u,
              (const double*)&H->ctl->sums[4]);
}

void pois_body(mpfc_s* H, int, cudaStream_t s) {
  const mpfc_launch_shape& sh = H->pshape;
  const int lt = pois_tail_first(H);
  for (int l = 0; l < lt; ++l) {
    const DLev F = plev(H, l), C = plev(H, l + 1);
    pois_half(H, F, 1, nullptr, s);
    pois_half(H, F, 0, nullptr, s);
    pois_half(H, F, 1, nullptr, s);
    mpfc_launch(sh, k_pois_restrict, mpfc_grid_of(sh, C.m, C.n), mpfc_blk_for(sh, C.m, C.n), 0, s, F, C);
  }
  PoisTail A;
  memset(&A, 0, sizeof(A));
  A.nlev = H->nlev - lt;
  A.P = H->poisP;
  for (int i = 0; i < A.nlev; ++i) A.lv[i] = plev(H, lt + i);
  mpfc_launch(sh, k_pois_tail, dim3(1), dim3(kPoisThreads), pois_tail_smem(H, lt), s, A);
  for (int l = lt - 1; l >= 0; --l) {
    const DLev F = plev(H, l), C = plev(H, l + 1);
    mpfc_launch(sh, k_pois_prolong, mpfc_grid_of(sh, C.m, C.n), mpfc_blk_for(sh, C.m, C.n), 0, s, C, F);
    for (int sw = 0; sw < 2; ++sw)
      for (int color = 0; color < 2; ++color) pois_half(H, F, color, l == 0 && sw == 1 ? H->px[0] : nullptr, s);
  }
  const DLev L0 = plev(H, 0);
  const dim3 g(mpfc_reduce_blocks((size_t)L0.m * L0.n)), b(256);
  if (lt == 0) mpfc_launch(sh, k_pois_apply, g, b, 0, s, L0, H->px[0], (const double*)&H->ctl->sums[4]);
  const double h = H->lev[0].h;
  mpfc_launch(sh, k_pois_resid<false>, g, b, 0, s, (const double*)H->px[0], (const double*)H->pf[0], L0, h * h,
              1.0 / (h * h), H->ctl, H->partials, H->cur_handle);
}

}  // namespace

// Pseudo-inverse of the coarsest grid's 4 I - (neighbour sums) (with the boundary rule):
// (A + J / G)^-1 - J / G, J all ones, by Gauss-Jordan elimination with partial pivoting.
int mpfc_pois_init(mpfc_s* H) {
  const Lev& C = H->lev[H->nlev - 1];
  const int m = C.m, n = C.n, G = m * n, W = 2 * G;
  std::vector<double> A((size_t)G * W, 0.0);
  for (int j = 0; j < n; ++j)
    for (int i = 0; i < m; ++i) {
      const int r = j * m + i;
      A[(size_t)r * W + r] += 4.0;
      const int js = C.nyn ? (j > 0 ? j - 1 : 0) : (j + n - 1) % n, jn = C.nyn ? (j < n - 1 ? j + 1 : n - 1) : (j + 1) % n;
      const int nb[4] = {j * m + (i + m - 1) % m, j * m + (i + 1) % m, js * m + i, jn * m + i};
      for (int q = 0; q < 4; ++q) A[(size_t)r * W + nb[q]] -= 1.0;
      for (int q = 0; q < G; ++q) A[(size_t)r * W + q] += 1.0 / G;
      A[(size_t)r * W + G + r] = 1.0;
    }
  for (int c = 0; c < G; ++c) {
    int piv = c;
    for (int r = c + 1; r < G; ++r)
      if (fabs(A[(size_t)r * W + c]) > fabs(A[(size_t)piv * W + c])) piv = r;
    if (piv != c)
      for (int q = 0; q < W; ++q) {
        const double t = A[(size_t)c * W + q];
        A[(size_t)c * W + q] = A[(size_t)piv * W + q];
        A[(size_t)piv * W + q] = t;
      }
    const double rp = 1.0 / A[(size_t)c * W + c];
    for (int q = 0; q < W; ++q) A[(size_t)c * W + q] *= rp;
    for (int r = 0; r < G; ++r) {
      if (r == c) continue;
      const double f = A[(size_t)r * W + c];
      for (int q = 0; q < W; ++q) A[(size_t)r * W + q] -= f * A[(size_t)c * W + q];
    }
  }
  std::vector<float> P((size_t)G * G);
  for (int r = 0; r < G; ++r)
    for (int c = 0; c < G; ++c) P[(size_t)r * G + c] = (float)(A[(size_t)r * W + G + c] - 1.0 / G);
  H->pshape = mpfc_default_launch_shape(MPFC_FP32_INNER, false);
  cudaError_t e = cudaFuncSetAttribute(k_pois_tail, cudaFuncAttributeMaxDynamicSharedMemorySize, 128 * 1024);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(H->poisP, P.data(), P.size() * sizeof(float), cudaMemcpyHostToDevice, H->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(H->stream);
  if (e != cudaSuccess) {
    mpfc_set_cuda_error(e, "Poisson solve's coarsest grid", __FILE__, __LINE__);
    return MPFC_ERR_CUDA;
  }
  return MPFC_OK;
}

// Solves for psi^k (H->psik) on the handle's stream; the result is H->px[0].  Asynchronous.
int mpfc_pois_solve(mpfc_s* H) {
  if (!H->pois_exec) {
    cudaStream_t cs = H->cap_stream;
    cudaGraph_t graph = nullptr;
    cudaGraphConditionalHandle hnd;
    cudaError_t e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
    cudaStreamCaptureStatus st;
    const cudaGraphNode_t* deps = nullptr;
    size_t ndeps = 0;
    if (e == cudaSuccess) e = cudaStreamGetCaptureInfo(cs, &st, nullptr, &graph, &deps, nullptr, &ndeps);
    if (e == cudaSuccess) e = cudaGraphConditionalHandleCreate(&hnd, graph, 0, 0);
    if (e != cudaSuccess) {
      mpfc_set_cuda_error(e, "capture of the Poisson solve", __FILE__, __LINE__);
      mpfc_abort_capture(cs);
      return MPFC_ERR_CUDA;
    }
    const mpfc_launch_shape& sh = H->pshape;
    const int G = H->p.m * H->p.n;
    const dim3 g(mpfc_reduce_blocks((size_t)G)), b(256);
    const double h = H->lev[0].h;
    mpfc_launch(sh, k_sum1, g, b, 0, cs, (const double*)H->psik, G, H->ctl, H->partials);
    mpfc_launch(sh, k_pois_start, g, b, 0, cs, (const double*)H->psik, H->pf[0], H->px[0], G, h * h, H->ctl,
                H->partials);
    mpfc_launch(sh, k_pois_resid<true>, g, b, 0, cs, (const double*)H->px[0], (const double*)H->pf[0], plev(H, 0), h * h,
                1.0 / (h * h), H->ctl, H->partials, hnd);
    H->cur_handle = hnd;
    const int rc = mpfc_capture_while(H, cs, hnd, &pois_body, 0);
    if (rc != MPFC_OK) {
      mpfc_abort_capture(cs);
      return rc;
    }
    e = cudaStreamEndCapture(cs, &graph);
    if (e == cudaSuccess) {
      e = cudaGraphInstantiate(&H->pois_exec, graph, 0);
      cudaGraphDestroy(graph);
    }
    if (e != cudaSuccess) {
      H->pois_exec = nullptr;
      mpfc_set_cuda_error(e, "cudaGraphInstantiate(Poisson solve)", __FILE__, __LINE__);
      return MPFC_ERR_CUDA;
    }
  }
  const cudaError_t e = cudaGraphLaunch(H->pois_exec, H->stream);
  if (e != cudaSuccess) {
    mpfc_set_cuda_error(e, "cudaGraphLaunch(Poisson solve)", __FILE__, __LINE__);
    return MPFC_ERR_CUDA;
  }
  return MPFC_OK;
}
