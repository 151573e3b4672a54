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

#include "df_kernels.cuh"
#include "df_leg.cuh"
#include "mpfc_internal.h"

using namespace mpfc;

namespace {

// ---------------------------------------------------------------------------
// FP64 residual of the iterate (df_defect_pair), the scaled norm and the loop decision.
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

template <int SCH, bool MODE0, bool FIRST>
__global__ void __launch_bounds__(256, 5) k_df_defect(const __grid_constant__ DefectArgs A) {
  pdl_enter();
  DSum sum{0.0, df{0.f, 0.f}};
  const float scale = MODE0 ? 1.0f : df_norm_scale(A.ctl->res);
  bool bad = false;
  const int half = A.L.m >> 1;
  for (int j = blockIdx.y * blockDim.y + threadIdx.y; j < A.L.n; j += gridDim.y * blockDim.y)
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < half; x += gridDim.x * blockDim.x)
      df_defect_pair<SCH, MODE0, FIRST>(A.L, A.k, A.P, x, j, A.zero, scale, sum, bad);
  double v[1] = {df_warp_sum<MODE0>(sum, scale)};
  if (bad) atomicOr(&A.ctl->range, 1);
  if (!grid_sum<1, true>(v, A.partials, &A.ctl->counter)) return;
  Ctl* ctl = A.ctl;
  const double res = sqrt(v[0] / (3.0 * (double)(A.L.m * A.L.n)));
  const bool go = resnorm_next(ctl, res, A.mode);
  // residuals this small would lose the low parts' range
  const int range = *(volatile int*)&ctl->range | (go && res < kDfMinResidual);
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

// Bound by instruction issue (536 instructions per cell, slots 74 % busy: 13 us at 1024^2) on the
// levels that stay in L2 and by the memory traffic (52 B per cell and half sweep) on larger ones.
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

template <int SCH>
__global__ void __launch_bounds__(kDfTailThreads) k_df_coarse(const __grid_constant__ DPar P, const float* __restrict__ K3f) {
  extern __shared__ float2 csm[];
  pdl_enter();
  coarse_df_block<SCH>(P, K3f, csm);
}

struct DTailArgs {
  DTailDim d;
  const float* K3f;
  DPar lv[kDfTailMax];
};

template <int SCH, bool NY>
__global__ void __launch_bounds__(kDfTailThreads, 1) k_df_tail(const __grid_constant__ DTailArgs A) {
  extern __shared__ float2 tsm[];
  __shared__ DPar sl[kDfTailMax];
  df_tail_body<SCH, NY>(A.d, A.lv, A.K3f, tsm, sl, [] { pdl_enter(); });
}

DPar dpar(const mpfc_s* H, int scheme, int l) {
  DPar P;
  P.L = H->dlev[l];
  P.L.W = H->lev[l].W;
  P.k = df_coef_of(H->coef[scheme - 1][l], scheme, H->coef[scheme - 1][l]);
  P.kb = df_coef_of(H->coefb[scheme - 1][l], scheme, H->coef[scheme - 1][l]);
  return P;
}

UPlanes uplanes(const mpfc_s* H) {
  UPlanes U;
  U.u[0] = H->lev[0].phi;
  U.u[1] = H->lev[0].mu;
  U.u[2] = H->lev[0].ka;
  return U;
}

// Handles of at most 64^2 cells run the producers' extra work as launches of its own and take no
// one-launch ways, so that a level keeps the 11 launches that mpfc_launch_counts states for them
// (tests/test_gpu_fp64.py, test_launch_counts).  That is not the faster shape: four steps at 64^2
// take 1.59 ms with it and 1.24 without, with the same bits.
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
  A.d.nlev = H->nlev - lt;
  A.d.nu1 = H->p.nu1;
  A.d.nu2 = H->p.nu2;
  A.K3f = H->K3[SCH - 1];
  for (int i = 0; i < A.d.nlev; ++i) A.lv[i] = dpar(H, SCH, lt + i);
  while (A.d.staged < A.d.nlev && tail_smem(H, lt, A.d.staged) > kDfTailSmem) ++A.d.staged;
  const size_t smem = tail_smem(H, lt, A.d.staged);
  if (H->dlev[0].nyn) mpfc_launch(H->shape, k_df_tail<SCH, true>, dim3(1), dim3(kDfTailThreads), smem, s, A);
  else mpfc_launch(H->shape, k_df_tail<SCH, false>, dim3(1), dim3(kDfTailThreads), smem, s, A);
}

int df_tail_first(const mpfc_s* H) {
  int lt = mpfc_tail_first_level(H, H->shape);
  if (lt < H->nlev && H->nlev - lt > kDfTailMax) lt = H->nlev - kDfTailMax;
  return lt;
}

// Levels that take one launch a way (df_leg.cuh): those of at most kLegCells cells above the
// tail, with pre- and post-sweeps.  At 512^2 a launch's updates already take what the launch does and
// the halo's only add to them: two steps at 1024^2 in 3.12 ms with that level too, 3.03 without; at
// 512^2 3.04 and 2.84.
constexpr long long kLegCells = 256 * 256;
bool df_leg_level(const mpfc_s* H, int l) {
  const int nu1 = H->p.nu1, nu2 = H->p.nu2, lt = df_tail_first(H);
  return !df_unfused(H) && l < (lt < H->nlev ? lt : H->nlev - 1) && nu1 >= 1 && nu1 <= kLegMaxNu && nu2 >= 1 &&
         nu2 <= kLegMaxNu && (long long)H->dlev[l].m * H->dlev[l].n <= kLegCells;
}

dim3 leg_grid(const DLev& L) { return dim3((L.m + kLegTile - 1) / kLegTile, (L.n + kLegTile - 1) / kLegTile); }

template <int SCH>
void launch_down(mpfc_s* H, const DPar& F, const DPar& C, bool first, cudaStream_t s) {
  const size_t smem = leg_smem(H->p.nu1, SCH, F.L.W != nullptr, false);
  auto go = [&](auto* k) { mpfc_launch(H->shape, k, leg_grid(F.L), dim3(kLegThreads), smem, s, F, C, H->p.nu1); };
  if (F.L.nyn) go(first ? k_df_down<SCH, true, true> : k_df_down<SCH, true, false>);
  else go(first ? k_df_down<SCH, false, true> : k_df_down<SCH, false, false>);
}

// The way up of level l; returns the level with its correction's planes.
template <int SCH>
DPar launch_up(mpfc_s* H, int l, const DPar& C, cudaStream_t s) {
  DPar F = dpar(H, SCH, l);
  LegOut O;
  memset(&O, 0, sizeof(O));
  for (int c = 0; c < 3; ++c) {
    if (l == 0) O.u[c] = uplanes(H).u[c];
    else O.e[c] = H->de[l][c];
  }
  const size_t smem = leg_smem(H->p.nu2, SCH, F.L.W != nullptr, true);
  auto go = [&](auto* k) { mpfc_launch(H->shape, k, leg_grid(F.L), dim3(kLegThreads), smem, s, C, F, O, H->p.nu2); };
  if (F.L.nyn) go(k_df_up<SCH, true>);
  else go(k_df_up<SCH, false>);
  for (int c = 0; c < 3; ++c) F.L.d[c] = O.e[c];
  return F;
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
    const bool first = (!unfused && !df_leg_level(H, l + 1)) || l + 1 == lt;   // the tail expects its first red sweep done
    if (df_leg_level(H, l)) {
      launch_down<SCH>(H, F, C, first, s);
      continue;
    }
    if (p.nu1 > 0) {
      if (unfused) launch_half<SCH, kAll, false>(H, F, 0, s);
      launch_half<SCH, kOwn, false>(H, F, 1, s);
      for (int sw = 1; sw < p.nu1; ++sw)
        for (int color = 0; color < 2; ++color) launch_half<SCH, kGen, false>(H, F, color, s);
    }
    // the coarse level's correction starts at zero where no pre-smoothing forms it (the
    // coarsest solve writes all of it)
    const int zero = p.nu1 == 0 && l + 1 < L - 1;
    const dim3 g = mpfc_grid_of(sh, C.L.m, C.L.n), b = mpfc_blk_for(sh, C.L.m, C.L.n);
    if (unfused) {
      mpfc_launch(sh, k_df_base, g, b, 0, s, F, C);
      if (first) mpfc_launch(sh, k_df_restrict<SCH, true, false>, g, b, 0, s, F, C, zero);
      else mpfc_launch(sh, k_df_restrict<SCH, false, false>, g, b, 0, s, F, C, zero);
    } else {
      if (first) mpfc_launch(sh, k_df_restrict<SCH, true, true>, g, b, 0, s, F, C, zero);
      else mpfc_launch(sh, k_df_restrict<SCH, false, true>, g, b, 0, s, F, C, zero);
    }
  }
  {
    MpfcRange range(lt < L ? "coarse tail" : "coarsest solve");
    if (lt < L) {
      launch_df_tail<SCH>(H, lt, s);
    } else {
      const int G = H->lev[L - 1].m * H->lev[L - 1].n;
      mpfc_launch(sh, k_df_coarse<SCH>, dim3(1), dim3(kDfTailThreads), coarse_df_smem(G), s, dpar(H, SCH, L - 1),
                  (const float*)H->K3[SCH - 1]);
    }
  }
  DPar up = dpar(H, SCH, down);   // the level last finished, where its correction is
  for (int l = down - 1; l >= 0; --l) {
    MpfcRange range(mpfc_level_name(l));
    if (df_leg_level(H, l)) {
      up = launch_up<SCH>(H, l, up, s);
      continue;
    }
    const DPar F = dpar(H, SCH, l), C = up;
    mpfc_launch(sh, k_df_prolong, mpfc_grid_of(sh, C.L.m, C.L.n), mpfc_blk_for(sh, C.L.m, C.L.n), 0, s, C, F);
    up = F;
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
  const dim3 g = pair_grid(H->p.m, H->p.n), b(32, 8);
  // the tail expects its first red sweep done, also where the finest level is in it
  const bool first = (!df_unfused(H) && !df_leg_level(H, 0)) || df_tail_first(H) == 0;
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
bool mpfc_df_usable(const mpfc_params* p) {
  const int L = mpfc_num_levels(p->m, p->n, p->coarsest);
  if (p->precision != MPFC_FP64 || L < 2) return false;
  double h = p->h;
  for (int l = 0; l < L; ++l, h *= 2.0)
    for (int s = 1; s <= 2; ++s)
      if (!df_coef_ok(mpfc_coef(p, s, h, 4)) || !df_coef_ok(mpfc_coef(p, s, h, 3))) return false;
  return true;
}

// Whether a workspace with the correction form's planes (a third to two thirds more than without)
// leaves the device room for the fields a caller keeps beside it, three planes of about twenty;
// handles and batches too large for that keep the FP64 V-cycle and its smaller workspace.  Asked
// of the device's whole memory, so that the size and the handle made with it agree.
bool mpfc_df_fits(size_t workspace) {
  if (workspace < ((size_t)8 << 30)) return true;
  size_t free_bytes = 0, total = 0;
  if (cudaMemGetInfo(&free_bytes, &total) != cudaSuccess) {   // no device: the size alone is asked for
    (void)cudaGetLastError();
    return true;
  }
  return workspace <= total / 8 * 7;
}

// Planes of the correction form.  Level 0: corrections and rho in dr0, p0 and phi^k in the
// Poisson planes (used only by mpfc_energy); coarser levels in the FP64 V-cycle's planes, which
// it writes before it reads them, and a one-launch way up's result in planes of its own.
size_t mpfc_df_carve(mpfc_s* H, size_t* off, char* base, const Lev* lev, double* const* dr0,
                     double* px0, double* pf0, int nlev) {
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
      for (int c = 0; c < 3; ++c) {
        v.d[c] = reinterpret_cast<float2*>(dr0[c]);
        v.r[c] = reinterpret_cast<float2*>(dr0[3 + c]);
      }
      v.pb = reinterpret_cast<float2*>(px0);
      v.pk = reinterpret_cast<float2*>(pf0);
    } else {
      double* const d[3] = {lev[l].phi, lev[l].mu, lev[l].ka};
      double* const r[3] = {lev[l].S1, lev[l].S2, lev[l].S3};
      for (int c = 0; c < 3; ++c) {
        v.d[c] = reinterpret_cast<float2*>(d[c]);
        v.r[c] = reinterpret_cast<float2*>(r[c]);
      }
      v.pb = reinterpret_cast<float2*>(lev[l].b1);
      v.pk = reinterpret_cast<float2*>(lev[l].b2);
      for (int c = 0; c < 3; ++c) {
        float2* e = (long long)G <= kLegCells ? take(G) : nullptr;
        if (H && base) H->de[l][c] = e;
      }
    }
    if (H && base) H->dlev[l] = v;
  }
  return *off - start;
}

int mpfc_df_init(mpfc_s* H) {
  if (!H->df) return MPFC_OK;
  cudaError_t e = cudaSuccess;
  auto raise = [&](auto* k) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDfTailSmem);
  };
  raise(k_df_tail<1, false>);
  raise(k_df_tail<1, true>);
  raise(k_df_tail<2, false>);
  raise(k_df_tail<2, true>);
  auto raise_leg = [&](auto* k, int scheme) {
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)leg_smem(kLegMaxNu, scheme, scheme == 2, true));
  };
  raise_leg(k_df_down<1, false, false>, 1);
  raise_leg(k_df_down<1, false, true>, 1);
  raise_leg(k_df_down<1, true, false>, 1);
  raise_leg(k_df_down<1, true, true>, 1);
  raise_leg(k_df_down<2, false, false>, 2);
  raise_leg(k_df_down<2, false, true>, 2);
  raise_leg(k_df_down<2, true, false>, 2);
  raise_leg(k_df_down<2, true, true>, 2);
  raise_leg(k_df_up<1, false>, 1);
  raise_leg(k_df_up<1, true>, 1);
  raise_leg(k_df_up<2, false>, 2);
  raise_leg(k_df_up<2, true>, 2);
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
  int legs = 0;
  for (int l = 0; l < down; ++l) legs += df_leg_level(H, l);
  return (down - legs) * per + 2 * legs + 2 + ((down == 0 || nu2 == 0) ? 1 : 0);      // + tail or coarsest solve, + residual, (+ u += d)
}
