// One level's way down or up of the V-cycle in correction form as one launch, for levels whose
// launches do not fill the chip.
//
// A half sweep of such a level is a chain of about 1.3 k clocks (536 instructions a cell, most of
// them dependent) in a launch of 2.3 us, and a level takes ten launches.  Here a CTA owns
// kLegTile x kLegTile cells and sweeps them together with a halo in shared memory: every half sweep
// needs the one before it on one more ring of cells, so the ring is computed by both tiles that
// hold it, from the same values with the same cell functions (the bits are those of the
// per-level launches).  2 nu rings: 1.43 times the cell updates at nu = 2, which pays while the
// updates of a launch take less than the launch itself.  A way takes 11 k clocks after its
// predecessor (5.5 us at 32^2 as at 256^2), bound by the chain: copies in 1 to 2 k, each half sweep
// 1.5 to 2.1 k, the prolongation 1.5 k, the restriction 2 to 4 k; five launches took about 12 us.
// Four steps at 512^2 3.13 -> 2.86 ms, two at 1024^2 3.13 -> 3.00, pinned at 512 x 384 4.51 -> 4.04.
//
// Down: the first red half sweep (d = 0 before it), the others, and the restriction.  Up: the
// prolongation and the sweeps; the result goes to planes of its own (or is added to u on the
// finest level), since the neighbours read this level's d as their halo.
#pragma once

#include "df_cells.cuh"

namespace mpfc {

constexpr int kLegTile = 16;
constexpr int kLegThreads = 288;   // 24 x 24 staged cells (nu = 2) in two passes, 22 x 22 / 2 in one
constexpr int kLegMaxNu = 3;
constexpr int kLegCellsPerThread = ((kLegTile + 4 * kLegMaxNu) * (kLegTile + 4 * kLegMaxNu) + kLegThreads - 1) / kLegThreads;

// The staged cells' planes and (way up) the coarse correction under them with a ring.
inline size_t leg_smem(int nu, int scheme, bool pinned, bool up) {
  const size_t w = kLegTile + 4 * (size_t)nu, cw = w / 2 + 2;
  return sizeof(float2) * (w * w * (7 + (scheme == 2 ? 1 : 0) + (pinned ? 1 : 0)) + (up ? 3 * cw * cw : 0));
}

__device__ __forceinline__ void leg_copy8(void* smem, const void* gmem) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(smem)), "l"(gmem)
               : "memory");
}
__device__ __forceinline__ void leg_copies_done() {
  asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
}

struct LegOut {
  float2* e[3];   // the level's correction after the way up ...
  double* u[3];   // ... or, on the finest level, the iterate it is added to
};

template <int SCH, bool NY>
struct Leg {
  DPar P;         // the tile with its halo as a level of its own, in shared memory
  int x0, y0, ylo, W, rows;
  int go[kLegCellsPerThread];                // where this thread's staged cells are in the level's planes,
  int wg[kLegCellsPerThread], ws[kLegCellsPerThread];   // in the pinning weight and in its staged copy

  // Staged cell t (colour-split order) and its domain coordinates.
  __device__ __forceinline__ void cell(const DLev& F, int t, int& x, int& y) const {
    const int half = W >> 1, hc = half * rows, color = t >= hc, r = (t - color * hc) / half;
    const int q = t - color * hc - r * half;
    x = (x0 + 2 * q + ((r + color) & 1)) % F.m;   // x0: the staged columns' origin, brought to >= 0
    y = ylo + r;
    if (!(NY && F.nyn)) y %= F.n;
  }

  __device__ __forceinline__ void init(const DPar& F, int nu, float2* sm) {
    const int halo = 2 * nu, m = F.L.m, n = F.L.n;
    W = kLegTile + 2 * halo;
    x0 = (int)blockIdx.x * kLegTile - halo;
    y0 = (int)blockIdx.y * kLegTile;
    int yhi = y0 + kLegTile + halo;
    ylo = y0 - halo;
    if (NY && F.L.nyn) {   // no rows outside the domain: the staged edge row is the boundary row
      ylo = max(ylo, 0);
      yhi = min(yhi, n);
    }
    rows = yhi - ylo;
    const int cells = W * rows;
    P = F;
    P.L.m = W;
    P.L.n = rows;
    for (int c = 0; c < 3; ++c) {
      P.L.d[c] = sm + c * cells;
      P.L.r[c] = sm + (3 + c) * cells;
    }
    P.L.pb = sm + 6 * cells;
    P.L.pk = sm + 7 * cells;
    P.L.W = F.L.W ? reinterpret_cast<const double*>(sm + 8 * cells) : nullptr;
    // the tile's own rows relative to the staged ones
    y0 -= ylo;
    // periodic origins brought to >= 0 (multiples of the even m and n keep the colours)
    x0 = (x0 % m + m) % m;
    if (!(NY && F.L.nyn)) ylo = (ylo % n + n) % n;
  }

  // The offsets of the copies (integer divisions), before the wait for the previous kernel: four
  // steps at 512^2 in 2.86 ms, 2.92 with them after it.
  __device__ __forceinline__ void plan(const DLev& F) {
    const int half = W >> 1, hc = half * rows;
#pragma unroll
    for (int q = 0; q < kLegCellsPerThread; ++q) {
      const int t = threadIdx.x + q * kLegThreads;
      go[q] = wg[q] = ws[q] = 0;
      if (t >= 2 * hc) continue;
      int x, y;
      cell(F, t, x, y);
      go[q] = (int)dindex(F, x, y);
      if (SCH == 2 && F.W) {
        const int color = t >= hc, r = (t - color * hc) / half, i = 2 * (t - color * hc - r * half) + ((r + color) & 1);
        wg[q] = y * F.m + x;
        ws[q] = r * W + i;
      }
    }
  }
  // Starts the copies of the planes a sweep reads only, and (OWN) of d.
  template <bool OWN>
  __device__ __forceinline__ void load(const DLev& F) const {
    const int cells = W * rows;
#pragma unroll
    for (int q = 0; q < kLegCellsPerThread; ++q) {
      const int t = threadIdx.x + q * kLegThreads;
      if (t >= cells) continue;
      const int g = go[q];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        leg_copy8(P.L.r[c] + t, F.r[c] + g);
        if (OWN) leg_copy8(P.L.d[c] + t, F.d[c] + g);
      }
      leg_copy8(P.L.pb + t, F.pb + g);
      if (SCH == 2) {
        leg_copy8(P.L.pk + t, F.pk + g);
        if (F.W) leg_copy8(const_cast<double*>(P.L.W) + ws[q], F.W + wg[q]);
      }
    }
  }

  // Half sweep of colour `color` on the tile and `ring` rings of cells around it.
  __device__ __forceinline__ void half_sweep(int color, int ring) const {
    const int halo = (W - kLegTile) >> 1, per = kLegTile / 2 + ring;
    int lo = y0 - ring, hi = y0 + kLegTile + ring;
    if (NY && P.L.nyn) {
      lo = max(lo, 0);
      hi = min(hi, rows);
    }
    for (int t = threadIdx.x; t < (hi - lo) * per; t += blockDim.x) {
      const int r = t / per, j = lo + r;
      const int x = ((halo - ring + 1 - ((j + color) & 1)) >> 1) + t - r * per;
      df_smooth_cell<SCH, kGen, NY, false>(P, color, x, j);
    }
    __syncthreads();
  }
};

// FIRST: also the coarse level's first red half sweep.
template <int SCH, bool NY, bool FIRST>
__global__ void __launch_bounds__(kLegThreads) k_df_down(const __grid_constant__ DPar F, const __grid_constant__ DPar C,
                                                         int nu) {
  extern __shared__ float2 lsm[];
  Leg<SCH, NY> T;
  T.init(F, nu, lsm);
  T.plan(F.L);
  pdl_enter();
  T.template load<false>(F.L);
  const int half = T.W >> 1, red = half * T.rows;
  for (int t = threadIdx.x; t < red; t += blockDim.x)   // black cells: d = 0
#pragma unroll
    for (int c = 0; c < 3; ++c) T.P.L.d[c][red + t] = make_float2(0.f, 0.f);
  leg_copies_done();
  __syncthreads();
  for (int t = threadIdx.x; t < red; t += blockDim.x) {
    // all staged rows take part, so a boundary row is told by its place in the domain
    const int r = t / half, y = T.ylo + r;
    DCell c;
    df_load_static<SCH>(T.P.L, F.k, t, 2 * (t - r * half) + (r & 1), r, c);
    const df z{0.f, 0.f};
    if (NY && F.L.nyn && (y == 0 || y == F.L.n - 1)) df_update<SCH, kAll>(F.kb, z, z, z, c);
    else df_update<SCH, kAll>(F.k, z, z, z, c);
    T.P.L.d[0][t] = f2(c.p);
    T.P.L.d[1][t] = f2(c.m);
    T.P.L.d[2][t] = f2(c.k);
  }
  __syncthreads();
  for (int hs = 1; hs < 2 * nu; ++hs) T.half_sweep(hs & 1, 2 * nu - hs);
  const int bx = blockIdx.x * kLegTile, by = blockIdx.y * kLegTile;
  // the first warps restrict while the others store d
  constexpr int kRw = kLegTile * kLegTile / 4;
  if (threadIdx.x < kRw) {
    const int I = threadIdx.x % (kLegTile / 2), J = threadIdx.x / (kLegTile / 2), cI = bx / 2 + I, cJ = by / 2 + J;
    if (cI < C.L.m && cJ < C.L.n) df_restrict_cell<SCH, FIRST, true>(T.P, C, nu + I, T.y0 / 2 + J, 0, cI, cJ);
    return;
  }
  for (int t = threadIdx.x - kRw; t < kLegTile * kLegTile; t += blockDim.x - kRw) {
    // colour-split order: consecutive threads store consecutive columns of one colour
    const int color = t >> 7, r = (t >> 3) & (kLegTile - 1), i = 2 * (t & 7) + ((r + color) & 1);
    if (bx + i >= F.L.m || by + r >= F.L.n) continue;
    const size_t g = dindex(F.L, bx + i, by + r), q = dindex(T.P.L, 2 * nu + i, T.y0 + r);
#pragma unroll
    for (int c = 0; c < 3; ++c) F.L.d[c][g] = T.P.L.d[c][q];
  }
}

template <int SCH, bool NY>
__global__ void __launch_bounds__(kLegThreads) k_df_up(const __grid_constant__ DPar C, const __grid_constant__ DPar F,
                                                       const __grid_constant__ LegOut O, int nu) {
  extern __shared__ float2 lsm[];
  Leg<SCH, NY> T;
  T.init(F, nu, lsm);
  const int half = T.W >> 1, hc = half * T.rows, cw = half + 2, ch = (T.rows >> 1) + 2;
  T.plan(F.L);
  // the coarse correction under the staged cells with one ring, a cell a thread
  static_assert(((kLegTile + 4 * kLegMaxNu) / 2 + 2) * ((kLegTile + 4 * kLegMaxNu) / 2 + 2) <= kLegThreads, "");
  float2* const e = lsm + (7 + (SCH == 2 ? 1 + (F.L.W != nullptr) : 0)) * 2 * hc;
  int ge = -1;
  if (threadIdx.x < cw * ch) {
    const int cj = threadIdx.x / cw, I = (T.x0 / 2 - 1 + (int)threadIdx.x - cj * cw + C.L.m) % C.L.m;
    int J = T.ylo / 2 - 1 + cj;
    if (NY && C.L.nyn) J = min(max(J, 0), C.L.n - 1);
    else J = (J + C.L.n) % C.L.n;
    ge = (int)dindex(C.L, I, J);
  }
  pdl_enter();
  T.template load<true>(F.L);
  if (ge >= 0)
#pragma unroll
    for (int c = 0; c < 3; ++c) leg_copy8(e + c * cw * ch + threadIdx.x, C.L.d[c] + ge);
  leg_copies_done();
  __syncthreads();
  for (int t = threadIdx.x; t < 2 * hc; t += blockDim.x) {
    const int color = t >= hc, r = (t - color * hc) / half, i = 2 * (t - color * hc - r * half) + ((r + color) & 1);
    const int q = ((r >> 1) + 1) * cw + (i >> 1) + 1, dx = (i & 1) ? 1 : -1, dy = (r & 1) ? cw : -cw;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float2* f = e + c * cw * ch + q;
      float2* d = T.P.L.d[c] + t;
      *d = f2(add(ldd(d), df_prolonged(ldd(f), ldd(f + dx), ldd(f + dy), ldd(f + dx + dy))));
    }
  }
  __syncthreads();
  for (int hs = 0; hs < 2 * nu; ++hs) T.half_sweep(hs & 1, 2 * nu - 1 - hs);
  const int bx = blockIdx.x * kLegTile, by = blockIdx.y * kLegTile;
  for (int t = threadIdx.x; t < kLegTile * kLegTile; t += blockDim.x) {
    if (O.u[0]) {   // row-major
      const int i = t & (kLegTile - 1), r = t / kLegTile;
      if (bx + i >= F.L.m || by + r >= F.L.n) continue;
      const size_t g = (size_t)(by + r) * F.L.m + bx + i, q = dindex(T.P.L, 2 * nu + i, T.y0 + r);
#pragma unroll
      for (int c = 0; c < 3; ++c) O.u[c][g] += df_to_f64(ldd(T.P.L.d[c] + q));
    } else {
      const int color = t >> 7, r = (t >> 3) & (kLegTile - 1), i = 2 * (t & 7) + ((r + color) & 1);
      if (bx + i >= F.L.m || by + r >= F.L.n) continue;
      const size_t g = dindex(F.L, bx + i, by + r), q = dindex(T.P.L, 2 * nu + i, T.y0 + r);
#pragma unroll
      for (int c = 0; c < 3; ++c) O.e[c][g] = T.P.L.d[c][q];
    }
  }
}

}  // namespace mpfc
