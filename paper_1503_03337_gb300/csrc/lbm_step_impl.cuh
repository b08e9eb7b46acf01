// Step kernels of the single-domain path and their typed launchers.  Each
// lbm_step_q*.cu file instantiates them for one Q, so the variants compile in
// parallel.
#pragma once

#include <cmath>
#include <type_traits>

#include "lbm_internal.h"
#include "lbm_kernels.cuh"
#include "lbm_launch.cuh"

namespace lbm {

template <typename R>
Domain<R> to_domain(const DomainDesc& d, const double F[3]);

// Resident 256-thread blocks per SM the register budget is sized for: four
// (64 registers a thread) for Q = 14 and 18 with 4- or 2-byte storage, two
// for their FP64.  Q = 26 needs more: three for FP32 (80 registers, a few
// dozen bytes spilled, measured faster at 256^3 than two: 29.3 vs 28.2
// GLUPS), two for FP16 / BF16 (34.8 at three vs 36.2 at two), one for FP64.
// The wide kernels (64-bit offsets, Q*N >= 2^31) of Q = 14 and 18 take
// three blocks (80 registers): at four they spill 150-180 bytes.
template <int Q, typename S, bool WIDE = false>
constexpr int step_min_blocks() {
  if (Q == 26) return sizeof(S) == 8 ? 1 : (sizeof(S) == 4 ? 3 : 2);
  if (WIDE && sizeof(S) <= 4) return 3;
  return sizeof(S) == 8 ? 2 : 4;
}

// Cells by rows: nx a multiple of 32, or a small box (steps_in_line).
// WIDE: 64-bit population offsets, for domains with Q*N >= 2^31.  SOLIDS =
// false: d has no solid mask (odd steps then carry five addressing variants
// instead of nine).  The next launch is let in after the wait, not before it:
// a trigger before it makes several later grids resident, whose blocks take
// whatever slots are free and bunch on some SMs (33^3 D3Q14 FP32: 3.07 us a
// step with the trigger first, 2.87 so; boxes of many waves do not change).
// Boxes with extrapolation faces hold it back (holds_next).
template <int Q, typename S, bool ODD, bool FORCE, bool SR, bool WIDE, bool SOLIDS, bool SLAB>
__global__ void __launch_bounds__(256, step_min_blocks<Q, S, WIDE>()) k_step(Domain<float> d) {
  pdl_acquire();
  if (!d.hold) pdl_release();
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = plane_of<SLAB>(d);
  if (x >= d.nx || y >= d.ny) return;
  // a 32-wide x-range containing x; it is the calling warp's range when
  // blockDim.x is a multiple of 32 (then the path choice is warp-uniform)
  const int x_lo = blockIdx.x * blockDim.x + (threadIdx.x & ~31);
  const int x_hi = x_lo + 31;
  update_cell<Q, S, float, ODD, FORCE, SR, false, WIDE, SOLIDS>(d, static_cast<S*>(d.f), x, y, z,
                                                                x_lo, x_hi);
}

// The cells of a launch in linear order (k_step_line).
struct LineArgs {
  int first, cells;  // cells first .. first + cells - 1, past N going on at 0
  FastDiv by_x, by_y;
};

// One cell per thread, cells in linear order whatever row they are in, so that
// no lanes are left empty at the ends of rows; the warp votes on the
// addressing variant.  The step is bound by instruction issue in L2-sized
// boxes and with 2-byte storage, so what it gains is the padding: us a step by
// rows and so, lid-driven boxes with walls on every other face, 97x97x49 D3Q18
// FP32 10.8 and 9.6 (11.5 and 10.7 with a symmetry plane on a z face, whose
// mirrored addressing every row end then takes), 65^3 8.4 and 6.8, 129^3 47.2
// and 41.8, 200^3 154 and 146, 97^3 FP16 17.2 and 13.6, 161^3 FP16 75.9 and
// 67.4, 100^3 D3Q26 FP16 34.8 and 23.9.  The coordinates of a cell are formed
// before the wait for the previous step.  SOLIDS: d has a solid mask; every
// such box without 64-bit offsets runs here (100^3, 30 % solid, FP32: 20.9 and
// 17.8; 192^3, whose rows have no padding, 137.7 and 137.0), so of k_step's
// builds only those with 64-bit offsets need the solid code.
template <int Q, typename S, bool ODD, bool FORCE, bool SR, bool SOLIDS>
__global__ void __launch_bounds__(256, step_min_blocks<Q, S>()) k_step_line(Domain<float> d,
                                                                            LineArgs a) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= a.cells) return;
  unsigned u = (unsigned)a.first + (unsigned)t;
  const int i = (int)(u < (unsigned)d.N ? u : u - (unsigned)d.N);
  S* const f = static_cast<S*>(d.f);
  if constexpr (!ODD) {
    pdl_acquire();
    if (!d.hold) pdl_release();
    update_even<Q, S, float, FORCE, SR, false, false, SOLIDS>(d, f, d.F, &d.key, i);
  } else {
    const int r = a.by_x(i), z = a.by_y(r), x = i - r * d.nx, y = r - z * d.ny;
    const bool yz = y == 0 || y == d.ny - 1 || z == 0 || z == d.nz - 1;
    const bool bulk_yz = !warp_any(yz), bulk_x = !warp_any(x == 0 || x == d.nx - 1);
    pdl_acquire();
    if (!d.hold) pdl_release();
    update_odd<Q, S, float, FORCE, SR, false, false, SOLIDS>(d, f, d.F, &d.key, i, x, y, z,
                                                             bulk_yz, bulk_x);
  }
}

// FP64 storage: cells in linear order, one after another whatever row they
// are in.  This device updates two FP64 lanes per clock and SM, so a warp
// instruction takes 16 clocks however many of its lanes are active, and the
// step is bound by that pipe; rows rounded up to whole warps waste it (16-wide
// rows half of it, 65-wide ones a third), as does any branch that splits a
// warp, so every cell takes the general addressing.  Launched with one warp
// per block (default_block): the warps then spread evenly over the SMs.
// 16x16x32 D3Q18: 28.5 us a step with 32 x 8 blocks of rows, 8.0 so.
template <int Q, bool ODD, bool FORCE, bool WIDE>
__global__ void __launch_bounds__(256, step_min_blocks<Q, double>()) k_step_f64(Domain<double> d) {
  // No trigger: the next launch comes in as the blocks of this one end.  Blocks
  // that are let in earlier take whatever slots free first, so that some SMs
  // hold more of them than others, and an SM's time goes by its warps (us a
  // step with the trigger before the wait, after it and without: D3Q18
  // 16x16x32 8.3, 8.2, 8.0; 32^3 32.6, 14.8, 14.7; 256x256x1 38.2, 38.2, 28.5;
  // D3Q26 31^3 44.8, 44.7, 27.6; 64^3 and more the same).
  pdl_acquire();
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;  // N < 2^31
  if (t >= (unsigned)d.N) return;
  const int i = (int)t;
  double* const f = static_cast<double*>(d.f);
  if constexpr (!ODD) {
    if (d.solid && (d.solid[i] & kSolidCell)) return;
    update_with_links<Q, double, double, false, FORCE, false, false, true, false, WIDE>(
        d, f, i, Links{}, d.F, &d.key);
  } else {
    const int x = i % d.nx, r = i / d.nx;
    const Links L = make_links(d, x, r % d.ny, r / d.ny);
    if (L.solid & kSolidCell) return;
    if (d.sym)
      update_with_links<Q, double, double, true, FORCE, false, false, true, true, WIDE>(
          d, f, i, L, d.F, &d.key);
    else
      update_with_links<Q, double, double, true, FORCE, false, false, false, true, WIDE>(
          d, f, i, L, d.F, &d.key);
  }
}

// Even steps with two x-adjacent cells per thread (see update_pair_even; nx
// even); blockDim.x threads cover 2*blockDim.x cells of a row.  The 36
// packed values of a pair need more registers than one cell's 18: at three
// 256-thread blocks per SM (80 registers) a pair spills about 100 bytes a
// thread to local memory, and is still faster than at two blocks without
// spills (measured at 256^3: FP16 66.4 vs 62.7 GLUPS for Q18, 85.0 vs 81.7
// for Q14).
template <int Q, typename S, bool FORCE, bool SR, bool SLAB>
__global__ void __launch_bounds__(256, 3) k_step_pair(Domain<float> d) {
  pdl_acquire();
  if (!d.hold) pdl_release();
  const int x0 = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = plane_of<SLAB>(d);
  if (x0 >= d.nx || y >= d.ny) return;
  update_pair_even<Q, S, FORCE, SR>(d, static_cast<S*>(d.f), x0 + d.nx * (y + d.ny * z));
}

template <typename R>
void launch_one(void (*kernel)(Domain<R>), const Domain<R>& d, dim3 grid, dim3 block, bool pdl,
                cudaStream_t st) {
  launch_pdl(kernel, grid, block, pdl, st, d);
}

template <int Q>
void launch_f64(const Domain<double>& d, bool odd, bool force, bool wide, const BlockShape& b,
                cudaStream_t st) {
  auto kernel = wide ? (odd ? (force ? k_step_f64<Q, true, true, true>
                                     : k_step_f64<Q, true, false, true>)
                            : (force ? k_step_f64<Q, false, true, true>
                                     : k_step_f64<Q, false, false, true>))
                     : (odd ? (force ? k_step_f64<Q, true, true, false>
                                     : k_step_f64<Q, true, false, false>)
                            : (force ? k_step_f64<Q, false, true, false>
                                     : k_step_f64<Q, false, false, false>));
  const unsigned threads = b.bx * b.by;
  launch_one(kernel, d, dim3((unsigned)((d.N + threads - 1) / threads)), dim3(threads),
             b.pdl != 0, st);
}

// fn.operator()<ODD, FORCE>() for the two run-time flags.
template <typename Fn>
void by_flags(bool odd, bool force, Fn&& fn) {
  if (odd) {
    if (force) fn.template operator()<true, true>();
    else fn.template operator()<true, false>();
  } else {
    if (force) fn.template operator()<false, true>();
    else fn.template operator()<false, false>();
  }
}

template <int Q, typename S, bool SR>
void launch_parity(const Domain<float>& d, bool odd, bool force, bool wide, int planes,
                   const BlockShape& b, cudaStream_t st) {
  const bool pdl = b.pdl != 0;
  const dim3 block(b.bx, b.by);
  const int by = (d.ny + b.by - 1) / b.by;
  const dim3 grid((d.nx + b.bx - 1) / b.bx, by, planes);
  // only FP32 boxes are swept in slabs (slab_plan)
  constexpr bool kSlabs = sizeof(S) == 4;
  const bool slab = kSlabs && is_slab(d, planes);
  // Q*N >= 2^31: one cell per thread with 64-bit population offsets
  if (wide) {
    by_flags(odd, force, [&]<bool ODD, bool FORCE>() {
      launch_one(slab ? k_step<Q, S, ODD, FORCE, SR, true, true, kSlabs>
                      : k_step<Q, S, ODD, FORCE, SR, true, true, false>,
                 d, grid, block, pdl, st);
    });
    return;
  }
  // two cells per thread: even steps of FP32 / FP16 / BF16 storage with nx
  // even and no solid nodes, Q = 14 or 18 (the 52 packed values of a Q = 26
  // pair would not fit the registers); every other step runs one cell per
  // thread
  if constexpr (Q != 26) {
    if (b.cpt == 2 && !odd && d.nx % 2 == 0 && !d.solid) {
      const dim3 half((d.nx / 2 + b.bx - 1) / b.bx, by, planes);
      by_flags(false, force, [&]<bool ODD, bool FORCE>() {
        launch_one(slab ? k_step_pair<Q, S, FORCE, SR, kSlabs> : k_step_pair<Q, S, FORCE, SR, false>,
                   d, half, block, pdl, st);
      });
      return;
    }
  }
  if (d.solid || steps_in_line(Q, d.nx, d.ny, d.N)) {
    const int plane = d.nx * d.ny, cells = planes * plane;
    const unsigned threads = b.bx * b.by;
    const LineArgs a{d.z0 * plane, cells, FastDiv(d.nx), FastDiv(d.ny)};
    const dim3 blocks(((unsigned)cells + threads - 1) / threads);
    by_flags(odd, force, [&]<bool ODD, bool FORCE>() {
      launch_pdl(d.solid ? k_step_line<Q, S, ODD, FORCE, SR, true>
                         : k_step_line<Q, S, ODD, FORCE, SR, false>,
                 blocks, dim3(threads), pdl, st, d, a);
    });
    return;
  }
  // The odd D3Q18 BF16 stochastic kernel that carries the solid code is faster
  // than the one without it: 240.4 against 248.2 us a step at 256^3 (pairs on
  // even steps), 267.4 against 282.2 one cell a thread; no difference at 128^3.
  // Registers and spills are the same, the order of instructions is not, and
  // no other type shares it (D3Q14 210.0 against 197.6, D3Q18 FP16 equal).
  by_flags(odd, force, [&]<bool ODD, bool FORCE>() {
    constexpr bool kSolids = ODD && Q == 18 && SR && std::is_same_v<S, __nv_bfloat16>;
    launch_one(slab ? k_step<Q, S, ODD, FORCE, SR, false, kSolids, kSlabs>
                    : k_step<Q, S, ODD, FORCE, SR, false, kSolids, false>,
               d, grid, block, pdl, st);
  });
}

// Steps n .. n + count - 1, slab by slab (run_slabs).  The descriptor is
// built once; a launch changes only its planes, force and rounding key, so it
// costs the host 1.8 us where rebuilding the descriptor made it 5.5 us (16^3
// D3Q18 FP32: 6.0 us a step before, 2.0 us now).
template <int Q, typename S, bool SR>
cudaError_t launch_typed(const DomainDesc& dd, int64_t n, int64_t count, BlockShape b,
                         const SlabPlan& plan, cudaStream_t st, StepProgress* done) {
  using R = std::conditional_t<sizeof(S) == 8, double, float>;
  const double zero[3] = {0.0, 0.0, 0.0};
  // the force-carrying update whenever the amplitude is nonzero (also at the
  // steps where a periodic force passes through zero), as the batch does
  const bool force = dd.force[0] != 0.0 || dd.force[1] != 0.0 || dd.force[2] != 0.0;
  Domain<R> d = to_domain<R>(dd, zero);
  const bool wide = wide_offsets(dd.Q, dd.N);
  d.hold = holds_next(dd);
  return run_slabs(dd.nz, dd.per[2] != 0, plan, count, [&](int64_t s, int z0, int planes) {
    double F[3];
    force_at(dd, n + s, F);
    for (int c = 0; c < 3; ++c) d.F[c] = R(F[c]);
    d.key = step_key(n + s);
    d.z0 = z0;
    const bool odd = ((n + s) & 1) != 0;
    if constexpr (sizeof(S) == 8) launch_f64<Q>(d, odd, force, wide, b, st);
    else launch_parity<Q, S, SR>(d, odd, force, wide, planes, b, st);
    return cudaGetLastError();
  }, done);
}

#define LBM_STEP_UNIT(Q, S, SR)                                                              \
  template cudaError_t launch_typed<Q, S, SR>(const DomainDesc&, int64_t, int64_t, BlockShape, \
                                              const SlabPlan&, cudaStream_t, StepProgress*)
#define LBM_STEP_EXTERN(Q, S, SR) extern LBM_STEP_UNIT(Q, S, SR)

template <int Q>
cudaError_t launch_storage(const DomainDesc& d, int64_t n, int64_t count, BlockShape b,
                           const SlabPlan& plan, cudaStream_t st, StepProgress* done) {
  const bool sr = d.rounding == LBM_ROUND_STOCHASTIC;
  switch (d.storage) {
    case LBM_STORAGE_F64: return launch_typed<Q, double, false>(d, n, count, b, plan, st, done);
    case LBM_STORAGE_F32: return launch_typed<Q, float, false>(d, n, count, b, plan, st, done);
    case LBM_STORAGE_F16:
      return sr ? launch_typed<Q, __half, true>(d, n, count, b, plan, st, done)
                : launch_typed<Q, __half, false>(d, n, count, b, plan, st, done);
    case LBM_STORAGE_BF16:
      return sr ? launch_typed<Q, __nv_bfloat16, true>(d, n, count, b, plan, st, done)
                : launch_typed<Q, __nv_bfloat16, false>(d, n, count, b, plan, st, done);
  }
  return cudaErrorInvalidValue;
}

}  // namespace lbm
