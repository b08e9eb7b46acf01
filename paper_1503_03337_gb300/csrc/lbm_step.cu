// Single-domain step: descriptor conversion, force time level, default launch
// shape, and dispatch to the per-Q kernel files (lbm_step_q14*.cu, _q18*.cu,
// _q26*.cu).
#include <algorithm>
#include <cmath>

#include "lbm_internal.h"
#include "lbm_kernels.cuh"

namespace lbm {

template <typename R>
Domain<R> to_domain(const DomainDesc& d, const double F[3]) {
  Domain<R> o{};
  o.f = d.f;
  o.nx = d.nx;
  o.ny = d.ny;
  o.nz = d.nz;
  o.N = d.N;
  for (int k = 0; k < 3; ++k) o.per[k] = d.per[k];
  o.moving = d.moving;
  o.sym = d.sym;
  o.solid = d.solid;
  for (int face = 0; face < 6; ++face) {
    for (int k = 0; k < 3; ++k) o.uw[face][k] = R(d.uw[face][k]);
    o.edge_axis[face] = d.edge_axis[face];
    for (int k = 0; k < 2; ++k) o.edge_scale[face][k] = R(d.edge_scale[face][k]);
  }
  o.s.sc = R(d.s[0]);
  o.s.se = R(d.s[1]);
  o.s.sq = R(d.s[2]);
  o.s.snu = R(d.s[3]);
  o.s.spi = R(d.s[4]);
  o.s.st = R(d.s[5]);
  if (d.Q == 14) scale_rows<14>(o.s);
  else if (d.Q == 18) scale_rows<18>(o.s);
  else scale_rows<26>(o.s);
  for (int k = 0; k < 3; ++k) o.F[k] = R(F[k]);
  o.key = 0;
  if (d.Q == 14) fill_offsets<14>(o);
  else if (d.Q == 18) fill_offsets<18>(o);
  else fill_offsets<26>(o);
  return o;
}
template Domain<double> to_domain<double>(const DomainDesc&, const double*);
template Domain<float> to_domain<float>(const DomainDesc&, const double*);

void force_at(const DomainDesc& d, int64_t n, double F[3]) {
  const double c = d.period > 0.0 ? std::cos(2.0 * M_PI * (double)n / d.period) : 1.0;
  for (int k = 0; k < 3; ++k) F[k] = d.force[k] * c;
}

const char* set_faces(DomainDesc& d, const lbm_geom* g) {
  for (int f = 0; f < 6; ++f)
    if (g->face[f] < LBM_PERIODIC || g->face[f] > LBM_NEQ_PRESSURE) return "unknown face kind";
  for (int f = 0; f < 6; ++f) {
    const int n = f < 2 ? d.nx : (f < 4 ? d.ny : d.nz);
    if ((g->face[f] == LBM_NEQ_VELOCITY || g->face[f] == LBM_NEQ_PRESSURE) && n < 3)
      return "an extrapolation face needs at least 3 nodes along its axis";
  }
  int per[3];
  for (int k = 0; k < 3; ++k) {
    const bool lo = g->face[2 * k] == LBM_PERIODIC, hi = g->face[2 * k + 1] == LBM_PERIODIC;
    if (lo != hi) return "opposite faces must both be periodic or neither";
    per[k] = lo ? 1 : 0;
  }
  for (int f = 0; f < 6; ++f) {
    for (int k = 0; k < 3; ++k)
      if (!std::isfinite(g->u_wall[f][k])) return "wall velocity not finite";
    const int k = g->edge_axis[f];
    if (k == 0) continue;
    if (k < 0 || k > 3) return "edge_axis must be 0 (none) or an axis + 1";
    if (g->face[f] != LBM_MOVING_WALL) return "an edge profile needs a moving face";
    if (k - 1 == f / 2) return "an edge profile runs along an in-plane axis of its face";
    if (!std::isfinite(g->edge_scale[f][0]) || !std::isfinite(g->edge_scale[f][1]))
      return "edge scale not finite";
  }
  for (int k = 0; k < 3; ++k) d.per[k] = per[k];
  d.moving = d.sym = d.neq_vel = d.neq_pre = 0;
  for (int f = 0; f < 6; ++f) {
    if (g->face[f] == LBM_MOVING_WALL) d.moving |= 1 << f;
    if (g->face[f] == LBM_SYMMETRY) d.sym |= 1 << f;
    if (g->face[f] == LBM_NEQ_VELOCITY) d.neq_vel |= 1 << f;
    if (g->face[f] == LBM_NEQ_PRESSURE) d.neq_pre |= 1 << f;
    const bool has_u = g->face[f] == LBM_MOVING_WALL || g->face[f] == LBM_NEQ_VELOCITY;
    for (int k = 0; k < 3; ++k) d.uw[f][k] = has_u ? g->u_wall[f][k] : 0.0;
    d.edge_axis[f] = g->edge_axis[f];
    d.edge_scale[f][0] = g->edge_axis[f] ? g->edge_scale[f][0] : 1.0;
    d.edge_scale[f][1] = g->edge_axis[f] ? g->edge_scale[f][1] : 1.0;
  }
  return nullptr;
}

// When and how a box is swept in slabs.  Measured on D3Q18 FP32 boxes of
// 128 x 128 x nz (135 MB of L2): a sweep of the whole box runs at 60-62 GLUPS
// up to 76 MB of populations, 57 at 85, 52 at 94, 45 at 113 and 44 from 150 MB
// on, where every step goes to memory; slabs run at 56-58 throughout (nz = 128:
// 47.7 us a step in whole sweeps, 37.1 in slabs).  They pay from about 0.65
// of L2 on.  A slab may touch 0.62 of L2: 128^3 takes 37.1 us with 66-78 MB a
// slab, 39.4 with 55 or 90 MB; 256^3 takes 326 with 85, 331 with 75, 360 in
// whole sweeps.  A round is 3/8 of the planes a slab touches, at most 16: the
// round's steps share one trip to memory, but each costs the slab a plane and
// every launch about 2 us of ramp and tail (128^3: 4 steps 40.4 us, 8 38.1,
// 16 37.1, 32 37.4).  Fewer than 11 planes (D3Q18 planes above 320^2) leave
// rounds of three steps, which run_slabs sweeps whole (320^3, with 11, takes
// 656 us in slabs and 703 whole).  D3Q26 is bound by its registers as much as
// by memory and wants 18 planes: 160^3 132 us in slabs, 138 in whole sweeps,
// 208^3 281 and 287, 224^3 375 and 370, 256^3 568 and 536.  The other storage
// types are not bound by memory in a whole sweep: FP64 by its arithmetic, FP16
// and BF16 by their issue rate (256^3 D3Q18 FP16: 232 us in whole sweeps, 240
// in slabs).
SlabPlan slab_plan(const DomainDesc& d, int64_t l2_bytes) {
  // a boundary pass follows every step: nothing to run several steps of
  if (d.neq_vel | d.neq_pre) return {};
  if (d.storage != LBM_STORAGE_F32) return {};
  const int64_t plane = (int64_t)d.nx * d.ny * (d.Q * 4 + (d.solid ? 4 : 0));
  if (plane * d.nz * 100 < l2_bytes * 65) return {};
  const int touched = (int)std::min<int64_t>(l2_bytes * 62 / 100 / plane, d.nz);
  if (touched < (d.Q == 26 ? 18 : 11)) return {};
  SlabPlan p;
  p.depth = std::min(16, touched * 3 / 8);
  const int own = touched - p.depth, share = d.per[2] ? d.nz : d.nz - p.depth;
  p.slabs = (share + own - 1) / own;
  // every slab keeps a plane, also while the first one of a periodic box
  // shrinks from both sides
  if (p.slabs < 2 || share / p.slabs <= p.depth) return {};
  return p;
}

// Rows that are not whole warps leave lanes empty; linear order does not.  In
// boxes of fewer cells than fill the device it gains little or loses: us a
// step by rows and in line, D3Q18 FP32 70x70x17 (83 thousand cells) 3.9 and
// 4.6, 45^3 FP16 (91) 4.3 and 4.3, 49^3 (118) 5.1 and 4.6, 65^3 8.4 and 6.8.
// Blocks of four warps: 65^3 6.96 us with eight, 6.75 with four, 7.07 with
// two; 97^3 FP16 14.0, 13.6 and 16.5; 100^3 D3Q26 FP16 27.3, 23.9 and 24.6.
// Boxes with 64-bit population offsets go by rows, so they keep the row shape
// below: with one row a block, ny > 65535 would exceed the grid's y limit.
bool steps_in_line(int Q, int nx, int ny, int64_t N) {
  return nx % 32 != 0 && nx > 1 && ny > 1 && N >= 100000 && !wide_offsets(Q, N);
}

BlockShape default_block(int Q, int nx, int ny, int64_t N, int storage) {
  if (storage == LBM_STORAGE_F64) return {32, 1, 1};  // one warp each (k_step_f64)
  if (steps_in_line(Q, nx, ny, N)) return {128, 1, 1};
  int bx = 32;
  while (bx < nx && bx < 128) bx *= 2;
  int by = 256 / bx;
  while (by > 1 && by / 2 >= ny) by /= 2;
  return {bx, by, 1};
}

TuneKey tune_key(const DomainDesc& d, const SlabPlan& plan) {
  return {d.Q, d.storage, d.rounding, d.nx, d.ny, d.nz, d.solid != nullptr, plan.slabs, plan.depth};
}

bool tune_candidate(const DomainDesc& d, const BlockShape& b) {
  const int xmax = ((d.nx + 31) / 32) * 32;
  if (b.bx * b.cpt > xmax && b.bx > 32) return false;
  // where no step runs two cells per thread
  if (b.cpt == 2 && (d.storage == LBM_STORAGE_F64 || d.Q == 26 || d.solid ||
                     wide_offsets(d.Q, d.N)))
    return false;
  return true;
}

int tune_steps(int trials, const SlabPlan& plan) {
  int unit = plan.slabs > 1 ? plan.depth : 2;
  unit += unit & 1 ? unit : 0;
  return (trials + unit - 1) / unit * unit;
}

cudaError_t launch_step_q14(const DomainDesc& d, int64_t n, int64_t count, BlockShape b,
                            const SlabPlan& plan, cudaStream_t st, StepProgress* done);
cudaError_t launch_step_q18(const DomainDesc& d, int64_t n, int64_t count, BlockShape b,
                            const SlabPlan& plan, cudaStream_t st, StepProgress* done);
cudaError_t launch_step_q26(const DomainDesc& d, int64_t n, int64_t count, BlockShape b,
                            const SlabPlan& plan, cudaStream_t st, StepProgress* done);

cudaError_t launch_steps(const DomainDesc& d, int64_t n, int64_t count, BlockShape b,
                         const SlabPlan& plan, cudaStream_t st, StepProgress* done) {
  if (d.N == 0) return cudaSuccess;
  if (d.Q == 14) return launch_step_q14(d, n, count, b, plan, st, done);
  if (d.Q == 18) return launch_step_q18(d, n, count, b, plan, st, done);
  if (d.Q == 26) return launch_step_q26(d, n, count, b, plan, st, done);
  return cudaErrorInvalidValue;
}

}  // namespace lbm
