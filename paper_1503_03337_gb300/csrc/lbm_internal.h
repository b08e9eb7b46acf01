// Host-side internals shared by the library's translation units.
#pragma once

#include <cuda_runtime.h>

#include <array>
#include <cstdint>
#include <string>

#include "../../include/lbm.h"

namespace lbm {

// Number of FP64 statistics a reduction produces (layout of lbm_stats after
// the two step counters): 3 du, 3 u, 3 u_prev, P, 3 flux, max, nonfinite.
constexpr int kNumSums = 14;   // summed entries
constexpr int kNumStats = 15;  // plus the max
constexpr int kReduceBlocks = 608;  // at most, of a reduction: 4 x 152 SMs
constexpr int kReduceThreads = 256;

// Everything a kernel needs to know about one domain, in FP64; the launchers
// convert it to the arithmetic type of the storage.
struct DomainDesc {
  int Q, nx, ny, nz, storage;
  int64_t N;
  void* f;
  int per[3];
  int moving;  // bit f: face f is a moving wall
  int sym;     // bit f: face f is a symmetry plane
  int neq_vel; // bit f: face f is a non-equilibrium extrapolation velocity face
  int neq_pre; // bit f: ... pressure face
  double p_face[6], p_amp[6], p_period;  // pressure of the pressure faces
  const uint32_t* solid;  // device: per-cell solid-link bits (Domain::solid), or null
  double uw[6][3];
  int edge_axis[6];  // edge profiles of moving faces (lbm_geom)
  double edge_scale[6][2];
  double s[6];  // sc, se, sq, snu, spi, st
  double force[3];
  double period;
  double p_ref;
  int rounding;  // enum lbm_rounding
};

struct BlockShape {
  int bx, by;
  int cpt;      // cells per thread: 1, or 2 (pairs along x, FP32 arithmetic only)
  int pdl = 1;  // programmatic dependent launch of consecutive steps
};

// i / n for 0 <= i < 2^31 and n >= 1 as a multiplication: with n <= 2^s < 2 n
// and m = floor(2^(31+s) / n) + 1 < 2^32, i m >> (31 + s) is exact because
// i (m n - 2^(31+s)) <= i 2^s < 2^(31+s).
struct FastDiv {
  unsigned m;
  int shift;
  explicit FastDiv(int n) {
    int s = 0;
    while ((int64_t(1) << s) < n) ++s;
    m = (unsigned)((uint64_t(1) << (31 + s)) / (unsigned)n + 1);
    shift = 31 + s;
  }
  __host__ __device__ int operator()(int i) const {
    return (int)(((uint64_t)(unsigned)i * m) >> shift);
  }
};

// Q * N >= 2^31: 64-bit population offsets.
inline bool wide_offsets(int Q, int64_t N) { return Q * N >= (int64_t(1) << 31); }

// The default launch of a box; 4- and 2-byte storage runs its cells in linear
// order (k_step_line) or by rows (k_step).
BlockShape default_block(int Q, int nx, int ny, int64_t N, int storage);
bool steps_in_line(int Q, int nx, int ny, int64_t N);

// The face fields of d (per, moving, sym, neq_*, uw) from a geometry.
// Returns nullptr, or the reason the geometry is invalid (then d is
// unchanged).  d's sizes must be set (extrapolation faces need 3 nodes).
const char* set_faces(DomainDesc& d, const lbm_geom* g);

// Per-cell solid-link bits (Domain::solid) of the solid-node mask `bytes`
// (N device bytes, nonzero = solid) for d's geometry.
cudaError_t launch_solid_links(const DomainDesc& d, const uint8_t* bytes, uint32_t* links,
                               cudaStream_t st);

// Do d's step and boundary launches let the next one in only as their blocks
// end?  Blocks of a boundary pass that is let in early take the first slots
// that free as the step drains, bunch on a few SMs, and the nodes of x faces (a
// line of memory per lane) then take long.  us a step, let in early and held
// back: D3Q14 FP32 64^3 14.5 and 9.9, 128^3 with x faces 57.0 and 43.7; D3Q18
// FP16 64^3 21.1 and 12.7, 28^3 8.3 and 8.0.  In smaller boxes it costs more
// than it gains (D3Q26 FP32 12^3 8.1 and 8.8, D3Q18 FP32 20^3 6.2 and 6.5),
// except with FP64 storage, whose steps let nothing in early (k_step_f64).
inline bool holds_next(const DomainDesc& d) {
  return (d.neq_vel | d.neq_pre) && (d.storage == LBM_STORAGE_F64 || d.N >= 16384);
}

// Non-equilibrium extrapolation of the boundary nodes of d's LBM_NEQ_*
// faces, on the populations of step n (after the step n-1 -> n).
cudaError_t launch_neq(const DomainDesc& d, int64_t n, bool pdl, cudaStream_t st);

// Message returned by lbm_last_error() on the calling thread.
void set_last_error(const std::string& msg);

// F(t_n) of a domain.
void force_at(const DomainDesc& d, int64_t n, double F[3]);

// Slabs of planes that run several steps each while their populations stay
// in L2 (slabs = 1: every step sweeps the whole box).  Neighbouring planes may
// be one step apart and no more, so a slab moves down one plane per step:
//   slab k runs step s of a round on planes [begin(k) - s, begin(k + 1) - s),
// the first one from plane 0 on and the last one up to the top, and slab k
// finishes the round before slab k + 1 starts.  Every cell of plane z then
// takes step s after planes z - 1 and z + 1 have taken step s - 1 and before
// either takes step s + 1.  That is all the in-place update needs (the slots
// that a cell's step s touches are touched only by the cell's and its
// neighbours' steps s - 1 and s + 1), so results do not depend on the plan.
// In a box periodic in z the first slab moves up at its bottom,
// [s, begin(1) - s), and the last one ends with the planes that this leaves:
// past the top and round to plane s - 1.
struct SlabPlan {
  int slabs = 1;
  int depth = 1;  // steps of a round
};

// The slabs of d's steps on a device with l2_bytes of L2.
SlabPlan slab_plan(const DomainDesc& d, int64_t l2_bytes);

// lbm_autotune: what its choice for a box depends on (the step kernels of the
// box and the order they sweep it in), whether a block is a candidate of its
// own there, and how many of at least `trials` steps it times: whole rounds of
// slabs, as many even as odd steps.
using TuneKey = std::array<int, 9>;
TuneKey tune_key(const DomainDesc& d, const SlabPlan& plan);
bool tune_candidate(const DomainDesc& d, const BlockShape& b);
int tune_steps(int trials, const SlabPlan& plan);

// What was queued of a run of steps: `steps` of the whole box, and, if torn,
// some planes further on (a launch failed within a round of slabs).
struct StepProgress {
  int64_t steps = 0;
  bool torn = false;
};

// launch(s, z0, planes) for every step s of 0 .. count - 1 and slab, up to the
// first launch that fails; *done (if not null) tells how far it came.
template <typename Fn>
cudaError_t run_slabs(int nz, bool periodic, const SlabPlan& plan, int64_t count, Fn&& launch,
                      StepProgress* done = nullptr) {
  // begin(k) leaves every slab the same number of planes per round: (planes
  // to share out) / slabs, plus the depth-wide ramp at the bottom
  const int64_t share = periodic ? nz : nz - plan.depth;
  auto begin = [&](int k) { return k == 0 ? 0 : plan.depth + (int)(k * share / plan.slabs); };
  for (int64_t s0 = 0; s0 < count; s0 += plan.depth) {
    const int steps = (int)(count - s0 < plan.depth ? count - s0 : plan.depth);
    // two or three steps do not save what the extra launches cost
    const int slabs = steps >= 4 ? plan.slabs : 1;
    for (int k = 0; k < slabs; ++k)
      for (int s = 0; s < steps; ++s) {
        int lo = k == 0 ? 0 : begin(k) - s;
        int hi = k == slabs - 1 ? nz : begin(k + 1) - s;
        if (periodic && slabs > 1) {
          if (k == 0) lo = s;
          if (k == slabs - 1) hi = nz + s;
        }
        if (cudaError_t e = launch(s0 + s, lo, hi - lo)) {
          if (done) *done = slabs == 1 ? StepProgress{s0 + s, false}
                                       : StepProgress{s0, k > 0 || s > 0};
          return e;
        }
      }
  }
  if (done) *done = {count, false};
  return cudaSuccess;
}

// Queue the fused steps n .. n + count - 1 (parity of each its number's).
cudaError_t launch_steps(const DomainDesc& d, int64_t n, int64_t count, BlockShape b,
                         const SlabPlan& plan, cudaStream_t st, StepProgress* done);

// f = f_eq(p - p_ref, u) at every node, stored for step 0 (even layout).
cudaError_t launch_init(const DomainDesc& d, const double* u, const double* p,
                        cudaStream_t st);

// Canonical populations / u / p of step n into a device buffer.
cudaError_t launch_read(const DomainDesc& d, int64_t n, unsigned mask, void* dst,
                        int dtype, cudaStream_t st);

// Canonical FP64 populations into the storage layout of step n.
cudaError_t launch_write(const DomainDesc& d, int64_t n, const double* src,
                         cudaStream_t st);

// FP64 reductions at step n against the snapshot u_prev (valid if
// have_prev); writes the new snapshot if u_prev != nullptr, per-block
// partials to `partials` (kReduceBlocks * kNumStats doubles) and the final
// statistics (kNumStats doubles) to `out`.
cudaError_t launch_reduce(const DomainDesc& d, int64_t n, double* u_prev,
                          int have_prev, double* partials, double* out,
                          cudaStream_t st);

}  // namespace lbm
