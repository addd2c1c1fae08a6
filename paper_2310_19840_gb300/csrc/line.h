// line.h - programs of the one-dimensional FP32 step (line.cuh): a list of
// phases that one block, or a cluster of blocks, runs for one member, with a
// barrier between them.
#pragma once

#include "sbi_internal.h"

namespace sbi {

constexpr int kLineSlots = 6;          // physical fields held in shared memory
constexpr int kLineMaxBytes = 40960;   // largest program (it is copied into shared memory)
constexpr int kLineStages = 4;         // RK4 stages of a program

enum LinePhaseType : uint8_t {
  LP_INVERSE = 0,   // jobs: mixed sums -> slots, one transform each
  LP_FORWARD = 1,   // jobs: products of slots -> mixed, one transform each
  LP_COL = 2,       // per mode: sums of terms, outputs, pass-through sums
  LP_RK = 3,        // state update; the new working values go to slots 2 (eta) and 3 (phi)
  LP_WDOT = 4,      // physical dst <- (V + eta_x phi_x) / (1 + eta_x^2)
  LP_WMK = 5,       // surface pressure profile -> slot 5 (of the first block, which runs job 0)
};

// One transform.  Inverse: slot <- inverse of the sum of bufs [buf, buf + nsrc),
// also written to the physical bufs[phys] when phys >= 0.  Forward: bufs[buf] <-
// transform of coef eta^ea delta^eb w^ew slot (op ROP_PROD), or of the
// dynamic-condition / kinematic forms of slots slot, slot + 1, slot + 2 = V,
// eta_x, phi_x (op ROP_N2, ROP_VFW).
struct LineJob {
  uint8_t op, slot, ea, eb, ew, nsrc;
  uint8_t pg;            // ROP_N2: subtract the pressure of slot 5
  uint8_t pad_;
  int16_t buf, phys;
  float coef;
};
// One multiplier of a column sum or output: src/dst is bufs[buf].
struct LineTerm {
  const void* tab;
  int16_t buf;
  uint8_t acc, ph;       // accumulator, power of i
  int32_t pad_;
};
struct LinePhase {
  uint8_t type;
  uint8_t sync;                // 1: what the phases before left in global memory, or still read there,
                               // has to be ordered for every block of the cluster first
  int16_t begin, end;          // jobs; LP_COL: terms
  int16_t out_begin, out_end;  // LP_COL: outputs (terms); LP_RK: index of the RkParams in out_begin
  int16_t pass_begin, pass_end;  // LP_COL: pass-through bufs, added to the first output
  int16_t eta, delta, wgt;     // physical bufs (-1: none)
  int16_t dst;                 // LP_WDOT
  const int* active;           // per-member flags (nullptr: every member runs the phase)
};
struct LineWmk {
  const double *prof, *omega, *phase, *t;
  int J, stage;                // stage: of LineParams::offset
};
struct LineHeader {
  int bytes;                   // of the whole program
  int nphases, phases, jobs, terms, bufs, rks, wmks;   // byte offsets of the arrays
  int W;
  const void* tw;
};
// What depends on the step size is handed over with the launch: a program is the
// same for every step (of a scheme whose tables are).
struct LineParams {
  const void* program;
  int bytes;
  int exact;                   // half of the modes kept
  int member0, member1;        // members of this launch (one cluster of blocks each)
  int cluster;                 // blocks per member
  RkScalar cdt[kLineStages], dt6;   // RK_STAGE phases, by stage - 1
  double offset[kLineStages];       // stage time minus step start, by LineWmk::stage
};
// The most blocks per member: rows of 2048 points and more have too few groups
// of threads in one block for the products of a level (at 1024 points two
// blocks were 20 % slower than one).
constexpr int line_cluster(int nx) { return nx >= 4096 ? 8 : (nx >= 2048 ? 4 : 1); }

// Whether a group of n members of nx points takes this form.  A member fills an
// SM (up to 1024 points; longer ones as good as), so the time is that of a
// member for every 152 of them, while that of one launch per pass hardly grows
// until the members fill the GPU.  Microseconds of a step, one launch and one
// per pass:
//   points  members  flat bottom   variable bottom
//      256      304  214 and 332
//      256      608  417 and 352   507 and 473
//     1024      304  275 and 391
//     1024      608  543 and 476   749 and 700
//     2048      152  299 and 425   373 and 585
//     2048      304  577 and 491   736 and 770
//     4096      152  417 and 569   629 and 845
//     4096      304  835 and 807   1232 and 1397
// (2432 members of 256 points: 1633 and 432 with a flat bottom.)
constexpr bool line_pays(int nx, int n, bool variable_bottom) {
  return n <= kSMs * (nx <= 1024 ? 3 : (variable_bottom ? 2 : 1));
}

cudaError_t prepare_line_kernels(int nx);
cudaError_t line_clusters(int nx, int cluster, int* most);   // after prepare_line_kernels
cudaError_t launch_line(int nx, const LineParams& p, cudaStream_t st);

}  // namespace sbi
