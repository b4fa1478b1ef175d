// resident.cuh -- plan and launcher of the resident CG solve (resident.cu).
#pragma once
#include "pb_internal.cuh"

namespace pb {

struct ResPlan {  // how a grid is cut into bricks, one CTA each
  int build = 0;              // index of the kernel build
  int by = 0, bz = 0;         // rows and planes of a brick
  int nby = 0, nbz = 0, ctas = 0;
  int room = 0;               // CTAs of its build that the device holds at once
  int threads = 0, gpr = 0;   // groups of four x nodes per row
  int planes = 0;             // planes a thread can own (0: any number)
  int off_ap = 0;             // offset of Ap in shared memory (p before it)
};
struct ResArgs {  // kernel arguments
  const Inst *inst;
  void *packets;
  int *err, *resid_pending, *resid_list;
  void *z, *d, *ap, *p0, *p1;
  double *x64, *x64b;
  const uint8_t *code;
  const void *diag;
  int nx, ny, nz, px;
  uint32_t gpr_magic;  // for division by gpr
  int by, bz, nby, nbz, gpr, off_codes, off_ap;
  int slot;            // its place among the batch's instances
  int budget;          // iterations after which the launch leaves an inner solve in phase INNER
};
// The grids of a launch, a run of CTAs each: grid n has CTAs first[n] .. first[n + 1] - 1.
constexpr int RES_MAX_GRIDS = 16;
struct ResWave {
  int n;
  int first[RES_MAX_GRIDS + 1];
  ResArgs grid[RES_MAX_GRIDS];
};
struct ResOne {  // a launch over one grid
  ResArgs grid[1];
};

constexpr int RES_STATIC_SMEM = 16384;  // more than the kernel's static shared memory (half: of the builds in pairs)
constexpr int RES_MAX_PER_SM = 2;       // CTAs of a build on an SM at most

// Plan of a grid for num_sms SMs of max_smem bytes a CTA (the largest one CTA
// may ask for) and l2_bytes of L2; false: it does not fit (the two-pass form
// runs).
bool resident_plan(int nx, int ny, int nz, int mode, int coef, int num_sms, int max_smem, long l2_bytes, ResPlan *out);
size_t resident_packet_bytes(int ctas);  // of a launch
// Plan of a grid of a batch: for the most such grids at once (it does not depend
// on what else runs, and so neither do the grid's sums).  FP32 with packed codes only.
bool resident_batch_plan(int nx, int ny, int nz, int num_sms, int max_smem, ResPlan *out);
// Inner solves of n <= RES_MAX_GRIDS instances of a batch (slot[k], descriptor
// *I[k] on the host, plans of one build, all periodic or none) that are in
// their start phase, or that were left at the budget by an earlier launch, side by
// side, `budget` iterations of each at most: at most the plans' room CTAs together.
cudaError_t launch_resident_batch(int n, const ResPlan *const *P, const Inst *const *I, const int *slot,
                                  const Batch &B, void *packets, size_t packet_bytes, int budget, cudaStream_t st);
// One inner solve of the batch's only instance (I: its descriptor on the host)
// if it is in its start phase.
cudaError_t launch_resident(const ResPlan &P, const Inst &I, const Batch &B, void *packets, size_t packet_bytes,
                            cudaStream_t st);

}  // namespace pb
