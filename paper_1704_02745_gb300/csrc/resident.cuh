// resident.cuh -- plan and launcher of the resident CG solve (resident.cu).
#pragma once
#include "pb_internal.cuh"

namespace pb {

struct ResPlan {  // how a grid is cut into bricks, one CTA each
  int build = 0;              // index of the kernel build
  int by = 0, bz = 0;         // rows and planes of a brick
  int nby = 0, nbz = 0, ctas = 0;
  int threads = 0, gpr = 0;   // groups of four x nodes per row
  int off_codes = 0, off_ap = 0;
  size_t smem = 0;
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
};

constexpr int RES_STATIC_SMEM = 16384;  // more than the kernel's static shared memory

// Plan of a grid for num_sms SMs of max_smem bytes a CTA; false: the grid does
// not fit (the two-pass form runs).
bool resident_plan(int nx, int ny, int nz, int mode, int coef, int num_sms, int max_smem, ResPlan *out);
size_t resident_packet_bytes(int num_sms);
// One inner solve of the batch's only instance (I: its descriptor on the host)
// if it is in its start phase.
cudaError_t launch_resident(const ResPlan &P, const Inst &I, const Batch &B, void *packets, size_t packet_bytes,
                            cudaStream_t st);

}  // namespace pb
