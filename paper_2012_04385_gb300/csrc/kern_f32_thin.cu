// Mixed-precision stage kernels on slabs of two planes, for launches of few
// leaves; every variant but the learned selector's, whose decision words are laid
// out by slabs of four.  Same build flags as kern_f32.cu; the names of stage_f32.cuh
// are those of an inline namespace here.
#define SF_THIN
#include "mr.cuh"
#include "stage_f32.cuh"

namespace mrb {

template <int FLUX>
static void launch_recon(const Topo& t, const Phys& p, const Pool& pool, int cur, int stage, const double* dt,
                         double* rhs_out, cudaStream_t st, int level) {
  if (p.recon == 2) launch_stage_f32<FLUX + 2>(t, p, pool, cur, stage, dt, rhs_out, st, level);
  else if (p.recon == 3) launch_stage_f32<FLUX + 4>(t, p, pool, cur, stage, dt, rhs_out, st, level);
  else if (p.recon == 4) launch_stage_f32<FLUX + 5>(t, p, pool, cur, stage, dt, rhs_out, st, level);
  else launch_stage_f32<FLUX + 0>(t, p, pool, cur, stage, dt, rhs_out, st, level);
}

void launch_rhs_rk_f32_thin(const Topo& t, const Phys& p, const Pool& pool, int cur, int stage, const double* dt,
                            double* rhs_out, cudaStream_t st, int level) {
  if (p.mu > 0.0) launch_stage_f32<32>(t, p, pool, cur, stage, dt, rhs_out, st, level);
  else if (p.flux == 1) launch_recon<8>(t, p, pool, cur, stage, dt, rhs_out, st, level);
  else if (p.flux == 2) launch_recon<16>(t, p, pool, cur, stage, dt, rhs_out, st, level);
  else launch_recon<0>(t, p, pool, cur, stage, dt, rhs_out, st, level);
}

}  // namespace mrb
