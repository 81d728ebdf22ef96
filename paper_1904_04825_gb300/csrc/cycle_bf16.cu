// The one-launch GMRES solve with BF16 element blocks.
#include "cycle.cuh"

namespace frk {

int launch_cycle_bf16(const CycleArgs& a, int nblocks, int riemann, cudaStream_t s) {
  return cyc::launch<__nv_bfloat16, float>(a, nblocks, riemann, s);
}
int resident_cycle_bf16(int riemann, int device) { return cyc::resident<__nv_bfloat16, float>(riemann, device); }

}  // namespace frk
