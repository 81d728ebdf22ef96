// The one-launch GMRES solve with FP32 element blocks.
#include "cycle.cuh"

namespace frk {

int launch_cycle_f32(const CycleArgs& a, int nblocks, int riemann, cudaStream_t s) {
  return cyc::launch<float, float>(a, nblocks, riemann, s);
}
int resident_cycle_f32(int riemann, int device) { return cyc::resident<float, float>(riemann, device); }

}  // namespace frk
