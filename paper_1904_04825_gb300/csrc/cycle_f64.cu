// The one-launch GMRES solve with FP64 element blocks.
#include "cycle.cuh"

namespace frk {

int launch_cycle_f64(const CycleArgs& a, int nblocks, int riemann, cudaStream_t s) {
  return cyc::launch<double, double>(a, nblocks, riemann, s);
}
int resident_cycle_f64(int riemann, int device) { return cyc::resident<double, double>(riemann, device); }

}  // namespace frk
