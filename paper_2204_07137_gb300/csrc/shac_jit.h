// Run-time model-specialised builds of the batched kernels (shac_jit.cu).
#pragma once
#include <string>
#include <vector>

#include "../../include/shacsim.h"
#include "shac_kernels.cuh"

namespace shac {

// The forward and adjoint kernels (k_batched) of one
// build, as handles the runtime's launch and attribute calls accept, and the
// key the launch arguments must carry (BatchedArgs::spec_key).
struct JitKernels {
  const void* fwd = nullptr;
  const void* adj = nullptr;
  unsigned int key = 0;
};

// Build (or fetch from the process-wide cache) the kernels for model layout m,
// link parents `parent` (m.L entries) and DOF ancestor masks `masks` (m.nv
// entries) on `device` with team size `lanes`, register dense row capacity
// `rows` (0: the shared-memory dense stages), per-environment scratch stride
// `stride` and, when the team covers the model, the lane form.  SHAC_ERR_CUDA if the run-time
// compiler or the module load fails (the compiler's log in *log when given).
shac_status jit_kernels(int device, const DevModel& m, const std::vector<int>& parent, const std::vector<int>& masks,
                        int lanes, int rows, int stride, bool lane_form, JitKernels* out, std::string* log);

}  // namespace shac
