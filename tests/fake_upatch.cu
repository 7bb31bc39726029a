// One launch of the unstructured patch kernel (2D, degree 2, FP32) whose
// workspace slice takes `slice` bytes of shared memory (0: none).
#include "../paper_2510_17785_gb300/csrc/umesh_kern.cuh"

extern "C" int launch_upatch(int mode, size_t slice) {
  pmg::UPatchArgs<float> a = {};
  a.ws_shared = slice > 0;
  a.ws_stride = slice / sizeof(float);
  return pmg::upatch_launch_P<2, 2, float>(mode, a, 1, nullptr);
}
