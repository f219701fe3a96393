// ce_resident_f32.cu -- the resident multi-step kernel (ce_resident.cuh), FP32.
#include "ce_resident.cuh"

namespace ce {

ResidentPlan resident_plan_f32(int dims, int64_t N, int nf, int device, int sms) {
  return resident::plan<float>(dims, N, nf, device, sms);
}

cudaError_t launch_resident(const ResidentArgs<float>& a, int dims, int nf, cudaStream_t st) {
  return resident::launch<float>(a, dims, nf, st);
}

}  // namespace ce
