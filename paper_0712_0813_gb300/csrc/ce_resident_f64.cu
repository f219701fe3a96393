// ce_resident_f64.cu -- the resident multi-step kernel (ce_resident.cuh), FP64.
#include "ce_resident.cuh"

namespace ce {

ResidentPlan resident_plan_f64(int dims, int64_t N, int nf, int device, int sms) {
  return resident::plan<double>(dims, N, nf, device, sms);
}

cudaError_t launch_resident(const ResidentArgs<double>& a, int dims, int nf, cudaStream_t st) {
  return resident::launch<double>(a, dims, nf, st);
}

}  // namespace ce
