// fei_sf64.cu -- FP64 instances of the sum-factorised forward (fei_sf.cuh).
#include "fei_internal.cuh"
#include "fei_sf.cuh"

namespace fei {

fei_status launch_sf64_forward(int p, const fei_reference *ref, const FwdArgs &a, int64_t grid_work, cudaStream_t s,
                               int64_t grid_cap) {
  if (grid_work <= 0) return FEI_OK;
  switch (p) {
    case 2: return launch_sf<double, 2>(ref->sf64, a, grid_work, s, grid_cap);
    case 3: return launch_sf<double, 3>(ref->sf64, a, grid_work, s, grid_cap);
    case 4: return launch_sf<double, 4>(ref->sf64, a, grid_work, s, grid_cap);
    case 5: return launch_sf<double, 5>(ref->sf64, a, grid_work, s, grid_cap);
    case 6: return launch_sf<double, 6>(ref->sf64, a, grid_work, s, grid_cap);
    case 7: return launch_sf<double, 7>(ref->sf64, a, grid_work, s, grid_cap);
  }
  return set_error(FEI_ERR_UNSUPPORTED, "sum-factorised FP64 path for degree %d", p);
}

}  // namespace fei
