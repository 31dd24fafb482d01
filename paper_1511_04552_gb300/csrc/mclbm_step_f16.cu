// Step kernels of libmclbm for state storage type __half (one translation unit per storage
// type, so the build compiles them in parallel).
#include <algorithm>

#include "mclbm_cluster.cuh"
#include "mclbm_pair.cuh"
#include "mclbm_resident.cuh"

namespace mcl {

cudaError_t launch_step_f16(const StepArgs& a, const StepConfig& c, const CUtensorMap* map,
                           cudaStream_t st) {
  return pair::launch_pair_t<__half>(a, c, map, st);
}

cudaError_t prepare_tma_f16(StepConfig* c, const Layout& L) {
  return pair::prepare_pair_tma_t<__half>(c, L);
}

cudaError_t prepare_cluster_f16(StepConfig* c, const Layout& L, bool all, bool two,
                                cudaStream_t st) {
  return cluster::prepare<__half>(c, L, all, two, st);
}

cudaError_t launch_cluster_f16(const StepArgs& a, const StepConfig& c, int n, uint32_t steps0,
                              uint32_t* epoch, cudaStream_t st) {
  return cluster::launch<__half>(a, c, n, steps0, epoch, st);
}

cudaError_t prepare_resident_f16(StepConfig* c, const Layout& L, bool all, bool two) {
  return resident::prepare<__half>(c, L, all, two);
}

cudaError_t launch_resident_f16(const StepArgs& a, const StepConfig& c, int n, void* scratch,
                               uint32_t* epoch, cudaStream_t st) {
  return resident::launch<__half>(a, c, n, scratch, epoch, st);
}

}  // namespace mcl
