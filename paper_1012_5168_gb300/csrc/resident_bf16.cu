// The cluster-resident solver for bf16 storage.
#include "resident_launch.cuh"

namespace dl {

cudaError_t launch_resident_bf16(const ResArgs &a, int C, int n, int cg, cudaStream_t s) {
    return resident_go<bf16>(a, C, n, cg, s);
}
int resident_clusters_bf16(int C) { return resident_max_clusters(resident_kernel<bf16, 0>, sizeof(ResShared<Real<bf16>::type>), C); }

}  // namespace dl
