// The cluster-resident solver for float storage.
#include "resident_launch.cuh"

namespace dl {

cudaError_t launch_resident_f32(const ResArgs &a, int C, int n, int cg, cudaStream_t s) {
    return resident_go<float>(a, C, n, cg, s);
}
int resident_clusters_f32(int C) { return resident_max_clusters(resident_kernel<float, 0>, sizeof(ResShared<Real<float>::type>), C); }

}  // namespace dl
