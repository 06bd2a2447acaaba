// Launch of the cluster-resident solver (resident.cuh) and its link layout.
#include "launch.h"
#include "resident.cuh"

namespace dl {

// Links for the resident solver: [parity][tile of 32 sites][36][32] pairs, pair q of a site its
// elements 2 q and 2 q + 1 of the eight-link row (d = 2 mu: U_mu(x); d = 2 mu + 1:
// U_mu(x - mu), not conjugated), the time boundary factor t_bc on the links of
// the hops that cross it, rounded from the FP64 links.
template <typename S>
static __global__ void resident_links_kernel(const double2 *g64, const uint32_t *coords, Geom g, S *out) {
    typedef typename Real<S>::type T;
    const long total = 72L * g.Vh;
    for (long idx = (long)blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += (long)gridDim.x * blockDim.x) {
        const int cb = (int)(idx % g.Vh), pq = (int)(idx / g.Vh), p = pq / 36, q = pq % 36;
        const Site st = decode(coords[(size_t)p * g.Vh + cb], g);
        cx<T> two[2];
        for (int h = 0; h < 2; ++h) {
            const int d = (2 * q + h) / 9, k = (2 * q + h) % 9, mu = d >> 1;
            const size_t site = (d & 1) ? (size_t)(1 - p) * g.Vh + nbr_bwd(st, g, mu) : (size_t)p * g.Vh + cb;
            const double2 u = g64[(site * 4 + mu) * 9 + k];
            const double sg = (mu == 3 && g.t_bc < 0 && st.c[3] == ((d & 1) ? 0 : g.L[3] - 1)) ? -1.0 : 1.0;
            two[h] = mk((T)(sg * u.x), (T)(sg * u.y));
        }
        st_pack<S, 2>(out + (((size_t)(p * ((g.Vh + 31) >> 5) + (cb >> 5)) * 36 + q) * 32 + (cb & 31)) * 4, two);
    }
}

cudaError_t launch_resident_links(int prec, const double *g64, const uint32_t *coords, const Geom &g, void *out,
                                  int grid, cudaStream_t s) {
    const double2 *u = reinterpret_cast<const double2 *>(g64);
    if (prec == P_F32) resident_links_kernel<float><<<grid, 256, 0, s>>>(u, coords, g, (float *)out);
    else resident_links_kernel<bf16><<<grid, 256, 0, s>>>(u, coords, g, (bf16 *)out);
    return cudaGetLastError();
}

}  // namespace dl
