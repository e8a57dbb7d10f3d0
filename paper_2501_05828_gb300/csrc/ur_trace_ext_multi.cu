// The extended tracer's instantiations (rough boundaries, point-source transmits, convex arrays, meshes)
// for batches of several scenes.
#include "ur_trace.cuh"

namespace ur {

template <int GEO>
void launch_extended(const TraceP &P, bool debug, int block, int grid, cudaStream_t s) {
    debug ? k_trace<true, false, false, true, GEO><<<grid, block, 0, s>>>(P)
          : k_trace<false, false, false, true, GEO><<<grid, block, 0, s>>>(P);
}

template void launch_extended<0>(const TraceP &, bool, int, int, cudaStream_t);
template void launch_extended<kGeoConvex>(const TraceP &, bool, int, int, cudaStream_t);
template void launch_extended<kGeoEmit>(const TraceP &, bool, int, int, cudaStream_t);
template void launch_extended<kGeoConvex | kGeoEmit>(const TraceP &, bool, int, int, cudaStream_t);
template void launch_extended<kGeoMesh | kGeoEmit>(const TraceP &, bool, int, int, cudaStream_t);
template void launch_extended<kGeoConvex | kGeoMesh | kGeoEmit>(const TraceP &, bool, int, int, cudaStream_t);

}  // namespace ur
