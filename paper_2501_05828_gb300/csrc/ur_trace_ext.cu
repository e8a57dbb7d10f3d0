// The extended tracer's instantiations (rough boundaries, point-source transmits, convex arrays, meshes)
// for launches of one scene.
#include "ur_trace.cuh"

namespace ur {

template <int GEO>
void launch_extended(const TraceP &P, bool debug, int block, int grid, cudaStream_t s) {
    debug ? k_trace<true, false, false, true, GEO><<<grid, block, 0, s>>>(P)
          : k_trace<false, false, false, true, GEO><<<grid, block, 0, s>>>(P);
}

template void launch_extended<kGeoOne>(const TraceP &, bool, int, int, cudaStream_t);
template void launch_extended<kGeoConvex | kGeoOne>(const TraceP &, bool, int, int, cudaStream_t);
template void launch_extended<kGeoEmit | kGeoOne>(const TraceP &, bool, int, int, cudaStream_t);
template void launch_extended<kGeoConvex | kGeoEmit | kGeoOne>(const TraceP &, bool, int, int, cudaStream_t);
template void launch_extended<kGeoMesh | kGeoEmit | kGeoOne>(const TraceP &, bool, int, int, cudaStream_t);
template void launch_extended<kGeoConvex | kGeoMesh | kGeoEmit | kGeoOne>(const TraceP &, bool, int, int, cudaStream_t);

}  // namespace ur
