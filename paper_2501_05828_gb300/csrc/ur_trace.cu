// The tracer's plane-wave instantiations and the choice among all of them.
#include "ur_trace.cuh"

namespace ur {

int trace_occupancy(int block, bool debug) {
    int n = 0;
    if (debug)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_trace<true, false, false, false, 0>, block, 0);
    else
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_trace<false, false, false, false, 0>, block, 0);
    return n > 0 ? n : 1;
}

namespace {

// What a launch's scenes, array and transmits ask of the tracer.
struct Needs {
    bool split = false, mesh = false, rough;
    Needs(const TraceP &P, bool point_waves) : rough(point_waves || P.radius > 0.f) {   // convex arrays: extended tracer
        for (int q = 0; q < P.n_scenes && q < kMaxScenes; ++q) {
            split = split || P.S[q].split_sampling != 0;
            mesh = mesh || P.S[q].n_tri > 0;
            for (int b = 0; b < P.S[q].n_bnd; ++b) rough = rough || P.S[q].bnd[b].alpha > 0.f;
        }
    }
    bool extended(bool emit) const { return rough || mesh || emit; }
};

}  // namespace

int trace_idle_min(const TraceP &P, bool point_waves, bool emit) {
    return Needs(P, point_waves).extended(emit) ? kIdleMinExtended : kIdleMin;
}

template <int ONE>
void launch_trace_of(const TraceP &P, bool debug, int block, int grid, cudaStream_t s, bool point_waves, bool emit) {
    const Needs needs(P, point_waves);
    const bool split = needs.split, mesh = needs.mesh;
    if (needs.extended(emit)) {
        const int cvx = P.radius > 0.f ? kGeoConvex : 0;
        if (mesh) {
            if (cvx) launch_extended<kGeoConvex | kGeoMesh | kGeoEmit | ONE>(P, debug, block, grid, s);
            else launch_extended<kGeoMesh | kGeoEmit | ONE>(P, debug, block, grid, s);
        } else if (emit) {
            if (cvx) launch_extended<kGeoConvex | kGeoEmit | ONE>(P, debug, block, grid, s);
            else launch_extended<kGeoEmit | ONE>(P, debug, block, grid, s);
        } else {
            if (cvx) launch_extended<kGeoConvex | ONE>(P, debug, block, grid, s);
            else launch_extended<ONE>(P, debug, block, grid, s);
        }
        return;
    }
    if (debug) {
        split ? k_trace<true, true, false, false, ONE><<<grid, block, 0, s>>>(P)
              : k_trace<true, false, false, false, ONE><<<grid, block, 0, s>>>(P);
    } else if (P.record) {
        split ? k_trace<false, true, true, false, ONE><<<grid, block, 0, s>>>(P)
              : k_trace<false, false, true, false, ONE><<<grid, block, 0, s>>>(P);
    } else {
        split ? k_trace<false, true, false, false, ONE><<<grid, block, 0, s>>>(P)
              : k_trace<false, false, false, false, ONE><<<grid, block, 0, s>>>(P);
    }
}

void launch_trace(const TraceP &P, bool debug, int block, int grid, cudaStream_t s, bool point_waves, bool emit) {
    if (P.n_scenes == 1)
        launch_trace_of<kGeoOne>(P, debug, block, grid, s, point_waves, emit);
    else
        launch_trace_of<0>(P, debug, block, grid, s, point_waves, emit);
}

}  // namespace ur
