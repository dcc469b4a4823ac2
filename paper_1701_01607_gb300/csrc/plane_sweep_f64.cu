// Shifted-plane sweep (plane_sweep.cuh), FP64 instances, and the host-side
// helpers shared by both precisions.
#include <algorithm>

#include "plane_sweep.cuh"

namespace mg3d {

bool plane_np_supported(int np) {
    for (int i = 0; i < kPlaneNpCount; ++i)
        if (kPlaneNp[i] == np) return true;
    return false;
}

// A band with more nodes than threads is walked two rows at a time: the rows
// share the x interpolation of the row between them.  A band with spare threads
// takes one row per thread and spreads the slots of a node over the spare ones.
PlaneLayout plane_layout(int prec, int np, int rows, int nx, int threads) {
    PlaneLayout l{};
    const int vw = prec == 0 ? 2 : 4;                 // elements per 16-byte vector
    const int nv = (np + 2 + vw - 1) / vw;            // chi0, S and np intensities
    const size_t es = prec == 0 ? 8 : 4;
    l.item_rows = (long)rows * nx > threads ? 2 : 1;
    l.ipad = ((rows + l.item_rows - 1) / l.item_rows * nx + 31) / 32 * 32;
    l.chunks = prec == 0 ? std::max(1, std::min(threads / l.ipad, nv - 1)) : 1;
    l.smem = 2ull * nv * (rows + 1) * nx * 16 + 2ull * rows * sizeof(plane::RowTarget);
    const size_t next = 6ull * rows * nx * es, sums = 4ull * l.chunks * rows * nx * es;
    if (l.chunks > 1) {
        if (l.smem + sums <= plane_smem_max(prec == 0)) l.smem += sums;
        else l.chunks = 1;
    }
    l.ahead = l.smem + next <= plane_smem_max(prec == 0) ? 1 : 0;
    if (l.ahead) l.smem += next;
    return l;
}

cudaError_t launch_plane_sweep_f64(const PlaneArgs<double> &a, const SweepShape &s,
                                   cudaStream_t st) {
    if (s.plane == 2) return launch_plane_async_f64(a, s, st);
    return plane_dispatch<double, false>(&a, s, a.nx, st, nullptr);
}

cudaError_t plane_active_clusters_f32(const SweepShape &s, int nx, int *n);

cudaError_t plane_active_clusters(int prec, const SweepShape &s, int nx, int *n) {
    *n = 0;
    if (prec != 0) return plane_active_clusters_f32(s, nx, n);
    if (s.plane == 2) return plane_async_clusters_f64(s, nx, n);
    return plane_dispatch<double, false>(nullptr, s, nx, 0, n);
}

}  // namespace mg3d
