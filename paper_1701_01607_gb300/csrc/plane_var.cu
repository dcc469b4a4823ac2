// Shifted-plane sweep of the two-level variants (plane_var.cuh): instances and
// host helpers.
#include <algorithm>

#include "plane_var.cuh"

namespace mg3d {

// As plane_layout, for np slots of two channels each and the fields copied ahead.
PlaneLayout plane_var_layout(int prec, int prd, int np, int rows, int nx, int threads) {
    PlaneLayout l{};
    const int spv = prec == 0 ? 1 : 2;   // slots per 16-byte vector
    const int nv = 1 + (np + spv - 1) / spv;
    const size_t es = prec == 0 ? 8 : 4;
    l.item_rows = (long)rows * nx > threads ? 2 : 1;
    l.ipad = ((rows + l.item_rows - 1) / l.item_rows * nx + 31) / 32 * 32;
    l.chunks = std::max(1, std::min(threads / l.ipad, nv - 1));
    l.smem = 2ull * nv * (rows + 1) * nx * 16 + 2ull * rows * sizeof(plane::RowDest);
    const size_t next = 3ull * (prd ? 1 : 4) * rows * nx * es;
    const size_t sums = 4ull * l.chunks * rows * nx * es;
    if (l.chunks > 1) {
        if (l.smem + sums <= plane_smem_max(prec == 0)) l.smem += sums;
        else l.chunks = 1;
    }
    l.ahead = l.smem + next <= plane_smem_max(prec == 0) ? 1 : 0;
    if (l.ahead) l.smem += next;
    return l;
}

cudaError_t launch_plane_var_f64(const PlaneVarArgs<double> &a, const SweepShape &s,
                                 cudaStream_t st) {
    return plane_var_dispatch<double>(&a, s, a.nx, st, nullptr);
}

cudaError_t launch_plane_var_f32(const PlaneVarArgs<float> &a, const SweepShape &s,
                                 cudaStream_t st) {
    return plane_var_dispatch<float>(&a, s, a.nx, st, nullptr);
}

cudaError_t plane_var_clusters(int prec, const SweepShape &s, int nx, int *n) {
    *n = 0;
    return prec == 0 ? plane_var_dispatch<double>(nullptr, s, nx, 0, n)
                     : plane_var_dispatch<float>(nullptr, s, nx, 0, n);
}

}  // namespace mg3d
