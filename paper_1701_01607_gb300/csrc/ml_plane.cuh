// Multi-level formal solution with shifted plane storage: the linear
// short-characteristics sweep (Sec. 3) of a static atmosphere, laid out as
// the two-level shifted-plane sweep (plane_sweep.cuh) is.
//
// The upwind crossing of a (ray, step) lies at the same horizontal offset from
// every node of the plane (periodic boundaries, Sec. 4.2), so each ray's
// finished plane is stored shifted by the offset of the step that reads it and
// a node finds its four upwind corners at fixed offsets (x, y), (x+1, y),
// (x, y+1), (x+1, y+1) of its ray's stored frame.  In the multi-level atom the
// opacity and source function differ from frequency to frequency, so they ride
// along as channels beside the intensity: per node, ray and frequency (I, chi,
// S), NF frequencies per block, padded to whole 16-byte vectors (vector v of all
// nodes of a frame contiguous: conflict-free 16-byte loads).
//
// One thread-block cluster per (group of NF frequencies of the chunk, group of
// rays of one hemisphere); its blocks split the stored frames in bands of
// rows, each with a halo row, and a block holds one frame per ray of its group (double buffered).  A thread owns an item, one column of two
// neighbouring rows, for the whole sweep and walks the group's rays at it, so
// the angle sums over the group are complete in registers and written once per
// (slot, frequency, node), the slot layout of the other multi-level sweep:
//   Jx = sum (I - w0 S) + sc sum w0,   Ux = sum u + oc sum w0,   Jm = sum I
// (times the ray weight; sc, oc: the parts of S and the opacity share the
// transition does not set), all sums of non-negative terms.  Writes go to the
// block owning the shifted row (distributed shared memory) with a copy into the
// halo row, at row addresses that are tabulated once per step (a store per
// ray and node would otherwise be mostly address arithmetic); one cluster
// barrier per plane orders them, its two halves on either side of the stores
// of the angle sums.
//
// The interpolation (the two rows of an item share the x interpolation of the
// row between them) and the FP64 weights in integer arithmetic are those of
// plane_sweep.cuh.
#pragma once

#include "plane_sweep.cuh"

namespace mg3d {

namespace mlplane {

// 16-byte vectors per node: I, chi, S of nf frequencies
template <typename T>
__host__ __device__ constexpr int vectors(int nf) {
    return (3 * nf + plane::vec_width<T>() - 1) / plane::vec_width<T>();
}

}  // namespace mlplane

template <typename T, int NF>
__device__ __forceinline__ void ml_plane_body(const MlPlaneArgs<T> &a) {
    using namespace plane;
    constexpr bool F64 = sizeof(T) == 8;
    constexpr int VW = vec_width<T>();
    constexpr int NV = mlplane::vectors<T>(NF);
    constexpr int R = NF == 4 ? 1 : 2;   // rows of an item (four frequencies fill the registers)

    const int g = blockIdx.y, slot = blockIdx.z;
    const int rpb = a.rpb, groups = 12 / rpb;
    const int hemi = slot / groups;
    const int r0 = hemi * 12 + (slot - hemi * groups) * rpb;   // rays 0-11 point up
    const bool up = hemi == 0;
    const int f0 = g * NF;
    const int nfl = min(NF, a.nfreq - f0);   // active frequencies of the group
    const int nb = a.bands;
    const bool cl = nb > 1;
    const int rank = (int)cluster_rank();
    const int nx = a.nx, ny = a.ny, nz = a.nz, rows = a.rows;
    const int y0 = rank * rows;
    const int myrows = min(rows, ny - y0);
    const int lastrows = ny - (nb - 1) * rows;
    const unsigned nxb = (unsigned)nx * 16, pitch = nxb;   // one stored row of a vector, bytes
    const unsigned vs = (unsigned)(rows + 1) * pitch;   // one vector of a ray's frame
    const unsigned ray_b = NV * vs;                     // one ray's stored frame
    const unsigned frame = (unsigned)rpb * ray_b;       // all rays of one buffer
    const int nplane = nx * ny;
    const long nvox = (long)nplane * nz;
    // a block's shared memory may be addressed by its cluster once the block runs:
    // arrive here, wait before the first store into another block
    if (cl) cluster_arrive_relaxed();

    extern __shared__ __align__(16) unsigned char smem_raw[];
    const unsigned buf_addr = smem_addr(smem_raw);
    __shared__ fx::u64 fx_tab[F64 ? 2 * fx::kTab : 1];   // tables of the integer weights
    // the rays' constants of step t in [t & 3], three steps ahead: the row
    // table of step t + 1 is made during step t, when all copies but the latest
    // group have landed
    __shared__ __align__(16) PlaneLerp<T> sstep[4][12];
    // where the band's rows go at the end of step t: [t & 1][ray][row]
    RowDest *dest = reinterpret_cast<RowDest *>(smem_raw + 2 * (size_t)frame);
    if (F64)
        for (int i = threadIdx.x; i < 2 * fx::kTab; i += blockDim.x) fx_tab[i] = a.fx_tab[i];
    auto fetch_steps = [&](int t) {
        constexpr int NC = sizeof(PlaneLerp<T>) / 16;
        for (int i = threadIdx.x; i < rpb * NC; i += blockDim.x) {
            const int j = i / NC, c = i - j * NC;
            cp_async16(reinterpret_cast<unsigned char *>(&sstep[t & 3][j]) + 16 * c,
                       reinterpret_cast<const unsigned char *>(&a.steps[(long)(r0 + j) * nz + t]) +
                           16 * c);
        }
        cp_async_commit();
    };
    fetch_steps(0);
    if (nz > 1) fetch_steps(1);
    if (nz > 2) fetch_steps(2);
    if (nz > 3) fetch_steps(3);
    cp_async_wait();
    __syncthreads();
    const T wray = T(1.0 / kRays);

    const int nth = blockDim.x;
    const int items = (myrows + R - 1) / R * nx;
    auto item_at = [&](int q, int &x, int &yl0, int &nr) {
        const int gy = band_of(q, a.xmagic);
        x = q - gy * nx;
        yl0 = gy * R;
        nr = min(R, myrows - yl0);
    };

    // The destinations of the band's rows in the frames of step t + 1, shifted by
    // each ray's sy: the block that owns the row and, where it is that block's
    // first row, the halo row of the band before it.  Made one step ahead; the
    // barrier between orders them.
    auto fill_dest = [&](int t) {
        for (int i = threadIdx.x; i < rpb * myrows; i += blockDim.x) {
            const int j = i / myrows, yl = i - j * myrows;
            int ys = y0 + yl - sstep[t & 3][j].sy;
            ys += ys < 0 ? ny : 0;
            const int ob = cl ? band_of(ys, a.rmagic) : 0;
            const int lr = ys - ob * rows;
            const unsigned col = (t & 1) * frame + (unsigned)j * ray_b;
            const int hb = ob == 0 ? nb - 1 : ob - 1;   // the band whose halo row is ys
            RowDest d;
            d.base = cluster_addr(buf_addr, (unsigned)ob) + col + (unsigned)lr * pitch;
            d.halo = lr != 0 ? kNoHalo
                             : cluster_addr(buf_addr, (unsigned)hb) + col +
                                   (unsigned)(hb == nb - 1 ? lastrows : rows) * pitch;
            dest[(t & 1) * rpb * rows + j * rows + yl] = d;
        }
    };
    // channels of row yl, column offset xs (bytes, shifted) for ray j
    auto put = [&](const T *cv, const RowDest &d, unsigned xs) {
        const unsigned base = d.base + xs;
#pragma unroll
        for (int v = 0; v < NV; ++v) st16(base + v * vs, cv + v * VW);
        if (d.halo != kNoHalo) {
#pragma unroll
            for (int v = 0; v < NV; ++v) st16(d.halo + xs + v * vs, cv + v * VW);
        }
    };
    // column x of the plane's frames shifted by sx, in bytes
    auto shifted = [&](unsigned xb, int sx) {
        const int xs = (int)xb - sx * 16;
        return (unsigned)(xs < 0 ? xs + (int)nxb : xs);
    };

    // chi and S of item q's nodes on the plane of step t
    auto load_nodes = [&](int t, int x, int yl0, int nr, T (*chi)[NF], T (*S)[NF]) {
        const long kp = (long)(up ? t : nz - 1 - t) * nplane;
#pragma unroll
        for (int j = 0; j < R; ++j)
#pragma unroll
            for (int k = 0; k < NF; ++k)
                if (j < nr && k < nfl) {
                    const long o = (long)(f0 + k) * nvox + kp + (y0 + yl0 + j) * nx + x;
                    chi[j][k] = a.chi[o];
                    S[j][k] = a.S[o];
                } else {
                    chi[j][k] = S[j][k] = T(0);
                }
    };

    // ---- entering boundary plane: I prescribed (bottom: Planck at the local
    // temperature, top: zero), w0 = 0
    if (nz > 1) {
        fill_dest(0);
        if (nz > 2) fill_dest(1);
        __syncthreads();
    }
    if (cl) cluster_wait();   // every block of the cluster has started
    {
        const long k0 = (long)(up ? 0 : nz - 1) * nplane;
        for (int q = threadIdx.x; q < items; q += nth) {
            int x, yl0, nr;
            item_at(q, x, yl0, nr);
            T chi[R][NF], S[R][NF];
            load_nodes(0, x, yl0, nr, chi, S);
#pragma unroll
            for (int i = 0; i < R; ++i) {
                if (i >= nr) continue;
                const int node = (y0 + yl0 + i) * nx + x;
                T cv[NV * VW];
#pragma unroll
                for (int c = 0; c < NV * VW; ++c) cv[c] = T(0);
#pragma unroll
                for (int k = 0; k < NF; ++k) {
                    if (k >= nfl) continue;
                    const T Ib = up ? a.ib[(long)(f0 + k) * nplane + node] : T(0);
                    cv[3 * k] = Ib;
                    cv[3 * k + 1] = chi[i][k];
                    cv[3 * k + 2] = S[i][k];
                    const long o = ((long)slot * a.nfreq + f0 + k) * nvox + k0 + node;
                    a.jx[o] = T(rpb) * wray * Ib;
                    a.ux[o] = T(rpb) * wray;
                    if (a.jm) a.jm[o] = T(rpb) * wray * Ib;
                }
                if (nz > 1)
                    for (int j = 0; j < rpb; ++j)
                        put(cv, dest[j * rows + yl0 + i],
                            shifted((unsigned)x * 16, sstep[0][j].sx));
            }
        }
    }
    // chi and S of the thread's first item, loaded one step ahead
    int x0i = 0, yl0i = 0, nr0i = 0;
    T nchi[R][NF], nS[R][NF];
    if ((int)threadIdx.x < items) {
        item_at(threadIdx.x, x0i, yl0i, nr0i);
        if (nz > 1) load_nodes(1, x0i, yl0i, nr0i, nchi, nS);
    }
    if (cl) cluster_barrier();
    else __syncthreads();

    for (int t = 1; t < nz; ++t) {
        const long kp = (long)(up ? t : nz - 1 - t) * nplane;
        const unsigned prev = buf_addr + ((t - 1) & 1) * frame;
        const bool write = t + 1 < nz;
        if (t + 3 < nz) fetch_steps(t + 3);
        if (t + 2 < nz) fill_dest(t + 1);
        const RowDest *dst = dest + (t & 1) * rpb * rows;
        // angle sums of the first item, stored after the barrier's first half
        T kj[R][NF], ku[R][NF], km[R][NF];
        for (int q = threadIdx.x; q < items; q += nth) {
            const bool first = q == (int)threadIdx.x;
            int x = x0i, yl0 = yl0i, nr = nr0i;
            T chi[R][NF], S[R][NF];
            if (first) {
#pragma unroll
                for (int i = 0; i < R; ++i)
#pragma unroll
                    for (int k = 0; k < NF; ++k) {
                        chi[i][k] = nchi[i][k];
                        S[i][k] = nS[i][k];
                    }
                if (write) load_nodes(t + 1, x, yl0, nr, nchi, nS);
            } else {
                item_at(q, x, yl0, nr);
                load_nodes(t, x, yl0, nr, chi, S);
            }
            const unsigned xb = (unsigned)x * 16, xb1 = x + 1 == nx ? 0u : xb + 16;
            T sp[R][NF], su[R][NF], sw[R][NF], si[R][NF];
#pragma unroll
            for (int i = 0; i < R; ++i)
#pragma unroll
                for (int k = 0; k < NF; ++k) sp[i][k] = su[i][k] = sw[i][k] = si[i][k] = T(0);
#pragma unroll 1
            for (int j = 0; j < rpb; ++j) {
                const PlaneLerp<T> st = sstep[t & 3][j];
                // H of a row; FP64 walks the item's rows from the nearer outer one
                const unsigned xn = (st.near & 1) ? xb1 : xb, xf = (st.near & 1) ? xb : xb1;
                bool down = false;
                if constexpr (F64) down = st.near & 2;
                const unsigned row0 = prev + (unsigned)j * ray_b +
                                      (unsigned)(down ? yl0 + nr : yl0) * pitch;
                const unsigned dpitch = down ? 0u - pitch : pitch;
                auto row_h = [&](int k, T *h) {
                    const unsigned pn = row0 + k * dpitch + xn, pf = row0 + k * dpitch + xf;
#pragma unroll
                    for (int v = 0; v < NV; ++v) {
                        T A[VW], B[VW];
                        lds16(pn + v * vs, A);
                        lds16(pf + v * vs, B);
#pragma unroll
                        for (int e = 0; e < VW; ++e) h[v * VW + e] = fma(st.rx, B[e], A[e]);
                    }
                };
                const unsigned xs = shifted(xb, st.sx);
                // node n of the item from its upwind channels V
                auto node = [&](auto n_tag, T *V) {
                    constexpr int n = decltype(n_tag)::value;
#pragma unroll
                    for (int k = 0; k < NF; ++k) {
                        if (k >= nfl) continue;
                        T cex, w0, wup, u, S_up;   // FP64: V and cex carry the factor c
                        if constexpr (F64) {
                            S_up = V[3 * k + 2] * st.c;
                            const T xt = fma(st.c, V[3 * k + 1], chi[n][k]) * st.half_s;
                            if (fx::in_range(xt)) {
                                fx::u64 m, cm;
                                int e, ce;
                                fx::unpack(xt, &m, &e);
                                fx::unpack(st.c, &cm, &ce);
                                fx::Weights w;
                                if (e <= fx::kThinExp) {
                                    w = fx::thin(m, e);
                                    u = fx::pack(w.u, 0);
                                } else {
                                    w = fx::closed(fx::mulhi(m, fx::kLog2e), e + 1, fx::recip(m),
                                                   1 - e, fx::Tables{fx_tab, fx_tab + fx::kTab});
                                    u = fx::pack32(w.um, w.ue);
                                }
                                cex = w.E ? fx::pack62(fx::mulhi(w.E, cm), ce - w.n) : 0.0;
                                w0 = w.w0;
                                wup = w.wup;
                            } else {
                                const Weights64 w = weights64(xt);
                                cex = st.c * w.ex;
                                w0 = w.w0;
                                wup = w.wup;
                                u = w.u;
                            }
                        } else {
                            S_up = V[3 * k + 2];
                            Weights32::eval((V[3 * k + 1] + chi[n][k]) * st.half_s, cex, w0, wup,
                                            u);
                        }
                        const T part = fma(V[3 * k], cex, wup * S_up);   // I - w0 S
                        const T I = fma(w0, S[n][k], part);
                        sp[n][k] += part;
                        su[n][k] += u;
                        sw[n][k] += w0;
                        if (a.jm) si[n][k] += I;
                        V[3 * k] = I;
                        V[3 * k + 1] = chi[n][k];
                        V[3 * k + 2] = S[n][k];
                    }
                    if (write) put(V, dst[j * rows + yl0 + n], xs);
                };
                using N0 = std::integral_constant<int, 0>;
                using N1 = std::integral_constant<int, 1>;
                T h0[NV * VW], h1[NV * VW], V[NV * VW];
                row_h(0, h0);
                row_h(1, h1);
                auto mix = [&](const T *ha, const T *hb) {   // rows in the walk's order
#pragma unroll
                    for (int c = 0; c < NV * VW; ++c) {
                        if constexpr (F64) V[c] = c < 3 * NF ? fma(st.ry, hb[c], ha[c]) : T(0);
                        else V[c] = c < 3 * NF ? fma(st.wy1, hb[c], st.wy0 * ha[c]) : T(0);
                    }
                };
                mix(h0, h1);
                if constexpr (R == 1) {
                    node(N0{}, V);
                } else {
                    if (down && nr == 2) node(N1{}, V);
                    else node(N0{}, V);
                    if (nr == 2) {
                        row_h(2, h0);
                        mix(h1, h0);
                        if (down) node(N0{}, V);
                        else node(N1{}, V);
                    }
                }
            }
#pragma unroll
            for (int i = 0; i < R; ++i) {
                if (i >= nr) continue;
#pragma unroll
                for (int k = 0; k < NF; ++k) {
                    if (k >= nfl) continue;
                    const long v = (long)(f0 + k) * nvox + kp + (y0 + yl0 + i) * nx + x;
                    const T vj = wray * (sp[i][k] + a.sc[v] * sw[i][k]);
                    const T vu = wray * (su[i][k] + a.oc[v] * sw[i][k]);
                    if (first) {
                        kj[i][k] = vj;
                        ku[i][k] = vu;
                        km[i][k] = wray * si[i][k];
                    } else {
                        const long o = (long)slot * a.nfreq * nvox + v;
                        a.jx[o] = vj;
                        a.ux[o] = vu;
                        if (a.jm) a.jm[o] = wray * si[i][k];
                    }
                }
            }
        }
        // the constants of step t + 2 are there before the barrier
        if (t + 3 < nz) cp_async_wait_but_last();
        else cp_async_wait();
        if (write) {
            if (cl) cluster_arrive();
            else __syncthreads();
        }
#pragma unroll
        for (int i = 0; i < R; ++i)
#pragma unroll
            for (int k = 0; k < NF; ++k)
                if (i < nr0i && k < nfl) {
                    const long o = ((long)slot * a.nfreq + f0 + k) * nvox + kp +
                                   (y0 + yl0i + i) * nx + x0i;
                    a.jx[o] = kj[i][k];
                    a.ux[o] = ku[i][k];
                    if (a.jm) a.jm[o] = km[i][k];
                }
        if (write && cl) cluster_wait_acquire();
    }
}

// MAXT threads at most, 128 registers (65536 / (MAXT x MINB)): two blocks of
// 256 or four of 128 can share an SM where shared memory allows
template <typename T, int NF, int MAXT>
__global__ void __launch_bounds__(MAXT, 512 / MAXT) ml_plane_kernel(const MlPlaneArgs<T> a) {
    ml_plane_body<T, NF>(a);
}

template <typename T, int NF>
inline size_t ml_plane_smem_t(int rows, int nx, int rpb) {
    return ml_plane_smem_bytes(sizeof(T) == 8 ? 0 : 1, NF, rows, nx, rpb);
}

// launch (a non-null) or occupancy query (a null: *n = clusters, or blocks
// per SM for one band, the GPU holds at once)
template <typename T, int NF, int MAXT>
static cudaError_t ml_plane_go(const MlPlaneArgs<T> *a, int bands, int rows, int nx, int rpb,
                               int nfreq, int threads, cudaStream_t st, int *n) {
    cudaError_t e = cudaFuncSetAttribute(ml_plane_kernel<T, NF, MAXT>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kMlPlaneMaxSmem);
    if (e == cudaSuccess && bands > kPortableBands)
        e = cudaFuncSetAttribute(ml_plane_kernel<T, NF, MAXT>,
                                 cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(bands, (nfreq + NF - 1) / NF, 2 * (12 / rpb));
    cfg.blockDim = dim3(threads, 1, 1);
    cfg.dynamicSmemBytes = ml_plane_smem_t<T, NF>(rows, nx, rpb);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = bands;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = bands > 1 ? 1 : 0;
    if (a) return cudaLaunchKernelEx(&cfg, ml_plane_kernel<T, NF, MAXT>, *a);
    if (bands == 1)
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            n, ml_plane_kernel<T, NF, MAXT>, threads, cfg.dynamicSmemBytes);
    return cudaOccupancyMaxActiveClusters(n, ml_plane_kernel<T, NF, MAXT>, &cfg);
}

template <typename T>
static cudaError_t ml_plane_dispatch(const MlPlaneArgs<T> *a, int nf_block, int bands, int rows,
                                     int nx, int rpb, int nfreq, int threads, cudaStream_t st,
                                     int *n) {
    if (threads < 32 || threads > 512 || threads % 32 || rpb < 1 || 12 % rpb)
        return cudaErrorInvalidValue;
    auto go = [&](auto nf_tag) -> cudaError_t {
        constexpr int NF = decltype(nf_tag)::value;
        if constexpr (sizeof(T) == 8 && NF > 1) {
            // FP64 with more than one frequency per block spills at 128 registers
            return cudaErrorInvalidValue;
        } else {
            if (threads <= 128)
                return ml_plane_go<T, NF, 128>(a, bands, rows, nx, rpb, nfreq, threads, st, n);
            if (threads <= 256)
                return ml_plane_go<T, NF, 256>(a, bands, rows, nx, rpb, nfreq, threads, st, n);
            return ml_plane_go<T, NF, 512>(a, bands, rows, nx, rpb, nfreq, threads, st, n);
        }
    };
    switch (nf_block) {
        case 1: return go(std::integral_constant<int, 1>{});
        case 2: return go(std::integral_constant<int, 2>{});
        case 4: return go(std::integral_constant<int, 4>{});
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace mg3d
