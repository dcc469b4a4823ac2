// Shifted-plane sweep of the two-level atom's variants: partial redistribution
// and moving atmospheres (linear upwind interpolation).
//
// The layout of plane_sweep.cuh: every finished plane is stored shifted by the
// offset of the step that reads it, so a node finds its upwind corners in its
// own block, two neighbouring rows at a time, and the FP64 weights are formed in
// integer arithmetic (fixed_weights.cuh).  What differs is that a slot carries a
// second channel beside its intensity:
//   partial redistribution: chi0 is common to the slots, a slot's channel is its
//     source function rho_f S.  The atmosphere is static, so a slot stands for a
//     mirror pair of frequencies, solved once (R is symmetric in x, so rho and
//     the intensity are even in x up to rounding); the new mean intensity gets it
//     in both frequencies' places.
//   moving atmosphere: S is common, a slot (one frequency: the flow breaks the
//     mirror symmetry) carries its Doppler-shifted opacity chi0 phi(x_f - u_r).
// Stored vectors: vector 0 the common channel, then one slot (I, Q) per vector
// in FP64 and two in FP32; the loop over vectors is not unrolled, so one
// instance serves every slot count.
//
// Bounds (GB300, one sweep): the band sweep these variants shared before read its
// corners through generic addresses of peer blocks, evaluated every frequency's
// weights (FP64: 32 FP64 operations a frequency) and interpolated one row at a
// time.  PRD FP64 32x32x65, 17 frequencies: 2.19 -> 0.50 ms, FP64 pipe; moving FP32
// 48x48x97, 17 frequencies: 0.97 -> 0.50 ms, issue slots and the plane step's chain.
#pragma once

#include "plane_sweep.cuh"

namespace mg3d {

// Body for ray blockIdx.z and slot group blockIdx.y.  R: rows of a thread's
// item; MODE: kSweepPrd or kSweepMoving.
template <typename T, int R, int MODE>
__device__ __forceinline__ void plane_var_body(const PlaneVarArgs<T> &a) {
    using namespace plane;
    constexpr bool F64 = sizeof(T) == 8;
    constexpr bool PRD = MODE == kSweepPrd;
    constexpr int VW = vec_width<T>();
    constexpr int SPV = VW / 2;          // slots per vector
    constexpr int NA = PRD ? 1 : 4;      // fields copied ahead

    const int r = blockIdx.z, g = blockIdx.y;
    const int nb = a.bands;
    const bool cl = nb > 1;
    const int rank = (int)cluster_rank();
    const int nx = a.nx, ny = a.ny, nz = a.nz, rows = a.rows;
    const int y0 = rank * rows;
    const int myrows = min(rows, ny - y0);
    const int lastrows = ny - (nb - 1) * rows;
    const int s0 = g * a.np;                              // first slot of the group
    const int nslot = min(a.np, a.nslots - s0);
    const int nv = 1 + (a.np + SPV - 1) / SPV;            // vectors of a frame
    const int nv_used = 1 + (nslot + SPV - 1) / SPV;
    const unsigned pitch = (unsigned)nx * 16;
    const unsigned vs = (unsigned)(rows + 1) * pitch;
    const unsigned frame = (unsigned)nv * vs;
    const int nplane = nx * ny;
    const int nvox = nplane * nz;
    const bool up = (a.up_mask >> r) & 1u;
    const long slot = (long)r * a.ngroups + g;
    T *__restrict__ pj = a.pj + slot * nvox;
    T *__restrict__ pu = a.pu + slot * nvox;
    const T wray = T(1.0 / kRays);
    // a block's shared memory may be addressed by its cluster once the block runs:
    // arrive here, wait before the first store into another block
    if (cl) cluster_arrive_relaxed();

    extern __shared__ __align__(16) unsigned char smem_raw[];
    const unsigned buf_addr = smem_addr(smem_raw);
    RowDest *dest = reinterpret_cast<RowDest *>(smem_raw + 2 * (size_t)frame);   // [2][rows]
    // the node fields two steps ahead: [3][NA][rows * nx]
    T *ahead = reinterpret_cast<T *>(smem_raw + 2 * (size_t)frame +
                                     2 * rows * sizeof(RowDest));
    const int chunks = a.chunks;
    T *red = ahead + (a.ahead ? 3 * NA * rows * nx : 0);   // [2][chunks][rows * nx][2]
    __shared__ fx::u64 fx_tab[F64 ? 2 * fx::kTab : 1];
    __shared__ __align__(16) PlaneLerp<T> step_ring[4];
    const fx::Tables ft{fx_tab, fx_tab + fx::kTab};
    if (F64)
        for (int i = threadIdx.x; i < 2 * fx::kTab; i += blockDim.x) fx_tab[i] = a.fx_tab[i];

    const int nth = blockDim.x;
    const int items = (myrows + R - 1) / R * nx;
    const int chunk = chunks > 1 ? (int)threadIdx.x / a.ipad : 0;
    const int q0 = threadIdx.x - chunk * a.ipad;
    const int qend = chunk < chunks ? items : 0;
    const int v_begin = 1 + (nv_used - 1) * chunk / chunks;
    const int v_end = 1 + (nv_used - 1) * (chunk + 1) / chunks;
    auto item_at = [&](int q, int &x, int &yl0, int &nr) {
        const int gy = band_of(q, a.xmagic);
        x = q - gy * nx;
        yl0 = gy * R;
        nr = min(R, myrows - yl0);
    };
    auto plane_of = [&](int t) { return (up ? t : nz - 1 - t) * nplane + y0 * nx; };
    // Jeff and U of the plane of step t from the chunks' sums, in chunk order
    auto flush_sums = [&](int t) {
        const int kp = plane_of(t);
        const T *src = red + (t & 1) * 2 * chunks * rows * nx;
        for (int o = threadIdx.x; o < myrows * nx; o += nth) {
            T j = src[2 * o], u = src[2 * o + 1];
            for (int c = 1; c < chunks; ++c) {
                j += src[2 * (c * rows * nx + o)];
                u += src[2 * (c * rows * nx + o) + 1];
            }
            pj[kp + o] = j;
            pu[kp + o] = u;
        }
    };
    // field i of the nodes: chi0; moving: also S, the projected velocity and the
    // profile normalisation of the ray
    auto field = [&](int i) {
        return i == 0 ? a.chi0
                      : i == 1 ? a.S : (i == 2 ? a.uproj : a.vnorm) + (long)r * nvox;
    };
    // The constants of step t, three steps ahead: the row table of step t + 1 is
    // made during step t, when all copies but the latest group have landed.
    auto fetch_step = [&](int t) {
        constexpr int NC = sizeof(PlaneLerp<T>) / 16;
        if (threadIdx.x < NC)
            cp_async16(reinterpret_cast<unsigned char *>(&step_ring[t & 3]) + 16 * threadIdx.x,
                       reinterpret_cast<const unsigned char *>(&a.steps[(long)r * nz + t]) +
                           16 * threadIdx.x);
    };
    auto prefetch = [&](int t, int part) {
        if (t + 1 < nz) fetch_step(t + 1);
        if (a.ahead) {
            const int kp = plane_of(t);
            T *dst = ahead + part * NA * rows * nx;
            for (int o = threadIdx.x; o < myrows * nx; o += nth)
#pragma unroll
                for (int i = 0; i < NA; ++i) cp_async(dst + i * rows * nx + o, field(i) + kp + o);
        }
        cp_async_commit();
    };
    auto local = [&](int i, int t, int part, int o) {
        return a.ahead ? ahead[(part * NA + i) * rows * nx + o] : field(i)[plane_of(t) + o];
    };
    // where the band's rows go at the end of step t (row shift sy)
    auto fill_dest = [&](int t, int sy) {
        for (int yl = threadIdx.x; yl < myrows; yl += nth) {
            int ys = y0 + yl - sy;
            ys += ys < 0 ? ny : 0;
            const int ob = cl ? band_of(ys, a.rmagic) : 0;
            const int lr = ys - ob * rows;
            const int hb = ob == 0 ? nb - 1 : ob - 1;   // the band whose halo row is ys
            RowDest d;
            d.base = cluster_addr(buf_addr, (unsigned)ob) + (t & 1) * frame + (unsigned)lr * pitch;
            d.halo = lr != 0 ? kNoHalo
                             : cluster_addr(buf_addr, (unsigned)hb) + (t & 1) * frame +
                                   (unsigned)(hb == nb - 1 ? lastrows : rows) * pitch;
            dest[(t & 1) * rows + yl] = d;
        }
    };
    auto put = [&](const RowDest &d, unsigned xs, int v, const T *cv) {
        st16(d.base + xs + v * vs, cv);
        if (d.halo != kNoHalo) st16(d.halo + xs + v * vs, cv);
    };
    auto shifted = [&](int x, int sx) {
        const int xs = x - sx;
        return (unsigned)(xs < 0 ? xs + nx : xs) * 16u;
    };
    auto exp_neg_of = [&](T x) {
        if constexpr (F64) return fx::exp_neg_fx(x, ft);
        else return __expf(-x);
    };
    // profile of frequency f at velocity u along the ray
    auto profile = [&](int f, T u) {
        const T d = a.xf[f] - u;
        return T(0.56418958354775628) * exp_neg_of(d * d);
    };
    // the mean intensity of slot p's frequencies gets I at node v
    auto store_j = [&](int p, int v, T I) {
        const int m = a.nf - 1 - p;
        T *j = a.jnu + (long)r * a.nf * nvox + v;
        j[(long)p * nvox] = wray * I;
        if (m != p) j[(long)m * nvox] = wray * I;
    };

    // ---- entering boundary plane: I prescribed, w0 = 0
    if (nz > 1) {
        fetch_step(1);
        prefetch(1, 1);
    }
    if (nz > 2) prefetch(2, 2);
    __syncthreads();   // fx_tab
    if (nz > 1) fill_dest(0, a.steps[(long)r * nz].sy);
    __syncthreads();
    if (cl) cluster_wait();   // every block of the cluster has started
    {
        const int k0 = plane_of(0);
        const int sx = a.steps[(long)r * nz].sx;
        for (int o = threadIdx.x; o < myrows * nx; o += nth) {
            const int yl = band_of(o, a.xmagic), x = o - yl * nx, v = k0 + o;
            const T Ib = up ? a.bbot[y0 * nx + o] : T(0);
            const T c0 = a.chi0[v];
            const T u = PRD ? T(0) : field(2)[v], nrm = PRD ? T(0) : field(3)[v];
            const RowDest d = dest[yl];
            const unsigned xs = shifted(x, sx);
            T cv[VW];
#pragma unroll
            for (int e = 0; e < VW; ++e) cv[e] = T(0);
            cv[0] = PRD ? c0 : a.S[v];
            if (nz > 1) put(d, xs, 0, cv);
            T wsum = 0;
            for (int vv = 1; vv < nv_used; ++vv) {
#pragma unroll
                for (int e = 0; e < SPV; ++e) {
                    const int p = (vv - 1) * SPV + e;
                    T q = 0;
                    if (p < nslot) {
                        if constexpr (PRD) {
                            q = a.rhoS[(long)(s0 + p) * nvox + v];
                            wsum += a.slots[s0 + p].w;
                            store_j(s0 + p, v, Ib);
                        } else {
                            const T prof = profile(s0 + p, u);
                            q = c0 * prof;
                            wsum += a.wq[s0 + p] * prof * nrm;
                        }
                    }
                    cv[2 * e] = Ib;
                    cv[2 * e + 1] = q;
                }
                if (nz > 1) put(d, xs, vv, cv);
            }
            pj[v] = Ib * wsum;
            pu[v] = wsum;
        }
    }
    cp_async_wait();
    if (cl) cluster_barrier();
    else __syncthreads();

    int part = 1;   // t mod 3
    if (nz > 2) {
        fill_dest(1, step_ring[1].sy);
        __syncthreads();
    }
    for (int t = 1; t < nz; ++t) {
        const int kp = plane_of(t);
        const unsigned prev = buf_addr + ((t - 1) & 1) * frame;
        const PlaneLerp<T> sp = step_ring[t & 3];
        const bool write = t + 1 < nz;
        if (t + 2 < nz) {
            prefetch(t + 2, part == 0 ? 2 : part - 1);
            fill_dest(t + 1, step_ring[(t + 1) & 3].sy);
        }
        if (chunks > 1 && t > 1) flush_sums(t - 1);
        bool down = false;   // FP64: the nearer row is the higher one
        fx::u64 cm = 0;      // FP64: c = (cm, ce)
        int ce = 0;
        if constexpr (F64) {
            down = sp.near & 2;
            fx::unpack(sp.c, &cm, &ce);
        }
        // sums of the thread's first item, stored after the barrier's first half
        T kj[R], ku[R];
        int ko[R], nk = 0;
        for (int q = q0; q < qend; q += nth) {
            int x, yl0, nr;
            item_at(q, x, yl0, nr);
            const unsigned xb = (unsigned)x * 16, xb1 = x + 1 == nx ? 0u : xb + 16;
            const unsigned xn = (sp.near & 1) ? xb1 : xb, xf = (sp.near & 1) ? xb : xb1;
            const unsigned row0 = prev + (unsigned)(down ? yl0 + nr : yl0) * pitch;
            const unsigned dpitch = down ? 0u - pitch : pitch;
            auto row_h = [&](int v, int k, T *h) {
                const unsigned p = row0 + k * dpitch + v * vs;
                T A[VW], B[VW];
                lds16(p + xn, A);
                lds16(p + xf, B);
#pragma unroll
                for (int e = 0; e < VW; ++e) h[e] = fma(sp.rx, B[e], A[e]);
            };
            // vector v at the item's nodes, in the walk's order (FP64: without c)
            auto upwind = [&](int v, T (*o)[VW]) {
                T h0[VW], h1[VW];
                row_h(v, 0, h0);
#pragma unroll
                for (int j = 0; j < R; ++j)
                    if (j < nr) {
                        row_h(v, j + 1, h1);
#pragma unroll
                        for (int e = 0; e < VW; ++e) {
                            if constexpr (F64) o[j][e] = fma(sp.ry, h1[e], h0[e]);
                            else o[j][e] = fma(sp.wy1, h1[e], sp.wy0 * h0[e]);
                            h0[e] = h1[e];
                        }
                    }
            };
            T V0[R][VW];
            upwind(0, V0);
            const unsigned xs = shifted(x, sp.sx);
            RowDest dst[R];
            int node[R];
            T chi_loc[R], S_loc[R], S_up[R], u[R], nrm[R], dtau0[R], cj[R], cu[R];
            fx::u64 dm[R], dr[R];
            int de[R];
#pragma unroll
            for (int j = 0; j < R; ++j) {
                if (j >= nr) continue;
                const int yl = down ? yl0 + nr - 1 - j : yl0 + j, o = yl * nx + x;
                node[j] = kp + o;
                dst[j] = dest[(t & 1) * rows + yl];
                chi_loc[j] = local(0, t, part, o);
                cj[j] = cu[j] = T(0);
                T common;
                if constexpr (PRD) {
                    if constexpr (F64) {
                        dtau0[j] = fma(sp.c, V0[j][0], chi_loc[j]) * sp.half_s;
                        fx::unpack(dtau0[j], &dm[j], &de[j]);
                        dr[j] = fx::recip(dm[j]);
                    } else {
                        dtau0[j] = (V0[j][0] + chi_loc[j]) * sp.half_s;
                    }
                    common = chi_loc[j];
                } else {
                    S_loc[j] = local(1, t, part, o);
                    u[j] = local(2, t, part, o);
                    nrm[j] = local(3, t, part, o);
                    S_up[j] = V0[j][0];
                    if constexpr (F64) S_up[j] *= sp.c;
                    common = S_loc[j];
                }
                if (write && chunk == 0) {
                    T cv[VW];
#pragma unroll
                    for (int e = 0; e < VW; ++e) cv[e] = e == 0 ? common : T(0);
                    put(dst[j], xs, 0, cv);
                }
            }
#pragma unroll 1
            for (int v = v_begin; v < v_end; ++v) {
                T V[R][VW];
                upwind(v, V);
#pragma unroll
                for (int j = 0; j < R; ++j) {
                    if (j >= nr) continue;
#pragma unroll
                    for (int e = 0; e < SPV; ++e) {
                        const int p = (v - 1) * SPV + e;
                        if (p >= nslot) {
                            V[j][2 * e] = V[j][2 * e + 1] = T(0);
                            continue;
                        }
                        const int f = s0 + p;
                        T Q = V[j][2 * e + 1];
                        // weights; FP64: cex = c e^-x, as the intensity lacks c
                        T cex, w0, wup, uu;
                        T Q_loc, rho = T(1), w;
                        if constexpr (PRD) {
                            Q_loc = a.rhoS[(long)f * nvox + node[j]];
                            rho = a.rho[(long)f * nvox + node[j]];
                            w = a.slots[f].w;
                        } else {
                            const T prof = profile(f, u[j]);
                            Q_loc = chi_loc[j] * prof;
                            w = a.wq[f] * prof * nrm[j];
                        }
                        if constexpr (F64) {
                            bool ok;
                            T xt;
                            fx::u64 m = 0, Y = 0, rc = 0;
                            int em = 0, ey = 0, er = 0;
                            if constexpr (PRD) {
                                const PlaneSlot<T> &sl = a.slots[f];
                                xt = dtau0[j] * sl.phi;
                                ok = fx::in_range(dtau0[j]) && sl.fx;
                                m = fx::mulhi(dm[j], sl.pm);
                                em = de[j] + sl.pe;
                                Y = fx::mulhi(dm[j], sl.ym);
                                ey = de[j] + sl.ye;
                                rc = fx::mulhi(dr[j], sl.im);
                                er = 1 - de[j] + sl.ie;
                            } else {
                                xt = fma(sp.c, Q, Q_loc) * sp.half_s;
                                ok = fx::in_range(xt);
                                fx::unpack(xt, &m, &em);
                                Y = fx::mulhi(m, fx::kLog2e);
                                ey = em + 1;
                                rc = fx::recip(m);
                                er = 1 - em;
                            }
                            if (ok) {
                                fx::Weights wt;
                                if (em <= fx::kThinExp) {
                                    wt = fx::thin(m, em);
                                    uu = fx::pack(wt.u, 0);
                                } else {
                                    wt = fx::closed(Y, ey, rc, er, ft);
                                    uu = fx::pack32(wt.um, wt.ue);
                                }
                                cex = wt.E ? fx::pack62(fx::mulhi(wt.E, cm), ce - wt.n) : 0.0;
                                w0 = wt.w0;
                                wup = wt.wup;
                            } else {
                                const Weights64 wt = weights64(xt);
                                cex = sp.c * wt.ex;
                                w0 = wt.w0;
                                wup = wt.wup;
                                uu = wt.u;
                            }
                        } else {
                            T xt;
                            if constexpr (PRD) xt = dtau0[j] * a.slots[f].phi;
                            else xt = (Q + Q_loc) * sp.half_s;
                            Weights32::eval(xt, cex, w0, wup, uu);
                        }
                        T I;
                        if constexpr (PRD) {
                            if constexpr (F64) Q *= sp.c;
                            const T ps = fma(V[j][2 * e], cex, wup * Q);   // I - w0 S
                            I = fma(w0, Q_loc, ps);
                            cj[j] = fma(w, ps, cj[j]);
                            cu[j] = fma(w, fma(-w0, rho, T(1)), cu[j]);
                            store_j(f, node[j], I);
                        } else {
                            const T ps = fma(V[j][2 * e], cex, wup * S_up[j]);
                            I = fma(w0, S_loc[j], ps);
                            cj[j] = fma(w, ps, cj[j]);
                            cu[j] = fma(w, uu, cu[j]);
                        }
                        V[j][2 * e] = I;
                        V[j][2 * e + 1] = Q_loc;
                    }
                    if (write) put(dst[j], xs, v, V[j]);
                }
            }
#pragma unroll
            for (int j = 0; j < R; ++j) {
                if (j >= nr) continue;
                if (chunks > 1) {
                    T *dr2 = red + 2 * (((t & 1) * chunks + chunk) * rows * nx + node[j] - kp);
                    dr2[0] = cj[j];
                    dr2[1] = cu[j];
                } else if (q == q0) {
                    kj[j] = cj[j];
                    ku[j] = cu[j];
                    ko[j] = node[j];
                    nk = j + 1;
                } else {
                    pj[node[j]] = cj[j];
                    pu[node[j]] = cu[j];
                }
            }
        }
        // before the barrier, since any thread may read the next plane's values:
        // the copies for step t + 1 are done
        if (t + 2 < nz) cp_async_wait_but_last();
        else cp_async_wait();
        if (write) {
            if (cl) cluster_arrive();
            else __syncthreads();
        }
#pragma unroll
        for (int j = 0; j < R; ++j)
            if (j < nk) {
                pj[ko[j]] = kj[j];
                pu[ko[j]] = ku[j];
            }
        if (write && cl) cluster_wait_acquire();
        part = part == 2 ? 0 : part + 1;
    }
    if (chunks > 1 && nz > 1) {
        __syncthreads();
        flush_sums(nz - 1);
    }
}

template <typename T, int MAXT, int R, int MODE>
__global__ void __launch_bounds__(MAXT) plane_var_kernel(const PlaneVarArgs<T> a) {
    plane_var_body<T, R, MODE>(a);
}

template <typename T, int MAXT, int R, int MODE>
static cudaError_t plane_var_go(const PlaneVarArgs<T> *a, const SweepShape &s,
                                const PlaneLayout &lay, cudaStream_t st, int *n) {
    cudaError_t e = cudaFuncSetAttribute(plane_var_kernel<T, MAXT, R, MODE>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)plane_smem_max(sizeof(T) == 8));
    if (e == cudaSuccess && s.bands > kPortableBands)
        e = cudaFuncSetAttribute(plane_var_kernel<T, MAXT, R, MODE>,
                                 cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[1];
    cfg.gridDim = dim3(s.bands, s.ngroups, kRays);
    cfg.blockDim = dim3(s.threads, 1, 1);
    cfg.dynamicSmemBytes = lay.smem;
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = s.bands;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = s.bands > 1 ? 1 : 0;   // one band: a plain launch
    if (a) {
        PlaneVarArgs<T> b = *a;
        b.ahead = lay.ahead;
        b.chunks = lay.chunks;
        b.ipad = lay.ipad;
        return cudaLaunchKernelEx(&cfg, plane_var_kernel<T, MAXT, R, MODE>, b);
    }
    if (s.bands == 1)
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            n, plane_var_kernel<T, MAXT, R, MODE>, s.threads, cfg.dynamicSmemBytes);
    return cudaOccupancyMaxActiveClusters(n, plane_var_kernel<T, MAXT, R, MODE>, &cfg);
}

// launch (a non-null) or occupancy query (a null)
template <typename T>
static cudaError_t plane_var_dispatch(const PlaneVarArgs<T> *a, const SweepShape &s, int nx,
                                      cudaStream_t st, int *n) {
    const PlaneLayout lay =
        plane_var_layout(sizeof(T) == 8 ? 0 : 1, s.prd, s.np, s.rows, nx, s.threads);
    auto go = [&](auto max_tag, auto r_tag) {
        constexpr int MAXT = decltype(max_tag)::value, R = decltype(r_tag)::value;
        return s.prd ? plane_var_go<T, MAXT, R, kSweepPrd>(a, s, lay, st, n)
                     : plane_var_go<T, MAXT, R, kSweepMoving>(a, s, lay, st, n);
    };
    using M256 = std::integral_constant<int, 256>;
    using M512 = std::integral_constant<int, 512>;
    using R1 = std::integral_constant<int, 1>;
    using R2 = std::integral_constant<int, 2>;
    if (s.threads <= 256) return lay.item_rows == 2 ? go(M256{}, R2{}) : go(M256{}, R1{});
    return lay.item_rows == 2 ? go(M512{}, R2{}) : go(M512{}, R1{});
}

}  // namespace mg3d
