// Formal solution with shifted plane storage: the linear short-characteristics
// sweep of a static atmosphere in complete redistribution (Sec. 3), laid out
// so that every node finds its upwind corners at fixed offsets from itself.
//
// The upwind crossing of a (ray, step) lies at the same horizontal offset
// (ix0 + tx, iy0 + ty) cells from every node of the plane (periodic in x and
// y, Sec. 4.2).  So when plane k is finished, each node's values are stored
// already shifted by the offset of the step that will read them: node (x, y)
// goes to position ((x - ix0') mod nx, (y - iy0') mod ny) of the stored frame,
// where (ix0', iy0') belongs to the next step.  The next step then reads the
// four corners of node (x, y) at positions (x, y), (x + 1, y), (x, y + 1) and
// (x + 1, y + 1) of that frame: the same four offsets for every node, with no
// wrap, band or peer arithmetic on the reading side.
//
// One thread-block cluster per (ray, group of frequencies): the cluster's
// blocks split the stored frame in bands of rows.  A block owns rows
// [rank*rows, rank*rows + myrows) of the frame, plus one halo row (the first
// row of the next band, or row 0 after the last band), so all four corners of
// its nodes are in its own shared memory (column nx is column 0).  Writes carry
// the shift instead: a node's values go to the block that owns its stored row
// (distributed shared memory, st.shared::cluster) and, for the first row of a
// band, also to the halo row that duplicates it; the addresses are tabulated
// a row and step.  Two planes are kept (read k-1, write k); one cluster barrier
// per plane orders the writes of a step before the reads of
// the next and the reads of a step before the overwrite two steps later.
//
// A second completion scheme (stage 3) replaces the barrier's release fence
// with transaction-counted stores: values bound for another block go by
// st.async, which counts its bytes on an mbarrier in the receiving block, and
// each block waits on its own mbarrier for the bytes its plane receives from
// other blocks (stores within a block are ordered by __syncthreads).  The
// reads of a step must still end, cluster-wide, before the plane they came
// from is overwritten two steps later; a relaxed cluster barrier (no fence)
// arrives at the end of a step and waits just before the first store of the
// next.  Every wait on an mbarrier is bounded in time: past the bound the
// kernel records MG3D_STATUS_WAIT in the status word, stops waiting and runs
// to the end, so the host reports an error instead of a hung launch.
//
// Slots: for the two-level atom in complete redistribution phi(x) = phi(-x)
// and S does not depend on frequency, so in a static atmosphere the transfer
// equation, its boundary values and its coefficients are the same at x and -x
// and so is the intensity, bit for bit.  A slot stands for such a mirror pair
// (or for the line centre): its intensity is solved once and enters the sums
// with the weight of both frequencies.
//
// Channels: per stored node chi0 and S of the node's plane (their upwind values
// come from the same corners), then the intensities of the group's slots,
// padded to whole 16-byte vectors.  Vector v of all nodes of a frame is
// contiguous, so the 16-byte loads and stores of a warp's consecutive nodes do
// not conflict in banks and a frame holds no padding between nodes.
//
// Interpolation.  The bilinear weights are the same for all nodes of a step, so
// the two directions are taken one after the other: H = A + rx B along x, scaled
// by the larger weight, and in FP64 V = H + ry H' along y the same way, upwind
// value = c V (0 <= rx, ry <= 1, 1/4 <= c <= 1); FP32 takes V = wy0 H + wy1 H'.
// A thread takes two nodes of neighbouring rows, which share the H of the row
// between them: 2.5 fused multiply-adds and 3 corner loads per channel and node
// instead of 4 and 4.
//
// What bounds it, and what it measured (GB300, one sweep, 9 frequencies; before:
// the pairs solved twice, one row per thread, FP64 weights in FP64):
//   FP64 64x64x129: 45 FP64 operations per node and ray (before 154) on a pipe
//     that issues one warp instruction in 18 clocks; 5.01 -> 1.79 ms.  Small
//     FP64 planes are the latency of one warp's slots, which the chunks below
//     run side by side: 16x16x33 220 -> 104 us.
//   FP32: issue slots and the wait for the slowest block of a plane; 64x64x129
//     344 -> 282 us, 128x128x129 1527 -> 825 us (980 with every node's destination
//     computed from its row instead of read from the row table).
//
// Per node the block accumulates, over its slots,
//   Jeff = sum w phi (I - w0 S)   and   U = sum w phi (1 - w0)
// (Sec. 2.1, the diagonal operator of MALI) into the partial slot of its
// (ray, group); the rate kernel adds the slots in a fixed order.
//
// chi0 and S of the block's own nodes on the next plane are copied to shared
// memory two steps ahead (cp.async), the step's constants three, so their latency
// overlaps the steps before; where the shape
// leaves no room for that they are read from global memory where used.
#pragma once

#include <cooperative_groups.h>

#include <type_traits>

#include "fixed_weights.cuh"
#include "mg3d_internal.h"
#include "sc_step.cuh"

namespace mg3d {

namespace plane {

template <typename T>
__host__ __device__ constexpr int vec_width() { return 16 / (int)sizeof(T); }
// 16-byte vectors per node: chi0, S and NP intensities
template <typename T, int NP>
__host__ __device__ constexpr int vectors() {
    return (NP + 2 + vec_width<T>() - 1) / vec_width<T>();
}

// where a row of the band is stored: in the block that owns it, and in the halo
// row of the block before (or kNoHalo)
struct RowDest {
    unsigned base, halo;
};
constexpr unsigned kNoHalo = ~0u;
// the same with the mbarriers of the async scheme (kNoBar: a row of this block)
constexpr unsigned kNoBar = ~0u;
struct __align__(16) RowTarget {
    unsigned base, halo, bar, hbar;
};

__device__ __forceinline__ unsigned smem_addr(const void *p) {
    return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ unsigned cluster_addr(unsigned a, unsigned rank) {
    unsigned r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// 16-byte store of (v[0..VW-1]) at a shared::cluster address (this block's
// or another block's shared memory; a launch without clusters is a cluster of
// one block).  No memory clobber: the
// stores go to the plane being written, which no thread reads before the
// barrier (whose asm carries the clobber) that ends the step.
__device__ __forceinline__ void st16(unsigned a, const float *v) {
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v[0]),
                 "f"(v[1]), "f"(v[2]), "f"(v[3]));
}
__device__ __forceinline__ void st16(unsigned a, const double *v) {
    asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(a), "d"(v[0]), "d"(v[1]));
}
// one 16-byte vector at an address of this block's shared memory
__device__ __forceinline__ void lds16(unsigned a, float *o) {
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(o[0]), "=f"(o[1]), "=f"(o[2]), "=f"(o[3])
                 : "r"(a));
}
__device__ __forceinline__ void lds16(unsigned a, double *o) {
    asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(o[0]), "=d"(o[1]) : "r"(a));
}
// one 16-byte vector of shared memory into registers
__device__ __forceinline__ void ld16(const float *p, float *o) {
    const float4 v = *reinterpret_cast<const float4 *>(p);
    o[0] = v.x;
    o[1] = v.y;
    o[2] = v.z;
    o[3] = v.w;
}
__device__ __forceinline__ void ld16(const double *p, double *o) {
    const double2 v = *reinterpret_cast<const double2 *>(p);
    o[0] = v.x;
    o[1] = v.y;
}
// The barrier in two halves: the release waits until the thread's earlier
// stores are performed, so stores to global memory that no other block reads
// go between the halves.
__device__ __forceinline__ void cluster_arrive() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait_acquire() {
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_barrier() {
    asm volatile(
        "barrier.cluster.arrive.release.aligned;\n\t"
        "barrier.cluster.wait.acquire.aligned;" ::
            : "memory");
}

// Split phases of a cluster barrier without memory ordering (the async
// scheme orders its data through mbarriers and __syncthreads)
__device__ __forceinline__ void cluster_arrive_relaxed() {
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
}
// 16-byte store into another block's shared memory that completes 16 bytes of
// the transaction count of the mbarrier at `bar` (a shared::cluster address
// in the same block)
__device__ __forceinline__ void st16_async(unsigned a, const float *v, unsigned bar) {
    asm volatile(
        "st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], "
        "{%1, %2, %3, %4}, [%5];" ::"r"(a),
        "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void st16_async(unsigned a, const double *v, unsigned bar) {
    asm volatile(
        "st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f64 [%0], "
        "{%1, %2}, [%3];" ::"r"(a),
        "d"(v[0]), "d"(v[1]), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void mbar_init(unsigned bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_init_fence() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
// the one arrival of a phase, with the bytes the phase is to receive
__device__ __forceinline__ void mbar_arrive_expect(unsigned bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool mbar_test(unsigned bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// Waits until the phase of parity `parity` of the mbarrier completes, at most
// kWaitLimitNs; false when the bound ran out.
constexpr unsigned long long kWaitLimitNs = 2000000000ull;
static __device__ __noinline__ bool mbar_wait_bounded(unsigned bar, unsigned parity) {
    if (mbar_test(bar, parity)) return true;
    const unsigned long long t0 = global_ns();
    for (unsigned it = 1;; ++it) {
        if (mbar_test(bar, parity)) return true;
        if ((it & 63u) == 0 && global_ns() - t0 > kWaitLimitNs) return false;
    }
}

// 4- or 8-byte copy from global to this block's shared memory
__device__ __forceinline__ void cp_async(float *dst, const float *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async(double *dst, const double *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_addr(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async_wait() {   // all of the thread's copies are done
    asm volatile("cp.async.wait_all;" ::: "memory");
}
__device__ __forceinline__ void cp_async_commit() {
    asm volatile("cp.async.commit_group;" ::: "memory");
}
__device__ __forceinline__ void cp_async_wait_but_last() {   // all but the last group
    asm volatile("cp.async.wait_group 1;" ::: "memory");
}

__device__ __forceinline__ float ex2_approx(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Short-characteristics weights of optical path x (>= 0) for the linear
// step I = I_up e^-x + w_up S_up + w0 S0:  u = (1 - e^-x)/x, w0 = 1 - u,
// w_up = u - e^-x.  Below a threshold the closed form cancels, and the
// Taylor series of w0 and w_up (FP32: w_up = x u - w0) replace it.
//   FP32: e^-x = 2^(-x log2 e) and 1/x by the hardware approximations (within
//   2 ulp, ample for the FP32 formal solution); series below x = 0.1.
//   FP64: 64-bit integer arithmetic (fixed_weights.cuh).
struct Weights32 {
    static __device__ __forceinline__ void series(float x, float &ex, float &w0, float &wup,
                                                  float &u) {
        // w0 + w_up = 1 - e^-x = x u
        w0 = x * (0.5f - x * (1.0f / 6.0f - x * (1.0f / 24.0f -
                                                 x * (1.0f / 120.0f - x * (1.0f / 720.0f)))));
        u = 1.0f - w0;
        wup = fmaf(x, u, -w0);
        ex = u - wup;
    }
    static __device__ __forceinline__ void closed(float x, float &ex, float &w0, float &wup,
                                                  float &u) {
        ex = ex2_approx(x * -1.44269504088896341f);
        const float ix = rcp_approx(x);
        u = fmaf(-ex, ix, ix);
        w0 = 1.0f - u;
        wup = u - ex;
    }
    static __device__ __forceinline__ void eval(float x, float &ex, float &w0, float &wup,
                                                float &u) {
        if (x < 0.1f) series(x, ex, w0, wup, u);
        else closed(x, ex, w0, wup, u);
    }
};

// FP64 weights for the arguments the integer weights (fixed_weights.cuh) leave
// out: optical paths that are zero, denormal, beyond 2^700, negative or NaN.  The
// series (below 1e-3, tested on the high word of x) as products with rounded
// reciprocals.
struct Weights64 {
    double ex, w0, wup, u;
};
static __device__ __noinline__ Weights64 weights64(double x) {
    Weights64 w;
    if (__double2hiint(x) < 0x3F50624D) {
        w.w0 = x * (0.5 - x * (1.0 / 6.0 - x * (1.0 / 24.0 - x * (1.0 / 120.0 - x * (1.0 / 720.0)))));
        w.wup = x * (0.5 - x * (1.0 / 3.0 - x * (1.0 / 8.0 - x * (1.0 / 30.0 - x * (1.0 / 144.0)))));
        w.u = 1.0 - w.w0;
        w.ex = w.u - w.wup;
    } else {
        const double ix = 1.0 / x;
        w.ex = exp(-x);
        w.u = fma(-w.ex, ix, ix);
        w.w0 = 1.0 - w.u;
        w.wup = w.u - w.ex;
    }
    return w;
}

}  // namespace plane

// The body of the kernel for ray blockIdx.z and frequency group blockIdx.y.
// R: rows of a thread's item.
template <typename T, int NP, int R, bool AS>
__device__ __forceinline__ void plane_sweep_body(const PlaneArgs<T> &a) {
    using namespace plane;
    constexpr int VW = vec_width<T>();
    constexpr int NV = vectors<T, NP>();
    constexpr bool F64 = sizeof(T) == 8;

    const int r = blockIdx.z, g = blockIdx.y;
    const int nb = a.bands;
    const bool cl = nb > 1;
    const bool as = AS && cl;               // the async completion scheme
    const int rank = (int)cluster_rank();   // 0 in a launch without clusters
    const int nx = a.nx, ny = a.ny, nz = a.nz, rows = a.rows;
    const int y0 = rank * rows;
    const int myrows = min(rows, ny - y0);
    const int lastrows = ny - (nb - 1) * rows;   // rows of the last band
    const unsigned pitch = (unsigned)nx * 16;            // one stored row of a vector, bytes
    const unsigned vs = (unsigned)(rows + 1) * pitch;    // one vector of a frame
    const unsigned frame = NV * vs;                      // one stored frame
    const int nplane = nx * ny;                  // the host keeps nvox below 2^31
    const bool up = (a.up_mask >> r) & 1u;
    const long slot = (long)r * a.ngroups + g;
    T *__restrict__ pj = a.pj + slot * (long)nplane * nz;
    T *__restrict__ pu = a.pu + slot * (long)nplane * nz;
    const PlaneSlot<T> *__restrict__ gs = a.slots + (long)g * NP;
    // a block's shared memory may be addressed by its cluster once the block runs:
    // arrive here, wait before the first store into another block
    if (cl && !as) cluster_arrive_relaxed();

    extern __shared__ __align__(16) unsigned char smem_raw[];
    const unsigned buf_addr = smem_addr(smem_raw);
    RowTarget *dest = reinterpret_cast<RowTarget *>(smem_raw + 2 * (size_t)frame);   // [2][rows]
    // chi0 and S of the band's nodes two steps ahead: [3][2][rows * nx]
    T *ahead = reinterpret_cast<T *>(smem_raw + 2 * (size_t)frame + 2 * rows * sizeof(RowTarget));
    // 16-byte copies: every band of every plane starts on such a boundary
    constexpr int CW = 16 / (int)sizeof(T);
    const bool wide = nplane % CW == 0 && (rows * nx) % CW == 0 &&
                      ((reinterpret_cast<size_t>(a.chi0) | reinterpret_cast<size_t>(a.S)) & 15) == 0;
    __shared__ fx::u64 fx_tab[F64 ? 2 * fx::kTab : 1];   // tables of the integer weights
    __shared__ PlaneSlot<T> stab[NP];
    // step constants up to three steps ahead
    __shared__ __align__(16) PlaneLerp<T> step_ring[4];
    // async scheme: one mbarrier per plane buffer, one phase per filling
    __shared__ __align__(8) unsigned long long full_bar[2];
    const unsigned bar_addr = smem_addr(full_bar);
    if (as && threadIdx.x == 0) {
        mbar_init(bar_addr, 1);
        mbar_init(bar_addr + 8, 1);
        mbar_init_fence();
    }
    if (F64)
        for (int i = threadIdx.x; i < 2 * fx::kTab; i += blockDim.x) fx_tab[i] = a.fx_tab[i];
    for (int i = threadIdx.x; i < NP; i += blockDim.x) stab[i] = gs[i];
    __syncthreads();
    const int nslot = g == a.ngroups - 1 ? a.nslot_last : NP;
    T wsum = 0;
#pragma unroll
    for (int p = 0; p < NP; ++p) wsum += stab[p].w;

    // FP32 keeps the slot tables in registers, an inactive slot as one of weight
    // zero, and knows the dtau0 from which all slots take the closed form or
    // below which all take the series (0.1 over the smallest and largest phi).
    T r_phi[F64 ? 1 : NP], r_w[F64 ? 1 : NP], d_closed = 0, d_series = 0;
    if constexpr (!F64) {
        T lo = stab[0].phi, hi = stab[0].phi;
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            r_phi[p] = p < nslot ? stab[p].phi : stab[0].phi;
            r_w[p] = stab[p].w;
            lo = min(lo, r_phi[p]);
            hi = max(hi, r_phi[p]);
        }
        d_closed = T(0.1) / lo;
        d_series = T(0.1) / hi;
    }

    // A thread's item is column x of rows yl0 .. yl0 + nr - 1 of the band.  With
    // more than one chunk (small bands) `ipad` threads take the items of each
    // chunk of the slots, so that the slots of a node run side by side; their
    // sums meet in shared memory one step later.
    const int nth = blockDim.x;
    const int items = (myrows + R - 1) / R * nx;
    const int chunks = a.chunks;
    const int ipad = a.ipad;
    const int chunk = chunks > 1 ? (int)threadIdx.x / ipad : 0;
    const int q0 = threadIdx.x - chunk * ipad;
    const int qend = chunk < chunks ? items : 0;
    // vectors 1 .. NV-1 of the chunk (the first chunk also takes vector 0)
    const int v_begin = 1 + (NV - 1) * chunk / chunks;
    const int v_end = 1 + (NV - 1) * (chunk + 1) / chunks;
    T *red = ahead + (a.ahead ? 6 * rows * nx : 0);   // [2][chunks][rows * nx][2]
    auto item_at = [&](int q, int &x, int &yl0, int &nr) {
        const int gy = band_of(q, a.xmagic);
        x = q - gy * nx;
        yl0 = gy * R;
        nr = min(R, myrows - yl0);
    };
    // Jeff and U of the plane of step t from the chunks' sums, in chunk order
    auto flush_sums = [&](int t) {
        const int kp = (up ? t : nz - 1 - t) * nplane + y0 * nx;
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

    // Where the band's rows go in the frame stored at step t, whose reader's row
    // shift is sy: one entry a row and step, instead of the modulo, band and
    // peer arithmetic at every node.
    auto fill_dest = [&](int t, int sy) {
        const unsigned par = t & 1;
        for (int yl = threadIdx.x; yl < myrows; yl += nth) {
            int ys = y0 + yl - sy;
            ys += ys < 0 ? ny : 0;
            const int ob = cl ? band_of(ys, a.rmagic) : 0;
            const int lr = ys - ob * rows;
            const int hb = ob == 0 ? nb - 1 : ob - 1;   // the band whose halo row is ys
            RowTarget d;
            d.base = cluster_addr(buf_addr, (unsigned)ob) + par * frame + (unsigned)lr * pitch;
            d.halo = lr != 0 ? kNoHalo
                             : cluster_addr(buf_addr, (unsigned)hb) + par * frame +
                                   (unsigned)(hb == nb - 1 ? lastrows : rows) * pitch;
            d.bar = as && ob != rank ? cluster_addr(bar_addr + 8u * par, (unsigned)ob) : kNoBar;
            d.hbar = as && hb != rank ? cluster_addr(bar_addr + 8u * par, (unsigned)hb) : kNoBar;
            dest[par * rows + yl] = d;
        }
    };
    auto shifted = [&](int x, int sx) {   // byte offset of the stored column
        const int xs = x - sx;
        return (unsigned)(xs < 0 ? xs + nx : xs) * 16u;
    };
    // vectors v0 .. v0+N-1 of the node's channels; to another block in the async
    // scheme: st.async counted on that block's mbarrier of the buffer
    auto put = [&](auto n_tag, const RowTarget &d, unsigned xs, int v0, const T *cv) {
        constexpr int N = decltype(n_tag)::value;
        if (AS && d.bar != kNoBar) {
#pragma unroll
            for (int v = 0; v < N; ++v)
                st16_async(d.base + xs + (v0 + v) * vs, cv + v * VW, d.bar);
        } else {
#pragma unroll
            for (int v = 0; v < N; ++v) st16(d.base + xs + (v0 + v) * vs, cv + v * VW);
        }
        if (d.halo != kNoHalo) {
            if (AS && d.hbar != kNoBar) {
#pragma unroll
                for (int v = 0; v < N; ++v)
                    st16_async(d.halo + xs + (v0 + v) * vs, cv + v * VW, d.hbar);
            } else {
#pragma unroll
                for (int v = 0; v < N; ++v) st16(d.halo + xs + (v0 + v) * vs, cv + v * VW);
            }
        }
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
    using One = std::integral_constant<int, 1>;
    using All = std::integral_constant<int, NV>;

    // chi0 and S of step t's plane into part t mod 3 of the ring, and the
    // constants of step t + 1
    auto prefetch = [&](int t, int part) {
        if (t + 1 < nz) fetch_step(t + 1);
        if (a.ahead) {
            const int kp = (up ? t : nz - 1 - t) * nplane + y0 * nx;
            T *dst = ahead + part * 2 * rows * nx;
            if (wide) {
                for (int o = CW * threadIdx.x; o < myrows * nx; o += CW * nth) {
                    cp_async16(dst + o, a.chi0 + kp + o);
                    cp_async16(dst + rows * nx + o, a.S + kp + o);
                }
            } else {
                for (int o = threadIdx.x; o < myrows * nx; o += nth) {
                    cp_async(dst + o, a.chi0 + kp + o);
                    cp_async(dst + rows * nx + o, a.S + kp + o);
                }
            }
        }
        cp_async_commit();
    };
    // chi0 and S of node o of the band on the plane of step t, part t mod 3
    auto local = [&](int t, int part, int o, T &chi, T &S) {
        if (a.ahead) {
            const T *src = ahead + part * 2 * rows * nx;
            chi = src[o];
            S = src[rows * nx + o];
        } else {
            const int kp = (up ? t : nz - 1 - t) * nplane + y0 * nx;
            chi = a.chi0[kp + o];
            S = a.S[kp + o];
        }
    };

    // Async scheme: the bytes buffer `par` of this block receives from other
    // blocks when the plane is stored with row shift sy.  Stored row ys (a
    // row of the band, or the halo row: the next band's first row, row 0
    // after the last band) holds source row (ys + sy) mod ny, all of its nx
    // nodes, written by the block that owns that row.  Warp
    // 0 counts the rows with another owner; its lane 0 posts the phase's one
    // arrival with the byte count.
    auto expect_fill = [&](int sy, int par) {
        if (threadIdx.x >= 32) return;
        int cnt = 0;
        for (int j = threadIdx.x; j <= myrows; j += 32) {
            const int ys = j < myrows ? y0 + j : (rank == nb - 1 ? 0 : y0 + rows);
            int ysrc = ys + sy;
            ysrc -= ysrc >= ny ? ny : 0;
            cnt += band_of(ysrc, a.rmagic) != rank ? 1 : 0;
        }
        cnt = __reduce_add_sync(0xffffffffu, cnt);
        if (threadIdx.x == 0)
            mbar_arrive_expect(bar_addr + 8u * par, (unsigned)(cnt * nx * NV * 16));
    };
    bool waits_ok = true;   // false once a bounded wait ran out
    auto wait_fill = [&](int s) {   // buffer s & 1 holds the plane stored at step s
        if (waits_ok && !mbar_wait_bounded(bar_addr + 8u * (s & 1), (unsigned)((s >> 1) & 1))) {
            waits_ok = false;
            if (a.status) atomicOr(a.status, kPlaneStatusWait);
        }
    };
    if (as && nz > 1) {
        // every block's mbarriers are initialised before any store reaches them
        cluster_barrier();
        expect_fill(a.steps[(long)r * nz].sy, 0);
    }

    // ---- entering boundary plane: I prescribed (bottom: Planck at the local
    // temperature, top: zero), so w0 = 0 and 1 - w0 = 1
    if (nz > 1) {
        fetch_step(1);
        prefetch(1, 1);
    }
    if (nz > 2) prefetch(2, 2);
    if (nz > 1) fill_dest(0, a.steps[(long)r * nz].sy);
    __syncthreads();
    if (cl && !as) cluster_wait();   // every block of the cluster has started
    {
        const int k0 = (up ? 0 : nz - 1) * nplane + y0 * nx;
        const PlaneLerp<T> sp = a.steps[(long)r * nz];
        for (int q = threadIdx.x; q < items; q += nth) {
            int x, yl0, nr;
            item_at(q, x, yl0, nr);
            for (int j = 0; j < nr; ++j) {
                const int o = (yl0 + j) * nx + x;
                const T Ib = up ? a.bbot[y0 * nx + o] : T(0);
                pj[k0 + o] = Ib * wsum;
                pu[k0 + o] = wsum;
                if (nz > 1) {
                    T cv[NV * VW];
#pragma unroll
                    for (int e = 0; e < NV * VW; ++e) cv[e] = Ib;
                    cv[0] = a.chi0[k0 + o];
                    cv[1] = a.S[k0 + o];
                    put(All{}, dest[yl0 + j], shifted(x, sp.sx), 0, cv);
                }
            }
        }
    }
    cp_async_wait();
    if (cl && !as) cluster_barrier();
    else __syncthreads();

    int part = 1;   // t mod 3
    if (nz > 2) {
        fill_dest(1, step_ring[1].sy);
        __syncthreads();
    }
    for (int t = 1; t < nz; ++t) {
        const int kp = (up ? t : nz - 1 - t) * nplane + y0 * nx;
        const unsigned char *prev = smem_raw + ((t - 1) & 1) * (size_t)frame;
        const PlaneLerp<T> sp = step_ring[t & 3];
        const bool write = t + 1 < nz;
        // part (t + 2) mod 3 was last read at step t - 1
        if (t + 2 < nz) {
            prefetch(t + 2, part == 0 ? 2 : part - 1);
            fill_dest(t + 1, step_ring[(t + 1) & 3].sy);
        }
        if (chunks > 1 && t > 1) flush_sums(t - 1);
        if (as) {
            // the other blocks' part of the plane stored at step t - 1
            wait_fill(t - 1);
            if (write) {
                expect_fill(sp.sy, t & 1);
                // every block's reads of this buffer (step t - 1) are over
                if (t >= 2) cluster_wait();
            }
        }
        // the nearer column and row first: H = A + rx B, V = H + ry H'
        bool down = false;   // FP64: the nearer row is the higher one
        fx::u64 cm = 0;      // FP64: c = (cm, ce)
        int ce = 0;
        if constexpr (F64) {
            down = sp.near & 2;
            fx::unpack(sp.c, &cm, &ce);
        }
        // Jeff and U of the thread's first item, stored after the barrier's first half
        T kj[R], ku[R];
        int ko[R], nk = 0;
        for (int q = q0; q < qend; q += nth) {
            int x, yl0, nr;
            item_at(q, x, yl0, nr);
            // rows in the order they are needed: node j of the item lies
            // between row j (nearer) and row j + 1 of the walk
            const unsigned char *row0 =
                prev + (unsigned)(down ? yl0 + nr : yl0) * pitch;
            const unsigned xb = (unsigned)x * 16, xb1 = x + 1 == nx ? 0u : xb + 16;
            const unsigned near_x = (sp.near & 1) ? xb1 : xb, far_x = (sp.near & 1) ? xb : xb1;
            const unsigned xs = shifted(x, sp.sx);
            const int dpitch = down ? -(int)pitch : (int)pitch;
            auto row_h = [&](int v, int k, T *h) {
                const unsigned char *p = row0 + k * dpitch + v * vs;
                T A[VW], B[VW];
                ld16(reinterpret_cast<const T *>(p + near_x), A);
                ld16(reinterpret_cast<const T *>(p + far_x), B);
#pragma unroll
                for (int e = 0; e < VW; ++e) h[e] = fma(sp.rx, B[e], A[e]);
            };
            if constexpr (!F64) {
                // FP32: all channels of a node at once, the slots unrolled
                T h0[NV * VW], h1[NV * VW];
#pragma unroll
                for (int v = 0; v < NV; ++v) row_h(v, 0, h0 + v * VW);
#pragma unroll
                for (int j = 0; j < R; ++j) {
                    if (j >= nr) break;
#pragma unroll
                    for (int v = 0; v < NV; ++v) row_h(v, j + 1, h1 + v * VW);
                    T ch[NV * VW];
#pragma unroll
                    for (int c = 0; c < NV * VW; ++c) {
                        ch[c] = c < NP + 2 ? fma(sp.wy1, h1[c], sp.wy0 * h0[c]) : T(0);
                        h0[c] = h1[c];
                    }
                    const int yl = yl0 + j;
                    T chi_loc, S_loc;
                    local(t, part, yl * nx + x, chi_loc, S_loc);
                    const T dtau0 = (ch[0] + chi_loc) * sp.half_s;
                    const T S_up = ch[1];
                    T cj = 0, cu = 0;
                    // every slot in closed form (0), by series (1), or each its own
                    auto slots = [&](auto mode_tag) {
                        constexpr int MODE = decltype(mode_tag)::value;
#pragma unroll
                        for (int p = 0; p < NP; ++p) {
                            T ex, w0, wup, u;
                            const T xt = dtau0 * r_phi[p];
                            if (MODE == 0) Weights32::closed(xt, ex, w0, wup, u);
                            else if (MODE == 1) Weights32::series(xt, ex, w0, wup, u);
                            else Weights32::eval(xt, ex, w0, wup, u);
                            cu = fma(r_w[p], u, cu);
                            const T part = fma(ch[2 + p], ex, wup * S_up);   // I - w0 S
                            cj = fma(r_w[p], part, cj);
                            ch[2 + p] = fma(w0, S_loc, part);
                        }
                    };
                    if (dtau0 >= d_closed) slots(std::integral_constant<int, 0>{});
                    else if (dtau0 < d_series) slots(std::integral_constant<int, 1>{});
                    else slots(std::integral_constant<int, 2>{});
                    const int o = yl * nx + x;
                    if (q == q0) {
                        kj[j] = cj;
                        ku[j] = cu;
                        ko[j] = kp + o;
                        nk = j + 1;
                    } else {
                        pj[kp + o] = cj;
                        pu[kp + o] = cu;
                    }
                    if (write) {
                        ch[0] = chi_loc;
                        ch[1] = S_loc;
                        put(All{}, dest[(t & 1) * rows + yl], xs, 0, ch);
                    }
                }
            } else {
            // vector v interpolated at the item's nodes (without the factor c)
            auto upwind = [&](int v, T (*o)[VW]) {
                T h0[VW], h1[VW];
                row_h(v, 0, h0);
#pragma unroll
                for (int j = 0; j < R; ++j) {
                    if (j < nr) {
                        row_h(v, j + 1, h1);
#pragma unroll
                        for (int e = 0; e < VW; ++e) {
                            o[j][e] = fma(sp.ry, h1[e], h0[e]);
                            h0[e] = h1[e];
                        }
                    }
                }
            };
            T V0[R][VW];
            upwind(0, V0);
            T S_up[R], S_loc[R], chi_loc[R], dtau0[R], cj[R], cu[R];
            // FP64: dtau0 = (dm, de), 1/dtau0 = (dr, 1 - de), the sum of the
            // slots' (w/phi)(1 - e^-x) in units of 2^(ea - 64)
            fx::u64 dm[R], dr[R], ud[R];
            int de[R];
            bool dok[R];
            RowTarget dst[R];
#pragma unroll
            for (int j = 0; j < R; ++j) {
                if (j < nr) {
                    const int yl = down ? yl0 + nr - 1 - j : yl0 + j;
                    local(t, part, yl * nx + x, chi_loc[j], S_loc[j]);
                    S_up[j] = V0[j][1] * sp.c;
                    dtau0[j] = fma(sp.c, V0[j][0], chi_loc[j]) * sp.half_s;
                    dok[j] = fx::in_range(dtau0[j]);
                    fx::unpack(dtau0[j], &dm[j], &de[j]);
                    dr[j] = fx::recip(dm[j]);
                    ud[j] = 0;
                    cj[j] = cu[j] = T(0);
                    if (write) dst[j] = dest[(t & 1) * rows + yl];
                }
            }
            // slot p's new intensity at node j from the upwind sum i (without c)
            auto step = [&](int j, int p, T i) {
                const PlaneSlot<T> &sl = stab[p];
                T cex, w0, wup;   // c e^-x, w0, w_up
                if (dok[j] && sl.fx) {
                    const int ex = de[j] + sl.pe;
                    fx::Weights w;
                    if (ex <= fx::kThinExp) {
                        w = fx::thin(fx::mulhi(dm[j], sl.pm), ex);
                        cu[j] = fma(sl.w, fx::pack(w.u, 0), cu[j]);
                    } else {
                        w = fx::closed(fx::mulhi(dm[j], sl.ym), de[j] + sl.ye,
                                       fx::mulhi(dr[j], sl.im), 1 - de[j] + sl.ie,
                                       fx::Tables{fx_tab, fx_tab + fx::kTab});
                        ud[j] += fx::mulhi(sl.aq, w.D);
                    }
                    cex = w.E ? fx::pack62(fx::mulhi(w.E, cm), ce - w.n) : 0.0;
                    w0 = w.w0;
                    wup = w.wup;
                } else {
                    const Weights64 w = weights64(dtau0[j] * sl.phi);
                    cu[j] = fma(sl.w, w.u, cu[j]);
                    cex = sp.c * w.ex;
                    w0 = w.w0;
                    wup = w.wup;
                }
                const T part = fma(i, cex, wup * S_up[j]);   // I - w0 S
                cj[j] = fma(sl.w, part, cj[j]);
                return fma(w0, S_loc[j], part);
            };
#pragma unroll
            for (int j = 0; j < R; ++j)
                if (j < nr && chunk == 0) {
                    V0[j][0] = chi_loc[j];
                    V0[j][1] = S_loc[j];
                    if (write) put(One{}, dst[j], xs, 0, V0[j]);
                }
#pragma unroll 1
            for (int v = v_begin; v < v_end; ++v) {
                T V[R][VW];
                upwind(v, V);
#pragma unroll
                for (int j = 0; j < R; ++j)
                    if (j < nr) {
#pragma unroll
                        for (int e = 0; e < VW; ++e) {
                            const int p = v * VW + e - 2;
                            V[j][e] = p < nslot ? step(j, p, V[j][e]) : T(0);
                        }
                        if (write) put(One{}, dst[j], xs, v, V[j]);
                    }
            }
#pragma unroll
            for (int j = 0; j < R; ++j)
                if (j < nr) {
                    const int o = (down ? yl0 + nr - 1 - j : yl0 + j) * nx + x;
                    // + (sum of (w/phi)(1 - e^-x)) / dtau0
                    if (ud[j] >> 32)
                        cu[j] = fma(fx::pack(dr[j], 1 - de[j] + stab[0].ea),
                                    fx::pack32(ud[j], 0), cu[j]);
                    if (chunks > 1) {
                        T *dr = red + 2 * (((t & 1) * chunks + chunk) * rows * nx + o);
                        dr[0] = cj[j];
                        dr[1] = cu[j];
                    } else if (q == q0) {
                        kj[j] = cj[j];
                        ku[j] = cu[j];
                        ko[j] = kp + o;
                        nk = j + 1;
                    } else {
                        pj[kp + o] = cj[j];
                        pu[kp + o] = cu[j];
                    }
                }
            }
        }
        // before the barrier, since any thread may read the next plane's values:
        // the copies for step t + 1 are done
        if (t + 2 < nz) cp_async_wait_but_last();
        else cp_async_wait();
        if (write) {
            if (as) {
                __syncthreads();
                if (t + 2 < nz) cluster_arrive_relaxed();
            } else if (cl) {
                cluster_arrive();
            } else {
                __syncthreads();
            }
        }
#pragma unroll
        for (int j = 0; j < R; ++j)
            if (j < nk) {
                pj[ko[j]] = kj[j];
                pu[ko[j]] = ku[j];
            }
        if (write && cl && !as) cluster_wait_acquire();
        part = part == 2 ? 0 : part + 1;
    }
    if (chunks > 1 && nz > 1) {
        __syncthreads();
        flush_sums(nz - 1);
    }
    // no block leaves while another may still address its shared memory
    if (as && nz > 1) cluster_barrier();
}

// MAXT: block-size bound the kernel is compiled for; MINB: resident blocks
// per SM it must fit (the register budget); R: rows of a thread's item.
template <typename T, int NP, int MAXT, int MINB, int R, bool AS>
__global__ void __launch_bounds__(MAXT, MINB) plane_sweep_kernel(const PlaneArgs<T> a) {
    plane_sweep_body<T, NP, R, AS>(a);
}

// ------------------------------------------------------------- launching

// Kernel attributes and the launch configuration of shape s (dynamic shared
// memory, clusters of `bands` blocks).
template <typename T, int NP, int MAXT, int MINB, int R, bool AS>
static cudaError_t plane_config(const SweepShape &s, size_t smem, cudaStream_t st,
                                cudaLaunchConfig_t *cfg, cudaLaunchAttribute *attr) {
    // the limit is the same for every launch, so a CUDA graph that captured a
    // launch needing more shared memory than a later one still replays
    cudaError_t e = cudaFuncSetAttribute(plane_sweep_kernel<T, NP, MAXT, MINB, R, AS>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)plane_smem_max(sizeof(T) == 8));
    if (e == cudaSuccess && s.bands > kPortableBands)
        e = cudaFuncSetAttribute(plane_sweep_kernel<T, NP, MAXT, MINB, R, AS>,
                                 cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    *cfg = cudaLaunchConfig_t{};
    cfg->gridDim = dim3(s.bands, s.ngroups, kRays);
    cfg->blockDim = dim3(s.threads, 1, 1);
    cfg->dynamicSmemBytes = smem;
    cfg->stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = s.bands;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg->attrs = attr;
    cfg->numAttrs = s.bands > 1 ? 1 : 0;   // one band: a plain launch
    return cudaSuccess;
}

// launch (a non-null) or occupancy query (a null: *n = clusters, or blocks
// per SM for one band, the GPU holds at once)
template <typename T, int NP, int MAXT, int MINB, int R, bool AS>
static cudaError_t plane_go_r(const PlaneArgs<T> *a, const SweepShape &s, const PlaneLayout &lay,
                              cudaStream_t st, int *n) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    cudaError_t e = plane_config<T, NP, MAXT, MINB, R, AS>(s, lay.smem, st, &cfg, attr);
    if (e != cudaSuccess) return e;
    if (a) {
        PlaneArgs<T> b = *a;
        b.ahead = lay.ahead;
        b.chunks = lay.chunks;
        b.ipad = lay.ipad;
        return cudaLaunchKernelEx(&cfg, plane_sweep_kernel<T, NP, MAXT, MINB, R, AS>, b);
    }
    if (s.bands == 1)
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            n, plane_sweep_kernel<T, NP, MAXT, MINB, R, AS>, s.threads, cfg.dynamicSmemBytes);
    return cudaOccupancyMaxActiveClusters(n, plane_sweep_kernel<T, NP, MAXT, MINB, R, AS>, &cfg);
}

template <typename T, int NP, int MAXT, int MINB, bool AS>
static cudaError_t plane_go(const PlaneArgs<T> *a, const SweepShape &s, int nx, cudaStream_t st,
                            int *n) {
    const PlaneLayout lay =
        plane_layout(sizeof(T) == 8 ? 0 : 1, NP, s.rows, nx, s.threads);
    return lay.item_rows == 2 ? plane_go_r<T, NP, MAXT, MINB, 2, AS>(a, s, lay, st, n)
                              : plane_go_r<T, NP, MAXT, MINB, 1, AS>(a, s, lay, st, n);
}

// register budget: lean 0 the full budget of MAXT threads (one block per SM),
// lean 1 (FP32 only) two blocks of 512 or four of 256 per SM (64 registers);
// FP32 blocks of up to 1024 threads for one or two slots
template <typename T, int NP, bool AS>
static cudaError_t plane_go_np(const PlaneArgs<T> *a, const SweepShape &s, int nx,
                               cudaStream_t st, int *n) {
    if constexpr (sizeof(T) == 4) {
        if (s.threads > 512) {
            // 1024 threads (64 registers): small slot counts only
            if constexpr (NP <= 2) {
                if (s.lean == 0) return plane_go<T, NP, 1024, 1, AS>(a, s, nx, st, n);
            }
            return cudaErrorInvalidValue;
        }
        if (s.lean == 1)
            return s.threads <= 256 ? plane_go<T, NP, 256, 4, AS>(a, s, nx, st, n)
                                    : plane_go<T, NP, 512, 2, AS>(a, s, nx, st, n);
        return s.threads <= 256 ? plane_go<T, NP, 256, 1, AS>(a, s, nx, st, n)
                                : plane_go<T, NP, 512, 1, AS>(a, s, nx, st, n);
    } else {
        // the FP64 body does not fit 64 registers without spilling: no lean variant
        if (s.lean != 0 || s.threads > 512) return cudaErrorInvalidValue;
        return s.threads <= 256 ? plane_go<T, NP, 256, 1, AS>(a, s, nx, st, n)
                                : plane_go<T, NP, 512, 1, AS>(a, s, nx, st, n);
    }
}

template <typename T, bool AS>
static cudaError_t plane_dispatch(const PlaneArgs<T> *a, const SweepShape &s, int nx,
                                  cudaStream_t st, int *n) {
    if (s.threads < 32 || s.threads > kPlaneMaxThreads || s.threads % 32 || s.lean < 0 ||
        s.lean > 1)
        return cudaErrorInvalidValue;
    switch (s.np) {
        case 1: return plane_go_np<T, 1, AS>(a, s, nx, st, n);
        case 2: return plane_go_np<T, 2, AS>(a, s, nx, st, n);
        case 3: return plane_go_np<T, 3, AS>(a, s, nx, st, n);
        case 5: return plane_go_np<T, 5, AS>(a, s, nx, st, n);
        case 8: return plane_go_np<T, 8, AS>(a, s, nx, st, n);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace mg3d
