// Collide-and-stream of whole lattice rows staged in shared memory by bulk
// copies (cp.async.bulk, the 1D form of TMA).
//
// Under A-A a node reads and writes the same 19 locations: at even steps its
// own slots, at odd steps slot k of x + c_k.  For the nodes of one row these
// are 19 whole rows of the slot arrays: (y, z) at even steps, row
// (y + c_ky, z + c_kz) of slot k at odd ones, where node x finds its element
// at x + c_kx, cyclic in the row (x is periodic).  No other row touches them.  So
// a unit of one or more rows is 19 (x rows) aligned copies in, arithmetic in
// place in shared memory, and 19 copies out: the one-node shifts of the odd
// parity become shared-memory offsets, no address is formed per node and
// direction, and loads run ahead of the arithmetic instead of being bounded
// by the registers of the warps in flight.  Solid nodes' elements go back as
// they came.
//
// A persistent CTA of consumer warps (one node per thread) and one producer
// warp works through the units u = blockIdx.x, + gridDim.x, ...: lane k of
// the producer owns buffer k of every stage, issues its loads, and when the
// consumers have finished a stage its stores; a stage is loaded again when
// its stores have read it.  Every wait is bounded; a producer that gives one up
// waits (bounded again) for the loads it has in flight before it leaves the
// shared memory they write to (a lane that gives up leaves the kernel, so no
// __syncwarp of the others waits for it for longer).
#pragma once

#include "lbm_collide_node.cuh"

namespace lbm {

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint32_t bar, int count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint32_t bar, int bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// False if the phase did not complete within the poll limit (each poll is
// itself a wait of up to some microseconds).
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
    for (int i = 0; i < (1 << 20); ++i) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.b32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, int bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void bulk_store(void *dst, uint32_t src, int bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(src), "r"(bytes)
                 : "memory");
}

constexpr int kRowStages = 4;    // most stages of a CTA
constexpr int kRowPitch = 1024;  // bytes of one slot buffer of a stage

// Units of a lattice: `rows` consecutive rows of one plane (fewer at its
// end), and the launch that works through them.
struct RowPlan {
    int rows, per_plane, units, stages;
    int consumers;  // threads, a multiple of 32
    FastDiv dpp, dnx;
};

// One unit: rows y0 .. y0 + nrow - 1 of plane z of a lattice.
template <typename T>
struct RowUnit {
    const Lat &L;
    const Phys &ph;
    T *f;
    uint8_t *flag;
    int *status;
    FastDiv dnx;
    int y0, z, nrow;
    __device__ __forceinline__ RowUnit(const Lat &l, const Phys &p, T *ff, uint8_t *fl, int *st, const FastDiv &dx,
                                       const FastDiv &dpp, int per_plane, int rows, int u)
        : L(l), ph(p), f(ff), flag(fl), status(st), dnx(dx) {
        z = (int)dpp.div((unsigned)u);
        y0 = (u - z * per_plane) * rows;
        nrow = min(rows, l.ny - y0);
    }
};

// A producer lane that gave up a wait at unit `it`: the status, and a wait for
// the loads of the units up to `loaded`.  Out of line: inlined, it cost the
// FP16 form half a percent.
static __device__ __noinline__ void rows_give_up(int *status, uint32_t full0, int it, int loaded, int nst, int lane) {
    if (lane == 0) atomicOr(status, ST_TIMEOUT);
    for (; it < loaded; ++it) mbar_wait(full0 + 8 * (it % nst), (it / nst) & 1);
}

// The units 0 .. units - 1 that get(u) describes (a RowUnit).  A stage's slot
// buffers lie a fixed pitch apart, so that a node's 19 elements are one base
// and immediate offsets.
template <int ODD, typename T, typename Get>
__device__ __forceinline__ void rows_body(Get get, const int units, const int nst, const int consumers) {
    extern __shared__ __align__(128) unsigned char rows_buf[];
    __shared__ __align__(8) unsigned long long bars[2 * kRowStages];
    constexpr int kStage = Q * kRowPitch, kP = kRowPitch / (int)sizeof(T);
    const uint32_t full0 = smem_addr(bars), done0 = full0 + 8 * kRowStages;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, cwarps = consumers >> 5;
    if (threadIdx.x == 0) {
        for (int s = 0; s < nst; ++s) {
            mbar_init(full0 + 8 * s, 1);
            mbar_init(done0 + 8 * s, cwarps);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const int mine = ((int)blockIdx.x < units) ? (units - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    if (warp == cwarps) {  // producer
        const uint32_t buf = smem_addr(rows_buf) + lane * kRowPitch;
        const int k = lane < Q ? lane : 0, oy = ODD ? rcy(k) : 0, oz = ODD ? rcz(k) : 0;
        // calls fn(global, shared, bytes) for the runs of rows of unit `it` in this lane's slot array
        auto rows = [&](int it, auto fn) {
            const RowUnit<T> r = get(blockIdx.x + it * gridDim.x);
            const int bytes = r.L.nx * (int)sizeof(T);
            T *base = r.f + ((size_t)k * r.L.S + (size_t)r.L.plane * (r.z + oz + 1));
            const uint32_t b = buf + (it % nst) * kStage;
            const int y1 = r.y0 + oy;
            if (y1 >= 0 && y1 + r.nrow <= r.L.ny) {  // rows of a plane follow each other
                fn(base + (size_t)r.L.nx * y1, b, r.nrow * bytes);
            } else {
                for (int j = 0; j < r.nrow; ++j) {
                    int y = y1 + j;
                    y = y < 0 ? y + r.L.ny : (y >= r.L.ny ? y - r.L.ny : y);
                    fn(base + (size_t)r.L.nx * y, b + j * bytes, bytes);
                }
            }
        };
        auto load = [&](int it) {
            const uint32_t bar = full0 + 8 * (it % nst);
            if (lane == 0) {
                const RowUnit<T> r = get(blockIdx.x + it * gridDim.x);
                mbar_expect(bar, Q * r.nrow * r.L.nx * (int)sizeof(T));
            }
            __syncwarp();
            if (lane < Q) rows(it, [&](T *g, uint32_t s, int bytes) { bulk_load(s, g, bytes, bar); });
        };
        bool ok = true;
        int loaded = min(nst, mine), it = 0;  // units whose loads have been issued; the unit at work
        for (int i = 0; i < loaded; ++i) load(i);
        for (; it < mine; ++it) {
            ok = mbar_wait(done0 + 8 * (it % nst), (it / nst) & 1);
            if (!ok) break;
            if (lane < Q) rows(it, [&](T *g, uint32_t s, int bytes) { bulk_store(g, s, bytes); });
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
            // the stage before this one has been read by its stores: load it again
            if (it > 0 && it - 1 + nst < mine) {
                asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                __syncwarp();
                load(it - 1 + nst);
                loaded = it + nst;
            }
        }
        if (!ok) rows_give_up(get(blockIdx.x).status, full0, it, loaded, nst, lane);
        asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    } else {
        for (int it = 0; it < mine; ++it) {
            const RowUnit<T> r = get(blockIdx.x + it * gridDim.x);
            const Lat &L = r.L;
            const int s = it % nst, nx = L.nx, count = r.nrow * nx, z = r.z;
            T *st = (T *)(rows_buf + s * kStage);
            // the flag of this thread's node, while the rows arrive
            uint8_t *flag = r.flag + (size_t)nx * (r.y0 + (size_t)L.ny * z);
            uint8_t fl = (int)threadIdx.x < count ? flag[threadIdx.x] : (uint8_t)1;
            if (!mbar_wait(full0 + 8 * s, (it / nst) & 1)) {
                if (lane == 0) atomicOr(r.status, ST_TIMEOUT);
                break;
            }
            for (int l = threadIdx.x; l < count; l += consumers) {
                if (l >= consumers) fl = flag[l];
                if (fl & 1) continue;
                if (fl) flag[l] = 0;  // refilled this step: plain fluid from now on
                const int j = (int)r.dnx.div((unsigned)l), x = l - j * nx;
                // element of slot k for this node: the node's own at even steps, x + c_kx at odd ones
                T *e[3];
                e[1] = st + l;
                e[0] = ODD ? (x == 0 ? e[1] + (nx - 1) : e[1] - 1) : e[1];
                e[2] = ODD ? (x == nx - 1 ? e[1] - (nx - 1) : e[1] + 1) : e[1];
                float d[Q];
#pragma unroll
                for (int i = 0; i < Q; ++i) {
                    const int k = ODD ? opp(i) : i;
                    d[i] = Store<T>::ld(e[cx(k) + 1] + k * kP);
                }
                collide_node(r.ph, d, r.status);
#pragma unroll
                for (int i = 0; i < Q; ++i) {
                    const int k = ODD ? i : opp(i);
                    Store<T>::st(e[cx(k) + 1] + k * kP, d[i]);
                }
                // Walls: as in sc_node, into slots that no row holds
                if (z == 0 || z == L.nz - 1) {
                    const Nbr nb(L, x, r.y0 + j);
                    T *g = r.f + ((size_t)nx * (r.y0 + (size_t)L.ny * z) + l + L.plane);
#pragma unroll
                    for (int k = 1; k < Q; ++k) {
                        if (cz(k) == 0) continue;
                        if (z != (cz(k) > 0 ? 0 : L.nz - 1)) continue;
                        const float v = wall_push(k, Store<T>::rt(d[opp(k)]), cz(k) > 0 ? r.ph.ulo : r.ph.uhi);
                        Store<T>::st(g + (ODD ? k * L.S : opp(k) * L.S + nb.off(-cx(k), -cy(k), -cz(k))), v);
                    }
                }
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(done0 + 8 * s);
        }
    }
}

}  // namespace lbm
