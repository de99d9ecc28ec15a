// Fused collide-and-stream kernels (Sect. 2.2) on the one-array A-A layout:
// the plain step, the far / near split of the overlapped schedule and the
// batched form.  The per-node bodies are in lbm_stream.cuh.
//
// Per fluid node: read the 19 pre-collision deviations d_i = f_i - w_i, form
// rho (Eq. 5) and the force-shifted velocity (Eq. 6, u = sum f c / rho + g/2),
// the non-equilibrium momentum flux Pi_ab = sum c_a c_b (f - f^eq) against the
// equilibrium of Eq. (9), the Smagorinsky relaxation time of Eq. (18)
//   tau* = tau0 + 1/2 [sqrt(tau0^2 + 18 sqrt(2) C^2 Q / rho) - tau0],
//   Q = sqrt(Pi_ab Pi_ab),
// relax (Eq. 12) and add the body-force source of Guo, Zheng & Shi (2002),
//   (1 - 1/(2 tau*)) w_i [3 (c_i - u).F + 9 (c_i.u)(c_i.F)],  F = rho g,
// then write the 19 post-collision deviations in place (A-A, so streaming is
// implicit in the addressing of the next step).  Nodes next to the z walls
// also write the halfway bounce-back value of Eqs. (19, 21) with q = 1/2,
//   f_k(x, t+1) = f^c_opp(k)(x) + 6 w_k (c_k . u_wall),
// straight into the slot the next step reads for the population arriving
// from the wall, so no separate wall pass is needed.  Sphere links are
// completed afterwards by the link kernel.
//
// Roofline: HBM-bound.  Algorithmic traffic per fluid node and step is
// 19 loads + 19 stores of the stored type plus one flag byte.
#include <algorithm>

#include "lbm_rows.cuh"
#include "lbm_stream.cuh"

namespace lbm {

// Every fluid node, one thread each, one block per row segment.  Resident
// blocks per SM: the even parity fits 48 registers without spills and at 5
// blocks keeps more loads in flight (FP32 collide 0.435 -> 0.422 ms per
// step over both parities; 6 blocks at 40 registers spill and lose); the
// odd parity's shifted addressing needs 64 (at 48 it spills 112 bytes and
// the step's collide took 0.477 ms).
#ifndef LBM_SC_MINB_EVEN
#define LBM_SC_MINB_EVEN 5
#endif
#ifndef LBM_SC_MINB_ODD
#define LBM_SC_MINB_ODD 4
#endif
template <int ODD, typename T>
__global__ void __launch_bounds__(256, ODD ? LBM_SC_MINB_ODD : LBM_SC_MINB_EVEN) k_stream_collide(const Lat L, const Phys ph, T *f, uint8_t *flag,
                                                        int *status, const int down) {
    // the link kernel reads the marks before its wait: it may start once every
    // block here has seen the refill (and so the marks) complete
    step_wait();
    step_next();
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y, z = down ? L.nz - 1 - (int)blockIdx.z : (int)blockIdx.z;
    if (x >= L.nx) return;
    const int row = y + L.ny * z;
    const int n = x + L.nx * row;
    sc_node<ODD, T>(L, ph, f, flag, status, x, y, z, n, flag[n]);
}

// The nodes of the groups in a list (the near groups of the overlapped
// schedule), *count groups, grid-stride with one thread per node, so a
// warp covers whole 32-byte sectors of each slot row; coordinates by exact
// multiply-high division.
template <int ODD, typename T>
__global__ void __launch_bounds__(256, 4) k_collide_list(const Lat L, const Phys ph, T *__restrict__ f,
                                                      uint8_t *__restrict__ flag, int *__restrict__ status,
                                                      const int *__restrict__ list, const int *__restrict__ count,
                                                      const int ngx, const int shift, const FastDiv dngx,
                                                      const FastDiv dny) {
    const int total = *count << shift;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
        const int g = list[t >> shift];
        const int row = (int)dngx.div((unsigned)g);
        const int x = ((g - row * ngx) << shift) | (t & ((1 << shift) - 1));
        if (x >= L.nx) continue;
        const int z = (int)dny.div((unsigned)row);
        const int n = x + L.nx * row;
        sc_node<ODD, T>(L, ph, f, flag, status, x, row - z * L.ny, z, n, flag[n]);
    }
}

// 16-bit storage: the same with one node pair per thread (sc_pair); the
// groups hold 2^shift nodes, 2^(shift - 1) pairs.  Requires even nx.
template <int ODD, typename T>
__global__ void __launch_bounds__(256, 4) k_collide_list2(const Lat L, const Phys ph, T *__restrict__ f,
                                                       uint8_t *__restrict__ flag, int *__restrict__ status,
                                                       const int *__restrict__ list, const int *__restrict__ count,
                                                       const int ngx, const int shift, const FastDiv dngx,
                                                       const FastDiv dny) {
    const int ps = shift - 1;  // pairs per group: 2^ps
    const int total = *count << ps;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
        const int g = list[t >> ps];
        const int row = (int)dngx.div((unsigned)g);
        const int xp = ((g - row * ngx) << ps) | (t & ((1 << ps) - 1));
        if (2 * xp >= L.nx) continue;
        const int z = (int)dny.div((unsigned)row);
        sc_pair<ODD, T>(L, ph, f, flag, status, xp, row - z * L.ny, z);
    }
}

// Rows through shared memory (lbm_rows.cuh), three CTAs per SM of 256
// consumers.  HBM-bound in FP32: 256^3 with 2000 spheres, us per launch at
// even / odd parity 394 / 394 (6.4 TB/s, 94% of a copy) where a thread per
// node with global loads took 385 / 452; collide phase 422 -> 396 us at 256^3,
// two CTAs 464, four (56 registers) 477.
//
// Where: the lattice has to exceed L2 (FP32 256x256x16, 80 MB: 26.6 us per
// step node-wise, 28.7 by rows; x 24: 45.4 and 43.6; 128^3: 57.7 both; FP16 /
// BF16 512x96x80, 150 MB: 78.4 / 77.0 by the pair kernel, 80.8 / 81.4 by
// rows) and whole rows fill 7/8 of a 1 KB buffer (FP32 128x256x256: 213 ->
// 208, 240x200x200 260 -> 253; four rows of 64: 106.6 -> 109.0, 160 of 256
// nodes filled: 110.5 -> 130).  Rows of more than a buffer in buffers of 2 KB,
// two CTAs per SM, lose (one FP32 row of 512: 112.6 -> 159; FP16 without
// spheres 640x256x128 428 -> 639, 1024x128x80 209 -> 271).
// 16-bit storage is bound by instruction issue, and the pair kernel does the
// conversions of two nodes from one word: two rows of 512 bytes in a buffer
// lose to it (297 us against 320 at four CTAs, 325 at three), one row of 896
// to 1024 bytes wins among spheres, whose solid halves the pair kernel stores
// element by element (us per step, pair / rows: 512x256x256 with 4000 spheres
// FP16 880 / 783, BF16 845 / 785; 448x256x256 823 / 747, 794 / 746;
// 480x256x256 870 / 787, 837 / 786; 512x256x128 without 318 / 313, 311 / 315).
constexpr long long kRowsFrom = 1ll << 23;  // bytes of a slot array
constexpr int kRowCtas = 3;
constexpr int kRowSmem = 226 * 1024 / kRowCtas - 1536;
constexpr int kRowThreads = 256;  // consumers at most

// f may carry __restrict__ here: it is read by bulk copies only, which no
// load can be made of (FP16 512x256x256 among spheres 617 -> 614 us).
template <int ODD, typename T>
__global__ void __launch_bounds__(kRowThreads + 32, kRowCtas)
    k_collide_rows(const Lat L, const Phys ph, T *__restrict__ f, uint8_t *flag, int *__restrict__ status, const RowPlan pl, const int down) {
    step_wait();  // as in k_stream_collide
    step_next();
    rows_body<ODD, T>(
        [&](int u) {
            return RowUnit<T>(L, ph, f, flag, status, pl.dnx, pl.dpp, pl.per_plane, pl.rows,
                              down ? pl.units - 1 - u : u);
        },
        pl.units, pl.stages, pl.consumers);
}

// The plan of a lattice whose rows can be copied whole (16-byte multiples)
// and fill a buffer (see above), else stages = 0.
static RowPlan rows_plan(const Lat &L, size_t esize) {
    RowPlan p{};
    const int fit = kRowPitch / (int)esize, rows = std::max(1, fit / L.nx);  // nodes and rows of a buffer
    if (L.nx * esize % 16 != 0 || L.N * (long long)esize < kRowsFrom) return p;
    if (rows * L.nx > fit || 8 * rows * L.nx < 7 * fit || L.nx < (esize == 4 ? 112 : fit / 2 + 1)) return p;
    p.rows = std::min(rows, L.ny);
    const int U = p.rows * L.nx, passes = (U + kRowThreads - 1) / kRowThreads;
    p.consumers = ((U + passes - 1) / passes + 31) / 32 * 32;
    p.stages = std::min(kRowStages, kRowSmem / (Q * kRowPitch));
    p.per_plane = (L.ny + p.rows - 1) / p.rows;
    p.units = p.per_plane * L.nz;
    p.dpp = FastDiv((unsigned)p.per_plane);
    p.dnx = FastDiv((unsigned)L.nx);
    return p;
}

// Batched form: every node of every instance, one persistent launch.  Chunk
// c = (instance, first node) covers TPB consecutive nodes of one instance
// (a block's threads, coalesced); block b takes the contiguous chunk range
// [b n / G, (b + 1) n / G).  The current instance's descriptor is staged in
// shared memory (read on use, not held in registers).  MINB resident blocks
// per SM bound the registers (64 per thread at TPB * MINB = 1024, 85 at
// 768); the autotuner picks both.
template <int ODD, typename T, int TPB, int MINB>
__global__ void __launch_bounds__(TPB, MINB) k_collide_batch(const Inst *__restrict__ I,
                                                                   const int2 *__restrict__ chunks, const int nchunks) {
    __shared__ __align__(16) unsigned char si_raw[sizeof(Inst)];
    Inst &si = *reinterpret_cast<Inst *>(si_raw);
    const int c0 = (int)((long long)nchunks * blockIdx.x / gridDim.x);
    const int c1 = (int)((long long)nchunks * (blockIdx.x + 1) / gridDim.x);
    int cur = -1;
    for (int c = c0; c < c1; ++c) {
        const int2 ch = chunks[c];
        if (ch.x != cur) {
            __syncthreads();
            const unsigned *src = (const unsigned *)(I + ch.x);
            unsigned *dst = (unsigned *)&si;
            for (int w = threadIdx.x; w < (int)(sizeof(Inst) / 4); w += TPB) dst[w] = src[w];
            __syncthreads();
            cur = ch.x;
        }
        const int n = ch.y + (int)threadIdx.x;
        if (n >= (int)si.L.N) continue;
        const int row = (int)si.dnx.div((unsigned)n);
        const int z = (int)si.dny.div((unsigned)row);
        sc_node<ODD, T>(si.L, si.ph, (T *)si.f, si.flag, si.status, n - row * si.L.nx, row - z * si.L.ny, z, n,
                        si.flag[n]);
    }
}

// The same with the instances' parameters in a kernel-parameter table (up to
// kCollideTable members): no shared-memory staging, and the constants are
// read through the constant cache as in the single-instance kernel.
template <int ODD, typename T, int TPB, int MINB>
__global__ void __launch_bounds__(TPB, MINB) k_collide_batch_tab(const __grid_constant__ CollideTable tab,
                                                                  const int2 *__restrict__ chunks,
                                                                  const int nchunks) {
    const int c0 = (int)((long long)nchunks * blockIdx.x / gridDim.x);
    const int c1 = (int)((long long)nchunks * (blockIdx.x + 1) / gridDim.x);
    for (int c = c0; c < c1; ++c) {
        const int2 ch = chunks[c];
        const CInst &ci = tab.c[ch.x];
        const int n = ch.y + (int)threadIdx.x;
        if (n >= (int)ci.L.N) continue;
        const int row = (int)ci.dnx.div((unsigned)n);
        const int z = (int)ci.dny.div((unsigned)row);
        sc_node<ODD, T>(ci.L, ci.ph, (T *)ci.f, ci.flag, ci.status, n - row * ci.L.nx, row - z * ci.L.ny, z, n,
                        ci.flag[n]);
    }
}

// 16-bit storage: two nodes per thread (sc_pair).  Requires even nx.
template <int ODD, typename T>
__global__ void __launch_bounds__(128, 8) k_stream_collide2(const Lat L, const Phys ph, T *f, uint8_t *flag,
                                                            int *status, const int down) {
    step_wait();  // as in k_stream_collide
    step_next();
    const int xp = blockIdx.x * blockDim.x + threadIdx.x;
    if (xp >= (L.nx >> 1)) return;
    sc_pair<ODD, T>(L, ph, f, flag, status, xp, blockIdx.y, down ? L.nz - 1 - (int)blockIdx.z : (int)blockIdx.z);
}

// Whether the collide of this parity goes through the planes from the top
// down: the planes the step before ended with are still in L2.  Us per step
// one way / alternating: 201x150x101 91.8 / 81.1, 160^3 110.5 / 101.2, 256^3
// 404 / 401, 256^3 BF16 312 / 308; lattices that fit L2 the same.  The link
// kernel in between takes L2 for its own scattered blocks: 160^3 with 400
// spheres of radius 4 158.7 / 155.7, 256^3 with 2000 533.6 / 534.8.  The line
// between the two, 760,000 links of spheres of the handle's largest radius
// (120 MB at the 158 bytes per link measured in FP32), is a measured one for
// this GPU's 129 MB of L2; smaller spheres than the handle allows, and 16-bit
// storage, reach it early and keep the one-way sweep.
static int sweep_down(const lbm_s *h, int parity) {
    const double r = h->p.max_radius, link_bytes = h->pt.np * 72.0 * r * r * 158.0;
    return parity && link_bytes < 120e6;
}

template <int ODD, typename T>
static int launch_rows(lbm_s *h, const RowPlan &p, bool pdl) {
    const auto k = k_collide_rows<ODD, T>;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kRowSmem) != cudaSuccess) return LBM_ERR_CUDA;
    const int grid = std::min(p.units, h->sms * kRowCtas);
    return launch_step(k, dim3(grid), dim3(p.consumers + 32), p.stages * Q * kRowPitch, h->stream, pdl, h->L, h->ph,
                       (T *)h->f, h->flag, h->status, p, sweep_down(h, ODD)) == cudaSuccess
               ? LBM_OK
               : LBM_ERR_CUDA;
}

template <int ODD, typename T>
static int launch_sc(lbm_s *h, bool pdl) {
    const int bx = h->L.nx >= 256 ? 256 : ((h->L.nx + 31) / 32) * 32;
    const dim3 grid((h->L.nx + bx - 1) / bx, h->L.ny, h->L.nz);
    return launch_step(k_stream_collide<ODD, T>, grid, dim3(bx), 0, h->stream, pdl, h->L, h->ph, (T *)h->f, h->flag,
                       h->status, sweep_down(h, ODD)) == cudaSuccess
               ? LBM_OK
               : LBM_ERR_CUDA;
}

template <int ODD, typename T>
static int launch_sc2(lbm_s *h, bool pdl) {
    const int hx = h->L.nx / 2;
    const int bx = hx >= 128 ? 128 : ((hx + 31) / 32) * 32;
    const dim3 grid((hx + bx - 1) / bx, h->L.ny, h->L.nz);
    return launch_step(k_stream_collide2<ODD, T>, grid, dim3(bx), 0, h->stream, pdl, h->L, h->ph, (T *)h->f, h->flag,
                       h->status, sweep_down(h, ODD)) == cudaSuccess
               ? LBM_OK
               : LBM_ERR_CUDA;
}

template <int ODD, typename T>
static int launch_parity(lbm_s *h, bool pdl) {
    const RowPlan p = rows_plan(h->L, sizeof(T));
    if (p.stages >= 2) return launch_rows<ODD, T>(h, p, pdl);
    if constexpr (sizeof(T) == 2) {
        if ((h->L.nx % 2) == 0) return launch_sc2<ODD, T>(h, pdl);
    }
    return launch_sc<ODD, T>(h, pdl);
}

template <typename T>
static int launch_type(lbm_s *h, int parity, bool pdl) {
    const int rc = parity ? launch_parity<1, T>(h, pdl) : launch_parity<0, T>(h, pdl);
    if (rc) cudaGetLastError();
    return rc;
}

bool collides_by_rows(const lbm_s *h) { return rows_plan(h->L, h->esize).stages >= 2; }

int launch_stream_collide(lbm_s *h, int parity, bool pdl) {
    switch (h->precision) {
        case LBM_FP32: return launch_type<float>(h, parity, pdl);
        case LBM_BF16_DEV: return launch_type<__nv_bfloat16>(h, parity, pdl);
        case LBM_FP16_DEV: return launch_type<__half>(h, parity, pdl);
    }
    return LBM_ERR_ARG;
}

template <typename T>
static int launch_list_type(lbm_s *h, int parity, const int *list, const int *count, cudaStream_t st) {
    const FastDiv dngx((unsigned)h->near_ngx), dny((unsigned)h->L.ny);
    const int grid = h->sms * 4, ngx = h->near_ngx, sh = h->near_shift;
    if constexpr (sizeof(T) == 2) {
        if ((h->L.nx % 2) == 0 && sh >= 1) {  // node pairs
            if (parity)
                k_collide_list2<1, T><<<grid, 256, 0, st>>>(h->L, h->ph, (T *)h->f, h->flag, h->status, list, count,
                                                             ngx, sh, dngx, dny);
            else
                k_collide_list2<0, T><<<grid, 256, 0, st>>>(h->L, h->ph, (T *)h->f, h->flag, h->status, list, count,
                                                             ngx, sh, dngx, dny);
            return cudaGetLastError() == cudaSuccess ? LBM_OK : LBM_ERR_CUDA;
        }
    }
    if (parity)
        k_collide_list<1, T><<<grid, 256, 0, st>>>(h->L, h->ph, (T *)h->f, h->flag, h->status, list, count, ngx, sh,
                                                   dngx, dny);
    else
        k_collide_list<0, T><<<grid, 256, 0, st>>>(h->L, h->ph, (T *)h->f, h->flag, h->status, list, count, ngx, sh,
                                                   dngx, dny);
    return cudaGetLastError() == cudaSuccess ? LBM_OK : LBM_ERR_CUDA;
}

int launch_collide_list(lbm_s *h, int parity, const int *list, const int *count, cudaStream_t stream) {
    cudaStream_t st = stream ? stream : h->stream;
    switch (h->precision) {
        case LBM_FP32: return launch_list_type<float>(h, parity, list, count, st);
        case LBM_BF16_DEV: return launch_list_type<__nv_bfloat16>(h, parity, list, count, st);
        case LBM_FP16_DEV: return launch_list_type<__half>(h, parity, list, count, st);
    }
    return LBM_ERR_ARG;
}

template <int ODD, typename T, int TPB, int MINB>
static cudaError_t collide_batch_t(const lbm_batch_s *b, int grid, const int2 *chunks, int nchunks) {
    if (b->ctab)
        k_collide_batch_tab<ODD, T, TPB, MINB><<<grid, TPB, 0, b->stream>>>(*b->ctab, chunks, nchunks);
    else
        k_collide_batch<ODD, T, TPB, MINB><<<grid, TPB, 0, b->stream>>>(b->dinst, chunks, nchunks);
    return cudaGetLastError();
}

// Launch shapes of the batched collide: (threads per block, minimum resident
// blocks per SM), i.e. 64 or 85 registers per thread.
#define LBM_BATCH_SHAPES(X) X(128, 8) X(128, 6) X(256, 4) X(256, 3) X(512, 2) X(512, 1)

template <int ODD, typename T>
static cudaError_t collide_batch_p(const lbm_batch_s *b, int tpb, int minb, int grid, const int2 *chunks,
                                   int nchunks) {
#define LBM_CASE(t, m) \
    if (tpb == t && minb == m) return collide_batch_t<ODD, T, t, m>(b, grid, chunks, nchunks);
    LBM_BATCH_SHAPES(LBM_CASE)
#undef LBM_CASE
    return cudaErrorInvalidValue;
}

template <typename T>
static cudaError_t collide_batch_ty(const lbm_batch_s *b, int P, int tpb, int minb, int grid, const int2 *chunks,
                                    int nchunks) {
    return P ? collide_batch_p<1, T>(b, tpb, minb, grid, chunks, nchunks)
             : collide_batch_p<0, T>(b, tpb, minb, grid, chunks, nchunks);
}

int launch_collide_batch(const lbm_batch_s *b, int P, int tpb, int minb, int grid, const int2 *chunks, int nchunks) {
    if (nchunks == 0) return LBM_OK;
    cudaError_t e = cudaErrorInvalidValue;
    switch (b->precision) {
        case LBM_FP32: e = collide_batch_ty<float>(b, P, tpb, minb, grid, chunks, nchunks); break;
        case LBM_BF16_DEV: e = collide_batch_ty<__nv_bfloat16>(b, P, tpb, minb, grid, chunks, nchunks); break;
        case LBM_FP16_DEV: e = collide_batch_ty<__half>(b, P, tpb, minb, grid, chunks, nchunks); break;
    }
    if (e != cudaSuccess) cudaGetLastError();
    return e == cudaSuccess ? LBM_OK : (e == cudaErrorInvalidValue ? LBM_ERR_ARG : LBM_ERR_CUDA);
}

template <int ODD, typename T, int TPB, int MINB>
static cudaError_t occ_t(int *bps, bool table) {
    return table ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(bps, k_collide_batch_tab<ODD, T, TPB, MINB>, TPB, 0)
                 : cudaOccupancyMaxActiveBlocksPerMultiprocessor(bps, k_collide_batch<ODD, T, TPB, MINB>, TPB, 0);
}

template <typename T>
static cudaError_t occ_ty(int P, int tpb, int minb, int *bps, bool table) {
#define LBM_CASE(t, m) \
    if (tpb == t && minb == m) return P ? occ_t<1, T, t, m>(bps, table) : occ_t<0, T, t, m>(bps, table);
    LBM_BATCH_SHAPES(LBM_CASE)
#undef LBM_CASE
    return cudaErrorInvalidValue;
}

int collide_batch_occupancy(int precision, int P, int tpb, int minb, int *blocks_per_sm, bool table) {
    cudaError_t e = cudaErrorInvalidValue;
    switch (precision) {
        case LBM_FP32: e = occ_ty<float>(P, tpb, minb, blocks_per_sm, table); break;
        case LBM_BF16_DEV: e = occ_ty<__nv_bfloat16>(P, tpb, minb, blocks_per_sm, table); break;
        case LBM_FP16_DEV: e = occ_ty<__half>(P, tpb, minb, blocks_per_sm, table); break;
    }
    if (e != cudaSuccess) cudaGetLastError();
    return e == cudaSuccess ? LBM_OK : LBM_ERR_CUDA;
}

}  // namespace lbm
