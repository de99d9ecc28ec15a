// Link kernels (Sect. 2.3): one CTA per sphere, run after the collide
// kernel of a step; the per-sphere body is in lbm_links.cuh.
#include <cmath>

#include "lbm_links.cuh"

namespace lbm {

// GI: compiled with the Galilean-invariant momentum exchange (taken where
// the handle asks for it).
// Bound by scattered DRAM blocks on thousands of spheres, by latency on a
// few.  64 registers (4 CTAs per SM, no spills) with three links per thread
// in flight, link phase in us on 256^3 with 2000 spheres / with 8136 /
// 512x256x256 with 7911 (FP16): 106.2 / 368 / 466; two links 108.9 / 377 /
// 476, five 107.4 / 373 / 473; 5 CTAs at 48 registers (spills) 118.7 / 416 /
// 499 with two and 112.0 / 402 / 514 with one, 6 CTAs 117 / 405 / 504.  With
// node codes per byte, links found per node and direction and three integer
// divisions per link, the same took 110.7 / 374 / 467 and 18.3 instead of
// 15.4 on 64^3 with 31 spheres (the step 60.1 -> 48.4 us there).  A thread's
// links, and so the sums, are in the same order for any batch.
#ifndef LBM_LINK_MINB
#define LBM_LINK_MINB 4  // resident CTAs per SM the register budget is set for
#endif
#ifndef LBM_LINK_BATCH
#define LBM_LINK_BATCH 3  // links per thread whose populations are loaded together
#endif

template <typename T, bool GI>
__global__ void __launch_bounds__(256, LBM_LINK_MINB) k_links(const Lat L, const Parts pt, const SFrame *__restrict__ fcur,
                                               T *f, const uint8_t *__restrict__ flag,
                                               const int32_t *__restrict__ owner, const int P, const int ext,
                                               const int cap, int *status, unsigned long long *ctr) {
    links_body<T, GI, LBM_LINK_BATCH>(L, pt, fcur, f, flag, owner, P, ext, cap, status, ctr, pt.order[blockIdx.x]);
}

// Batched: instance blockIdx.y; parity P is also the step parity.
// 64 sweep members, us per step: 2533 at 4 CTAs per SM with three links in
// flight, 2564 with two, 2587 at 3 CTAs with four.
#ifndef LBM_LINK_B_MINB
#define LBM_LINK_B_MINB 4
#endif
#ifndef LBM_LINK_B_BATCH
#define LBM_LINK_B_BATCH 3
#endif
template <typename T, bool GI>
__global__ void __launch_bounds__(256, LBM_LINK_B_MINB) k_links_b(const Inst *__restrict__ I, const int P,
                                                                  const int ext, const int cap) {
    const Inst &a = I[blockIdx.y];
    if ((int)blockIdx.x >= a.pt.np) return;
    links_body<T, GI, LBM_LINK_B_BATCH>(a.L, a.pt, a.pt.frame[P], (T *)a.f, a.flag, a.owner, P, ext, cap, a.status,
                                        a.ctr, a.pt.order[blockIdx.x]);
}

int link_capacity(double max_radius) {
    const double r = max_radius < 1.0 ? 1.0 : max_radius;
    return (int)std::ceil(80.0 * r * r) + 64;
}

size_t link_smem(int ext, int cap) {
    const LinkTile tl(ext);
    return 8 * (size_t)tl.B * tl.B + 4 * (size_t)cap + 2 * (size_t)tl.ncap(cap);
}

// Raise (never lower: other handles may need more) a kernel's dynamic
// shared memory limit to smem bytes.
template <typename K>
static cudaError_t raise_smem(K kernel, size_t smem) {
    cudaFuncAttributes at;
    cudaError_t e = cudaFuncGetAttributes(&at, kernel);
    if (e == cudaSuccess && at.maxDynamicSharedSizeBytes < (int)smem)
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    return e;
}

template <bool GI>
static cudaError_t raise_all(size_t smem) {
    cudaError_t e = raise_smem(k_links<float, GI>, smem);
    if (e == cudaSuccess) e = raise_smem(k_links<__nv_bfloat16, GI>, smem);
    if (e == cudaSuccess) e = raise_smem(k_links<__half, GI>, smem);
    if (e == cudaSuccess) e = raise_smem(k_links_b<float, GI>, smem);
    if (e == cudaSuccess) e = raise_smem(k_links_b<__nv_bfloat16, GI>, smem);
    if (e == cudaSuccess) e = raise_smem(k_links_b<__half, GI>, smem);
    return e;
}

int links_setup(int ext, int cap) {
    const size_t smem = link_smem(ext, cap);
    cudaError_t e = raise_all<false>(smem);
    if (e == cudaSuccess) e = raise_all<true>(smem);
    if (e != cudaSuccess) cudaGetLastError();
    return e == cudaSuccess ? LBM_OK : LBM_ERR_CUDA;
}

template <typename T, bool GI>
static void links_launch(lbm_s *h, int parity, size_t smem, const SFrame *fcur, int ext, int cap, bool pdl) {
    launch_step(k_links<T, GI>, dim3(h->pt.np), dim3(256), smem, h->stream, pdl, h->L, h->pt, fcur, (T *)h->f, h->flag,
                h->owner, parity, ext, cap, h->status, h->ctr);
}

template <typename T>
static void links_launch_t(lbm_s *h, int parity, size_t smem, const SFrame *fcur, int ext, int cap, bool pdl) {
    if (h->pt.gimea) links_launch<T, true>(h, parity, smem, fcur, ext, cap, pdl);
    else links_launch<T, false>(h, parity, smem, fcur, ext, cap, pdl);
}

int launch_links(lbm_s *h, int parity, bool pdl) {
    const int ext = h->tile_ext, cap = h->link_cap;
    const size_t smem = link_smem(ext, cap);
    const SFrame *fcur = h->pt.frame[h->steps & 1];
    switch (h->precision) {
        case LBM_FP32: links_launch_t<float>(h, parity, smem, fcur, ext, cap, pdl); break;
        case LBM_BF16_DEV: links_launch_t<__nv_bfloat16>(h, parity, smem, fcur, ext, cap, pdl); break;
        case LBM_FP16_DEV: links_launch_t<__half>(h, parity, smem, fcur, ext, cap, pdl); break;
        default: return LBM_ERR_ARG;
    }
    return cudaGetLastError() == cudaSuccess ? LBM_OK : LBM_ERR_CUDA;
}

int links_setup_batch(int ext, int cap) { return links_setup(ext, cap); }

// A batch with any member on the Galilean-invariant exchange takes the GI
// kernels; each instance still follows its own setting.
template <typename T>
static void links_launch_batch(const lbm_batch_s *b, int P, size_t smem, int ext, int cap) {
    bool gi = false;
    for (int i = 0; i < b->n; ++i) gi = gi || b->m[i]->pt.gimea != 0;
    const dim3 grid(b->max_np, b->n);
    if (gi) k_links_b<T, true><<<grid, 256, smem, b->stream>>>(b->dinst, P, ext, cap);
    else k_links_b<T, false><<<grid, 256, smem, b->stream>>>(b->dinst, P, ext, cap);
}

int launch_links_batch(const lbm_batch_s *b, int P) {
    if (b->max_np == 0) return LBM_OK;
    const int ext = b->ext, cap = b->cap;
    const size_t smem = link_smem(ext, cap);
    switch (b->precision) {
        case LBM_FP32: links_launch_batch<float>(b, P, smem, ext, cap); break;
        case LBM_BF16_DEV: links_launch_batch<__nv_bfloat16>(b, P, smem, ext, cap); break;
        case LBM_FP16_DEV: links_launch_batch<__half>(b, P, smem, ext, cap); break;
        default: return LBM_ERR_ARG;
    }
    return cudaGetLastError() == cudaSuccess ? LBM_OK : LBM_ERR_CUDA;
}

}  // namespace lbm
