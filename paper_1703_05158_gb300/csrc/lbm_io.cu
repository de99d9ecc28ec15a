// Gather / scatter between the A-A storage and the natural layout of the ABI
// ([19][N] FP64 populations, FP32 density and velocity, owner ids).  The
// pre-collision population f_k(x) of the current time sits at
// in_slot(parity, k, x); values are w_k + stored deviation.
//
// The FP64 pipe runs at 1/64 of the FP32 rate: a convert and an add per
// population took 2.1x the time of the memory traffic (160^3: 293 us read,
// 274 us set; now 139 and 140, 6.7 TB/s).  Within a binade the bits of a double count its ulps, so
// w + d is an integer add to the bits of w, and f - w the difference of two
// bit patterns; whatever leaves that range (and zeros, subnormals, infinities,
// NaN) takes the FP64 operations, so every result is theirs.
#include <type_traits>

#include "lbm_internal.cuh"

namespace lbm {

// (double)d + w_k, k a direction of weight class w36 = W36.
template <int W36>
__device__ __forceinline__ double add_w(float d) {
    constexpr double w = (double)W36 / 36.0;
    constexpr int kExp = W36 == 12 ? -2 : (W36 == 2 ? -5 : -6);  // 2^kExp <= w < 2^(kExp + 1)
    const unsigned u = __float_as_uint(d), e = (u >> 23) & 255u;
    // |d| = m 2^(e - 150), an ulp of w is 2^(kExp - 52)
    const int sh = (int)e - (98 + kExp);
    const long long wb = __double_as_longlong(w);
    if ((u << 1) == 0u) return w;
    if (sh >= 0 && sh <= 29 && e != 0u) {
        const long long m = (long long)((u & 0x7fffffu) | 0x800000u) << sh;
        const long long r = wb + ((int)u < 0 ? -m : m);
        if ((int)(r >> 52) == (int)(wb >> 52)) return __longlong_as_double(r);
    }
    return w + (double)d;
}

// (float)(f - w_k).
template <int W36>
__device__ __forceinline__ float sub_w(double f) {
    constexpr double w = (double)W36 / 36.0;
    constexpr int kExp = W36 == 12 ? -2 : (W36 == 2 ? -5 : -6);
    const long long fb = __double_as_longlong(f), wb = __double_as_longlong(w);
    // the difference of two numbers of one binade is exact in FP64, and a
    // whole number of ulps: one rounding either way.  A 64-bit conversion
    // would take the FP64 pipe (421 us): the leading 32 bits with the lost
    // ones as a sticky bit round the same.
    if ((int)(fb >> 52) == (int)(wb >> 52)) {
        const long long n = fb - wb;
        const unsigned long long u = (unsigned long long)(n < 0 ? -n : n);
        const int sh = 32 - __clz((int)(unsigned)(u >> 32));  // 0 .. 20
        unsigned v = (unsigned)(u >> sh);
        v |= ((unsigned)u & ((1u << sh) - 1u)) != 0u;
        const float r = __fmul_rn(__uint2float_rn(v), __uint_as_float((unsigned)(127 + kExp - 52 + sh) << 23));
        return n < 0 ? -r : r;
    }
    return (float)(f - w);
}

// Node index -> coordinates without integer division.
struct Coords {
    FastDiv dnx, dny;
    explicit Coords(const Lat &L) : dnx((unsigned)L.nx), dny((unsigned)L.ny) {}
};

// Offset (from slot 0 of the node's storage index s) of the slot that holds
// pre-collision population K at parity P.
template <int P, int K>
__device__ __forceinline__ long long in_off(const Lat &L, const Nbr &nb) {
    return P == 0 ? K * L.S : opp(K) * L.S + nb.off(-cx(K), -cy(K), -cz(K));
}

// Compile-time loop over the directions.
template <int K = 0, typename F>
__device__ __forceinline__ void each_dir(F f) {
    if constexpr (K < Q) {
        f(std::integral_constant<int, K>());
        each_dir<K + 1>(f);
    }
}

// The output kernels also leave the status word in pinned host memory, so
// that the call's one synchronisation brings it.
__device__ __forceinline__ void post_status(const int *st, volatile int *host) {
    if (blockIdx.x == 0 && threadIdx.x == 0) *host = *st;
}

template <typename T, int P>
__global__ void __launch_bounds__(256) k_get_populations(const Lat L, const Coords C, const T *__restrict__ f,
                                                         const uint8_t *__restrict__ flag, double *__restrict__ out,
                                                         const int *st, int *host) {
    post_status(st, host);
    const int n = blockIdx.x * 256 + threadIdx.x;
    if (n >= L.N) return;
    const int row = (int)C.dnx.div((unsigned)n), z = (int)C.dny.div((unsigned)row);
    const bool solid = flag[n] & 1;
    const Nbr nb(L, n - row * L.nx, row - z * L.ny);
    const T *a = f + (n + L.plane);
    float d[Q];
    each_dir([&](auto k) { d[k] = Store<T>::ld(a + in_off<P, k>(L, nb)); });
    each_dir([&](auto k) { __stcs(out + (k * L.N + n), solid ? 0.0 : add_w<w36(k)>(d[k])); });
}

template <typename T, int P>
__global__ void __launch_bounds__(256) k_set_populations(const Lat L, const Coords C, T *__restrict__ f,
                                                         const uint8_t *__restrict__ flag,
                                                         const double *__restrict__ in) {
    const int n = blockIdx.x * 256 + threadIdx.x;
    if (n >= L.N) return;
    if (flag[n] & 1) return;
    const int row = (int)C.dnx.div((unsigned)n), z = (int)C.dny.div((unsigned)row);
    const Nbr nb(L, n - row * L.nx, row - z * L.ny);
    T *a = f + (n + L.plane);
    double v[Q];
    each_dir([&](auto k) { v[k] = __ldcs(in + (k * L.N + n)); });
    each_dir([&](auto k) { Store<T>::st(a + in_off<P, k>(L, nb), sub_w<w36(k)>(v[k])); });
}

template <typename T, int P>
__global__ void __launch_bounds__(256) k_fields(const Lat L, const Coords C, const Phys ph, const T *__restrict__ f,
                                                const uint8_t *__restrict__ flag, float *__restrict__ rho,
                                                float *__restrict__ u, const int *st, int *host) {
    post_status(st, host);
    const int n = blockIdx.x * 256 + threadIdx.x;
    if (n >= L.N) return;
    float r = 0.f, ux = 0.f, uy = 0.f, uz = 0.f;
    if (!(flag[n] & 1)) {
        const int row = (int)C.dnx.div((unsigned)n), z = (int)C.dny.div((unsigned)row);
        const Nbr nb(L, n - row * L.nx, row - z * L.ny);
        const T *a = f + (n + L.plane);
        float d[Q];
        each_dir([&](auto k) { d[k] = Store<T>::ld(a + in_off<P, k>(L, nb)); });
        float dr = 0.f, jx = 0.f, jy = 0.f, jz = 0.f;
        each_dir([&](auto k) {
            dr += d[k];
            jx += cx(k) * d[k];
            jy += cy(k) * d[k];
            jz += cz(k) * d[k];
        });
        r = 1.f + dr;
        ux = jx / r + 0.5f * ph.g[0];
        uy = jy / r + 0.5f * ph.g[1];
        uz = jz / r + 0.5f * ph.g[2];
    }
    if (rho) rho[n] = r;
    if (u) {
        u[n] = ux;
        u[L.N + n] = uy;
        u[2 * L.N + n] = uz;
    }
}

__global__ void k_owner(const long long N, const uint8_t *__restrict__ flag, const int32_t *__restrict__ owner,
                        int32_t *__restrict__ out, const int *st, int *host) {
    post_status(st, host);
    const long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (n >= N) return;
    out[n] = (flag[n] & 1) ? owner[n] : -1;
}

__global__ void k_count_fluid(const Lat L, const uint8_t *__restrict__ flag, unsigned long long *__restrict__ ctr) {
    const long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const unsigned fluid = (n < L.N && !(flag[n] & 1)) ? 1u : 0u;
    const unsigned c = __popc(__ballot_sync(0xffffffffu, fluid));
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(ctr + 2, (unsigned long long)c);
}

// Loads and state of the spheres: n values per array, each array to its own
// place (null: skipped).  One launch where five small copies took about 10 us
// each (one sphere, idle stream: 58 -> 19 us per call into host arrays,
// through pinned memory).
struct StateOut {
    double *p[5];
};
__global__ void k_state(const Parts pt, const int n, const StateOut o, const int *st, int *host) {
    post_status(st, host);
    const double *src[5] = {pt.Fh, pt.Th, pt.X, pt.V, pt.W};
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
#pragma unroll
    for (int k = 0; k < 5; ++k)
        if (o.p[k]) o.p[k][i] = src[k][i];
}

// External load of the spheres from F and T (null: zero).
__global__ void k_load(const Parts pt, const int n, const double *F, const double *T) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    pt.Fx[i] = F ? F[i] : 0.0;
    pt.Tx[i] = T ? T[i] : 0.0;
}

int launch_state(lbm_s *h, double *const *out) {
    StateOut o;
    for (int k = 0; k < 5; ++k) o.p[k] = out[k];
    const int n = 3 * h->pt.np;
    k_state<<<(n + 127) / 128, 128, 0, h->stream>>>(h->pt, n, o, h->status, h->status_host);
    return cudaGetLastError() == cudaSuccess ? LBM_OK : LBM_ERR_CUDA;
}

int launch_load(lbm_s *h, const double *F, const double *T) {
    const int n = 3 * h->pt.np;
    k_load<<<(n + 127) / 128, 128, 0, h->stream>>>(h->pt, n, F, T);
    return cudaGetLastError() == cudaSuccess ? LBM_OK : LBM_ERR_CUDA;
}

static inline unsigned blocks_of(long long N) { return (unsigned)((N + 255) / 256); }

template <typename T, int P>
static void get_t(lbm_s *h, double *out) {
    k_get_populations<T, P><<<blocks_of(h->L.N), 256, 0, h->stream>>>(h->L, Coords(h->L), (const T *)h->f, h->flag, out,
                                                                      h->status, h->status_host);
}
template <typename T, int P>
static void set_t(lbm_s *h, const double *in) {
    k_set_populations<T, P><<<blocks_of(h->L.N), 256, 0, h->stream>>>(h->L, Coords(h->L), (T *)h->f, h->flag, in);
}
template <typename T, int P>
static void fields_t(lbm_s *h, float *rho, float *u) {
    k_fields<T, P><<<blocks_of(h->L.N), 256, 0, h->stream>>>(h->L, Coords(h->L), h->ph, (const T *)h->f, h->flag, rho, u,
                                                             h->status, h->status_host);
}

// fn<T, P>(args) for the handle's storage type and parity P.
#define LBM_BY_TYPE(fn, ...)                                                                        \
    switch (h->precision) {                                                                         \
        case LBM_FP32: P ? fn<float, 1>(__VA_ARGS__) : fn<float, 0>(__VA_ARGS__); break;            \
        case LBM_BF16_DEV: P ? fn<__nv_bfloat16, 1>(__VA_ARGS__) : fn<__nv_bfloat16, 0>(__VA_ARGS__); break; \
        case LBM_FP16_DEV: P ? fn<__half, 1>(__VA_ARGS__) : fn<__half, 0>(__VA_ARGS__); break;      \
        default: return LBM_ERR_ARG;                                                                \
    }                                                                                               \
    return cudaGetLastError() == cudaSuccess ? LBM_OK : LBM_ERR_CUDA

int launch_get_populations(lbm_s *h, double *out, int P) { LBM_BY_TYPE(get_t, h, out); }

int launch_set_populations(lbm_s *h, const double *in, int P) { LBM_BY_TYPE(set_t, h, in); }

int launch_fields(lbm_s *h, float *rho, float *u, int P) { LBM_BY_TYPE(fields_t, h, rho, u); }

int launch_owner(lbm_s *h, int32_t *out) {
    k_owner<<<blocks_of(h->L.N), 256, 0, h->stream>>>(h->L.N, h->flag, h->owner, out, h->status, h->status_host);
    return cudaGetLastError() == cudaSuccess ? LBM_OK : LBM_ERR_CUDA;
}

int launch_count_fluid(lbm_s *h) {
    k_count_fluid<<<blocks_of(h->L.N), 256, 0, h->stream>>>(h->L, h->flag, h->ctr);
    return cudaGetLastError() == cudaSuccess ? LBM_OK : LBM_ERR_CUDA;
}

}  // namespace lbm
