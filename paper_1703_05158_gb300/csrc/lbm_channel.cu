// Differentiation form: the mean plate drag of a channel flow and its
// gradient by a hand-written adjoint (reverse) of the stream-collide step
// with bounce-back, with checkpoint and recompute.
//
// Problem (lattice units).  D3Q19, x from an inlet plane (x = 0) to an
// outlet plane (x = nx - 1), y periodic, halfway walls at z = -1/2 and
// nz - 1/2, a fixed plate (node box) and fixed spheres.  Step s = 1 .. S:
//   f^s = P(G^{s-1}):  streaming (Eq. 13) into interior fluid nodes, with
//        bounce-back on cut links: walls and plate q = 1/2, spheres Bouzidi
//        (Eq. 19) with q the smallest root of |x + q c_j - X| = R, all at
//        rest; inlet nodes f = f^eq(rho(1, y, z), u_in(z)), u_in = u_peak
//        4 zh (1 - zh) x^, zh = (z + 1/2)/nz; outlet nodes f = f^eq(1,
//        u(nx - 2, y, z)) with u the force-shifted velocity of Eq. (6);
//   G^s = C(f^s):  the collision of the production kernels (collide_node:
//        BGK, Smagorinsky tau of Eq. 18, Guo source) at interior fluid
//        nodes; G = f at inlet and outlet nodes;
//   D^s = sum over plate links (x, j) of (G_j^s(x) + f_opp(j)^{s+1}(x)) c_j,x
//        = 2 G_j^s(x) c_j,x (momentum exchange, Eq. 25, on a halfway wall).
// f^0 = w (rest), J = mean of D^s over s in [avg_from, S], and the gradient
// is taken with respect to theta = (u_peak, g_x, C).
//
// Populations are stored as FP32 deviations from w, like the production
// path; the pull rules are affine with weights summing to 1 and w_opp(j) =
// w_j, so they apply to deviations unchanged.  Geometry (node classes and
// link fractions) is decided once in FP64 with round-to-nearest intrinsics
// in the order the FP64 oracle uses, so both classify every node alike.
//
// Reverse.  With lambda^s = dJ/df^s and gbar^s = dJ/dG^s:
//   gbar^s = (dD^s/dG^s) [s in the window] / n + P'(G^s)^T lambda^{s+1}
//   lambda^s = C'(f^s)^T gbar^s  (identity at inlet and outlet nodes)
//   dJ/dtheta = sum_s gbar^s . dC/dtheta + lambda^{s+1} . dP/dtheta
// Cut links.  A pull of interior fluid node x along a cut link c_j would read
// population i = opp(j) of the solid node (or wall ghost) x + c_j: a slot no
// node owns.  Before each step one thread per cut link (k_chan_flinks) puts
// the bounced-back population there, so the step itself is a plain pull of
// 19 slots.  The reverse step gathers lambda_i at x + c_i, the transpose of
// that pull; before it, one thread per cut link (k_chan_rlinks) applies the
// transpose of the bounce-back to lambda^{s+1} in place (see k_chan_lists),
// so the gather is as plain.  The geometry is fixed, so both lists are made
// once.  C^T is the analytic vector-Jacobian product of collide_node
// (chan_collide_vjp).  The forward run keeps f^s every K steps; the reverse
// sweep recomputes each K-step segment from its checkpoint, keeping its f^s,
// and runs the segment backwards.  The planes next to the inlet and outlet
// ride in edge blocks of the same launches, which also do the inlet / outlet
// equilibria of a forward step and add their adjoint to lambda^s of a reverse
// step.  Parameter gradients are summed per warp into the warp's own slots
// and added up once at the end of the sweep.
#include <cmath>
#include <vector>

#include "lbm_collide_node.cuh"
#include "lbm_sum.cuh"

namespace lbm {
namespace {

enum : uint8_t { CH_FLUID = 0, CH_SOLID = 1, CH_INLET = 2, CH_OUTLET = 3, CH_PLATE = 4 };

// Populations G and adjoints lambda have one ghost plane below z = 0 and one
// above z = nz - 1 (the slots of the wall links) and slot stride Ng; the
// recorded states f^s are [Q][N].
struct ChanGeo {
    int nx, ny, nz, N;
    int plane;              // nx ny
    size_t Ng;              // nx ny (nz + 2)
    const uint8_t *type;    // [N] node class
    const uint32_t *plate;  // [N]: bit j set if x -> x + c_j ends in the plate
};

__device__ __forceinline__ int wrapy(int y, int ny) { return y < 0 ? y + ny : (y >= ny ? y - ny : y); }

__device__ __forceinline__ bool is_fluid_type(uint8_t t) { return t != CH_SOLID && t != CH_PLATE; }

// ---- geometry ---------------------------------------------------------------

__device__ __forceinline__ double offs(double xi, double Xc, int n, bool periodic) {
    double d = __dsub_rn(xi, Xc);
    if (periodic) {
        if (d > 0.5 * n) d = __dsub_rn(d, (double)n);
        if (d < -0.5 * n) d = __dadd_rn(d, (double)n);
    }
    return d;
}

__device__ __forceinline__ double sq3(double a, double b, double c) {
    return __dadd_rn(__dadd_rn(__dmul_rn(a, a), __dmul_rn(b, b)), __dmul_rn(c, c));
}

__device__ __forceinline__ bool in_box(const int *lo, const int *hi, int x, int y, int z) {
    return x >= lo[0] && x <= hi[0] && y >= lo[1] && y <= hi[1] && z >= lo[2] && z <= hi[2];
}

struct PlateBox {
    int lo[3], hi[3];
};

__device__ uint8_t node_type(int nx, int ny, int x, int y, int z, const PlateBox &pb, int np, const double *X,
                             const double *R) {
    if (x == 0) return CH_INLET;
    if (x == nx - 1) return CH_OUTLET;
    if (in_box(pb.lo, pb.hi, x, y, z)) return CH_PLATE;
    for (int a = 0; a < np; ++a) {
        const double dx = offs(x, X[3 * a], nx, false), dy = offs(y, X[3 * a + 1], ny, true);
        const double dz = __dsub_rn((double)z, X[3 * a + 2]);
        if (sq3(dx, dy, dz) < __dmul_rn(R[a], R[a])) return CH_SOLID;
    }
    return CH_FLUID;
}

__global__ void k_chan_types(const int nx, const int ny, const int nz, const PlateBox pb, const int np,
                             const double *__restrict__ X, const double *__restrict__ R, uint8_t *__restrict__ type) {
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= nx * ny * nz) return;
    const int x = n % nx, y = (n / nx) % ny, z = n / (nx * ny);
    type[n] = node_type(nx, ny, x, y, z, pb, np, X, R);
}

// Cut links of every fluid node (the branch q < 1/2 is decided in FP64 and
// kept when q is rounded to FP32).  A link with q < 1/2 whose second point
// x - c_j is not fluid takes the halfway rule f = G_j(x), which is the
// q >= 1/2 rule at q = 1/2 exactly, so it is stored as q = 1/2.
__global__ void k_chan_links(const int nx, const int ny, const int nz, const int np, const double *__restrict__ X,
                             const double *__restrict__ R, const uint8_t *__restrict__ type, float *__restrict__ qout,
                             uint32_t *__restrict__ plate) {
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    const int N = nx * ny * nz;
    if (n >= N) return;
    const int x = n % nx, y = (n / nx) % ny, z = n / (nx * ny);
    uint32_t pm = 0;
    qout[n] = -1.f;  // j = 0
    for (int j = 1; j < Q; ++j) {
        float qf = -1.f;
        if (is_fluid_type(type[n])) {
            const int xx = x + rcx(j), zz = z + rcz(j);
            if (zz < 0 || zz >= nz) {
                qf = 0.5f;
            } else if (xx >= 0 && xx < nx) {
                const int m = xx + nx * (wrapy(y + rcy(j), ny) + ny * zz);
                if (type[m] == CH_PLATE) {
                    qf = 0.5f;
                    pm |= 1u << j;
                } else if (type[m] == CH_SOLID) {
                    double best = 2.0;
                    for (int a = 0; a < np; ++a) {
                        const double dx = offs(x, X[3 * a], nx, false), dy = offs(y, X[3 * a + 1], ny, true);
                        const double dz = __dsub_rn((double)z, X[3 * a + 2]);
                        const double ex = __dadd_rn(dx, (double)rcx(j)), ey = __dadd_rn(dy, (double)rcy(j));
                        const double ez = __dadd_rn(dz, (double)rcz(j));
                        if (!(sq3(ex, ey, ez) < __dmul_rn(R[a], R[a]))) continue;
                        const double aa = (double)(rcx(j) * rcx(j) + rcy(j) * rcy(j) + rcz(j) * rcz(j));
                        const double b = __dadd_rn(__dadd_rn(rcx(j) * dx, rcy(j) * dy), rcz(j) * dz);
                        const double c0 = __dsub_rn(sq3(dx, dy, dz), __dmul_rn(R[a], R[a]));
                        double disc = __dsub_rn(__dmul_rn(b, b), __dmul_rn(aa, c0));
                        if (disc < 0.0) disc = 0.0;
                        const double t = __ddiv_rn(c0, __dadd_rn(-b, __dsqrt_rn(disc)));
                        if (t < best) best = t;
                    }
                    if (best > 1.0) best = 1.0;
                    if (best < 0.0) best = 0.0;
                    qf = (float)best;
                    if (best < 0.5 && !(qf < 0.5f)) qf = 0.49999997f;  // keep the FP64 branch
                    const int bx = x - rcx(j), bz = z - rcz(j);
                    const bool second = bx >= 0 && bx < nx && bz >= 0 && bz < nz &&
                                        is_fluid_type(type[bx + nx * (wrapy(y - rcy(j), ny) + ny * bz)]);
                    if (!second && qf < 0.5f) qf = 0.5f;
                }
            }
        }
        qout[(size_t)j * N + n] = qf;
    }
    plate[n] = pm;
}

// The cut links of the interior fluid nodes as lists, grouped by direction
// (count[j] links along c_j; FILL places them from cursor[j] on; the order
// within a direction does not matter, no two records of a list write the
// same slot).  Slots are element indices i Ng + storage index.
//
// Forward record of link (x, j), i = opp(j): f_i(x) from G_j(x) and either
// G_j(x2), x2 = x - c_j (q < 1/2), or G_i(x): (i0, i1, the slot of i at
// x + c_j, q).
//
// Reverse record: with e = lambda_i(x) the transpose adds
//   a e to gbar_j(x),    a = 2q (q < 1/2) or 1/(2q): through the slot of j at
//                        x + c_j, which only x gathers;
//   (1-2q) e to gbar_j(x2)           (q < 1/2): through the slot of j at x;
//   (2q-1)/(2q) e to gbar_i(x)       (q > 1/2): through the slot of i at x2.
// A slot is gathered by one node, and e is never one of the slots written
// (x + c_j is not fluid), so the records are independent but for two cases,
// which the record of the q > 1/2 link leaves to a special record (value
// c0 lambda[s0] + c1 lambda[s1], added to the slot or assigned):
//   x2 is not an interior fluid node: the slot of i at x2 carries nothing,
//     or the a e of the link (x, i);
//   the link (x2, i) is cut with q < 1/2 and adds to the same slot.
struct ChanSpecial {
    uint32_t dst, s0, s1;
    float c0, c1;
    int add;
};
constexpr uint32_t kNoSlot = 0xffffffffu;

template <bool FILL>
__global__ void k_chan_lists(const ChanGeo G, const float *__restrict__ q, uint32_t *__restrict__ cursor,
                             uint4 *__restrict__ fl, uint4 *__restrict__ rl, ChanSpecial *__restrict__ sp) {
    const int n = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
    const bool in = n < G.N && G.type[n < G.N ? n : 0] == CH_FLUID;
    const int x = n % G.nx, y = (n / G.nx) % G.ny, z = n / G.plane;
    auto qof = [&](int j, int m) { return q[(size_t)j * G.N + m]; };
    auto slot = [&](int i, int xx, int yy, int zz) {
        return (uint32_t)((size_t)i * G.Ng + xx + (size_t)G.nx * (wrapy(yy, G.ny) + (size_t)G.ny * (zz + 1)));
    };
    for (int j = 1; j < Q; ++j) {
        const float qj = in ? qof(j, n) : -1.f;
        const unsigned bal = __ballot_sync(0xffffffffu, qj >= 0.f);
        if (bal) {
            uint32_t base = 0;
            if (lane == 0) base = atomicAdd(cursor + j, (uint32_t)__popc(bal));
            base = __shfl_sync(0xffffffffu, base, 0);
            if (qj >= 0.f) {
                const int i = ropp(j), x2 = x - rcx(j), y2 = y - rcy(j), z2 = z - rcz(j);
                const bool box2 = z2 >= 0 && z2 < G.nz;  // x2 in [0, nx): x is interior
                const int n2 = box2 ? x2 + G.nx * (wrapy(y2, G.ny) + G.ny * z2) : -1;
                const bool fluid2 = box2 && G.type[n2] == CH_FLUID;
                const float qi = qof(i, n);               // the link (x, i)
                const float q2 = fluid2 ? qof(i, n2) : -1.f;  // the link (x2, i)
                const bool low = qj < 0.5f, high = qj > 0.5f;
                // the slot (i, x2) of a high link is special (see above)
                const bool special = high && (!fluid2 || (q2 >= 0.f && q2 < 0.5f));
                if (special) {
                    const uint32_t k = atomicAdd(cursor, 1u);
                    if (FILL) {
                        ChanSpecial r;
                        r.dst = slot(i, x2, y2, z2);
                        r.s1 = slot(i, x, y, z);
                        r.c1 = __fdiv_rn(2.f * qj - 1.f, 2.f * qj);
                        r.add = fluid2;
                        r.s0 = fluid2 ? slot(j, x2, y2, z2) : slot(j, x, y, z);
                        r.c0 = fluid2 ? 1.f - 2.f * q2
                                      : (qi < 0.f ? 0.f : (qi < 0.5f ? 2.f * qi : __fdiv_rn(1.f, 2.f * qi)));
                        sp[k] = r;
                    }
                }
                if (FILL) {
                    const uint32_t k = base + __popc(bal & ((1u << lane) - 1u));
                    const uint32_t here = slot(j, x, y, z);
                    const uint32_t second = low ? slot(j, x2, y2, z2) : (high ? slot(i, x, y, z) : here);
                    fl[k] = make_uint4(here, second, slot(i, x + rcx(j), y + rcy(j), z + rcz(j)), __float_as_uint(qj));
                    // x + c_j is not fluid: the link (x, i), if cut with q > 1/2, has a special record for this slot
                    const uint32_t da = qi > 0.5f ? kNoSlot : slot(j, x + rcx(j), y + rcy(j), z + rcz(j));
                    // the link (x2, i), if cut with q > 1/2, has a special record for the slot (j, x) of a low link
                    const uint32_t du = low ? (q2 > 0.5f ? kNoSlot : here)
                                            : (high && !special ? slot(i, x2, y2, z2) : kNoSlot);
                    rl[k] = make_uint4(slot(i, x, y, z), da, du, __float_as_uint(qj));
                }
            }
        }
    }
}

// ---- forward -----------------------------------------------------------------

// Deviation of f^eq_i(rho, u) (Eq. 9) from w_i.
__device__ __forceinline__ float feq_dev(int i, float rho, float ux, float uy, float uz) {
    const float cu = rcx(i) * ux + rcy(i) * uy + rcz(i) * uz, uu = ux * ux + uy * uy + uz * uz;
    const float w = (float)rw36(i) / 36.f;
    return w * (rho * (1.f + 3.f * cu + 4.5f * cu * cu - 1.5f * uu) - 1.f);
}

__device__ __forceinline__ void moments(const float *d, float &rho, float &jx, float &jy, float &jz) {
    rho = 1.f;
    jx = jy = jz = 0.f;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        rho += d[i];
        jx += rcx(i) * d[i];
        jy += rcy(i) * d[i];
        jz += rcz(i) * d[i];
    }
}

// Warp sums of three values added to the warp's own slots dst[0..2] (the
// same warp of the same block adds to them every reverse step, on one
// stream; no block barrier).
__device__ __forceinline__ void warp_part(double a, double b, double c, double *dst) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
        c += __shfl_xor_sync(0xffffffffu, c, o);
    }
    if ((threadIdx.x & 31) == 0) {
        dst[0] += a;
        dst[1] += b;
        dst[2] += c;
    }
}

// Warp sum of a plate-drag contribution, one FP64 atomic per warp that has
// any (most warps have none).
__device__ __forceinline__ void warp_add(double v, double *dst) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0 && v != 0.0) atomicAdd(dst, v);
}

// Launch shape of the per-node kernels: a block covers kChanTx consecutive
// nodes of one x row; grid (ceil(nx / kChanTx), ny, nz), so that (x, y, z)
// come from the block and thread indices without integer division.
constexpr int kChanTx = 128;
// Resident blocks per SM of k_chan_step and k_chan_adj.  With the cut links
// in kernels of their own both are straight code that waits on its 19 (38)
// loads, and fewer blocks without spills win: 128x64x64 nodes, 200 spheres,
// 500 steps, ms per gradient with step / adj at 6 / 4 blocks 43.4, 6 / 5
// 43.4, 6 / 6 42.6, 5 / 5 43.4, 7 / 5 44.3; before the inlet and outlet rows
// moved into the collision's adjoint 12 / 10 took 71.3, 6 / 6 51.4, 5 / 5
// 50.2 (the links tested per direction inside the node kernels: 110.8; walked
// per node: 79 at best).  Recorded states are written and read once, dozens
// of steps apart: streaming stores and loads keep them from evicting G and
// lambda (2 x 40 MB) from L2 (51.9 -> 51.4 ms).
#ifndef LBM_CHAN_ADJ_MINB
#define LBM_CHAN_ADJ_MINB 6
#endif
#ifndef LBM_CHAN_STEP_MINB
#define LBM_CHAN_STEP_MINB 6
#endif

// A kernel of a channel run is a programmatic dependent of the one before
// it on the stream: it may start once every block of that one has started,
// reads the static geometry of its nodes, and touches populations, adjoints
// and sums only after chan_wait (the completion of the kernel before), through
// pointers without __restrict__ (see step_wait).
__device__ __forceinline__ void chan_wait() {
    asm volatile("griddepcontrol.launch_dependents;");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// The node of a thread of the per-node kernels.  Blocks of the first
// gridDim.z - nz slabs (`edge`, dispatched first) take the nodes next to the
// inlet (x = 1) and to the outlet (x = nx - 2), one thread per (side, y, z);
// the others one node each of the lattice, from the top plane down where down
// is set: steps alternate, so that one begins with the planes the step before
// ended with, which are still in L2 (a gradient of 500 steps at 128x64x64, whose
// states of 40 MB do not all fit, 42.6 -> 41.7 ms; 48x20x24 the same).
struct ChanNode {
    int x, y, z, n;
    int ym, yp;  // element offsets of y - 1 and y + 1 (periodic)
    bool edge, in;
    __device__ __forceinline__ ChanNode(const ChanGeo &G, const int down) {
        const int ex = (int)gridDim.z - G.nz;
        edge = (int)blockIdx.z < ex;
        if (edge) {
            const int P = G.ny * G.nz;
            const int k = ((blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x) * kChanTx + threadIdx.x;
            const int yz = k < P ? k : k - P;
            in = k < 2 * P;
            x = k < P ? 1 : G.nx - 2;
            z = yz / G.ny;
            y = yz - z * G.ny;
        } else {
            x = blockIdx.x * kChanTx + threadIdx.x;
            y = blockIdx.y;
            z = (int)blockIdx.z - ex;
            if (down) z = G.nz - 1 - z;
            in = x < G.nx;
        }
        n = x + G.nx * (y + G.ny * z);
        ym = y == 0 ? G.nx * (G.ny - 1) : -G.nx;
        yp = y == G.ny - 1 ? -G.nx * (G.ny - 1) : G.nx;
    }
    // element offset of x + s c_i (s = +1 or -1)
    __device__ __forceinline__ int off(const ChanGeo &G, int i, int s) const {
        const int dy = s * cy(i);
        return s * cx(i) + (dy > 0 ? yp : (dy < 0 ? ym : 0)) + s * cz(i) * G.plane;
    }
};

// The bounced-back population of each cut link (Eq. 19), into the slot that
// the node's pull reads: f_i(x) = 2q G_j(x) + (1-2q) G_j(x - c_j) for q < 1/2,
// else G_j(x)/(2q) + (2q-1)/(2q) G_i(x), i = opp(j).
constexpr int kLinkTx = 128;
__global__ void __launch_bounds__(kLinkTx) k_chan_flinks(const uint4 *__restrict__ list, const int count,
                                                         float *G) {
    const int t = blockIdx.x * kLinkTx + threadIdx.x;
    const uint4 r = t < count ? list[t] : make_uint4(0u, 0u, 0u, 0u);
    chan_wait();
    if (t >= count) return;
    const float g0 = G[r.x], g1 = G[r.y], q = __uint_as_float(r.w), q2 = 2.f * q;
    G[r.z] = q < 0.5f ? __fmaf_rn(q2, g0, __fmul_rn(__fsub_rn(1.f, q2), g1))
                      : __fmaf_rn(__fdiv_rn(__fsub_rn(q2, 1.f), q2), g1, __fdiv_rn(g0, q2));
}

// One step at the interior fluid nodes (PULL: f^s pulled from G^{s-1}) or at
// every fluid node (!PULL: f^s = fin, the stored state): record f^s in frec
// (may be null), G^s = C(f^s) into Gout (G = f at inlet and outlet nodes),
// plate drag of G^s added to *drag (may be null).  With PULL the launch's
// edge blocks (see ChanNode) pull at the planes next to the inlet and the
// outlet as well and write the equilibria of Eq. (9) at the inlet (x = 0) and
// outlet (x = nx - 1) nodes; G = f there.
template <bool PULL>
__global__ void __launch_bounds__(kChanTx, LBM_CHAN_STEP_MINB) k_chan_step(const ChanGeo G, const Phys ph, const float u_peak,
                                                       const float *Gin, const float *fin, float *frec, float *Gout,
                                                       double *drag, int *status, const int down) {
    const ChanNode c(G, down);
    const int n = c.n;
    const uint8_t t = c.in ? G.type[n] : (uint8_t)CH_SOLID;
    const bool live = PULL ? t == CH_FLUID : is_fluid_type(t);
    const uint32_t pm = live && drag ? G.plate[n] : 0u;
    chan_wait();
    double D = 0.0;
    if (live) {
        float d[Q];
        if (!PULL) {
#pragma unroll
            for (int i = 0; i < Q; ++i) d[i] = fin[(size_t)i * G.N + n];
        } else {
#pragma unroll
            for (int i = 0; i < Q; ++i) d[i] = Gin[i * G.Ng + (n + G.plane + c.off(G, i, -1))];
        }
        if (PULL && c.edge) {
            float rho, jx, jy, jz;
            moments(d, rho, jx, jy, jz);
            if (c.x == 1) {
                const float zh = (c.z + 0.5f) / G.nz;
                const float ux = u_peak * 4.f * zh * (1.f - zh);
#pragma unroll
                for (int i = 0; i < Q; ++i) d[i] = feq_dev(i, rho, ux, 0.f, 0.f);
            } else {
                const float ux = jx / rho + 0.5f * ph.g[0], uy = jy / rho + 0.5f * ph.g[1], uz = jz / rho + 0.5f * ph.g[2];
#pragma unroll
                for (int i = 0; i < Q; ++i) d[i] = feq_dev(i, 1.f, ux, uy, uz);
            }
            const int nb = c.x == 1 ? n - 1 : n + 1;  // the inlet or outlet node
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                if (frec) __stcs(frec + (size_t)i * G.N + nb, d[i]);
                Gout[i * G.Ng + (nb + G.plane)] = d[i];
            }
        } else {
            if (frec)
#pragma unroll
                for (int i = 0; i < Q; ++i) __stcs(frec + (size_t)i * G.N + n, d[i]);
            if (t == CH_FLUID) collide_node(ph, d, status);
#pragma unroll
            for (int i = 0; i < Q; ++i) Gout[i * G.Ng + (n + G.plane)] = d[i];
            if (pm && !c.edge)
#pragma unroll
                for (int j = 1; j < Q; ++j)
                    if (((pm >> j) & 1u) && rcx(j) != 0)
                        D += 2.0 * rcx(j) * ((double)d[j] + (double)rw36(j) / 36.0);
        }
    }
    if (__any_sync(0xffffffffu, pm != 0u)) warp_add(D, drag);
}

// ---- reverse -----------------------------------------------------------------

// The adjoint of the inlet or outlet row of P at step s that ends at fluid
// node n, given lambda^s at the row's inlet or outlet node (row): that node's
// populations are read by the pulls of the five directions with c_x = side
// only (x = 1 and x = nx - 2 hold interior fluid nodes only).  Both depend on
// the populations at n through rho and j alone, so the row adds a part equal
// in all directions (all) and one proportional to c_i (dir) to lambda^s at n,
// where the gathers of step s - 1 find it.
//
// Written as additions to what the collision's adjoint had just stored, the
// row read f^s (19 loads), then lambda^s (19 loads) again and stored it
// twice, in the blocks that the launch waits for: a reverse step of 48x20x24
// nodes (with its share of the recomputed forward run) took 26.9 us and then,
// with the row inside the collision's adjoint, 17.2 us, 79.9 and 64.6 us for
// 128x64x64 nodes (17.7 and 62.2 now).
constexpr int kRow = 5;  // directions with c_x = 1 (or -1)
struct RowBar {
    float all = 0.f, dir[3] = {0.f, 0.f, 0.f};
    double gup = 0.0, ggx = 0.0;  // the row's parts of dJ/du_peak and dJ/dg_x
};

// inlet: f_i(0) = rho_1 fe_i(1, u_in)
__device__ __forceinline__ void fold_inlet(const ChanGeo &G, const float u_peak, const float (&row)[kRow], const int z,
                                           const float rho1, RowBar &r) {
    const float zh = (z + 0.5f) / G.nz, sh = 4.f * zh * (1.f - zh), ux = u_peak * sh;
    float ub = 0.f;
    int k = 0;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        if (cx(i) != 1) continue;
        const float w = (float)rw36(i) / 36.f, cu = rcx(i) * ux, l = row[k++];
        r.all += l * w * (1.f + 3.f * cu + 4.5f * cu * cu - 1.5f * ux * ux);
        ub += l * w * (3.f * rcx(i) + 9.f * cu * rcx(i) - 3.f * ux);
    }
    r.gup = (double)ub * rho1 * sh;
}

// outlet: f_i(nx-1) = f^eq_i(1, u(nx-2)), u = j / rho + g / 2 (1 / rho rounded,
// not the approximate one of the collision's adjoint)
__device__ __forceinline__ void fold_outlet(const Phys &ph, const float (&row)[kRow], const float (&j)[3],
                                            const float rho, RowBar &r) {
    const float ir = __fdiv_rn(1.f, rho);
    const float u[3] = {j[0] * ir + 0.5f * ph.g[0], j[1] * ir + 0.5f * ph.g[1], j[2] * ir + 0.5f * ph.g[2]};
    float uba[3] = {0.f, 0.f, 0.f};
    int k = 0;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        if (cx(i) != -1) continue;
        const float w = (float)rw36(i) / 36.f, l = row[k++];
        const float cu = rcx(i) * u[0] + rcy(i) * u[1] + rcz(i) * u[2];
        uba[0] += l * w * (3.f * rcx(i) + 9.f * cu * rcx(i) - 3.f * u[0]);
        uba[1] += l * w * (3.f * rcy(i) + 9.f * cu * rcy(i) - 3.f * u[1]);
        uba[2] += l * w * (3.f * rcz(i) + 9.f * cu * rcz(i) - 3.f * u[2]);
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        r.dir[a] = ir * uba[a];
        r.all -= r.dir[a] * (j[a] * ir);
    }
    r.ggx = 0.5 * (double)uba[0];
}

// Vector-Jacobian product of collide_node at deviations d: lam = C'(d)^T gb,
// and the products with dC/dg_x and dC/dsmag (smag = 18 sqrt(2) C^2).
//
// The collision is g_k = (1 - om) d_k + om E_k + sk S_k with
//   E_k = w_k (drho - 1.5 rho u.u + 4.5 rho (c_k.u)^2 + 3 rho c_k.u),
//   S_k = w_k rho g_x (3 c_kx - 3 u_x + 9 (c_k.u) c_kx),  sk = 1 - om/2,
// and E, S and om depend on d only through drho, j and Pi.  So every sum
// over k that the chain rule needs is a moment of gb: with
//   N0 = sum w_k gb_k,  N1 = sum w_k gb_k c_k,  N2 = sum w_k gb_k c_k c_k,
// sum w gb (c.u) = u.N1, sum w gb (c.u)^2 = u.N2.u, sum w gb (c.u) c = N2 u.
// The result is lam_i = (1 - om) gb_i + A + B.c_i + M:c_i c_i, taken by
// opposite pairs (i, i + 9) like the forward collision.  Divisions and
// square roots use the hardware approximations (a few ulp): the adjoint
// only has to carry the gradient to well within its 1e-3 tolerance.  The deviations are
// read pair by pair from f (slot stride N; null: the rest state) and the
// result is written to lam (slot stride Ng), so that only gb is held whole.
// side 1 (-1): n is the fluid end of the inlet (outlet) row, whose adjoint is
// added (see RowBar).
__device__ __forceinline__ void chan_collide_vjp(const ChanGeo &G, const Phys &ph, const float u_peak,
                                                 const float *__restrict__ f, const float (&gb)[Q],
                                                 float *__restrict__ lam, const int side, const float (&row)[kRow],
                                                 const int z, float &gx_bar, float &smag_bar, RowBar &rowb) {
    const size_t N = (size_t)G.N, Ng = G.Ng;
    // forward intermediates (the moments of d, by opposite pairs)
    const float d0 = f ? __ldcs(f) : 0.f;
    float drho = d0, j[3] = {0.f, 0.f, 0.f}, m[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};  // m: xx yy zz xy xz yz
    float N0 = wf(0) * gb[0], N1[3] = {0.f, 0.f, 0.f}, N2[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, gd = gb[0] * d0;
#pragma unroll
    for (int i = 1; i <= 9; ++i) {
        const int k = i + 9;  // opp(i)
        const float di = f ? __ldcs(f + i * N) : 0.f, dk = f ? __ldcs(f + k * N) : 0.f;
        const float sp = di + dk, dm = di - dk;
        const float gs = wf(i) * (gb[i] + gb[k]), gm = wf(i) * (gb[i] - gb[k]);
        drho += sp;
        N0 += gs;
        gd += gb[i] * di + gb[k] * dk;
        if (cx(i)) { j[0] += cx(i) * dm; N1[0] += cx(i) * gm; m[0] += sp; N2[0] += gs; }
        if (cy(i)) { j[1] += cy(i) * dm; N1[1] += cy(i) * gm; m[1] += sp; N2[1] += gs; }
        if (cz(i)) { j[2] += cz(i) * dm; N1[2] += cz(i) * gm; m[2] += sp; N2[2] += gs; }
        if (cx(i) * cy(i)) { m[3] += cx(i) * cy(i) * sp; N2[3] += cx(i) * cy(i) * gs; }
        if (cx(i) * cz(i)) { m[4] += cx(i) * cz(i) * sp; N2[4] += cx(i) * cz(i) * gs; }
        if (cy(i) * cz(i)) { m[5] += cy(i) * cz(i) * sp; N2[5] += cy(i) * cz(i) * gs; }
    }
    const float rho = 1.f + drho, ir = __fdividef(1.f, rho);
    const float u[3] = {j[0] * ir + 0.5f * ph.g[0], j[1] * ir + 0.5f * ph.g[1], j[2] * ir + 0.5f * ph.g[2]};
    const float uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    float P6[6], Qn = 0.f, inner = ph.tau0 * ph.tau0, tau = ph.tau0;
    const bool les = ph.smag > 0.f;
    if (les) {
        const float t3 = drho * (1.f / 3.f);
        P6[0] = m[0] - t3 - rho * u[0] * u[0];
        P6[1] = m[1] - t3 - rho * u[1] * u[1];
        P6[2] = m[2] - t3 - rho * u[2] * u[2];
        P6[3] = m[3] - rho * u[0] * u[1];
        P6[4] = m[4] - rho * u[0] * u[2];
        P6[5] = m[5] - rho * u[1] * u[2];
        const float q2 = P6[0] * P6[0] + P6[1] * P6[1] + P6[2] * P6[2] +
                         2.f * (P6[3] * P6[3] + P6[4] * P6[4] + P6[5] * P6[5]);
        Qn = q2 > 0.f ? q2 * rsqrtf(q2) : 0.f;
        inner = ph.smag * Qn * ir + ph.tau0 * ph.tau0;
        tau = ph.tau0 + 0.5f * (inner * rsqrtf(inner) - ph.tau0);
    }
    const float om = __fdividef(1.f, tau), sk = 1.f - 0.5f * om, gx = ph.g[0];
    // moments of gb contracted with u
    const float N2u[3] = {N2[0] * u[0] + N2[3] * u[1] + N2[4] * u[2], N2[3] * u[0] + N2[1] * u[1] + N2[5] * u[2],
                          N2[4] * u[0] + N2[5] * u[1] + N2[2] * u[2]};
    const float uN1 = u[0] * N1[0] + u[1] * N1[1] + u[2] * N1[2];
    const float uN2u = u[0] * N2u[0] + u[1] * N2u[1] + u[2] * N2u[2];
    const float eq = -1.5f * uu * N0 + 4.5f * uN2u + 3.f * uN1;  // sum w gb (E/w - drho)/rho
    const float sx = 3.f * N1[0] - 3.f * u[0] * N0 + 9.f * N2u[0];  // sum gb S / (rho g_x)
    // om_bar = sum gb (E - d - S/2)
    const float om_bar = drho * N0 + rho * eq - gd - 0.5f * rho * gx * sx;
    float drho_bar = om * N0;
    float rho_bar = om * eq + sk * gx * sx;
    float ub[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) ub[a] = om * rho * (-3.f * u[a] * N0 + 9.f * N2u[a] + 3.f * N1[a]);
    const float ks = sk * rho * gx;
    ub[0] += ks * (-3.f * N0 + 9.f * N2[0]);
    ub[1] += ks * 9.f * N2[3];
    ub[2] += ks * 9.f * N2[4];
    gx_bar = sk * rho * sx;
    // om = 1 / tau, tau = tau0 + (sqrt(inner) - tau0) / 2, inner = smag Q / rho + tau0^2
    float ir_bar = 0.f, mb[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    smag_bar = 0.f;
    if (les) {
        const float tau_bar = -om_bar * om * om;
        const float in_bar = tau_bar * 0.25f * rsqrtf(inner);
        smag_bar = in_bar * Qn * ir;
        ir_bar += in_bar * ph.smag * Qn;
        const float Q_bar = in_bar * ph.smag * ir;
        const float q2_bar = Qn > 0.f ? __fdividef(Q_bar, 2.f * Qn) : 0.f;
#pragma unroll
        for (int k = 0; k < 3; ++k) mb[k] = 2.f * P6[k] * q2_bar;
#pragma unroll
        for (int k = 3; k < 6; ++k) mb[k] = 4.f * P6[k] * q2_bar;
        drho_bar -= (mb[0] + mb[1] + mb[2]) * (1.f / 3.f);
        rho_bar -= mb[0] * u[0] * u[0] + mb[1] * u[1] * u[1] + mb[2] * u[2] * u[2] + mb[3] * u[0] * u[1] +
                   mb[4] * u[0] * u[2] + mb[5] * u[1] * u[2];
        ub[0] -= rho * (2.f * mb[0] * u[0] + mb[3] * u[1] + mb[4] * u[2]);
        ub[1] -= rho * (2.f * mb[1] * u[1] + mb[3] * u[0] + mb[5] * u[2]);
        ub[2] -= rho * (2.f * mb[2] * u[2] + mb[4] * u[0] + mb[5] * u[1]);
    }
    // u = j / rho + g / 2
    float jb[3] = {ub[0] * ir, ub[1] * ir, ub[2] * ir};
    ir_bar += ub[0] * j[0] + ub[1] * j[1] + ub[2] * j[2];
    gx_bar += 0.5f * ub[0];
    rho_bar -= ir_bar * ir * ir;
    float dtot = drho_bar + rho_bar;  // rho = 1 + drho
    if (side) {
        if (side > 0) fold_inlet(G, u_peak, row, z, rho, rowb);
        else fold_outlet(ph, row, j, rho, rowb);
        dtot += rowb.all;
#pragma unroll
        for (int a = 0; a < 3; ++a) jb[a] += rowb.dir[a];
    }
    const float keep = 1.f - om;
    lam[0] = keep * gb[0] + dtot;
#pragma unroll
    for (int i = 1; i <= 9; ++i) {
        const int k = i + 9;
        float even = dtot, odd = 0.f;
        if (cx(i)) { even += mb[0]; odd += cx(i) * jb[0]; }
        if (cy(i)) { even += mb[1]; odd += cy(i) * jb[1]; }
        if (cz(i)) { even += mb[2]; odd += cz(i) * jb[2]; }
        if (cx(i) * cy(i)) even += cx(i) * cy(i) * mb[3];
        if (cx(i) * cz(i)) even += cx(i) * cz(i) * mb[4];
        if (cy(i) * cz(i)) even += cy(i) * cz(i) * mb[5];
        lam[i * Ng] = keep * gb[i] + even + odd;
        lam[k * Ng] = keep * gb[k] + even - odd;
    }
}

// Transpose of the bounce-back on lambda^{s+1}, in place (see k_chan_lists):
// the list's links, then its special records.
__global__ void __launch_bounds__(kLinkTx) k_chan_rlinks(const uint4 *__restrict__ list, const int count,
                                                         const ChanSpecial *__restrict__ sp, const int nsp,
                                                         float *lam) {
    const int t = blockIdx.x * kLinkTx + threadIdx.x;
    const uint4 r = t < count ? list[t] : make_uint4(0u, kNoSlot, kNoSlot, 0u);
    chan_wait();
    if (t < count) {
        const float e = lam[r.x], q = __uint_as_float(r.w), q2 = 2.f * q;
        const float u = r.z != kNoSlot ? lam[r.z] : 0.f;
        const bool low = q < 0.5f;
        if (r.y != kNoSlot) lam[r.y] = __fmul_rn(low ? q2 : __fdiv_rn(1.f, q2), e);
        if (r.z != kNoSlot)
            lam[r.z] = __fmaf_rn(low ? __fsub_rn(1.f, q2) : __fdiv_rn(__fsub_rn(q2, 1.f), q2), e, u);
    } else if (t - count < nsp) {
        const ChanSpecial c = sp[t - count];
        const float v0 = lam[c.s0], v1 = lam[c.s1];
        const float v = c.add ? __fmaf_rn(c.c0, v0, lam[c.dst]) : __fmul_rn(c.c0, v0);
        lam[c.dst] = __fmaf_rn(c.c1, v1, v);
    }
}

// Reverse step s: lambda^s from lambda^{s+1} (lam1) and f^s (fs; null for
// the rest state f^0 = w), weight wd of D^s in J (0 outside the window).  The
// gather gbar_i(x) = lambda_i(x + c_i) is the whole transpose of the pull once
// k_chan_rlinks has run on lambda^{s+1}; lambda is 0 in the slots of nodes
// that are neither interior fluid nor the end of a cut link.  lambda^{s+1}
// also carries the adjoint of its step's inlet and outlet rows at x = 1 and
// x = nx - 2.  Those two planes are computed by the launch's edge blocks (see
// ChanNode), which with `fold` also gather lambda^s at the row's inlet or
// outlet node and fold its adjoint in for the next reverse step.  The parts
// of dJ/d(u_peak, g_x, smag) of each warp are added to its own slots over the
// steps in FP64 (no atomics): triples of the edge warps in gedge, pairs
// (g_x, smag) of the others in gpart.
__global__ void __launch_bounds__(kChanTx, LBM_CHAN_ADJ_MINB) k_chan_adj(
    const ChanGeo G, const Phys ph, const float u_peak, const float *lam1, const float *fs, const float wd,
    float *lam0, const int fold, double *gpart, double *gedge, const int down) {
    const ChanNode c(G, down);
    // the planes x = 1 and x = nx - 2 belong to the edge blocks
    const bool in = c.in && (c.edge || !(c.x == 1 || c.x == G.nx - 2));
    const int n = c.n;
    float gxb = 0.f, smb = 0.f;
    RowBar rowb;
    const bool live = in && G.type[n] == CH_FLUID;
    const uint32_t pm = live && wd != 0.f ? G.plate[n] : 0u;
    const int warp = (blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z)) * (kChanTx / 32) + (threadIdx.x >> 5);
    const int part = 2 * warp + (threadIdx.x & 1);
    chan_wait();
    const double sum0 = c.edge ? 0.0 : gpart[part];  // early: nothing hides its latency at the end
    if (live) {
        float gb[Q], row[kRow] = {0.f, 0.f, 0.f, 0.f, 0.f};
        const float *l1 = lam1 + (n + G.plane);
#pragma unroll
        for (int i = 0; i < Q; ++i) gb[i] = l1[(ptrdiff_t)(i * G.Ng) + c.off(G, i, 1)];
        const int side = !c.edge || !fold ? 0 : (c.x == 1 ? 1 : -1);  // c_x of the pulls that read the row's end
        if (side) {
            int k1 = 0, k2 = 0;
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                const float *l = l1 + (ptrdiff_t)(i * G.Ng) + c.off(G, i, 1);
                if (cx(i) == 1) {
                    if (side > 0) row[k1] = l[-1];
                    ++k1;
                }
                if (cx(i) == -1) {
                    if (side < 0) row[k2] = l[1];
                    ++k2;
                }
            }
        }
        if (pm)
#pragma unroll
            for (int i = 0; i < Q; ++i)
                if ((pm >> i) & 1u) gb[i] += wd * 2.f * rcx(i);
        chan_collide_vjp(G, ph, u_peak, fs ? fs + n : nullptr, gb, lam0 + (n + G.plane), side, row, c.z, gxb, smb, rowb);
    }
    if (c.edge) {
        warp_part(rowb.gup, rowb.ggx + (double)gxb, (double)smb, gedge + 3 * warp);
    } else {
        const double s = warp_sum2(gxb, smb);
        if ((threadIdx.x & 31) < 2) gpart[part] = sum0 + s;
    }
}

// grad[0..2] += the sums of the warps' parts: ne FP64 triples of the edge
// warps, nb pairs (g_x, smag) from warp ne on.
__global__ void __launch_bounds__(256) k_chan_gsum(const double *gedge, int ne, const double *gpart, int nb,
                                                   double *grad) {
    chan_wait();
    double a[3] = {0.0, 0.0, 0.0};
    for (int k = threadIdx.x; k < ne; k += blockDim.x)
#pragma unroll
        for (int c = 0; c < 3; ++c) a[c] += gedge[3 * k + c];
    for (int k = ne + threadIdx.x; k < ne + nb; k += blockDim.x) {
        a[1] += gpart[2 * k];
        a[2] += gpart[2 * k + 1];
    }
    __shared__ double sh[3][8];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a[c] += __shfl_xor_sync(0xffffffffu, a[c], o);
        if ((threadIdx.x & 31) == 0) sh[c][threadIdx.x >> 5] = a[c];
    }
    __syncthreads();
    if (threadIdx.x == 0)
        for (int c = 0; c < 3; ++c) {
            for (int w = 1; w < (int)(blockDim.x >> 5); ++w) a[c] += sh[c][w];
            grad[c] += a[c];
        }
}

}  // namespace
}  // namespace lbm

using namespace lbm;

struct lbm_channel_s {
    lbm_channel_params p;
    int N = 0, np = 0, K = 0, nck = 0;
    uint8_t *type = nullptr;
    uint32_t *plate = nullptr;
    uint4 *flist = nullptr, *rlist = nullptr;  // cut links of a forward / reverse step
    ChanSpecial *special = nullptr;
    int nlinks = 0, nspecial = 0;
    // per-warp parts of dJ/d(g_x, smag), of the edge warps of dJ/d(u_peak, g_x, smag) (k_chan_adj)
    double *gpart = nullptr, *gedge = nullptr;
    double *X = nullptr, *R = nullptr;
    float *G[2] = {nullptr, nullptr}, *lam[2] = {nullptr, nullptr};
    float *seg = nullptr;   // K states f^s of a segment
    float *ckpt = nullptr;  // f^s at s = 0, K, 2K, ...
    float *fend = nullptr;  // f^S of the last forward
    double *drag = nullptr, *grad = nullptr;
    int *status = nullptr;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    Phys ph{};
    double theta[3] = {0.0, 0.0, 0.0};
    bool have_forward = false;
    size_t bytes = 0;
};

namespace {

ChanGeo geo_of(const lbm_channel_s *c) {
    ChanGeo g;
    g.nx = c->p.nx;
    g.ny = c->p.ny;
    g.nz = c->p.nz;
    g.N = c->N;
    g.type = c->type;
    g.plane = c->p.nx * c->p.ny;
    g.Ng = (size_t)c->N + 2 * (size_t)g.plane;
    g.plate = c->plate;
    return g;
}

void set_phys(lbm_channel_s *c) {
    c->ph = Phys{};
    c->ph.tau0 = (float)c->p.tau0;
    c->ph.smag = (float)(18.0 * std::sqrt(2.0) * c->theta[2] * c->theta[2]);
    c->ph.g[0] = (float)c->theta[1];
}

template <typename T>
int calloc_dev(lbm_channel_s *c, T **p, size_t n) {
    *p = nullptr;
    if (n == 0) return LBM_OK;
    if (cudaMalloc((void **)p, n * sizeof(T)) != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
        return LBM_ERR_NOMEM;
    }
    c->bytes += n * sizeof(T);
    return cudaMemsetAsync(*p, 0, n * sizeof(T), c->stream) == cudaSuccess ? LBM_OK : LBM_ERR_CUDA;
}

void chan_release(lbm_channel_s *c) {
    void *ptrs[] = {c->type, c->plate, c->flist, c->rlist, c->special, c->gpart, c->gedge, c->X, c->R, c->G[0], c->G[1], c->lam[0],
                    c->lam[1], c->seg, c->ckpt, c->fend, c->drag, c->grad, c->status};
    for (void *p : ptrs)
        if (p) cudaFree(p);
    if (c->own_stream && c->stream) cudaStreamDestroy(c->stream);
}

int chan_check(lbm_channel_s *c, int rc) {
    if (rc) {
        cudaGetLastError();
        return rc;
    }
    if (cudaStreamSynchronize(c->stream) != cudaSuccess) {
        cudaGetLastError();
        return LBM_ERR_CUDA;
    }
    int st = 0;
    if (cudaMemcpy(&st, c->status, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) {
        cudaGetLastError();
        return LBM_ERR_CUDA;
    }
    return (st & ST_DIVERGED) ? LBM_ERR_DIVERGED : LBM_OK;
}

int launch_ok() { return cudaGetLastError() == cudaSuccess ? LBM_OK : LBM_ERR_CUDA; }

// Slabs of edge blocks that lead the grid of a per-node launch (see ChanNode),
// their warps, and the grid.
int chan_slabs(const lbm_channel_params &p) {
    const long long per_slab = (long long)((p.nx + kChanTx - 1) / kChanTx) * p.ny * kChanTx, rows = 2ll * p.ny * p.nz;
    return (int)((rows + per_slab - 1) / per_slab);
}
dim3 chan_grid(const lbm_channel_params &p, int slabs) {
    return dim3((unsigned)((p.nx + kChanTx - 1) / kChanTx), p.ny, p.nz + slabs);
}
int chan_warps(const lbm_channel_params &p, int slabs) {
    return (int)((p.nx + kChanTx - 1) / kChanTx) * p.ny * slabs * (kChanTx / 32);
}

// Launch of a channel kernel as a programmatic dependent of the kernel
// before it on the stream (see chan_wait).
template <typename... P, typename... A>
int chan_launch(lbm_channel_s *c, void (*k)(P...), const dim3 grid, const int threads, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.stream = c->stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k, static_cast<P>(args)...);
    if (e != cudaSuccess) cudaGetLastError();
    return e == cudaSuccess ? LBM_OK : LBM_ERR_CUDA;
}

// Forward from f^{s0} (fin) over steps s0 + 1 .. s1: f^s recorded into
// rec(s) when it returns non-null; drag of G^s into drag[s - 1] when
// with_drag.
template <typename Rec>
int chan_run(lbm_channel_s *c, const float *fin, int s0, int s1, Rec rec, bool with_drag) {
    const ChanGeo g = geo_of(c);
    const dim3 grid = chan_grid(c->p, 0), grid_edge = chan_grid(c->p, chan_slabs(c->p));
    const float up = (float)c->theta[0];
    int rc = chan_launch(c, k_chan_step<false>, grid, kChanTx, g, c->ph, up, nullptr, fin, nullptr, c->G[s0 & 1],
                         with_drag && s0 >= 1 ? c->drag + (s0 - 1) : nullptr, c->status, s0 & 1);
    for (int s = s0 + 1; s <= s1 && !rc; ++s) {
        if (c->nlinks)
            rc = chan_launch(c, k_chan_flinks, dim3((c->nlinks + kLinkTx - 1) / kLinkTx), kLinkTx, c->flist, c->nlinks,
                             c->G[(s - 1) & 1]);
        if (!rc) rc = chan_launch(c, k_chan_step<true>, grid_edge, kChanTx, g, c->ph, up, c->G[(s - 1) & 1], nullptr, rec(s),
                         c->G[s & 1], with_drag ? c->drag + (s - 1) : nullptr, c->status, s & 1);
    }
    return rc;
}

}  // namespace

extern "C" {

int lbm_channel_create(const lbm_channel_params *prm, int32_t n, const double *pos, const double *radius,
                       lbm_channel *out) {
    if (!prm || !out || n < 0 || (n > 0 && (!pos || !radius))) return LBM_ERR_ARG;
    *out = nullptr;
    const lbm_channel_params &p = *prm;
    if (p.nx < 8 || p.ny < 1 || p.nz < 2 || !(p.tau0 > 0.5) || !(p.cs_smag >= 0.0)) return LBM_ERR_ARG;
    if (!std::isfinite(p.tau0) || !std::isfinite(p.cs_smag) || !std::isfinite(p.inlet_peak) ||
        !std::isfinite(p.body_accel_x))
        return LBM_ERR_ARG;
    if (p.steps < 1 || p.avg_from < 1 || p.avg_from > p.steps || p.checkpoint_every < 1) return LBM_ERR_ARG;
    if ((long long)p.nx * p.ny * p.nz * Q >= (1ll << 31)) return LBM_ERR_UNSUPPORTED;  // kernels index [Q][N] in int
    // grid rows (y, z) of the per-node kernels, plus at most nz / 64 + 1 slabs of extra blocks in z
    if (p.ny > 65535 || p.nz > 64000) return LBM_ERR_UNSUPPORTED;
    // obstacles stay clear of the inlet / outlet planes and their neighbours
    const bool plate = p.plate_lo[0] <= p.plate_hi[0] && p.plate_lo[1] <= p.plate_hi[1] && p.plate_lo[2] <= p.plate_hi[2];
    if (plate && (p.plate_lo[0] < 2 || p.plate_hi[0] > p.nx - 3)) return LBM_ERR_ARG;
    for (int a = 0; a < n; ++a) {
        const double *X = pos + 3 * a;
        if (!(radius[a] > 0.0) || !(X[0] - radius[a] > 1.0) || !(X[0] + radius[a] < p.nx - 2.0) ||
            !std::isfinite(X[1]) || !std::isfinite(X[2]))
            return LBM_ERR_ARG;
    }
    lbm_channel_s *c = new (std::nothrow) lbm_channel_s();
    if (!c) return LBM_ERR_NOMEM;
    c->p = p;
    c->N = p.nx * p.ny * p.nz;
    c->np = n;
    c->K = p.checkpoint_every;
    c->nck = p.steps / c->K + 1;
    c->theta[0] = p.inlet_peak;
    c->theta[1] = p.body_accel_x;
    c->theta[2] = p.cs_smag;
    set_phys(c);
    DeviceScope ds(p.device);
    int rc = cudaSetDevice(p.device) == cudaSuccess ? LBM_OK : LBM_ERR_CUDA;
    if (!rc) {
        if (p.cuda_stream) {
            c->stream = (cudaStream_t)p.cuda_stream;
        } else if (cudaStreamCreateWithFlags(&c->stream, cudaStreamNonBlocking) == cudaSuccess) {
            c->own_stream = true;
        } else {
            rc = LBM_ERR_CUDA;
        }
    }
    const size_t NQs = (size_t)c->N * Q, NQg = NQs + 2 * (size_t)Q * p.nx * p.ny;
    if (!rc) rc = calloc_dev(c, &c->type, (size_t)c->N);
    if (!rc) rc = calloc_dev(c, &c->plate, (size_t)c->N);
    if (!rc) rc = calloc_dev(c, &c->gpart, 2 * (size_t)chan_warps(p, chan_slabs(p) + p.nz));
    if (!rc) rc = calloc_dev(c, &c->gedge, 3 * (size_t)chan_warps(p, chan_slabs(p)));
    if (!rc) rc = calloc_dev(c, &c->X, 3 * (size_t)n);
    if (!rc) rc = calloc_dev(c, &c->R, (size_t)n);
    for (int k = 0; k < 2 && !rc; ++k) {
        rc = calloc_dev(c, &c->G[k], NQg);
        if (!rc) rc = calloc_dev(c, &c->lam[k], NQg);
    }
    if (!rc) rc = calloc_dev(c, &c->seg, NQs * c->K);
    if (!rc) rc = calloc_dev(c, &c->ckpt, NQs * c->nck);
    if (!rc) rc = calloc_dev(c, &c->fend, NQs);
    if (!rc) rc = calloc_dev(c, &c->drag, (size_t)p.steps);
    if (!rc) rc = calloc_dev(c, &c->grad, 3);
    if (!rc) rc = calloc_dev(c, &c->status, 1);
    if (!rc && n > 0 &&
        (cudaMemcpyAsync(c->X, pos, 3 * sizeof(double) * n, cudaMemcpyHostToDevice, c->stream) != cudaSuccess ||
         cudaMemcpyAsync(c->R, radius, sizeof(double) * n, cudaMemcpyHostToDevice, c->stream) != cudaSuccess))
        rc = LBM_ERR_CUDA;
    if (!rc) {
        PlateBox pb;
        for (int k = 0; k < 3; ++k) {
            pb.lo[k] = p.plate_lo[k];
            pb.hi[k] = p.plate_hi[k];
        }
        const int blocks = (c->N + 255) / 256;
        k_chan_types<<<blocks, 256, 0, c->stream>>>(p.nx, p.ny, p.nz, pb, n, c->X, c->R, c->type);
        rc = launch_ok();
        // link fractions (a temporary), counted and then placed in the lists
        float *q = nullptr;
        uint32_t *cursor = nullptr, cnt[Q] = {};
        if (!rc && (cudaMalloc((void **)&q, sizeof(float) * NQs) != cudaSuccess ||
                    cudaMalloc((void **)&cursor, sizeof(cnt)) != cudaSuccess)) {
            cudaGetLastError();
            rc = LBM_ERR_NOMEM;
        }
        auto ok = [](cudaError_t e) { return e == cudaSuccess ? LBM_OK : LBM_ERR_CUDA; };
        const ChanGeo g = geo_of(c);
        if (!rc) {
            k_chan_links<<<blocks, 256, 0, c->stream>>>(p.nx, p.ny, p.nz, n, c->X, c->R, c->type, q, c->plate);
            rc = launch_ok();
        }
        if (!rc) rc = ok(cudaMemsetAsync(cursor, 0, sizeof(cnt), c->stream));
        if (!rc) {
            k_chan_lists<false><<<blocks, 256, 0, c->stream>>>(g, q, cursor, nullptr, nullptr, nullptr);
            rc = launch_ok();
        }
        if (!rc) rc = ok(cudaMemcpyAsync(cnt, cursor, sizeof(cnt), cudaMemcpyDeviceToHost, c->stream));
        if (!rc) rc = ok(cudaStreamSynchronize(c->stream));
        if (!rc) {
            c->nspecial = (int)cnt[0];
            uint32_t at[Q] = {};
            for (int j = 1; j < Q; ++j) at[j] = (uint32_t)c->nlinks, c->nlinks += (int)cnt[j];
            rc = calloc_dev(c, &c->flist, (size_t)c->nlinks);
            if (!rc) rc = calloc_dev(c, &c->rlist, (size_t)c->nlinks);
            if (!rc) rc = calloc_dev(c, &c->special, (size_t)c->nspecial);
            if (!rc) rc = ok(cudaMemcpyAsync(cursor, at, sizeof(at), cudaMemcpyHostToDevice, c->stream));
            if (!rc) {
                k_chan_lists<true><<<blocks, 256, 0, c->stream>>>(g, q, cursor, c->flist, c->rlist, c->special);
                rc = launch_ok();
            }
            if (!rc) rc = ok(cudaStreamSynchronize(c->stream));
        }
        if (q) cudaFree(q);
        if (cursor) cudaFree(cursor);
    }
    rc = chan_check(c, rc);
    if (rc) {
        chan_release(c);
        delete c;
        return rc;
    }
    *out = c;
    return LBM_OK;
}

int lbm_channel_destroy(lbm_channel c) {
    if (!c) return LBM_ERR_ARG;
    DeviceScope ds(c->p.device);
    cudaStreamSynchronize(c->stream);
    chan_release(c);
    delete c;
    return LBM_OK;
}

int lbm_channel_set_theta(lbm_channel c, const double *theta) {
    if (!c || !theta || !std::isfinite(theta[0]) || !std::isfinite(theta[1]) || !(theta[2] >= 0.0) ||
        !std::isfinite(theta[2]))
        return LBM_ERR_ARG;
    for (int k = 0; k < 3; ++k) c->theta[k] = theta[k];
    set_phys(c);
    c->have_forward = false;
    return LBM_OK;
}

int lbm_channel_forward(lbm_channel c, double *J) {
    if (!c) return LBM_ERR_ARG;
    DeviceScope ds(c->p.device);
    const size_t NQs = (size_t)c->N * Q;
    const int S = c->p.steps, K = c->K;
    int rc = cudaMemsetAsync(c->drag, 0, sizeof(double) * S, c->stream) == cudaSuccess ? LBM_OK : LBM_ERR_CUDA;
    if (!rc && cudaMemsetAsync(c->ckpt, 0, sizeof(float) * NQs, c->stream) != cudaSuccess) rc = LBM_ERR_CUDA;  // f^0 = w
    auto rec = [&](int s) -> float * {
        if (s == S) return c->fend;
        return s % K == 0 ? c->ckpt + NQs * (s / K) : nullptr;
    };
    if (!rc) rc = chan_run(c, c->ckpt, 0, S, rec, true);
    if (!rc && S % K == 0 &&
        cudaMemcpyAsync(c->ckpt + NQs * (S / K), c->fend, sizeof(float) * NQs, cudaMemcpyDeviceToDevice, c->stream) !=
            cudaSuccess)
        rc = LBM_ERR_CUDA;
    std::vector<double> d((size_t)S);
    if (!rc &&
        cudaMemcpyAsync(d.data(), c->drag, sizeof(double) * S, cudaMemcpyDeviceToHost, c->stream) != cudaSuccess)
        rc = LBM_ERR_CUDA;
    rc = chan_check(c, rc);
    if (rc) return rc;
    double sum = 0.0;
    for (int s = c->p.avg_from; s <= S; ++s) sum += d[s - 1];
    if (J) *J = sum / (S - c->p.avg_from + 1);
    c->have_forward = true;
    return LBM_OK;
}

int lbm_channel_backward(lbm_channel c, double *grad) {
    if (!c || !grad) return LBM_ERR_ARG;
    if (!c->have_forward) return LBM_ERR_ARG;  // the checkpoints belong to another theta
    DeviceScope ds(c->p.device);
    const size_t NQs = (size_t)c->N * Q;
    const int S = c->p.steps, K = c->K;
    const int slabs = chan_slabs(c->p);
    const dim3 grid_edge = chan_grid(c->p, slabs);
    const int nedge = chan_warps(c->p, slabs), nwarps = chan_warps(c->p, c->p.nz);
    const ChanGeo g = geo_of(c);
    const float up = (float)c->theta[0];
    const float wd = (float)(1.0 / (S - c->p.avg_from + 1));
    int rc = cudaMemsetAsync(c->grad, 0, 3 * sizeof(double), c->stream) == cudaSuccess ? LBM_OK : LBM_ERR_CUDA;
    if (!rc && (cudaMemsetAsync(c->gpart, 0, 2 * sizeof(double) * (size_t)(nedge + nwarps), c->stream) != cudaSuccess ||
                cudaMemsetAsync(c->gedge, 0, 3 * sizeof(double) * (size_t)nedge, c->stream) != cudaSuccess))
        rc = LBM_ERR_CUDA;
    // lambda^{S+1} = 0, with no inlet / outlet adjoint
    if (!rc && cudaMemsetAsync(c->lam[(S + 1) & 1], 0, sizeof(float) * g.Ng * Q, c->stream) != cudaSuccess)
        rc = LBM_ERR_CUDA;
    for (int seg = S / K; seg >= 0 && !rc; --seg) {
        const int s0 = seg * K, s1 = std::min(s0 + K - 1, S);  // reverse steps s1 .. s0
        const float *f0 = c->ckpt + NQs * seg;                   // f^{s0}
        // f^{s0+1} .. f^{s1} into seg slots 0 .. K-2 (drag not needed again)
        auto rec = [&](int s) -> float * { return c->seg + NQs * (size_t)(s - s0 - 1); };
        if (s1 > s0) rc = chan_run(c, f0, s0, s1, rec, false);
        for (int s = s1; s >= s0 && !rc; --s) {
            const float *fs = s == s0 ? f0 : c->seg + NQs * (size_t)(s - s0 - 1);
            const float w = (s >= c->p.avg_from && s >= 1) ? wd : 0.f;
            // the edge blocks of reverse step s > 0 fold in the inlet / outlet adjoint that step s - 1 reads
            if (s < S && c->nlinks)
                rc = chan_launch(c, k_chan_rlinks, dim3((c->nlinks + c->nspecial + kLinkTx - 1) / kLinkTx), kLinkTx,
                                 c->rlist, c->nlinks, c->special, c->nspecial, c->lam[(s + 1) & 1]);
            if (!rc)
                rc = chan_launch(c, k_chan_adj, grid_edge, kChanTx, g, c->ph, up, c->lam[(s + 1) & 1], s == 0 ? nullptr : fs,
                             w, c->lam[s & 1], s > 0 ? 1 : 0, c->gpart, c->gedge, s & 1);
        }
    }
    if (!rc) rc = chan_launch(c, k_chan_gsum, dim3(1), 256, c->gedge, nedge, c->gpart, nwarps, c->grad);
    double gr[3] = {0.0, 0.0, 0.0};
    if (!rc && cudaMemcpyAsync(gr, c->grad, sizeof(gr), cudaMemcpyDeviceToHost, c->stream) != cudaSuccess)
        rc = LBM_ERR_CUDA;
    rc = chan_check(c, rc);
    if (rc) return rc;
    grad[0] = gr[0];
    grad[1] = gr[1];
    grad[2] = gr[2] * 36.0 * std::sqrt(2.0) * c->theta[2];  // d smag / d C
    return LBM_OK;
}

int lbm_channel_drag(lbm_channel c, double *drag) {
    if (!c || !drag || !c->have_forward) return LBM_ERR_ARG;
    DeviceScope ds(c->p.device);
    int rc = cudaMemcpyAsync(drag, c->drag, sizeof(double) * c->p.steps, cudaMemcpyDeviceToHost, c->stream) ==
                     cudaSuccess
                 ? LBM_OK
                 : LBM_ERR_CUDA;
    return chan_check(c, rc);
}

int lbm_channel_populations(lbm_channel c, double *f) {
    if (!c || !f || !c->have_forward) return LBM_ERR_ARG;
    DeviceScope ds(c->p.device);
    std::vector<float> h((size_t)c->N * Q);
    int rc = cudaMemcpyAsync(h.data(), c->fend, sizeof(float) * h.size(), cudaMemcpyDeviceToHost, c->stream) ==
                     cudaSuccess
                 ? LBM_OK
                 : LBM_ERR_CUDA;
    rc = chan_check(c, rc);
    if (rc) return rc;
    for (int i = 0; i < Q; ++i)
        for (int n = 0; n < c->N; ++n) f[(size_t)i * c->N + n] = (double)h[(size_t)i * c->N + n] + w36(i) / 36.0;
    return LBM_OK;
}

int lbm_channel_geometry(lbm_channel c, uint8_t *type) {
    if (!c || !type) return LBM_ERR_ARG;
    DeviceScope ds(c->p.device);
    int rc = cudaMemcpyAsync(type, c->type, (size_t)c->N, cudaMemcpyDeviceToHost, c->stream) == cudaSuccess
                 ? LBM_OK
                 : LBM_ERR_CUDA;
    return chan_check(c, rc);
}

}  // extern "C"
