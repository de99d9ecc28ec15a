// Interpolated bounce-back on sphere links and momentum exchange (Sect. 2.3)
// for one sphere per CTA, after the collide of its neighbourhood: the phases
// of the link kernels (lbm_links.cu).
//
// The CTA holds the fluid nodes of a cube around the sphere as one 64-bit
// row mask per (y, z) in shared memory.  Every pair (solid node s owned by the
// sphere, direction j) with x = s - c_j fluid is a cut link.  Its fraction q is the smallest root of
// |x + t c_j - X| = R in FP32, written as c0 / (-b + sqrt(b^2 - a c0)) and
// evaluated with the same round-to-nearest operations as the oracle.  The
// population k = opp(j) that x receives from the solid side is (Eq. 19 with
// the moving-boundary term of Eq. 21, deviations from w throughout):
//   q <  1/2, x - c_j fluid: 2q d^c_j(x) + (1-2q) d^c_j(x - c_j) + 6 w_j (c_k.u_b)
//   q <  1/2, otherwise:     d^c_j(x) + 6 w_j (c_k.u_b)
//   q >= 1/2:                d^c_j(x)/(2q) + (2q-1)/(2q) d^c_k(x) + (3/q) w_j (c_k.u_b)
// with u_b = V + Om x (x + q c_j - X).  It is written where the next step
// reads f_k(x).  All inputs are post-collision values of the finished step
// and all outputs are slots no other link reads, so links are independent.
//
// Momentum exchange (Eqs. 25, 26): the sphere receives
//   dP = (f^c_j(x) + f_k(x, t+1)) c_j,   torque (x_b - X) x dP,
// and with the Galilean-invariant option (Wen, Zhang & Fang 2014; not in the
// paper) also -(f^c_j(x) - f_k(x, t+1)) u_b.
// With f = w + d this splits into the deviation part (d^c_j + d_k) c_j,
// summed in FP32 per thread and per warp (shuffles), and the rest part
// 2 w_j c_j = (36 w_j / 18) c_j, counted exactly in integers; (x_b - X) x c_j
// = (x - X) x c_j since c_j x c_j = 0.  The CTA combines the warp sums in
// FP64 in a fixed order, so the force is deterministic.
#pragma once

#include "lbm_internal.cuh"

namespace lbm {

// Instruction budget.  One CTA handles ~1150 links of a sphere of radius 4;
// on a few spheres its latency is the step's, on thousands the SMs issue for
// half of the kernel's time while it waits on scattered DRAM blocks.  So the
// geometry is bit arithmetic on rows (a thread loads a row's flags as words,
// a node's 18 neighbour tests are 9 row words), a link carries its offsets and
// direction in its list entry, direction constants come from a shared table
// and only tiles that cross a periodic face wrap their coordinates (times
// beside k_links).

// Wrap a coordinate that is at most one box length outside [0, n).
__device__ __forceinline__ int wrap1(int x, int n) { return x < 0 ? x + n : (x >= n ? x - n : x); }

// The cube of a sphere with e = ceil(R): B nodes per edge at offsets lo ..
// lo + B - 1 from floor(X).  Its solid nodes have offsets -e + 1 .. e, the
// links' fluid nodes x = s - c_j and x - c_j lie within two more.
// A node index t = x + B (y + B z) is split by multiplying with mB = 2^32 / B
// + 1 and mB2 = 2^32 / B^2 + 1 and taking the high word: exact for t < B^3 <
// 2^16 (B <= 36), where a division by a run-time B costs some twenty
// instructions.
struct LinkTile {
    int lo, B;
    unsigned mB, mB2;
    __host__ __device__ __forceinline__ explicit LinkTile(int e, unsigned mb = 0u, unsigned mb2 = 0u)
        : lo(-e - 1), B(2 * e + 4), mB(mb), mB2(mb2) {}
    // row r = y + B z
    __device__ __forceinline__ void row_yz(int r, int &y, int &z) const {
        z = (int)__umulhi((unsigned)r, mB);
        y = r - z * B;
    }
    __device__ __forceinline__ void xyz(int t, int &x, int &y, int &z) const {
        z = (int)__umulhi((unsigned)t, mB2);
        const int r = t - z * B * B;
        y = (int)__umulhi((unsigned)r, mB);
        x = r - y * B;
    }
    // at most every node of the core, and every listed node has a link
    __host__ __device__ __forceinline__ int ncap(int cap) const {
        const int c = B - 4, c3 = c * c * c;
        return c3 < cap ? c3 : cap;
    }
};

// Shared memory of a link CTA: row masks of the fluid nodes (bit i of row
// y + B z: the node at offsets lo + (i, y, z)), the links (cap entries, packed
// as i | y << 6 | z << 12 | j << 18) and the node indexes of the owned nodes
// that have links, in (z, y, x) order.
struct LinkShared {
    unsigned long long *row;
    uint32_t *list;
    uint16_t *nodes;
    __device__ __forceinline__ LinkShared(unsigned char *smem, int cap, const LinkTile &tl)
        : row((unsigned long long *)smem), list((uint32_t *)(row + tl.B * tl.B)), nodes((uint16_t *)(list + cap)) {}
};

// Constants of direction j for the link loop.
struct LinkDir {
    float4 c;  // c_j, w_j
    int off;   // storage offset of c_j
    int js, ks;  // slot offsets of j and opp(j)
    int rx;    // row offset cy + B cz, shifted left by 2, | (c_x + 1)
};

__device__ __forceinline__ void link_dirs(const Lat &L, const LinkTile &tl, LinkDir *dir) {
    const int j = threadIdx.x;
    if (j >= Q) return;
    LinkDir d;
    d.c = make_float4((float)rcx(j), (float)rcy(j), (float)rcz(j), (float)rw36(j) * (1.f / 36.f));
    d.off = rcx(j) + L.nx * (rcy(j) + L.ny * rcz(j));
    d.js = j * (int)L.S;
    d.ks = ropp(j) * (int)L.S;
    d.rx = (rcy(j) + tl.B * rcz(j)) * 4 + (rcx(j) + 1);
    dir[j] = d;
}

// The solid bits of 4 flags.
__device__ __forceinline__ unsigned solid4(unsigned w) { return ((w & 0x01010101u) * 0x10204080u) >> 28; }

// 1. The fluid row masks of sphere p's cube (a node outside the box in z is
//    not fluid), and 2. its nodes with links: a row's owned nodes are its
//    solid ones in the core with owner p; those next to a fluid node (any of
//    the 18 directions) are listed.  One thread per row; the list keeps row
//    order (block scan).  Returns the number of nodes; ends with a barrier.
//    Flags and owners are read through L2.
__device__ __forceinline__ int link_nodes(const Lat &L, const int b[3], const uint8_t *__restrict__ flag,
                                          const int32_t *__restrict__ owner, const int p, const LinkTile &tl,
                                          const LinkShared &sh, const int ncap, int *__restrict__ status) {
    __shared__ int wsum[8];
    const int B = tl.B, BB = B * B, core = B - 4;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int x0 = b[0] + tl.lo;
    const int xs = wrap1(x0, L.nx);
    const unsigned long long full = (1ull << B) - 1ull;  // B <= 36
    // the solid bits of len nodes from n on, from aligned words (the flags are padded to a whole word)
    auto solid_bits = [&](const int n, const int len) {
        unsigned long long solid = 0ull;
        const int sh0 = n & 3;
        const unsigned *w = (const unsigned *)(flag + (n - sh0));
        constexpr int kW = 4;
        for (int k0 = 0; 4 * k0 < len + sh0; k0 += kW) {
            unsigned v[kW];
#pragma unroll
            for (int k = 0; k < kW; ++k) v[k] = 4 * (k0 + k) < len + sh0 ? __ldcg(w + k0 + k) : 0u;
#pragma unroll
            for (int k = 0; k < kW; ++k) {
                const unsigned long long m = solid4(v[k]);
                const int at = 4 * (k0 + k) - sh0;
                solid |= at >= 0 ? m << at : m >> -at;
            }
        }
        return solid & ((1ull << len) - 1ull);
    };
    for (int r = threadIdx.x; r < BB; r += blockDim.x) {
        int ty, tz;
        tl.row_yz(r, ty, tz);
        const int z = b[2] + tl.lo + tz;
        unsigned long long solid = full;
        if (z >= 0 && z < L.nz) {
            const int n0 = L.nx * (wrap1(b[1] + tl.lo + ty, L.ny) + L.ny * z);
            int n = n0 + xs, len = min(B, L.nx - xs);
            solid = 0ull;
#pragma unroll 1
            for (int at = 0; at < B; n = n0, len = B - at) {  // past a periodic face, the rest from the row's start
                solid |= solid_bits(n, len) << at;
                at += len;
            }
        }
        sh.row[r] = ~solid & full;
    }
    __syncthreads();
    int total = 0;
    for (int r0 = 0; r0 < BB; r0 += blockDim.x) {
        const int r = r0 + threadIdx.x;
        int y, z;
        tl.row_yz(r, y, z);
        unsigned long long s = 0ull;
        const int zb = b[2] + tl.lo + z;  // rows outside the box are solid, but nobody owns their nodes
        if (r < BB && y >= 2 && y < B - 2 && z >= 2 && z < B - 2 && zb >= 0 && zb < L.nz) {
            const unsigned long long *f = sh.row + r;
            const unsigned long long lines = f[-1] | f[1] | f[-B] | f[B], mid = f[0];
            const unsigned long long any = (mid | lines) << 1 | (mid | lines) >> 1 | lines |
                                           f[-1 - B] | f[1 - B] | f[-1 + B] | f[1 + B];
            s = any & ~mid & (((1ull << core) - 1ull) << 2);  // solid, next to a fluid node, in the core
            if (s) {
                const int n0 = L.nx * (wrap1(b[1] + tl.lo + y, L.ny) + L.ny * zb);
                unsigned long long own = 0ull, c = s;
                constexpr int kOwn = 8;
                while (c) {
                    int i[kOwn], o[kOwn];
#pragma unroll
                    for (int u = 0; u < kOwn; ++u) {
                        i[u] = c ? __ffsll((long long)c) - 1 : -1;
                        c &= c - 1ull;
                        o[u] = i[u] >= 0 ? __ldcg(owner + n0 + wrap1(x0 + i[u], L.nx)) : -1;
                    }
#pragma unroll
                    for (int u = 0; u < kOwn; ++u)
                        if (i[u] >= 0 && o[u] == p) own |= 1ull << i[u];
                }
                s = own;
            }
        }
        const int mine = __popcll(s);
        int incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        if (lane == 31) wsum[wid] = incl;
        __syncthreads();
        int pos = total + incl - mine, round = 0;
        for (int w = 0; w < nw; ++w) {
            if (w < wid) pos += wsum[w];
            round += wsum[w];
        }
        while (s) {
            const int i = __ffsll((long long)s) - 1;
            s &= s - 1ull;
            if (pos < ncap) sh.nodes[pos] = (uint16_t)(i + B * r);
            ++pos;
        }
        total += round;
        __syncthreads();
    }
    if (total > ncap && threadIdx.x == 0) atomicOr(status, ST_TILE);
    return min(total, ncap);
}

// Per-thread partial sums of a CTA's links: the deviation part in FP32, the
// rest part 2 w_j c_j in integers (36 w_j c_j summed, divided by 18 at the end).
struct LinkAcc {
    float Fd[3] = {0.f, 0.f, 0.f}, Td[3] = {0.f, 0.f, 0.f};
    int I[3] = {0, 0, 0}, J[3] = {0, 0, 0};
};

// Directions with c_axis = sign and weight class w36 = w, as a bit mask.
__host__ __device__ constexpr uint32_t dir_mask(int axis, int sign, int w) {
    uint32_t m = 0;
    for (int j = 1; j < Q; ++j)
        if ((axis == 0 ? cx(j) : (axis == 1 ? cy(j) : cz(j))) == sign && w36(j) == w) m |= 1u << j;
    return m;
}

// 3. Cut links of the listed nodes into sh.list in node order, direction
//    minor; returns their count (at most cap).  Thread i takes the nodes i,
//    i + T, ...: the 18 tests read the 9 rows around the node, one block scan
//    of the counts places the links.  The rest part of the momentum exchange
//    is a sum over the node's directions (bit counts), and its moment is
//    s x that sum, (x - X) x c_j and (s - X) x c_j being equal.  Ends with a
//    block barrier.
__device__ __forceinline__ int link_enumerate(const LinkShared &sh, const LinkTile &tl, const int nn, const int cap,
                                              LinkAcc &acc, int *__restrict__ status) {
    __shared__ int wsum[8];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5, B = tl.B;
    int total = 0;
    for (int k0 = 0; k0 < nn; k0 += blockDim.x) {
        const int k = k0 + threadIdx.x;
        uint32_t mask = 0u, t = 0u;
        if (k < nn) {
            int i, y, z;
            tl.xyz(sh.nodes[k], i, y, z);
            t = (uint32_t)(i | y << 6 | z << 12);
            const unsigned long long *f = sh.row + y + B * z;
            uint32_t win[3][3];  // bits 0, 1, 2: the nodes at x - 1, x, x + 1 of row (y + dy, z + dz)
#pragma unroll
            for (int dz = -1; dz <= 1; ++dz)
#pragma unroll
                for (int dy = -1; dy <= 1; ++dy) win[dz + 1][dy + 1] = (uint32_t)(f[dy + B * dz] >> (i - 1));
#pragma unroll
            for (int j = 1; j < Q; ++j) mask |= ((win[1 - cz(j)][1 - cy(j)] >> (1 - cx(j))) & 1u) << j;
            int I[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                I[a] = 2 * (__popc(mask & dir_mask(a, 1, 2)) - __popc(mask & dir_mask(a, -1, 2))) +
                       __popc(mask & dir_mask(a, 1, 1)) - __popc(mask & dir_mask(a, -1, 1));
                acc.I[a] += I[a];
            }
            const int sx = i + tl.lo, sy = y + tl.lo, sz = z + tl.lo;
            acc.J[0] += sy * I[2] - sz * I[1];
            acc.J[1] += sz * I[0] - sx * I[2];
            acc.J[2] += sx * I[1] - sy * I[0];
        }
        const int c = __popc(mask);
        int inc = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += v;
        }
        if (lane == 31) wsum[wid] = inc;
        __syncthreads();
        int pos = total + inc - c, round = 0;
        for (int w = 0; w < nw; ++w) {
            if (w < wid) pos += wsum[w];
            round += wsum[w];
        }
        while (mask) {
            const uint32_t j = __ffs(mask) - 1;
            mask &= mask - 1u;
            if (pos < cap) sh.list[pos] = t | j << 18;
            ++pos;
        }
        total += round;
        __syncthreads();
    }
    if (total > cap && threadIdx.x == 0) atomicOr(status, ST_TILE);
    return min(total, cap);
}

// 4. Bounce-back and momentum exchange of links l = threadIdx.x,
//    threadIdx.x + blockDim.x, ... < total of the sphere with frame Fr.  The
//    fraction q is the smallest root of |x + q c_j - X| = R as
//    c0 / (-b + sqrt(b^2 - a c0)), in FP32 with the oracle's operations.
//    BATCH links per thread per round have their populations in flight
//    together.  Every product and sum is an explicit round-to-nearest
//    operation, so each kernel that inlines this rounds alike.
template <typename T, bool GI, int BATCH>
__device__ __forceinline__ void link_apply(const Lat &L, const Parts &pt, const SFrame &Fr, T *__restrict__ f,
                                           const int P, const LinkTile &tl, const LinkShared &sh,
                                           const LinkDir *__restrict__ dir, const int total, LinkAcc &acc) {
    const int x0 = Fr.b[0] + tl.lo, y0 = Fr.b[1] + tl.lo, z0 = Fr.b[2] + tl.lo;
    // storage index of the cube's first node, as if nothing wrapped
    const int base = x0 + L.nx * (y0 + L.ny * (z0 + 1));
    const bool wraps = x0 < 0 || x0 + tl.B > L.nx || y0 < 0 || y0 + tl.B > L.ny;
    for (int l0 = threadIdx.x; l0 < total; l0 += BATCH * blockDim.x) {
        float ld[BATCH][2], lq[BATCH];
        uint32_t le[BATCH];
        int dst[BATCH], lbr[BATCH];
#pragma unroll
        for (int u = 0; u < BATCH; ++u) {
            const int l = l0 + u * blockDim.x;
            le[u] = 0u;
            if (l >= total) continue;
            const uint32_t t = sh.list[l];
            const int i = t & 63, y = (t >> 6) & 63, z = (t >> 12) & 63;
            const LinkDir d = dir[t >> 18];
            // x = s - c_j relative to X
            const float dx = __fsub_rn((float)(tl.lo + i) - d.c.x, Fr.fr[0]);
            const float dy = __fsub_rn((float)(tl.lo + y) - d.c.y, Fr.fr[1]);
            const float dz = __fsub_rn((float)(tl.lo + z) - d.c.z, Fr.fr[2]);
            const float d2 = __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
            const float qa = d.c.x * d.c.x + d.c.y * d.c.y + d.c.z * d.c.z;  // 1 or 2, exact
            const float qb = __fadd_rn(__fadd_rn(__fmul_rn(d.c.x, dx), __fmul_rn(d.c.y, dy)), __fmul_rn(d.c.z, dz));
            const float c0 = __fsub_rn(d2, Fr.R2);
            float disc = __fsub_rn(__fmul_rn(qb, qb), __fmul_rn(qa, c0));
            if (disc < 0.f) disc = 0.f;
            float q = __fdiv_rn(c0, __fadd_rn(-qb, __fsqrt_rn(disc)));
            q = fminf(fmaxf(q, 0.f), 1.f);
            // branch of Eq. (19): 0 interpolate with x - c_j, 1 halfway fallback (x - c_j not fluid), 2 q >= 1/2
            const int cjx = (d.rx & 3) - 1;
            const int i2 = i - 2 * cjx, r2 = y + tl.B * z - 2 * (d.rx >> 2);
            const int br = q < 0.5f ? ((sh.row[r2] >> i2) & 1ull ? 0 : 1) : 2;
            // storage indices of the solid node s, of x and of x - c_j
            int ss = base + i + L.nx * (y + L.ny * z), sx = ss - d.off, sb = sx - d.off;
            if (wraps) {
                const int cjy = (int)d.c.y, cjz = (int)d.c.z;
                const int xx = wrap1(x0 + i - cjx, L.nx), xy = wrap1(y0 + y - cjy, L.ny), xz = z0 + z - cjz + 1;
                sx = xx + L.nx * (xy + L.ny * xz);
                ss = wrap1(xx + cjx, L.nx) + L.nx * (wrap1(xy + cjy, L.ny) + L.ny * (xz + cjz));
                sb = wrap1(xx - cjx, L.nx) + L.nx * (wrap1(xy - cjy, L.ny) + L.ny * (xz - cjz));
            }
            // post-collision d^c_j(x) and, by branch, d^c_j(x - c_j) or d^c_k(x)
            const T *a0 = f + (P == 0 ? d.ks + sx : d.js + ss);
            const T *a1 = f + (br == 0 ? (P == 0 ? d.ks + sb : d.js + sx) : (P == 0 ? d.js + sx : d.ks + sb));
            ld[u][0] = Store<T>::ld(a0);
            ld[u][1] = br == 1 ? 0.f : Store<T>::ld(a1);
            dst[u] = P == 0 ? d.js + ss : d.ks + sx;  // where the next step reads f_k(x)
            le[u] = t;
            lq[u] = q;
            lbr[u] = br;
        }
        const float *V = Fr.V, *W = Fr.W;
#pragma unroll
        for (int u = 0; u < BATCH; ++u) {
            if (le[u] == 0u) continue;  // a link's direction is never 0
            const uint32_t t = le[u];
            const float4 c = dir[t >> 18].c;
            const float dx = __fsub_rn((float)(tl.lo + (int)(t & 63)) - c.x, Fr.fr[0]);
            const float dy = __fsub_rn((float)(tl.lo + (int)((t >> 6) & 63)) - c.y, Fr.fr[1]);
            const float dz = __fsub_rn((float)(tl.lo + (int)((t >> 12) & 63)) - c.z, Fr.fr[2]);
            const float q = lq[u], dcj = ld[u][0], wj = c.w;
            // boundary point x_b = x + q c_j relative to X, and its velocity u_b = V + Om x (x_b - X)
            const float lx = __fadd_rn(dx, c.x * q), ly = __fadd_rn(dy, c.y * q), lz = __fadd_rn(dz, c.z * q);
            const float ubx = __fadd_rn(V[0], __fsub_rn(__fmul_rn(W[1], lz), __fmul_rn(W[2], ly)));
            const float uby = __fadd_rn(V[1], __fsub_rn(__fmul_rn(W[2], lx), __fmul_rn(W[0], lz)));
            const float ubz = __fadd_rn(V[2], __fsub_rn(__fmul_rn(W[0], ly), __fmul_rn(W[1], lx)));
            const float cku = -__fadd_rn(__fadd_rn(c.x * ubx, c.y * uby), c.z * ubz);  // c_k = -c_j
            const float q2 = 2.f * q;  // exact
            float dn;
            if (lbr[u] == 0) {
                dn = __fadd_rn(__fadd_rn(__fmul_rn(q2, dcj), __fmul_rn(__fsub_rn(1.f, q2), ld[u][1])),
                               __fmul_rn(__fmul_rn(6.f, wj), cku));
            } else if (lbr[u] == 1) {
                dn = __fadd_rn(dcj, __fmul_rn(__fmul_rn(6.f, wj), cku));
            } else {
                const float i2q = __fdiv_rn(0.5f, q);
                dn = __fadd_rn(__fadd_rn(__fmul_rn(dcj, i2q), __fmul_rn(__fmul_rn(__fsub_rn(q2, 1.f), i2q), ld[u][1])),
                               __fmul_rn(__fmul_rn(__fdiv_rn(3.f, q), wj), cku));
            }
            Store<T>::st(f + dst[u], dn);

            const float m = __fadd_rn(dcj, dn);
            const float cxr[3] = {__fsub_rn(dy * c.z, dz * c.y), __fsub_rn(dz * c.x, dx * c.z),
                                  __fsub_rn(dx * c.y, dy * c.x)};  // (x - X) x c_j
            const float fj[3] = {c.x, c.y, c.z};
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                acc.Fd[a] = __fadd_rn(acc.Fd[a], m * fj[a]);
                acc.Td[a] = __fmaf_rn(m, cxr[a], acc.Td[a]);
            }
            if (GI && pt.gimea) {  // Galilean-invariant form: - (f^c_j - f_k) u_b, the weights cancel
                const float e = __fsub_rn(dcj, dn);
                const float ub[3] = {ubx, uby, ubz};
                const float lxu[3] = {__fsub_rn(__fmul_rn(ly, ubz), __fmul_rn(lz, uby)),
                                      __fsub_rn(__fmul_rn(lz, ubx), __fmul_rn(lx, ubz)),
                                      __fsub_rn(__fmul_rn(lx, uby), __fmul_rn(ly, ubx))};
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    acc.Fd[a] = __fmaf_rn(-e, ub[a], acc.Fd[a]);
                    acc.Td[a] = __fmaf_rn(-e, lxu[a], acc.Td[a]);
                }
            }
        }
    }
}

// 5. Warp sums in FP32, then FP64 across warps in a fixed order; thread 0
//    writes sphere p's load (plus the covered / uncovered-node momentum of
//    the step with the correction) and counts its links.
__device__ __forceinline__ void link_reduce_store(const Parts &pt, const int p, const int b[3], const LinkAcc &acc,
                                                  const int total, unsigned long long *__restrict__ ctr) {
    __shared__ float redf[8][6];
    __shared__ int redi[8][6];
    __shared__ double sh[12];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    float v[6] = {acc.Fd[0], acc.Fd[1], acc.Fd[2], acc.Td[0], acc.Td[1], acc.Td[2]};
    int iv[6] = {acc.I[0], acc.I[1], acc.I[2], acc.J[0], acc.J[1], acc.J[2]};
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int a = 0; a < 6; ++a) {
            v[a] = __fadd_rn(v[a], __shfl_xor_sync(0xffffffffu, v[a], o));
            iv[a] += __shfl_xor_sync(0xffffffffu, iv[a], o);
        }
    }
    if (lane == 0) {
        for (int a = 0; a < 6; ++a) {
            redf[wid][a] = v[a];
            redi[wid][a] = iv[a];
        }
    }
    __syncthreads();
    // lanes 0..11 of warp 0 each sum one component over the warps in FP64
    if (threadIdx.x < 12) {
        const int a = threadIdx.x;
        double sum = 0.0;
        for (int w = 0; w < nw; ++w) sum = __dadd_rn(sum, a < 6 ? (double)redf[w][a] : (double)redi[w][a - 6]);
        sh[a] = sum;
    }
    __syncthreads();
    if (threadIdx.x < 3) {  // one component each
        const int a = threadIdx.x, a1 = a == 2 ? 0 : a + 1, a2 = a == 0 ? 2 : a - 1;
        const double f1 = pt.X[3 * p + a1] - (double)b[a1], f2 = pt.X[3 * p + a2] - (double)b[a2];  // exact: X - floor(X)
        // rest part 2 w_j c_j: F = I/18, T = (J - frac x I)/18
        constexpr double i18 = 1.0 / 18.0;
        const double fxI = __dsub_rn(__dmul_rn(f1, sh[6 + a2]), __dmul_rn(f2, sh[6 + a1]));
        double Fa = __dadd_rn(sh[a], __dmul_rn(sh[6 + a], i18));
        double Ta = __dadd_rn(sh[3 + a], __dmul_rn(__dsub_rn(sh[9 + a], fxI), i18));
        if (pt.corr) {  // momentum of the nodes covered / uncovered this step
            Fa = __dadd_rn(Fa, pt.Fcorr[3 * p + a]);
            Ta = __dadd_rn(Ta, pt.Tcorr[3 * p + a]);
        }
        pt.Fh[3 * p + a] = Fa;
        pt.Th[3 * p + a] = Ta;
        if (a == 0) atomicAdd(ctr, (unsigned long long)total);
    }
}

// The links of sphere p in one pass (one CTA, at most 256 threads): node
// rows, link list, bounce-back and momentum exchange, per-sphere sums.  Run
// after the step's collide and refill.
template <typename T, bool GI, int BATCH = 6>
__device__ __forceinline__ void links_body(const Lat &L, const Parts &pt, const SFrame *__restrict__ fcur,
                                           T *f, const uint8_t *__restrict__ flag,
                                           const int32_t *__restrict__ owner, const int P, const int ext,
                                           const int cap, int *status, unsigned long long *ctr, const int p) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ LinkDir dir[Q];
    const SFrame Fr = fcur[p];
    // The sphere's own cube; ext (shared memory is sized for it) bounds it: a
    // small sphere among large ones scans only its own.  Nodes are listed in
    // (z, y, x) order whatever the extent, so the link list, and every sum
    // over it, is the same for any extent that holds the sphere.
    const int e = min(ext, (int)ceilf(Fr.R));
    const unsigned B = 2u * (unsigned)e + 4u;
    const LinkTile tl(e, 0xFFFFFFFFu / B + 1u, 0xFFFFFFFFu / (B * B) + 1u);
    const LinkShared sh(smem, cap, tl);
    link_dirs(L, tl, dir);
    LinkAcc acc;
    const int nn = link_nodes(L, Fr.b, flag, owner, p, tl, sh, tl.ncap(cap), status);
    const int total = link_enumerate(sh, tl, nn, cap, acc, status);
    // the rows and the list read only the marks (a refilled node's flag turns
    // from 2 to 0 in the collide, fluid either way): they may be made while
    // the collide's last blocks run, the populations are read after it
    step_wait();
    step_next();
    link_apply<T, GI, BATCH>(L, pt, Fr, f, P, tl, sh, dir, total, acc);
    link_reduce_store(pt, p, Fr.b, acc, total, ctr);
}

}  // namespace lbm
