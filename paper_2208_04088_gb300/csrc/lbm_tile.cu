// lbm_tile.cu -- temporally blocked time stepping in register tiles: up to
// kWaveK steps per launch (kWaveGradK when lambda != mu, whose source needs the
// density gradient), FP32 storage, two population buffers.
//
// A block owns a tile (ring) of W x H nodes and keeps the nine populations of
// every node in registers for all steps of the launch: a thread holds two
// adjacent columns of `rows` consecutive rows, as f32x2 pairs.  Streaming along
// x is one shuffle per population and pair, along y a renaming of the thread's
// rows plus one row exchanged with the neighbouring threads through shared
// memory.  The ring has a halo of kTileHalo nodes on each side that is not a
// box edge; what a step can no longer compute shrinks by one node per step
// (two when lambda != mu), so the core of every tile is exact and tiles overlap
// only in what they read.  Populations and displacements cross HBM once per
// launch.
//
// Boundary rules (Sec. 4).  Nodes that a rule reads (boundary nodes, and the
// upstream nodes of their links) publish their post-collision populations in
// shared memory; the cut links of the tile are then spread over all threads of
// the block, one link to a thread (cut_link_value, the function of every other
// boundary path), and the owners pick up the results.  Per node the arithmetic
// is that of the one-step kernels, so every stored value is bit-identical.
//
// What bounds it: FP32 issue in the tiles of a large lattice (a 64 x 64 tile
// updates 4096 nodes per step, 65 paired operations per pair and 12 per node
// for the displacement, of which the core's 48 x 48 count); on lattices of
// less than a few hundred thousand nodes the latency of one step (two block
// barriers, the collision's and a link's dependent chain) and of the launch.
#include <algorithm>
#include <cstdint>
#include <cstring>
#include <vector>

#include <cuda.h>
#include <cuda_runtime.h>

#include "lbm_async.cuh"
#include "lbm_device.cuh"
#include "lbm_internal.h"

namespace lbm {

namespace {

constexpr int kNT = kTileThreads;

// Shared memory of a tile: the populations as copied in, whose space is reused
// once they are in registers (row exchange, published nodes, link results,
// link rules, densities), the slot map, the displacement records.
template <int LPR, int R> struct Shape {
    static constexpr int G = kNT / LPR;  // groups of rows, one per LPR threads
    static constexpr int W = 2 * LPR, H = G * R;
    static constexpr int kSlots = TileShape{LPR, R}.slots();
    static constexpr size_t kStage = (size_t)W * H * 36;
    static constexpr size_t kEx = (size_t)2 * 2 * G * 3 * LPR * 8;  // parity, direction, group, plane
    static constexpr size_t kOffPub = kEx;
    static constexpr size_t kOffOut = kOffPub + (size_t)kSlots * 12 * 4;
    static constexpr int kRules = 1024;  // links whose rules are kept
    static constexpr size_t kOffRule = kOffOut + (size_t)kSlots * 8 * 4;
    static constexpr size_t kOffDen = kOffRule + (size_t)9 * kRules * 4;
    static constexpr size_t kAlias = kOffDen + (size_t)2 * G * LPR * 8;
    static constexpr size_t kOffSlot = ((kStage > kAlias ? kStage : kAlias) + 127) / 128 * 128;
    static constexpr size_t kOffCut = kOffSlot + (size_t)W * H * 2;
    static constexpr size_t kOffU = kOffCut + kSlots;
    static constexpr size_t kOffBar = kOffU + (size_t)W * H * 16;
    static constexpr size_t kSmem = kOffBar + 16;
    static_assert(kSmem <= 232448, "shared memory of one block");
    static_assert(W <= 256 && H <= 256, "copy box");
};

// The pair moved one column to the right (each node takes its left
// neighbour's value) or to the left.
template <int LPR> __device__ __forceinline__ F2 from_left(F2 v) {
    float lo, hi;
    f2_split(v, lo, hi);
    return f2(__shfl_up_sync(0xffffffffu, hi, 1, LPR), lo);
}
template <int LPR> __device__ __forceinline__ F2 from_right(F2 v) {
    float lo, hi;
    f2_split(v, lo, hi);
    return f2(hi, __shfl_down_sync(0xffffffffu, lo, 1, LPR));
}

__device__ __forceinline__ F2 as_f2(unsigned long long v) {
    F2 r;
    r.v = v;
    return r;
}

// Nine populations of a published node (48 bytes, 16-byte aligned).
__device__ __forceinline__ void put9(float *p, const float v[9]) {
    float4 *q = reinterpret_cast<float4 *>(p);
    q[0] = make_float4(v[0], v[1], v[2], v[3]);
    q[1] = make_float4(v[4], v[5], v[6], v[7]);
    p[8] = v[8];
}
__device__ __forceinline__ void get9(const float *p, float v[9]) {
    const float4 *q = reinterpret_cast<const float4 *>(p);
    const float4 a = q[0], b = q[1];
    v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w;
    v[4] = b.x, v[5] = b.y, v[6] = b.z, v[7] = b.w;
    v[8] = p[8];
}

// Programmatic launch order: the next launch of the stream may start its
// prologue now, and this one has waited for everything before it.
__device__ __forceinline__ void release_next() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void wait_for_previous() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// nsteps steps of one tile; the first is step `toff` after *time.
template <int LPR, int R, bool GRAD>
__device__ __forceinline__ void tile_steps(const CUtensorMap *tf, float *__restrict__ dst,
                                           float4 *__restrict__ uc,
                                           const uint8_t *__restrict__ cls, const TileRec &rec,
                                           const uint32_t *__restrict__ pubs,
                                           const TileLink *__restrict__ links,
                                           const BCDev *__restrict__ bcs, const Lattice &L,
                                           const int64_t *__restrict__ time, int toff, int nsteps,
                                           uint32_t *__restrict__ status, unsigned char *sm) {
    using S = Shape<LPR, R>;
    constexpr int W = S::W, H = S::H, G = S::G;
    const int tid = threadIdx.x, t = tid % LPR, g = tid / LPR;
    const int c0 = 2 * t, row0 = g * R;
    const uint32_t bar = smem_addr(sm + S::kOffBar);
    float4 *us = reinterpret_cast<float4 *>(sm + S::kOffU);
    volatile int *landed = reinterpret_cast<volatile int *>(sm + S::kOffBar + 8);

    // the previous launch writes nothing that is read up to wait_for_previous()
    constexpr uint32_t kNone = 0xffffu;
    const int npub = rec.npub, nlink = rec.nlink;
    uint8_t *cutm = sm + S::kOffCut;
    uint32_t slot[R];       // slots of the thread's published nodes (low, high half)
    uint32_t rowflag = 0;   // rows in which a lane of the warp has one (warp-uniform)
#pragma unroll
    for (int r = 0; r < R; ++r) slot[r] = 0xffffffffu;
    if (npub) {  // uniform over the block
        uint32_t *map = reinterpret_cast<uint32_t *>(sm + S::kOffSlot);
        for (int q = tid; q < W * H / 2; q += kNT) map[q] = 0xffffffffu;
        __syncthreads();
        for (int q = tid; q < npub; q += kNT) {
            const uint32_t p = pubs[rec.pub0 + q];
            reinterpret_cast<uint16_t *>(map)[((p >> 8) & 0xffu) * W + (p & 0xffu)] = (uint16_t)q;
            cutm[q] = (uint8_t)(p >> 16);
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < R; ++r) {
            slot[r] = map[((row0 + r) * W + c0) / 2];
            if (__ballot_sync(0xffffffffu, slot[r] != 0xffffffffu)) rowflag |= 1u << r;
        }
    }
    wait_for_previous();
    if (tid == 0) {
        mbar_init(bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        mbar_expect_tx(bar, (uint32_t)S::kStage);
        tma_load_3d(smem_addr(sm), tf, rec.x0, rec.y0, 0, bar);
    }
    // while the populations arrive: which of the thread's nodes are material
    // core nodes (bit 2 r + j), and their displacement records
    const float tb0 = (float)(*time + toff - 1);
    const int64_t k0 = (int64_t)(rec.y0 + row0) * L.pitch + rec.x0 + c0;
    const bool core_a = c0 >= rec.c0 && c0 < rec.c1, core_b = c0 + 1 >= rec.c0 && c0 + 1 < rec.c1;
    uint32_t mine = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        if (row0 + r < rec.r0 || row0 + r >= rec.r1 || !(core_a || core_b)) continue;
        const int64_t k = k0 + (int64_t)r * L.pitch;
        const uint32_t cc = __ldg(reinterpret_cast<const uint16_t *>(cls + k));
        if (core_a && (cc & 0xffu) != kVoid) mine |= 1u << (2 * r);
        if (core_b && (cc >> 8) != kVoid) mine |= 2u << (2 * r);
        if ((mine >> (2 * r)) & 1u) us[(2 * r) * kNT + tid] = uc[k];
        if ((mine >> (2 * r)) & 2u) us[(2 * r + 1) * kNT + tid] = uc[k + 1];
    }
    uint32_t corerow = 0;  // rows in which a lane of the warp has a core node (warp-uniform)
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (__ballot_sync(0xffffffffu, ((mine >> (2 * r)) & 3u) != 0)) corerow |= 1u << r;
    if (tid == 0)  // a limit of 0 gives up at once, whether or not the copy has landed
        *landed = L.wait_ns > 0 && mbar_wait(bar, 0, L.wait_ns);
    __syncthreads();
    if (!*landed) {
        // flag it, and keep the block's shared memory until the copy is over
        if (tid == 0) {
            atomicOr(status, 2u);
            mbar_wait(bar, 0, kDefaultWaitNs);
        }
        return;
    }
    F2 f[R][9];
    {
        const unsigned long long *st = reinterpret_cast<const unsigned long long *>(sm);
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int i = 0; i < 9; ++i) f[r][i] = as_f2(st[((i * H + row0 + r) * W + c0) / 2]);
    }
    __syncthreads();  // the copy's space is free

    unsigned long long *ex = reinterpret_cast<unsigned long long *>(sm);
    float *pub = reinterpret_cast<float *>(sm + S::kOffPub);
    float *out = reinterpret_cast<float *>(sm + S::kOffOut);
    float *rulef = reinterpret_cast<float *>(sm + S::kOffRule);  // [9][kRules]: attributes, LinkRule
    uint32_t *ruleu = reinterpret_cast<uint32_t *>(rulef);
    constexpr uint32_t kAttrRamp = 1u << 31;
    unsigned long long *den = reinterpret_cast<unsigned long long *>(sm + S::kOffDen);
    const F2 w2 = splat<F2>(L.omega), s32 = splat<F2>(rmul(L.src, 1.0f / 3.0f));
    float nonfinite = 0.0f;  // the last step's moments, summed: non-finite if any one is

#pragma unroll 1
    for (int l = 0; l < nsteps; ++l) {
        if (npub) {
            // the populations that the boundary rules read
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (!((rowflag >> r) & 1u)) continue;
                const uint32_t sa = slot[r] & 0xffffu, sb = slot[r] >> 16;
                float lo[9], hi[9];
#pragma unroll
                for (int i = 0; i < 9; ++i) f2_split(f[r][i], lo[i], hi[i]);
                if (sa != kNone) put9(pub + sa * 12, lo);
                if (sb != kNone) put9(pub + sb * 12, hi);
            }
        }
        // streaming along x
#pragma unroll
        for (int r = 0; r < R; ++r) {
            f[r][1] = from_left<LPR>(f[r][1]);
            f[r][5] = from_left<LPR>(f[r][5]);
            f[r][8] = from_left<LPR>(f[r][8]);
            f[r][3] = from_right<LPR>(f[r][3]);
            f[r][6] = from_right<LPR>(f[r][6]);
            f[r][7] = from_right<LPR>(f[r][7]);
        }
        // ... and along y: the outermost rows go to the neighbouring groups
        // (buffers alternate, so one barrier per step orders them)
        unsigned long long *eu = ex + (size_t)(l & 1) * 2 * G * 3 * LPR, *ed = eu + G * 3 * LPR;
        eu[(g * 3 + 0) * LPR + t] = f[R - 1][2].v;
        eu[(g * 3 + 1) * LPR + t] = f[R - 1][5].v;
        eu[(g * 3 + 2) * LPR + t] = f[R - 1][6].v;
        ed[(g * 3 + 0) * LPR + t] = f[0][4].v;
        ed[(g * 3 + 1) * LPR + t] = f[0][7].v;
        ed[(g * 3 + 2) * LPR + t] = f[0][8].v;
        __syncthreads();
        if (npub) {
            // one cut link to a thread; the part of its rule that the populations
            // do not enter is formed again only when its boundary data change
            // (a ramp, or the load coming on at time 0)
            const float tb = tb0 + (float)l;  // boundary data at the time of f^col
#pragma unroll 1
            for (int e = tid; e < nlink; e += kNT) {
                uint32_t attr;
                LinkRule rule;
                bool fresh = l == 0 || tb == 0.0f || e >= S::kRules;
                if (!fresh) {
                    attr = ruleu[e];
                    fresh = (attr & kAttrRamp) != 0;
                }
                if (fresh) {
                    const TileLink lk = links[rec.link0 + e];
                    const int i = lk.dir, kk = i <= 4 ? (i + 1) % 4 + 1 : (i - 3) % 4 + 5;
                    const BLink b{lk.q, lk.n0, lk.n1, lk.bc, lk.bc2};
                    // slots, direction, flags (an upstream node not read: the node itself)
                    attr = lk.own | (uint32_t)((lk.flags & kLinkUpstream) ? lk.up : lk.own) << 10 |
                           (uint32_t)kk << 20 | (uint32_t)lk.flags << 24;
                    if (bcs[lk.bc].profile == LBM_PROFILE_RAMP || bcs[lk.bc2].profile == LBM_PROFILE_RAMP)
                        attr |= kAttrRamp;
                    rule = link_rule(kk, lk.flags & kLinkMiss, lk.flags & kLinkDirichlet,
                                     lk.flags & kLinkCorner, b, bcs, tb, L);
                    if (e < S::kRules) {
                        ruleu[e] = attr;
                        const float v[8] = {rule.q, rule.kap, rule.fac, rule.t0,
                                            rule.t1, rule.c0, rule.c1, rule.c2};
#pragma unroll
                        for (int m = 0; m < 8; ++m) rulef[(1 + m) * S::kRules + e] = v[m];
                    }
                } else {
                    float v[8];
#pragma unroll
                    for (int m = 0; m < 8; ++m) v[m] = rulef[(1 + m) * S::kRules + e];
                    rule = LinkRule{v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7]};
                }
                const int k = (attr >> 20) & 15u, i = k <= 4 ? (k + 1) % 4 + 1 : (k - 3) % 4 + 5;
                const uint32_t flags = attr >> 24, own = attr & 1023u;
                const float *gp = pub + own * 12, *yp = pub + ((attr >> 10) & 1023u) * 12;
                float gx[9];
                get9(gp, gx);
                const Mom mx = moments(gx);
                float gy[9];
                get9(yp, gy);
                const Mom my = moments(gy);
                // kappa = 0 at a mid-link wall: its upstream population does not count
                const float gy_i = (flags & kLinkUpstream) ? yp[i] : 0.0f;
                out[own * 8 + k - 1] =
                    link_value(k, rule, flags & kLinkDirichlet, flags & kLinkCorner,
                               flags & kLinkExtrapolate, gp[k], gp[i], gy_i, mx.dr, mx.pxx, mx.pyy, mx.pxy, my.dr, my.pxx, my.pyy,
                               my.pxy, L);
            }
        }
#pragma unroll
        for (int r = R - 1; r > 0; --r) {
            f[r][2] = f[r - 1][2];
            f[r][5] = f[r - 1][5];
            f[r][6] = f[r - 1][6];
        }
#pragma unroll
        for (int r = 0; r < R - 1; ++r) {
            f[r][4] = f[r + 1][4];
            f[r][7] = f[r + 1][7];
            f[r][8] = f[r + 1][8];
        }
        {
            // the ring's outermost rows take some group's values: they are halo
            const int gm = g > 0 ? g - 1 : 0, gp = g < G - 1 ? g + 1 : g;
            f[0][2] = as_f2(eu[(gm * 3 + 0) * LPR + t]);
            f[0][5] = as_f2(eu[(gm * 3 + 1) * LPR + t]);
            f[0][6] = as_f2(eu[(gm * 3 + 2) * LPR + t]);
            f[R - 1][4] = as_f2(ed[(gp * 3 + 0) * LPR + t]);
            f[R - 1][7] = as_f2(ed[(gp * 3 + 1) * LPR + t]);
            f[R - 1][8] = as_f2(ed[(gp * 3 + 2) * LPR + t]);
        }
        if (npub) {
            __syncthreads();
            // the populations that arrive through cut links
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (!((rowflag >> r) & 1u)) continue;
                const uint32_t sa = slot[r] & 0xffffu, sb = slot[r] >> 16;
                // every lane reads (slot 0 where it has none): no lane waits for another
                const uint32_t ca = sa != kNone ? cutm[sa] : 0u, cb = sb != kNone ? cutm[sb] : 0u;
                const float4 *oa = reinterpret_cast<const float4 *>(out + (sa != kNone ? sa : 0u) * 8);
                const float4 *ob = reinterpret_cast<const float4 *>(out + (sb != kNone ? sb : 0u) * 8);
                const float4 a0 = oa[0], a1 = oa[1], b0 = ob[0], b1 = ob[1];
                const float va[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
                const float vb[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
                for (int k = 1; k < 9; ++k) {
                    float lo, hi;
                    f2_split(f[r][k], lo, hi);
                    lo = ((ca >> (opp(k) - 1)) & 1u) ? va[k - 1] : lo;
                    hi = ((cb >> (opp(k) - 1)) & 1u) ? vb[k - 1] : hi;
                    f[r][k] = f2(lo, hi);
                }
            }
        }
        F2 dn[GRAD ? R : 1], dbelow, dabove;
        if constexpr (GRAD) {
            // densities at this time level, for the gradient in the source
#pragma unroll
            for (int r = 0; r < R; ++r) dn[r] = density_of(f[r]);
            den[g * LPR + t] = dn[R - 1].v;
            den[(G + g) * LPR + t] = dn[0].v;
            __syncthreads();
            dbelow = as_f2(den[(g > 0 ? g - 1 : 0) * LPR + t]);
            dabove = as_f2(den[(G + (g < G - 1 ? g + 1 : g)) * LPR + t]);
        }
        const bool last = l == nsteps - 1;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            F2 sx = f2(L.fx, L.fx), sy = f2(L.fy, L.fy);
            if constexpr (GRAD) {
                const F2 rxp = from_right<LPR>(dn[r]), rxm = from_left<LPR>(dn[r]);
                const F2 ryp = r < R - 1 ? dn[r < R - 1 ? r + 1 : r] : dabove;
                const F2 rym = r > 0 ? dn[r > 0 ? r - 1 : 0] : dbelow;
                if ((rowflag >> r) & 1u) {
                    // one-sided where an axis neighbour is across a wall
                    const uint32_t sa = slot[r] & 0xffffu, sb = slot[r] >> 16;
                    const uint32_t ca = sa != kNone ? cutm[sa] : 0u, cb = sb != kNone ? cutm[sb] : 0u;
                    float d[2], xp[2], xm[2], yp[2], ym[2], hx[2], hy[2];
                    f2_split(dn[r], d[0], d[1]);
                    f2_split(rxp, xp[0], xp[1]);
                    f2_split(rxm, xm[0], xm[1]);
                    f2_split(ryp, yp[0], yp[1]);
                    f2_split(rym, ym[0], ym[1]);
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const uint32_t c = j ? cb : ca;
                        grad_source(d[j], xp[j], xm[j], yp[j], ym[j], !(c & 1u), !(c & 4u), !(c & 2u),
                                    !(c & 8u), L, hx[j], hy[j]);
                    }
                    sx = f2(hx[0], hx[1]);
                    sy = f2(hy[0], hy[1]);
                } else {
                    grad_source_open(dn[r], rxp, rxm, ryp, rym, L, sx, sy);
                }
            }
            F2 dr, jx, jy;
            collide_v(f[r], sx, sy, w2, s32, dr, jx, jy);
            if ((corerow >> r) & 1u) {
                // both nodes of every lane, without branches: records of nodes
                // outside the core are never stored
                float dra, drb, jxa, jxb, jya, jyb;
                f2_split(dr, dra, drb);
                f2_split(jx, jxa, jxb);
                f2_split(jy, jya, jyb);
                float4 *ua = us + (2 * r) * kNT + tid, *ub = ua + kNT;
                float4 wa = *ua, wb = *ub;
                integrate_u_value(wa, jxa, jya, L.rho0 + dra);
                integrate_u_value(wb, jxb, jyb, L.rho0 + drb);
                *ua = wa;
                *ub = wb;
                if (last) {
                    const uint32_t m = (mine >> (2 * r)) & 3u;
                    const float na = radd(radd(dra, jxa), jya), nb = radd(radd(drb, jxb), jyb);
                    nonfinite = radd(nonfinite, radd(m & 1u ? na : 0.0f, m & 2u ? nb : 0.0f));
                }
            }
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const uint32_t m = (mine >> (2 * r)) & 3u;
        if (!m) continue;
        const int64_t k = k0 + (int64_t)r * L.pitch;
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            float *o = dst + i * L.fplane + k;
            float lo, hi;
            f2_split(f[r][i], lo, hi);
            if (m == 3u) {
                *reinterpret_cast<float2 *>(o) = make_float2(lo, hi);
            } else if (m & 1u) {
                o[0] = lo;
            } else {
                o[1] = hi;
            }
        }
        if (m & 1u) uc[k] = us[(2 * r) * kNT + tid];
        if (m & 2u) uc[k + 1] = us[(2 * r + 1) * kNT + tid];
    }
    if (!isfinite(nonfinite)) flag_nonfinite(status, nonfinite, 0.0f, 0.0f);
}

template <int LPR, int R, bool GRAD>
__global__ void __launch_bounds__(kNT, 1)
    k_tile(const __grid_constant__ CUtensorMap tf, float *__restrict__ dst, float4 *__restrict__ uc,
           const uint8_t *__restrict__ cls, const TileRec *__restrict__ tiles,
           const uint32_t *__restrict__ pubs, const TileLink *__restrict__ links,
           const BCDev *__restrict__ bcs, Lattice L, const int64_t *__restrict__ time, int toff,
           int nsteps, uint32_t *__restrict__ status) {
    extern __shared__ __align__(1024) unsigned char sm[];
    release_next();
    const TileRec rec = tiles[blockIdx.x];
    tile_steps<LPR, R, GRAD>(&tf, dst, uc, cls, rec, pubs, links, bcs, L, time, toff, nsteps, status,
                             sm);
}

// The tiles of many lattices in one launch (a batch, lambda = mu): a tile's
// instance supplies its buffers, tables and lattice parameters.
template <int LPR, int R>
__global__ void __launch_bounds__(kNT, 1)
    k_tile_batch(const TileInst *__restrict__ insts, const TileRec *__restrict__ tiles,
                 const uint32_t *__restrict__ pubs, const TileLink *__restrict__ links, int cur,
                 int toff, int nsteps) {
    extern __shared__ __align__(1024) unsigned char sm[];
    __shared__ __align__(16) Lattice s_L;
    release_next();
    const TileRec rec = tiles[blockIdx.x];
    const TileInst *I = insts + rec.inst;
    constexpr int kWords = (int)(sizeof(Lattice) / 4);
    if (threadIdx.x < kWords)
        reinterpret_cast<uint32_t *>(&s_L)[threadIdx.x] =
            reinterpret_cast<const uint32_t *>(&I->L)[threadIdx.x];
    __syncthreads();
    tile_steps<LPR, R, false>(&I->map[cur], I->f[cur ^ 1], I->uc, I->cls, rec, pubs, links, I->bcs, s_L,
                              I->time, toff, nsteps, I->status, sm);
}

template <int LPR, int R> cudaError_t batch_shape(const TileBatch &B, int cur, int toff, int nsteps,
                                                  cudaStream_t s) {
    static const cudaError_t attr_set = cudaFuncSetAttribute(
        k_tile_batch<LPR, R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Shape<LPR, R>::kSmem);
    if (attr_set != cudaSuccess || B.ntiles <= 0) return attr_set;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)B.ntiles);
    cfg.blockDim = dim3(kNT);
    cfg.dynamicSmemBytes = Shape<LPR, R>::kSmem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_tile_batch<LPR, R>, B.insts, B.tiles, B.pubs, B.links, cur, toff,
                              nsteps);
}

template <int LPR, int R, bool GRAD>
cudaError_t launch_shape(const Lattice &L, const DevState &S, const TileDev &T, int cur, int toff,
                         int nsteps, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)T.ntiles);
    cfg.blockDim = dim3(kNT);
    cfg.dynamicSmemBytes = Shape<LPR, R>::kSmem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_tile<LPR, R, GRAD>, T.map[cur], static_cast<float *>(S.f[cur ^ 1]),
                              static_cast<float4 *>(S.ucomp), (const uint8_t *)S.cls, T.tiles, T.pubs,
                              T.links, (const BCDev *)S.bcs, L, (const int64_t *)S.time, toff, nsteps,
                              S.status);
}

template <int LPR, int R>
bool encode_shape(const Lattice &L, const DevState &S, CUtensorMap map[2]) {
    using Sh = Shape<LPR, R>;
    const cuuint64_t dims[3] = {(cuuint64_t)L.nx, (cuuint64_t)L.ny, 9};
    const cuuint64_t str[2] = {(cuuint64_t)L.pitch * 4, (cuuint64_t)L.fplane * 4};
    const cuuint32_t box[3] = {(cuuint32_t)Sh::W, (cuuint32_t)Sh::H, 9};
    for (int b = 0; b < 2; ++b)
        if (!encode(&map[b], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, S.f[b], dims, str, box)) return false;
    return true;
}

template <int LPR, int R> cudaError_t prepare_shape(const Lattice &L, const DevState &S, TileDev *T) {
    using Sh = Shape<LPR, R>;
    if (!encode_shape<LPR, R>(L, S, T->map)) return cudaErrorInvalidValue;
    return L.grad ? cudaFuncSetAttribute(k_tile<LPR, R, true>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Sh::kSmem)
                  : cudaFuncSetAttribute(k_tile<LPR, R, false>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Sh::kSmem);
}

}  // namespace

bool tile_supported() { return encoder() != nullptr; }

cudaError_t tile_prepare(const Lattice &L, const DevState &S, TileDev *T) {
    switch (T->shape) {
        case 0: return prepare_shape<16, 1>(L, S, T);
        case 1: return prepare_shape<32, 2>(L, S, T);
        case 2: return prepare_shape<32, 3>(L, S, T);
        default: return prepare_shape<32, 4>(L, S, T);
    }
}

cudaError_t launch_tile(const Lattice &L, const DevState &S, const TileDev &T, int cur, int toff,
                        int nsteps, cudaStream_t s) {
#define LBM_TILE(n, lpr, r)                                                                  \
    case n:                                                                                  \
        return L.grad ? launch_shape<lpr, r, true>(L, S, T, cur, toff, nsteps, s)            \
                      : launch_shape<lpr, r, false>(L, S, T, cur, toff, nsteps, s);
    switch (T.shape) {
        LBM_TILE(0, 16, 1)
        LBM_TILE(1, 32, 2)
        LBM_TILE(2, 32, 3)
        LBM_TILE(3, 32, 4)
    }
#undef LBM_TILE
    return cudaErrorInvalidValue;
}

bool tile_maps(const Lattice &L, const DevState &S, int shape, CUtensorMap map[2]) {
    switch (shape) {
        case 0: return encode_shape<16, 1>(L, S, map);
        case 1: return encode_shape<32, 2>(L, S, map);
        case 2: return encode_shape<32, 3>(L, S, map);
        default: return encode_shape<32, 4>(L, S, map);
    }
}

cudaError_t launch_tile_batch(const TileBatch &B, int cur, int toff, int nsteps, cudaStream_t s) {
    switch (B.shape) {
        case 0: return batch_shape<16, 1>(B, cur, toff, nsteps, s);
        case 1: return batch_shape<32, 2>(B, cur, toff, nsteps, s);
        case 2: return batch_shape<32, 3>(B, cur, toff, nsteps, s);
        default: return batch_shape<32, 4>(B, cur, toff, nsteps, s);
    }
}

}  // namespace lbm
