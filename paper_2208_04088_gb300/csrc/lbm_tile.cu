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
// Tiles without boundary nodes (most of a large lattice) take tile_interior:
// the populations of the block's next tile arrive while this one steps, and the
// block's warps meet at a split barrier.  Tiles with them take tile_steps.
//
// What bounds it: instruction issue in the tiles of a large lattice (a 64 x 64
// tile updates 4096 nodes per step, 42 paired operations per pair and 7 paired
// ones per node for the displacement, of which the core's 48 x 48 count; about
// as many moves, shuffles and address operations go with them).  One interior
// 64 x 64 tile, 8 steps: 14 us, of which 1.3 us a step (1350 cycles of FP32
// work in 2740).  On lattices of less than a few hundred thousand nodes it is
// the latency of one step (two block barriers, the collision's and a link's
// dependent chain: 2 us in a 32 x 32 tile) and of the launch.  2048^2 edge
// crack, 500 steps: 11.7 ms (strips 18.9); with lambda != mu 21.7 (one step per
// launch 44.8); 1024 x 512 plate with a hole, 600 steps: 2.57 (4.26).
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
    static constexpr size_t kEnd = kOffU + (size_t)W * H * 16;
    static_assert(W <= 256 && H <= 256, "copy box");
};

// Shared memory of a tile without boundary nodes: the populations of the next
// tile arrive while this one steps, so nothing shares their space; records of
// the core only; the row exchange in two buffers (one when lambda != mu, whose
// second barrier per step orders its reuse), and the densities' exchange.
template <int R, bool GRAD> struct Inner {
    using S = Shape<32, R>;
    static constexpr int CW = S::W - 2 * kTileHalo, CH = S::H - 2 * kTileHalo;
    static constexpr size_t kOffU = S::kStage;
    static constexpr size_t kOffEx = kOffU + (size_t)CW * CH * 16;
    static constexpr int kExOne = 2 * (S::G - 1) * 3 * 32;  // words of one buffer
    static constexpr size_t kOffDen = kOffEx + (size_t)(GRAD ? 1 : 2) * kExOne * 8;
    static constexpr size_t kEnd = kOffDen + (GRAD ? (size_t)2 * (S::G - 1) * 32 * 8 : 0);
};

// Barriers and block-wide values, behind the larger of the two layouts.
struct Control {
    unsigned long long load, step, den;  // mbarriers: copy landed, rows exchanged, densities exchanged
    int landed, next;                    // the copy landed in time; the block's next tile
    int lost, pad2;                      // a wait between the block's warps ran out
    TileRec rec;                         // its record
    float4 *uc;                          // and its displacement records
    int pitch, pad;
};
template <int LPR, int R, bool GRAD> __host__ __device__ constexpr size_t control_at() {
    if constexpr (LPR == 32)
        return ((Shape<LPR, R>::kEnd > Inner<R, GRAD>::kEnd ? Shape<LPR, R>::kEnd
                                                            : Inner<R, GRAD>::kEnd) + 127) / 128 * 128;
    else
        return (Shape<LPR, R>::kEnd + 127) / 128 * 128;
}
template <int LPR, int R, bool GRAD> constexpr size_t smem_bytes() {
    static_assert(control_at<LPR, R, GRAD>() + sizeof(Control) + 1024 <= 232448,
                  "shared memory of one block (with the static part of a batch)");
    return control_at<LPR, R, GRAD>() + sizeof(Control);
}

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

// The rule of a tile's link at boundary time tb, and its attributes: slots of
// its node and of the upstream node (the node itself if it is not read),
// direction it arrives in, flags, and whether its data change with time.
constexpr uint32_t kAttrRamp = 1u << 31;
__device__ __forceinline__ LinkRule make_rule(const TileLink &lk, const BCDev *__restrict__ bcs,
                                              float tb, const Lattice &L, uint32_t &attr) {
    const int i = lk.dir, k = i <= 4 ? (i + 1) % 4 + 1 : (i - 3) % 4 + 5;
    const BLink b{lk.q, lk.n0, lk.n1, lk.bc, lk.bc2};
    attr = lk.own | (uint32_t)((lk.flags & kLinkUpstream) ? lk.up : lk.own) << 10 | (uint32_t)k << 20 |
           (uint32_t)lk.flags << 24;
    if (bcs[lk.bc].profile == LBM_PROFILE_RAMP || bcs[lk.bc2].profile == LBM_PROFILE_RAMP)
        attr |= kAttrRamp;
    return link_rule(k, lk.flags & kLinkMiss, lk.flags & kLinkDirichlet, lk.flags & kLinkCorner, b, bcs,
                     tb, L);
}

// A wait that did not end at the first try, out of the step's code: 2048^2 crack
// 11.42 ms, 11.79 with it inline (lambda != mu keeps it inline: 21.7, 23.7).
__device__ __noinline__ bool wait_on(uint32_t bar, uint32_t parity, int64_t limit) {
    return mbar_wait(bar, parity, limit);
}

// Programmatic launch order: the next launch of the stream may start its
// prologue now, and this one has waited for everything before it.
__device__ __forceinline__ void release_next() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void wait_for_previous() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Between the two kernels of a launch (see Part): a block of the first counts
// itself in counter[kReady], with what the launch before wrote behind it; the
// second has all of that once it reads the count of every block.
constexpr int kReady = 2;
__device__ __forceinline__ void say_ready(int32_t *counter) {
    int before;
    asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], 1;"
                 : "=r"(before)
                 : "l"(counter + kReady)
                 : "memory");
    if (before >= 0) release_next();  // (always) not before the count has arrived
}
__device__ __forceinline__ bool all_ready(const int32_t *counter, int blocks) {
    int n;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(n) : "l"(counter + kReady) : "memory");
    return n == blocks;
}

// Copies a tile's populations into the space at the start of shared memory.
template <int LPR, int R>
__device__ __forceinline__ void issue_load(const CUtensorMap *tf, const TileRec &rec, uint32_t bar,
                                           unsigned char *sm) {
    // order the block's earlier shared-memory accesses before the copy
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    mbar_expect_tx(bar, (uint32_t)Shape<LPR, R>::kStage);
    tma_load_3d(smem_addr(sm), tf, rec.x0, rec.y0, 0, bar);
}

// Block-wide wait for the copy; false after the wait limit: the launch is
// flagged, and the copy waited out so that none is in flight when the block
// exits.  A limit of 0 gives up at once, whether or not the copy has landed.
__device__ __forceinline__ bool load_landed(Control *c, uint32_t bar, uint32_t parity,
                                            const Lattice &L, uint32_t *status) {
    if (threadIdx.x == 0) {
        const bool ok = L.wait_ns > 0 && mbar_wait(bar, parity, L.wait_ns);
        *reinterpret_cast<volatile int *>(&c->landed) = ok;
        if (!ok) {
            atomicOr(status, 2u);
            mbar_wait(bar, parity, kDefaultWaitNs);
        }
    }
    __syncthreads();
    return *reinterpret_cast<volatile int *>(&c->landed) != 0;
}
__device__ __forceinline__ bool is_lost(const Control *c) {
    return *reinterpret_cast<const volatile int *>(&c->lost) != 0;
}

// nsteps steps of one tile, any tile; the first is step `toff` after *time.
// `first`: the block's first tile (it waits for the previous launch once its
// tables are read).  Returns false when the copy did not land in time.
// ready: counter to release the next kernel with (say_ready) once the previous
// launch is over, or null (released before).
// SRC: the source S is not zero (a body force, or the gradient's).
template <int LPR, int R, bool GRAD, bool SRC>
__device__ __forceinline__ bool tile_steps(const CUtensorMap *tf, float *__restrict__ dst,
                                           float4 *__restrict__ uc,
                                           const uint8_t *__restrict__ cls, const TileRec &rec,
                                           const uint32_t *__restrict__ pubs,
                                           const TileLink *__restrict__ links,
                                           const BCDev *__restrict__ bcs, const Lattice &L,
                                           const int64_t *__restrict__ time, int toff, int nsteps,
                                           uint32_t *__restrict__ status, unsigned char *sm,
                                           Control *ctl, bool first, int32_t *ready,
                                           uint32_t load_parity) {
    using S = Shape<LPR, R>;
    constexpr int W = S::W, H = S::H, G = S::G;
    const int tid = threadIdx.x, t = tid % LPR, g = tid / LPR;
    const int c0 = 2 * t, row0 = g * R;
    const uint32_t bar = smem_addr(&ctl->load);
    float4 *us = reinterpret_cast<float4 *>(sm + S::kOffU);

    // the previous launch writes nothing that is read before wait_for_previous()
    constexpr uint32_t kNone = 0xffffu;
    const int npub = rec.npub, nlink = rec.nlink;
    // The rule of the thread's (first) link stays in registers where the tile
    // leaves room for it, in shared memory otherwise (350 cycles a step).
    constexpr bool kKeep = R == 1 || (R == 2 && !GRAD);
    // cut masks in registers likewise
    constexpr bool kCuts = !GRAD || R <= 2;
    uint8_t *cutm = sm + S::kOffCut;
    uint32_t slot[R];       // slots of the thread's published nodes (low, high half)
    uint32_t cuts[(R + 1) / 2];  // their cut masks, a byte per node (kCuts)
    uint32_t rowflag = 0;   // rows in which a lane of the warp has one (warp-uniform)
#pragma unroll
    for (int r = 0; r < R; ++r) slot[r] = 0xffffffffu;
#pragma unroll
    for (int r = 0; r < (R + 1) / 2; ++r) cuts[r] = 0;
    // The last warp starts the copy (in a block's first tile once the previous
    // launch is over) while the others read the tile's tables.
    constexpr int kReaders = kNT - 32;
    if (tid == kReaders) {
        if (first) wait_for_previous();
        issue_load<LPR, R>(tf, rec, bar, sm);
    }
    if (npub) {  // uniform over the block
        uint32_t *map = reinterpret_cast<uint32_t *>(sm + S::kOffSlot);
        if (tid < kReaders) {
            for (int q = tid; q < W * H / 2; q += kReaders) map[q] = 0xffffffffu;
            asm volatile("barrier.cta.sync 1, %0;" ::"n"(kReaders) : "memory");
            for (int q = tid; q < npub; q += kReaders) {
                const uint32_t p = pubs[rec.pub0 + q];
                reinterpret_cast<uint16_t *>(map)[((p >> 8) & 0xffu) * W + (p & 0xffu)] = (uint16_t)q;
                cutm[q] = (uint8_t)(p >> 16);
            }
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < R; ++r) {
            slot[r] = map[((row0 + r) * W + c0) / 2];
            const uint32_t sa = slot[r] & 0xffffu, sb = slot[r] >> 16;
            if (kCuts) cuts[r / 2] |= ((sa != kNone ? cutm[sa] : 0u) | (sb != kNone ? cutm[sb] : 0u) << 8)
                           << (16 * (r & 1));
            if (__ballot_sync(0xffffffffu, slot[r] != 0xffffffffu)) rowflag |= 1u << r;
        }
    }
    // the cut masks of row r's two nodes
    auto cut_masks = [&](int r) -> uint32_t {
        if (kCuts) return cuts[r / 2] >> (16 * (r & 1));
        const uint32_t sa = slot[r] & 0xffffu, sb = slot[r] >> 16;
        return (sa != kNone ? cutm[sa] : 0u) | (sb != kNone ? cutm[sb] : 0u) << 8;
    };
    TileLink my_link;
    if (kKeep && tid < nlink) my_link = links[rec.link0 + tid];
    if (first) wait_for_previous();
    if (ready && tid == 0) say_ready(ready);
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
    uint32_t my_attr = 0;
    LinkRule my_rule{};
    if (kKeep && tid < nlink) my_rule = make_rule(my_link, bcs, tb0, L, my_attr);
    if (!load_landed(ctl, bar, load_parity, L, status)) return false;
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
    unsigned long long *den = reinterpret_cast<unsigned long long *>(sm + S::kOffDen);
    const Relax<F2> rc = relax_of<F2>(L);
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
                uint32_t attr = my_attr;
                LinkRule rule = my_rule;
                const bool mine_kept = kKeep && e == tid;
                bool fresh = tb == 0.0f || (!mine_kept && (l == 0 || e >= S::kRules));
                if (!fresh) {
                    if (!mine_kept) attr = ruleu[e];
                    fresh = (attr & kAttrRamp) != 0;
                }
                if (fresh) {
                    // tb is rounded twice where tb0 is no longer exact (2^24)
                    const float at = tb0 < 16777216.0f ? tb : (float)(*time + toff - 1 + l);
                    rule = make_rule(links[rec.link0 + e], bcs, at, L, attr);
                    if (mine_kept) {
                        my_rule = rule;
                    } else if (e < S::kRules) {
                        ruleu[e] = attr;
                        const float v[8] = {rule.q, rule.kap, rule.fac, rule.t0,
                                            rule.t1, rule.c0, rule.c1, rule.c2};
#pragma unroll
                        for (int m = 0; m < 8; ++m) rulef[(1 + m) * S::kRules + e] = v[m];
                    }
                } else if (!mine_kept) {
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
                const Mom mx = moments<kSums32>(gx);
                float gy[9];
                get9(yp, gy);
                const Mom my = moments<kSums32>(gy);
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
                const uint32_t ca = cut_masks(r), cb = ca >> 8;
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
        const int reach = (GRAD ? 2 : 1) * (nsteps - 1 - l);  // rows around the core still needed
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (!__any_sync(0xffffffffu, row0 + r >= rec.r0 - reach && row0 + r < rec.r1 + reach))
                continue;
            F2 sx = f2(L.fx, L.fx), sy = f2(L.fy, L.fy);
            if constexpr (GRAD) {
                const F2 rxp = from_right<LPR>(dn[r]), rxm = from_left<LPR>(dn[r]);
                const F2 ryp = r < R - 1 ? dn[r < R - 1 ? r + 1 : r] : dabove;
                const F2 rym = r > 0 ? dn[r > 0 ? r - 1 : 0] : dbelow;
                if ((rowflag >> r) & 1u) {
                    // one-sided where an axis neighbour is across a wall
                    const uint32_t ca = cut_masks(r), cb = ca >> 8;
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
            collide_sums<SRC>(f[r], sx, sy, rc, dr, jx, jy);
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
    return true;
}

// Two adjacent records (32 bytes, aligned) in one store.
__device__ __forceinline__ void store_pair_records(float4 *p, const float4 &a, const float4 &b) {
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(a.x), "f"(a.y),
                 "f"(a.z), "f"(a.w), "f"(b.x), "f"(b.y), "f"(b.z), "f"(b.w)
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void copy16(uint32_t dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// nsteps steps of a tile without boundary nodes (every node of its ring is
// interior, its core the ring without the halo).  The block's warps meet once
// per step (twice when lambda != mu) at an mbarrier that they arrive at when
// their outermost rows are posted and wait at only when they need their
// neighbours': in between they update their inner rows, so no warp waits for
// the slowest one's whole step.  Thread 0 takes the block's next tile during
// the first steps (take_next fills ctl->next, rec, uc, pitch) and copies its
// populations in behind this tile's; each thread fetches the displacement
// records of its own nodes of the next tile as soon as those of this one are
// stored.  early: it does (a launch of too few steps takes the next tile
// afterwards); loaded: the tile before this one did.
//
// A wait of the warps for one another that runs out flags the block (ctl->lost),
// which flags the launch once the tile is over.  The warp goes on, arriving as
// before, so no later wait is longer than the limit either, but a phase may then
// end without every warp.  It cannot end so unseen: the flag is stored before the
// warp's next arrival, which releases it to whoever that arrival lets through.
// So a warp that finds the flag clear once its last wait is over has been given
// everything it used, its neighbours' rows and thread 0's words on the next tile;
// where the flag is set it stores nothing, copies nothing for the next tile, and
// the block takes no other one.
template <int R, bool GRAD, bool SRC, class Next>
__device__ __forceinline__ bool tile_interior(const CUtensorMap *tf, float *__restrict__ dst,
                                              float4 *__restrict__ uc, const TileRec &rec,
                                              const Lattice &L, int nsteps,
                                              uint32_t *__restrict__ status, unsigned char *sm,
                                              Control *ctl, bool first, bool loaded, bool early,
                                              uint32_t load_parity, uint32_t &phase,
                                              uint32_t &dphase,
                                              const Next &take_next) {
    using S = Shape<32, R>;
    using I = Inner<R, GRAD>;
    constexpr int W = S::W, H = S::H, G = S::G, HL = kTileHalo;
    const int tid = threadIdx.x, t = tid & 31, g = tid >> 5;
    const int c0 = 2 * t, row0 = g * R;
    const uint32_t bar = smem_addr(&ctl->load), bstep = smem_addr(&ctl->step), bden = smem_addr(&ctl->den);
    const bool core = c0 >= HL && c0 < W - HL;  // the core's edges lie between pairs
    // the thread's record of row r, column c0 + j: [core row][j][core pair]
    float4 *us = reinterpret_cast<float4 *>(sm + I::kOffU) + (row0 - HL) * I::CW +
                 (core ? t - HL / 2 : 0);
    unsigned long long *ex = reinterpret_cast<unsigned long long *>(sm + I::kOffEx);
    unsigned long long *den = reinterpret_cast<unsigned long long *>(sm + I::kOffDen);
    auto core_row = [&](int r) { return row0 + r >= HL && row0 + r < H - HL; };  // warp-uniform

    if (first) wait_for_previous();
    if (tid == 0 && !loaded) issue_load<32, R>(tf, rec, bar, sm);
    const int64_t k0 = (int64_t)(rec.y0 + row0) * L.pitch + rec.x0 + c0;
    if (!loaded && core && rec.c1 > rec.c0) {
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (core_row(r)) {
                copy16(smem_addr(us + r * I::CW), uc + k0 + (int64_t)r * L.pitch);
                copy16(smem_addr(us + r * I::CW + I::CW / 2), uc + k0 + (int64_t)r * L.pitch + 1);
            }
    }
    if (!load_landed(ctl, bar, load_parity, L, status) || is_lost(ctl)) {
        copy_wait();
        return false;
    }
    if (rec.c1 == rec.c0) return true;  // no material in the whole lattice, nothing copied behind it
    F2 f[R][9];
    {
        // pulled along y by the address (the ring's outermost rows, halo, by
        // whatever row is there)
        const unsigned long long *st = reinterpret_cast<const unsigned long long *>(sm);
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                int y = row0 + r - c_cy(i);
                if (r == 0 && c_cy(i) > 0) y = max(y, 0);
                if (r == R - 1 && c_cy(i) < 0) y = min(y, H - 1);
                f[r][i] = as_f2(st[((i * H + y) * W + c0) / 2]);
            }
    }
    auto shift_x = [&](int r) {
        f[r][1] = from_left<32>(f[r][1]);
        f[r][5] = from_left<32>(f[r][5]);
        f[r][8] = from_left<32>(f[r][8]);
        f[r][3] = from_right<32>(f[r][3]);
        f[r][6] = from_right<32>(f[r][6]);
        f[r][7] = from_right<32>(f[r][7]);
    };
    // the end of a phase of a barrier that the block's warps meet at
    auto meet = [&](uint32_t at, uint32_t parity) {
        if (GRAD ? !mbar_wait(at, parity, L.wait_ns)
                 : !mbar_try_wait(at, parity) && !wait_on(at, parity, L.wait_ns))
            *reinterpret_cast<volatile int *>(&ctl->lost) = 1;
    };
    // the outermost rows to the neighbouring warps
    auto post = [&](int l) {
        unsigned long long *eu = ex + (GRAD ? 0 : (l & 1) * I::kExOne) + t, *ed = eu + (G - 1) * 96;
        if (g < G - 1) {
            eu[(g * 3 + 0) * 32] = f[R - 1][2].v;
            eu[(g * 3 + 1) * 32] = f[R - 1][5].v;
            eu[(g * 3 + 2) * 32] = f[R - 1][6].v;
        }
        if (g > 0) {
            ed[(g * 3 - 3) * 32] = f[0][4].v;
            ed[(g * 3 - 2) * 32] = f[0][7].v;
            ed[(g * 3 - 1) * 32] = f[0][8].v;
        }
        __syncwarp();
        if (t == 0) mbar_arrive(bstep);
    };
    // rows one up and one down, the outermost from the neighbours
    auto take = [&](int l) {
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
        meet(bstep, phase);
        phase ^= 1;
        const unsigned long long *eu = ex + (GRAD ? 0 : (l & 1) * I::kExOne) + t, *ed = eu + (G - 1) * 96;
        if (g > 0) {
            f[0][2] = as_f2(eu[(g * 3 - 3) * 32]);
            f[0][5] = as_f2(eu[(g * 3 - 2) * 32]);
            f[0][6] = as_f2(eu[(g * 3 - 1) * 32]);
        }
        if (g < G - 1) {
            f[R - 1][4] = as_f2(ed[(g * 3 + 0) * 32]);
            f[R - 1][7] = as_f2(ed[(g * 3 + 1) * 32]);
            f[R - 1][8] = as_f2(ed[(g * 3 + 2) * 32]);
        }
    };
    const Relax<F2> rc = relax_of<F2>(L);
    float nonfinite = 0.0f;
    copy_wait();
#pragma unroll
    for (int r = 0; r < R; ++r) shift_x(r);
    auto step = [&](int l, auto is_last) {
        constexpr bool last = decltype(is_last)::value;
        const int reach = (GRAD ? 2 : 1) * (nsteps - 1 - l);  // rows around the core still needed
        F2 dn[GRAD ? R : 1], dbelow, dabove;
        if constexpr (GRAD) {
#pragma unroll
            for (int r = 0; r < R; ++r) dn[r] = density_of(f[r]);
            if (g < G - 1) den[g * 32 + t] = dn[R - 1].v;
            if (g > 0) den[(G - 1 + g - 1) * 32 + t] = dn[0].v;
            __syncwarp();
            if (t == 0) mbar_arrive(bden);
            meet(bden, dphase);
            dphase ^= 1;
            dbelow = g > 0 ? as_f2(den[(g - 1) * 32 + t]) : dn[0];
            dabove = g < G - 1 ? as_f2(den[(G - 1 + g) * 32 + t]) : dn[R - 1];
        }
        const bool keep = core && !(last && is_lost(ctl));
        // the thread's two outermost rows first
#pragma unroll
        for (int q = 0; q < R; ++q) {
            const int r = q == 0 ? 0 : (q == 1 ? R - 1 : q - 1);
            if (row0 + r >= HL - reach && row0 + r < H - HL + reach) {
                F2 sx = f2(L.fx, L.fx), sy = f2(L.fy, L.fy);
                if constexpr (GRAD) {
                    const F2 ryp = r < R - 1 ? dn[r < R - 1 ? r + 1 : r] : dabove;
                    const F2 rym = r > 0 ? dn[r > 0 ? r - 1 : 0] : dbelow;
                    grad_source_open(dn[r], from_right<32>(dn[r]), from_left<32>(dn[r]), ryp, rym, L, sx,
                                     sy);
                }
                F2 dr, jx, jy;
                collide_sums<SRC>(f[r], sx, sy, rc, dr, jx, jy);
                if (core_row(r)) {
                    float dra, drb, jxa, jxb, jya, jyb;
                    f2_split(dr, dra, drb);
                    f2_split(jx, jxa, jxb);
                    f2_split(jy, jya, jyb);
                    float4 *ua = us + r * I::CW, *ub = ua + I::CW / 2;
                    float4 wa = *ua, wb = *ub;
                    integrate_u_value(wa, jxa, jya, L.rho0 + dra);
                    integrate_u_value(wb, jxb, jyb, L.rho0 + drb);
                    if (keep) {
                        if (!last) {
                            *ua = wa;
                            *ub = wb;
                        } else {
                            const int64_t k = k0 + (int64_t)r * L.pitch;
                            store_pair_records(uc + k, wa, wb);
                            nonfinite = radd(nonfinite, radd(radd(radd(dra, jxa), jya),
                                                             radd(radd(drb, jxb), jyb)));
#pragma unroll
                            for (int i = 0; i < 9; ++i)
                                *reinterpret_cast<unsigned long long *>(dst + i * L.fplane + k) = f[r][i].v;
                            if (early && ctl->next >= 0 && ctl->rec.c1 > ctl->rec.c0) {
                                const float4 *un =
                                    ctl->uc + (int64_t)(ctl->rec.y0 + row0 + r) * ctl->pitch + ctl->rec.x0 + c0;
                                copy16(smem_addr(ua), un);
                                copy16(smem_addr(ub), un + 1);
                            }
                        }
                    }
                }
            }
            if (q == (R > 1 ? 1 : 0) && !last) {
                shift_x(0);
                if (R > 1) shift_x(R - 1);
                post(l + 1);
            }
        }
        if (!last) {
#pragma unroll
            for (int r = 1; r < R - 1; ++r) shift_x(r);
            take(l + 1);
        }
        if (tid == 0 && early) take_next(l);
    };
    if constexpr (GRAD) {  // two at a time: 2048^2 crack 175 us a launch without, 171 with
        int l = 0;
        if (!(nsteps & 1)) step(l++, std::false_type{});
#pragma unroll 1
        for (; l < nsteps - 1; l += 2) {
            step(l, std::false_type{});
            step(l + 1, std::false_type{});
        }
    } else {
#pragma unroll 1
        for (int l = 0; l < nsteps - 1; ++l) step(l, std::false_type{});
    }
    step(nsteps - 1, std::true_type{});
    if (!isfinite(nonfinite)) flag_nonfinite(status, nonfinite, 0.0f, 0.0f);
    return true;
}

// What a launch steps: one lattice, or the instances of a batch (their lattice
// parameters staged in shared memory when a block turns to another one).
struct OneLattice {
    const CUtensorMap *tf;
    float *out;
    float4 *u;
    const uint8_t *classes;
    const BCDev *bc;
    const Lattice &l;
    const int64_t *clock;
    uint32_t *flags;
    __device__ bool enter(int) { return false; }
    __device__ const CUtensorMap *map(int) const { return tf; }
    __device__ float *dst(int) const { return out; }
    __device__ float4 *uc(int) const { return u; }
    __device__ int pitch(int) const { return l.pitch; }
    __device__ const uint8_t *cls(int) const { return classes; }
    __device__ const BCDev *bcs(int) const { return bc; }
    __device__ const Lattice &L() const { return l; }
    __device__ const int64_t *time(int) const { return clock; }
    __device__ uint32_t *status(int) const { return flags; }
};
struct BatchLattices {
    const TileInst *insts;
    int cur;
    Lattice *l;  // shared memory
    int staged;
    // whether the block has met at a barrier in it
    __device__ bool enter(int i) {
        if (i == staged) return false;  // uniform over the block
        constexpr int kWords = (int)(sizeof(Lattice) / 4);
        __syncthreads();  // the last tile's reads are over
        if (threadIdx.x < kWords)
            reinterpret_cast<uint32_t *>(l)[threadIdx.x] =
                reinterpret_cast<const uint32_t *>(&insts[i].L)[threadIdx.x];
        __syncthreads();
        staged = i;
        return true;
    }
    __device__ const CUtensorMap *map(int i) const { return &insts[i].map[cur]; }
    __device__ float *dst(int i) const { return insts[i].f[cur ^ 1]; }
    __device__ float4 *uc(int i) const { return insts[i].uc; }
    __device__ int pitch(int i) const { return insts[i].L.pitch; }
    __device__ const uint8_t *cls(int i) const { return insts[i].cls; }
    __device__ const BCDev *bcs(int i) const { return insts[i].bcs; }
    __device__ const Lattice &L() const { return *l; }
    __device__ const int64_t *time(int i) const { return insts[i].time; }
    __device__ uint32_t *status(int i) const { return insts[i].status; }
};

// A launch is one kernel over all its tiles, or, where it has many without
// boundary rules (kSplitTiles), two: the first steps the tiles with rules, the
// second the others.  Each then has registers and code of its own: in the one
// kernel the interior tiles of the 2048^2 crack take 151 us a launch, alone 145,
// with lambda != mu 169 and 147.  But the second starts only when the launch
// before is over, where the one kernel has its blocks waiting.
//
// Order of the two: both read what the launch before wrote, and write disjoint
// cores.  A block of the first waits for the launch before, counts itself ready
// (a release, which passes on what that wait made visible to it) and only then
// releases the second kernel, whose blocks start as the first kernel's leave
// room.  Each of them acquires the count before it reads anything; should it not
// find all blocks in it, it waits for the first kernel to end.  They also wait
// for that kernel before they exit: whatever follows the second follows both.
// The plans with so many tiles take the larger shapes.
constexpr bool can_split(int lpr, int r) { return lpr == 32 && r >= 3; }
enum class Part { kAll, kRules, kInner };

// Tiles of 64 columns are taken by one block per SM, the first by block index
// and the others from a counter, which the last block to finish puts back to
// zero; the smallest tiles and those of Part::kRules go one to a block.  nrules:
// the blocks of the first of two kernels.
template <int LPR, int R, bool GRAD, bool SRC, Part P, class Ctx>
__device__ __forceinline__ void run_tiles(Ctx ctx, const TileRec *__restrict__ tiles, int ntiles,
                                          int nrules, int32_t *__restrict__ counter,
                                          const uint32_t *__restrict__ pubs,
                                          const TileLink *__restrict__ links, int toff, int nsteps,
                                          unsigned char *sm) {
    constexpr size_t kControl = control_at<LPR, R, GRAD>();
    Control *ctl = reinterpret_cast<Control *>(sm + kControl);
    if (P != Part::kRules) release_next();
    if (threadIdx.x == 0) {
        mbar_init(smem_addr(&ctl->load), 1);
        mbar_init(smem_addr(&ctl->step), kNT / 32);
        mbar_init(smem_addr(&ctl->den), kNT / 32);
        ctl->lost = 0;
        ctl->next = -1;
        if (P == Part::kInner) {
            if (!all_ready(counter, nrules)) wait_for_previous();
            // and before this thread's copies (asynchronous proxy) read it
            asm volatile("fence.proxy.async.global;" ::: "memory");
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    TileRec rec = tiles[blockIdx.x];
    ctx.enter(rec.inst);
    if constexpr (LPR != 32 || P == Part::kRules) {
        tile_steps<LPR, R, GRAD, SRC>(ctx.map(rec.inst), ctx.dst(rec.inst), ctx.uc(rec.inst), ctx.cls(rec.inst),
                                 rec, pubs, links, ctx.bcs(rec.inst), ctx.L(), ctx.time(rec.inst), toff,
                                 nsteps, ctx.status(rec.inst), sm, ctl, true,
                                 P == Part::kRules ? counter : nullptr, 0);
    } else {
        const bool more = ntiles > (int)gridDim.x;
        auto grab = [&]() {
            const int i = (int)gridDim.x + atomicAdd(counter, 1);
            return i < ntiles ? i : -1;
        };
        // the next tile of an interior one, in three parts a step apart (each
        // waits for what the one before asked for)
        auto take_next = [&](int part) {
            if (part == 0) {
                ctl->next = more ? grab() : -1;
            } else if (part == 1 && ctl->next >= 0) {
                ctl->rec = tiles[ctl->next];
                issue_load<LPR, R>(ctx.map(ctl->rec.inst), ctl->rec, smem_addr(&ctl->load), sm);
            } else if (part == 2 && ctl->next >= 0) {
                ctl->uc = ctx.uc(ctl->rec.inst);
                ctl->pitch = ctx.pitch(ctl->rec.inst);
            }
        };
        // whether the next tile is known to every thread before this one's last step
        const bool early = nsteps >= (GRAD ? 4 : 5);
        bool first = P == Part::kAll, loaded = false;
        uint32_t parity = 0, phase = 0, dphase = 0;
        // Where a wait between the warps ran out, threads leave as they see it (a
        // thread that has left counts as arrived at every later barrier of the
        // block); whoever goes on past a barrier that a thread has left sees it
        // too, behind that barrier.  Nothing is in flight then: neither this
        // thread's records nor, of thread 0, the copy of the next tile.
        bool inner;
        int i;
        auto leave = [&]() {
            if (!inner || !is_lost(ctl)) return false;
            if ((threadIdx.x & 31) == 0) atomicOr(ctx.status(i), 2u);
            copy_wait();
            if (threadIdx.x == 0 && loaded && ctl->next >= 0)
                mbar_wait(smem_addr(&ctl->load), parity, kDefaultWaitNs);
            return true;
        };
        for (;;) {
            bool ok;
            i = rec.inst;
            inner = P == Part::kInner || rec.npub == 0;
            // an empty core steps nothing, so it takes no tile meanwhile
            const bool ahead = inner && early && rec.c1 > rec.c0;
            if (inner) {
                ok = tile_interior<R, GRAD, SRC>(ctx.map(i), ctx.dst(i), ctx.uc(i), rec, ctx.L(), nsteps,
                                            ctx.status(i), sm, ctl, first, loaded, early, parity, phase,
                                            dphase, take_next);
            } else {
                ok = tile_steps<LPR, R, GRAD, SRC>(ctx.map(i), ctx.dst(i), ctx.uc(i), ctx.cls(i), rec, pubs,
                                              links, ctx.bcs(i), ctx.L(), ctx.time(i), toff, nsteps,
                                              ctx.status(i), sm, ctl, first, nullptr, parity);
            }
            if (!ok) break;
            first = false;
            parity ^= 1;
            loaded = ahead;
            if (leave()) break;
            if (!ahead) {
                if (!more) break;
                __syncthreads();
                if (threadIdx.x == 0) {
                    ctl->next = grab();
                    if (ctl->next >= 0) ctl->rec = tiles[ctl->next];
                }
                __syncthreads();
                if (leave()) break;
            }
            if (ctl->next < 0) break;
            rec = ctl->rec;
            if (ctx.enter(rec.inst) && leave()) break;
        }
        if (more && threadIdx.x == 0 && atomicAdd(counter + 1, 1) == (int)gridDim.x - 1) {
            counter[0] = 0;
            counter[1] = 0;
            counter[kReady] = 0;
        }
        if (P == Part::kInner) wait_for_previous();
    }
}

template <int LPR, int R, bool GRAD, bool SRC, Part P>
__global__ void __launch_bounds__(kNT, 1)
    k_tile(const __grid_constant__ CUtensorMap tf, float *__restrict__ dst, float4 *__restrict__ uc,
           const uint8_t *__restrict__ cls, const TileRec *__restrict__ tiles, int ntiles, int nrules,
           int32_t *__restrict__ counter, const uint32_t *__restrict__ pubs,
           const TileLink *__restrict__ links, const BCDev *__restrict__ bcs,
           const __grid_constant__ Lattice L, const int64_t *__restrict__ time, int toff, int nsteps,
           uint32_t *__restrict__ status) {
    extern __shared__ __align__(1024) unsigned char sm[];
    run_tiles<LPR, R, GRAD, SRC, P>(OneLattice{&tf, dst, uc, cls, bcs, L, time, status}, tiles, ntiles,
                                    nrules, counter, pubs, links, toff, nsteps, sm);
}

// The tiles of many lattices in one launch (a batch, lambda = mu).
template <int LPR, int R, bool SRC, Part P>
__global__ void __launch_bounds__(kNT, 1)
    k_tile_batch(const TileInst *__restrict__ insts, const TileRec *__restrict__ tiles, int ntiles,
                 int nrules, int32_t *__restrict__ counter, const uint32_t *__restrict__ pubs,
                 const TileLink *__restrict__ links, int cur, int toff, int nsteps) {
    extern __shared__ __align__(1024) unsigned char sm[];
    __shared__ __align__(16) Lattice s_L;
    run_tiles<LPR, R, false, SRC, P>(BatchLattices{insts, cur, &s_L, -1}, tiles, ntiles, nrules, counter, pubs, links,
                                     toff, nsteps, sm);
}

// `kernel` in programmatic order behind the one launched before it.
template <class... P, class... A>
cudaError_t launch_tiles(void (*kernel)(P...), int blocks, size_t smem, cudaStream_t s, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(kNT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// blocks for n tiles of one launch: one per SM, the smallest tiles one each
template <int LPR> int blocks_for(int n, int sms) { return LPR == 32 ? std::min(n, sms) : n; }

template <int LPR, int R, bool SRC>
cudaError_t batch_shape(const TileBatch &B, int cur, int toff, int nsteps, cudaStream_t s) {
    auto allow = [](auto kernel) {
        return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)smem_bytes<LPR, R, false>());
    };
    if (B.ntiles <= 0) {
        // at the creation of every batch: the limit is the current device's
        cudaError_t e = allow(k_tile_batch<LPR, R, SRC, Part::kAll>);
        if constexpr (can_split(LPR, R)) {
            if (e == cudaSuccess) e = allow(k_tile_batch<LPR, R, SRC, Part::kRules>);
            if (e == cudaSuccess) e = allow(k_tile_batch<LPR, R, SRC, Part::kInner>);
        }
        return e;
    }
    auto launch = [&](auto kernel, int blocks, int first, int n) {
        return launch_tiles(kernel, blocks, smem_bytes<LPR, R, false>(), s, B.insts, B.tiles + first, n,
                            B.nrules, B.counter, B.pubs, B.links, cur, toff, nsteps);
    };
    if constexpr (can_split(LPR, R)) {
        if (B.nrules > 0) {
            const int inner = B.ntiles - B.nrules;
            const cudaError_t e =
                launch(k_tile_batch<LPR, R, SRC, Part::kRules>, B.nrules, 0, B.nrules);
            return e != cudaSuccess ? e : launch(k_tile_batch<LPR, R, SRC, Part::kInner>,
                                                 blocks_for<LPR>(inner, B.sms), B.nrules, inner);
        }
    }
    return launch(k_tile_batch<LPR, R, SRC, Part::kAll>, blocks_for<LPR>(B.ntiles, B.sms), 0, B.ntiles);
}

template <int LPR, int R, bool GRAD, bool SRC>
cudaError_t launch_shape(const Lattice &L, const DevState &S, const TileDev &T, int cur, int toff,
                         int nsteps, cudaStream_t s) {
    auto launch = [&](auto kernel, int blocks, int first, int n) {
        return launch_tiles(kernel, blocks, smem_bytes<LPR, R, GRAD>(), s, T.map[cur],
                            static_cast<float *>(S.f[cur ^ 1]), static_cast<float4 *>(S.ucomp),
                            (const uint8_t *)S.cls, T.tiles + first, n, T.nrules, T.counter, T.pubs, T.links,
                            (const BCDev *)S.bcs, L, (const int64_t *)S.time, toff, nsteps, S.status);
    };
    if constexpr (can_split(LPR, R)) {
        if (T.nrules > 0) {
            const int inner = T.ntiles - T.nrules;
            const cudaError_t e =
                launch(k_tile<LPR, R, GRAD, SRC, Part::kRules>, T.nrules, 0, T.nrules);
            return e != cudaSuccess ? e : launch(k_tile<LPR, R, GRAD, SRC, Part::kInner>,
                                                 blocks_for<LPR>(inner, T.sms), T.nrules, inner);
        }
    }
    return launch(k_tile<LPR, R, GRAD, SRC, Part::kAll>, blocks_for<LPR>(T.ntiles, T.sms), 0, T.ntiles);
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

bool has_force(const Lattice &L) { return L.fx != 0.0f || L.fy != 0.0f; }

template <int LPR, int R, bool GRAD, bool SRC> cudaError_t allow_smem() {
    auto allow = [](auto kernel) {
        return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)smem_bytes<LPR, R, GRAD>());
    };
    cudaError_t e = allow(k_tile<LPR, R, GRAD, SRC, Part::kAll>);
    if constexpr (can_split(LPR, R)) {
        if (e == cudaSuccess) e = allow(k_tile<LPR, R, GRAD, SRC, Part::kRules>);
        if (e == cudaSuccess) e = allow(k_tile<LPR, R, GRAD, SRC, Part::kInner>);
    }
    return e;
}

template <int LPR, int R> cudaError_t prepare_shape(const Lattice &L, const DevState &S, TileDev *T) {
    if (!encode_shape<LPR, R>(L, S, T->map)) return cudaErrorInvalidValue;
    if constexpr (R < 4)
        if (L.grad) return allow_smem<LPR, R, true, true>();
    if (L.grad) return cudaErrorInvalidValue;
    return has_force(L) ? allow_smem<LPR, R, false, true>() : allow_smem<LPR, R, false, false>();
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
    // the plans with lambda != mu take no tile of four rows to a thread
#define LBM_TILE(n, lpr, r)                                                                      \
    case n:                                                                                      \
        if constexpr (r < 4)                                                                     \
            if (L.grad) return launch_shape<lpr, r, true, true>(L, S, T, cur, toff, nsteps, s);  \
        if (L.grad) break;                                                                       \
        return has_force(L) ? launch_shape<lpr, r, false, true>(L, S, T, cur, toff, nsteps, s)   \
                            : launch_shape<lpr, r, false, false>(L, S, T, cur, toff, nsteps, s);
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
#define LBM_TILE(n, lpr, r)                                                  \
    case n:                                                                  \
        return B.force ? batch_shape<lpr, r, true>(B, cur, toff, nsteps, s)  \
                       : batch_shape<lpr, r, false>(B, cur, toff, nsteps, s);
    switch (B.shape) {
        LBM_TILE(0, 16, 1)
        LBM_TILE(1, 32, 2)
        LBM_TILE(2, 32, 3)
        LBM_TILE(3, 32, 4)
    }
#undef LBM_TILE
    return cudaErrorInvalidValue;
}

}  // namespace lbm
