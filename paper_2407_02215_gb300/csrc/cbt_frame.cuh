// One frame of a batch in one launch (the Sec. 3.3 pipeline, Alg. 9): a
// persistent cooperative kernel, every block resident, whose phases are
// separated by grid-wide barriers instead of kernel boundaries.
//
//   P0 prep       frame counters, item-tile prefix, camera-relative roots
//   P1 classify   LOD wishes; what needs a walk listed, split costs bounded
//   P2 gate-sum   chain and group walks of what the gate could grant; cost sums
//   P3 gate       tile prefix from the tiles' cost sums, grants, chain marking
//   P4 alloc      fates, tile-local allocation prefixes, fill records; free list
//   P5 fill       new records, neighbour links, bitfield
//   P6 reduce     sum tree (the last word tile of an instance builds the top)
//   P7 compact    live list, and the vertices of the new triangulation
//
// The two prefix sums of the per-step kernels (decoupled look-back) become
// reduce-then-scan here: tile sums, a barrier, then each tile adds the sums
// before it (the gate), or the fill adds its tile's prefix (the allocation).
// State between phases lives in the slot arrays (command words, scan words);
// each block keeps its instance descriptor and frame parameters in shared
// memory across tiles and phases. A pool above the single-instance frame's
// tables is a batch of one with an instantiation of its own, whose classify and
// walks can take tiles in parts and whose export follows the compaction as a
// phase (P8). Reads of data other
// blocks wrote in an earlier phase follow a barrier whose fences order them.
// Every wait is bounded: a barrier that runs out sets the batch's abort word,
// every later wait then returns at once, and the instances report kErrTimeout.
#pragma once
#include "cbt_kernels.cuh"
#include "cbt_phases.cuh"

namespace cbtgpu {

namespace {

constexpr int kFThreads = 256;
constexpr int kFPer = 4;  // items per thread and tile: kFThreads * kFPer == kTileItems
static_assert(kFThreads * kFPer == (int)kTileItems, "tile shape");
constexpr uint32_t kFBuf = 4096;  // shared scratch words (lists, tree top, live slots)
constexpr uint32_t kRelRange = 256;  // root-table entries per warp range in P0
constexpr uint32_t kMinIpt = 4, kMaxIpt = 8;  // items per thread of a scan tile
constexpr int kBarrierSpin = 1 << 22;
constexpr uint32_t kBarriers = 7;  // grid barriers per frame (one more for a single instance)
constexpr int kAllocDone = 7;      // ticket counter: blocks done with the allocation phase

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ uint32_t ld_acquire_gpu(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void red_release_gpu(uint32_t* p, uint32_t v) {
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Grid-wide barrier k (1-based) of the launch: a monotonic arrival counter
// that never resets; barrier k of a launch that started at count `epoch` is
// passed once the count reaches epoch + k * gridDim.x (wrap-safe compare).
// Arrival is a release reduction of the block's writes (ordered after the
// whole block by __syncthreads); the spin is an acquire load. The launch is
// cooperative, so every block is resident and every arrival comes.
__device__ void grid_wait(BatchGlobals* bg, uint32_t target, int limit) {
    __syncthreads();
    if (threadIdx.x == 0) {
        red_release_gpu(&bg->bar_count, 1u);
        int it = 0;
        while ((int)(ld_acquire_gpu(&bg->bar_count) - target) < 0) {
            if (ld_volatile(&bg->abort)) break;
            if (++it > limit) {
                atomicExch(&bg->abort, 1u);
                break;
            }
            __nanosleep(32);
        }
    }
    __syncthreads();
}

__device__ __forceinline__ void grid_sync(BatchGlobals* bg, uint32_t epoch, uint32_t k) {
    grid_wait(bg, epoch + k * gridDim.x, kBarrierSpin);
}

__device__ __forceinline__ void stamp(const BatchDev& bt, int k) {
    if (bt.timing && blockIdx.x == 0 && threadIdx.x == 0) bt.bg->t[k] = global_ns();
}

// Per-block context: the instance of the current tile (descriptor and frame
// parameters reloaded only when the instance changes) and the tile's place.
struct FCtx {
    Inst I;
    FrameP fp;
    uint32_t b;       // cached instance, kNull before the first tile
    uint32_t nb, lt;  // instance and local index of the current tile
    uint32_t tb, te;  // the instance's tiles in the current partition
    uint32_t N, F;    // frame-start live and free counts of the cached instance
};

// Block-uniform; ends with __syncthreads.
__device__ __forceinline__ void ctx_tile(const BatchDev& bt, const uint32_t* base, uint32_t t, uint32_t T,
                                         FCtx& c) {
    if (threadIdx.x == 0) {
        if (bt.B == 1) {  // base[0] = 0, base[1] = T
            c.nb = 0;
            c.lt = t;
            c.tb = 0;
            c.te = T;
        } else {
            const uint32_t b = find_inst(base, bt.B, t);
            c.nb = b;
            c.lt = t - base[b];
            c.tb = base[b];
            c.te = base[b + 1];
        }
    }
    __syncthreads();
    const uint32_t b = c.nb;
    if (b != c.b) {
        load_tile_ctx(bt, b, &c.I, &c.fp);
        __syncthreads();
        if (threadIdx.x == 0) {
            c.b = b;
            c.N = c.I.g->N;
            c.F = c.I.g->F;
        }
    }
    __syncthreads();
}

// The tiles of a phase handed out as blocks finish: tile blockIdx.x first, then
// by a counter, taken while the current tile is worked on. What a tile costs
// differs and clusters (grants and chains at an instance's start, culled
// regions): with tiles dealt round robin the batch frame waited for its
// slowest blocks, and with four consecutive tiles at a time it was slower
// still (batch of 15M bisectors: 1744 and 1953 us; handed out 1684). With at
// most one of the T tiles per block there is nothing to hand out (the gate of
// 65k bisectors in a pool of 2^23 slots: 9.3 us with tickets, 8.1 without).
struct TileFeed {
    uint32_t* ticket;
    uint32_t* s;  // [2] in shared memory
    uint32_t T, p = 0, ahead = kNull;
    __device__ __forceinline__ TileFeed(uint32_t* t, uint32_t* shared, uint32_t tiles) : ticket(t), s(shared), T(tiles) {}
    __device__ __forceinline__ void take() {
        if (threadIdx.x == 0 && T > gridDim.x) ahead = gridDim.x + atomicAdd(ticket, 1u);
    }
    __device__ __forceinline__ uint32_t first() {
        take();
        return blockIdx.x;
    }
    // With the whole block, at the end of a tile.
    __device__ __forceinline__ uint32_t next() {
        if (T <= gridDim.x) return kNull;
        if (threadIdx.x == 0) s[p] = ahead;
        __syncthreads();
        const uint32_t t = s[p];
        p ^= 1u;
        take();
        return t;
    }
};
// Counters of the phases (tickets of the batch; kAllocDone is the last).
enum : int { kFeedClassify = 0, kFeedWalks, kFeedGate, kFeedAlloc, kFeedCompact, kFeeds };
static_assert(kFeeds <= kAllocDone, "counters of their own");

__device__ __forceinline__ unsigned long long pack_pair(Pair p) {
    return ((unsigned long long)p.a << 32) | (unsigned long long)p.b;
}
__device__ __forceinline__ Pair unpack_pair(unsigned long long v) {
    return Pair{(uint32_t)(v >> 32), (uint32_t)v};
}

// Block sums of two Pairs (s_red: 4 * (blockDim / 32) words); every thread
// gets both totals.
__device__ __forceinline__ void block_sum2(Pair& x, Pair& y, uint32_t* s_red) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (int)(blockDim.x >> 5);
    uint32_t v[4] = {x.a, x.b, y.a, y.b};
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_xor_sync(0xFFFFFFFFu, v[q], o);
    if (lane == 0)
#pragma unroll
        for (int q = 0; q < 4; ++q) s_red[4 * warp + q] = v[q];
    __syncthreads();
    uint32_t r[4] = {0, 0, 0, 0};
    for (int w = 0; w < nw; ++w)
#pragma unroll
        for (int q = 0; q < 4; ++q) r[q] += s_red[4 * w + q];
    __syncthreads();
    x = Pair{min(r[0], kSat), min(r[1], kSat)};
    y = Pair{min(r[2], kSat), min(r[3], kSat)};
}

// Sums of the tile aggregates of the current instance: before tile t, and
// over all its tiles.
__device__ __forceinline__ void tile_sums(const unsigned long long* agg, const FCtx& c, Pair& before, Pair& all,
                                          uint32_t* s_red) {
    const uint32_t t = c.tb + c.lt;
    before = Pair{0, 0};
    all = Pair{0, 0};
    for (uint32_t u = c.tb + threadIdx.x; u < c.te; u += blockDim.x) {
        const Pair v = unpack_pair(__ldcg(agg + u));
        all = padd(all, v);
        if (u < t) before = padd(before, v);
    }
    block_sum2(before, all, s_red);
}

// ------------------------------------------------------------------ phases

// P0: frame counters per instance; the item tiles (kTileItems live indices)
// and the scan tiles (kFThreads * ipt, one per block when the live total
// allows) laid out over the batch; the camera-relative root tables.
__device__ void phase_prep(const BatchDev& bt, Pair* s_warp, uint32_t* s_tmp) {
    if (blockIdx.x == 0) {
        if (threadIdx.x == 0) s_tmp[0] = s_tmp[1] = s_tmp[2] = 0;
        __syncthreads();
        for (uint32_t b = threadIdx.x; b < bt.B; b += blockDim.x) atomicAdd(&s_tmp[2], bt.inst[b].sums[1]);
        __syncthreads();
        const uint32_t per_round = gridDim.x * kFThreads;
        const uint32_t ipt = s_tmp[2] > kMinIpt * per_round ? kMaxIpt : kMinIpt;  // 16-byte loads per thread
        const uint32_t S = ipt * kFThreads;
        for (uint32_t b0 = 0; b0 < bt.B; b0 += blockDim.x) {
            const uint32_t b = b0 + threadIdx.x;
            uint32_t tiles = 0, stiles = 0;
            if (b < bt.B) {
                const Inst& I = bt.inst[b];
                const uint32_t N = I.sums[1];
                Globals* g = I.g;
                g->N = N;
                g->F = I.cap - N;
                g->A = 0;
                g->Mg = 0;
                g->Stot = 0;
                g->C = 0;
                g->done = 0;
                g->marks_clean = 0;
                g->freel_full = 0;
                tiles = (N + kTileItems - 1u) / kTileItems;
                stiles = (N + S - 1u) / S;
                g->ntiles = tiles;
                g->nstiles = stiles;
                for (int k = 0; k < kStCount; ++k) g->stats[k] = 0;
                g->stats[kStLiveBefore] = N;
                g->stats[kStFreeBefore] = I.cap - N;
                g->stats[kStFrame] = frame_of(bt, b).frame;
                pc_generation(g, frame_of(bt, b));
                if (bt.nout) bt.nout[b] = N;
            }
            Pair tot;
            const Pair ex = block_scan(Pair{stiles, tiles}, tot, s_warp);
            if (b < bt.B) {
                bt.tile_base[b] = s_tmp[0] + ex.b;
                bt.stile_base[b] = s_tmp[1] + ex.a;
            }
            __syncthreads();
            if (threadIdx.x == 0) {
                s_tmp[0] += tot.b;
                s_tmp[1] += tot.a;
            }
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            bt.tile_base[bt.B] = s_tmp[0];
            bt.stile_base[bt.B] = s_tmp[1];
            bt.bg->total_tiles = s_tmp[0];
            bt.bg->total_stiles = s_tmp[1];
            bt.bg->scan_ipt = ipt;
            bt.bg->live_total = s_tmp[2];
            bt.bg->t[kFramePhases] = 0;
            for (int k = 0; k < 8; ++k) bt.bg->tickets[k] = 0;
        }
    }
    // block 0 sets up the instances; the others share the root tables in
    // warp ranges (a multiple of 32 entries, at most kRelRange, enough ranges
    // for every warp)
    if (gridDim.x == 1 || blockIdx.x > 0) {
        const uint32_t nb = gridDim.x > 1 ? gridDim.x - 1u : 1u, bb = gridDim.x > 1 ? blockIdx.x - 1u : 0u;
        const uint32_t nw = nb * (kFThreads / 32), wid = bb * (kFThreads / 32) + threadIdx.x / 32u;
        const uint32_t per = min(kRelRange, ((bt.Trel + nw - 1u) / nw + 31u) & ~31u);
        for (uint32_t e = wid * per; e < bt.Trel; e += nw * per) rel_range(bt, e, min(bt.Trel, e + per));
        // the tiles' sums: costs per scan tile, lower bounds per item tile and
        // per 32 item tiles
        const uint32_t sums = 2u * bt.Titems + bt.Twords;
        for (uint32_t t = bb * kFThreads + threadIdx.x; t < sums; t += nb * kFThreads) bt.status[t] = 0ull;
    }
}

// Lower-bound costs of the split wishes, per item tile of the batch and per 32
// item tiles of instance b (after the scan tiles' sums; an instance has at
// least as many word tiles as it has 32 item tiles).
__device__ __forceinline__ unsigned long long* bound_sums(const BatchDev& bt) { return bt.status + bt.Titems; }
__device__ __forceinline__ unsigned long long* bound_groups(const BatchDev& bt, uint32_t b) {
    return bt.status + 2u * bt.Titems + (bt.B == 1 ? 0u : bt.wtile_base[b]);
}
// A warp's 128 items of a tile: their walk entries (16 bits each: item, bit 7
// for a split wish, bit 8 for one whose root halfedge has a Twin) from the
// second word of the items' fill records (written only in P4), the number of
// entries in the first.
constexpr uint32_t kSubItems = kTileItems / (kFThreads / 32);
static_assert(kSubItems == 128u, "7-bit items");
__device__ __forceinline__ uint32_t* walk_region(const Inst& I, uint32_t i) {
    return reinterpret_cast<uint32_t*>(I.chgr + i);
}
// Whether a split of bisector j has an allocation bound of 4, else 2: every
// bisector under a root whose halfedge has a Twin has one (its refinement
// edge is inside the root triangle, on an edge to the face's centroid, or on
// that halfedge), and its chain then costs itself and the Twin's pair.
__device__ __forceinline__ bool has_twin_bound(const Inst& I, uint64_t j) {
    const int d = depth_of(j, I.ch);
    const uint32_t h = d >= 0 ? (uint32_t)((j >> d) - (1ull << I.ch)) : kNull;
    return h < I.H && !((__ldg(I.rbnd + (h >> 5)) >> (h & 31u)) & 1u);
}

// Whether classify takes a single instance's T item tiles in four parts of 256
// items, a warp one round of 32, or whole, a warp four rounds: whole tiles of
// a pool that holds few bisectors leave blocks idle beside others that run
// four rounds in a row. The parts' shared lists cost FP32 more than they give
// once half of the blocks have a tile, the forms with longer evaluations once
// every block has two (2^23-slot pools, 608 blocks; whole and in parts, us: FP32,
// 65k live 18.0 and 7.4, 239k 17.6 and 14.4, 562k 26.6 and 27.5; fixed point,
// 366k 47 and 36, 1.0M 100 and 90; projected, 107k 140 and 39, 814k 294 and 199,
// 2.3M 541 and 535; displaced, 567k 143 and 118, 1.4M 290 and 291).
template <int F>
__device__ __forceinline__ bool classify_in_parts(uint32_t T) {
    return F == kFormF32 ? 2u * T <= gridDim.x : T < 2u * gridDim.x;
}
// The same for the walks, each of whose parts adds up the bounds before its
// tile: while every part has a block of its own (65k live, 64 tiles: 11.6 and
// 8.2 us; 239k 12.9 and 17.2).
__device__ __forceinline__ bool walks_in_parts(uint32_t T) { return T * (uint32_t)kFPer <= gridDim.x; }

// P1: wishes of every live bisector (Sec. 3.3 GenerateCommands with the R8
// LOD reading) over item tiles, each warp on its own 128 items of the tile;
// the items that need a walk listed in place, and the split wishes' lower
// bounds summed for the walks.
template <int F, bool kParts>
__device__ void phase_classify(const BatchDev& bt, FCtx& c, uint32_t* s_tab, uint32_t* s_cnt) {
    const uint32_t T = bt.bg->total_tiles, S = kFThreads * bt.bg->scan_ipt;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const uint32_t rounds = kParts ? 1u : (uint32_t)kFPer, units = kParts ? T * kFPer : T;
    __shared__ uint32_t s_feed[2], s_part[2];
    TileFeed feed(&bt.bg->tickets[kFeedClassify], s_feed, units);
    for (uint32_t u = feed.first(); u < units; u = feed.next()) {
        const uint32_t t = kParts ? u / kFPer : u, q = kParts ? u % kFPer : 0u;
        if (threadIdx.x < 2) s_part[threadIdx.x] = 0;
        stats_reset(s_cnt);
        ctx_tile(bt, bt.tile_base, t, T, c);
        const Inst& I = c.I;
        const FrameP& fp = c.fp;
        const uint32_t N = c.N;
        const bool chain = fp.gate != 1;
        const bool cache = vc_form<F>(fp) && fp.vout;
        const uint64_t key = splitmix64(((uint64_t)fp.seed << 32) | (uint64_t)fp.frame);
        // the warp's 128 items and its first round of 32 in them
        const uint32_t w0 = c.lt * kTileItems + kSubItems * (kParts ? 2u * q + (warp >> 2) : warp);
        const uint32_t k0 = kParts ? warp & 3u : 0u;
        uint32_t sl[kFPer];
        uint64_t hj[kFPer];
#pragma unroll
        for (int k = 0; k < kFPer; ++k) {
            const uint32_t i = w0 + 32u * (k0 + (uint32_t)k) + lane;
            sl[k] = (uint32_t)k < rounds && i < N ? I.live[i] : kNull;
        }
#pragma unroll
        for (int k = 0; k < kFPer; ++k) hj[k] = sl[k] != kNull ? I.heap[sl[k]] : 0ull;
        uint32_t n = 0, bound = 0, paper = 0;
        if (w0 < N) {
            uint32_t* const reg = walk_region(I, w0);
            uint16_t* const list = reinterpret_cast<uint16_t*>(reg + 1);
#pragma unroll 1
            for (uint32_t k = k0; k < k0 + rounds; ++k) {
                const uint32_t x = 32u * k + lane, i = w0 + x;
                bool split = false, walk = false, twin = false;
                uint32_t cost = 0;
                if (i < N) {
                    const uint32_t cmd = classify_item<F>(I, fp, key, i, sl[0], hj[0], s_tab, s_cnt, cache);
                    split = (cmd & kSplitWish) != 0u;
                    twin = split && has_twin_bound(I, hj[0]);
                    walk = (split && chain) || ((cmd & kMergeWish) && !(cmd & kHeapOdd));
                    // the paper's gate: the cost classify_item has set, without a walk
                    if (split && !chain) cost = 3u * (uint32_t)depth_of(hj[0], I.ch) + 4u;
                }
                const unsigned wm = __ballot_sync(0xFFFFFFFFu, walk);
                if (kParts) {  // the four warps of the 128 items append to one list
                    if (lane == 0) n = atomicAdd(&s_part[warp >> 2], (uint32_t)__popc(wm));
                    n = __shfl_sync(0xFFFFFFFFu, n, 0);
                }
                if (walk)
                    list[n + __popc(wm & ((1u << lane) - 1u))] =
                        (uint16_t)(x | (split ? 128u : 0u) | (twin ? 256u : 0u));
                n += __popc(wm);
                if (chain)
                    bound += 2u * (__popc(__ballot_sync(0xFFFFFFFFu, split)) + __popc(__ballot_sync(0xFFFFFFFFu, twin)));
                else
                    paper += __reduce_add_sync(0xFFFFFFFFu, cost);
#pragma unroll
                for (int q = 0; q + 1 < kFPer; ++q) {  // constant indices: registers, not local memory
                    sl[q] = sl[q + 1];
                    hj[q] = hj[q + 1];
                }
            }
            if (lane == 0) {
                if (!kParts) reg[0] = n;
                if (bound) {
                    atomicAdd(bound_sums(bt) + t, (unsigned long long)bound);
                    atomicAdd(bound_groups(bt, c.b) + (c.lt >> 5), (unsigned long long)bound);
                }
                if (paper) atomicAdd(bt.status + (bt.B == 1 ? 0u : bt.stile_base[c.b]) + w0 / S, (unsigned long long)paper);
            }
        }
        __syncthreads();
        if (kParts && lane == 0 && k0 == 0u && w0 < N) *walk_region(I, w0) = s_part[warp >> 2];
        stats_flush(s_cnt, I.g, kStSplitWishes);
        __syncthreads();
    }
}

// Alg. 4 group of s1 (heap ID j1, a merge wish) on the frame-start state,
// walked only while s1 can be its smallest member and every member wishes
// to merge: true when both hold, with the members (m[0] = s1, m[1] its
// sibling, m[2] the bisector across the outer half of the refinement edge,
// m[3] its sibling) and the parents' count.
static __device__ bool group_if_mergeable(const Inst& I, uint32_t s1, uint64_t j1, Group& g) {
    if (depth_of(j1, I.ch) < 1) return false;
    const uint4 r1 = I.nb[s1];
    const bool bit = j1 & 1ull;
    const uint32_t s2 = bit ? r1.z : r1.y;
    const uint32_t s3 = bit ? r1.y : r1.z;
    if (s2 == kNull || bad_slot(I, s2, kErrLink)) return false;
    if (s3 != kNull && bad_slot(I, s3, kErrLink)) return false;
    const uint64_t j2 = I.heap[s2];
    const uint32_t c2 = *cmd_ptr(I, s2);
    uint64_t j3 = 0ull;
    uint4 r3 = make_uint4(kNull, kNull, kNull, 0u);
    uint32_t c3 = 0u;
    if (s3 != kNull) {
        j3 = I.heap[s3];
        r3 = I.nb[s3];
        c3 = *cmd_ptr(I, s3);
    }
    if ((j2 >> 1) != (j1 >> 1) || j2 < j1 || !(c2 & kMergeWish)) return false;
    g.m[0] = s1;
    g.m[1] = s2;
    g.m[2] = g.m[3] = kNull;
    g.n = 2;
    g.np = 1;
    g.imin = 0;
    if (s3 != kNull) {
        // the other pair's smaller member is its even one
        if (bitlen64(j3) != bitlen64(j1) || (j3 >> 1) == (j1 >> 1) || (j3 & ~1ull) < j1 || !(c3 & kMergeWish))
            return false;
        const uint32_t s4 = bit ? r3.y : r3.z;
        if (s4 == kNull || bad_slot(I, s4, kErrLink)) return false;
        const uint64_t j4 = I.heap[s4];
        const uint32_t c4 = *cmd_ptr(I, s4);
        if ((j4 >> 1) != (j3 >> 1) || !(c4 & kMergeWish)) return false;
        g.m[2] = s3;
        g.m[3] = s4;
        g.n = 4;
        g.np = 2;
    }
    return true;
}

// P2: the walks, per item tile. A split wish is denied whatever its cost when
// the lower bounds (2, or 4 with a Twin) of the instance's split wishes before
// its tile plus its own exceed the free slots F: in a tile where the bounds
// before it do so alone, no split here or later can be granted and their
// costs are left out; else the bound stands in for such a wish's cost, so that
// the splits after it are denied on these costs as on the true ones. The
// other splits walk their chains (command form of Alg. 3: cost, members for
// the marking). A merge wish with an even heap ID walks its Alg. 4 group
// while it can be a candidate with this wish its smallest member, which then
// records the members. Costs go to the scan tile's sums.
// Without the bounds every wish of a full pool walked its chain only to be
// denied: 6.6M wishes of a batch of 15M bisectors, 0.7M granted; its classify
// with the walks took 680 us and the gate's sums 67, these two phases 427 and 343 (in a
// nearly full 2^23-slot pool 290 and 10, now 165 and 110).
template <bool kParts>
__device__ void phase_walks(const BatchDev& bt, FCtx& c, uint32_t* s_cnt, unsigned long long* s_red, uint32_t* s_tmp,
                            uint32_t* s_n) {
    const uint32_t T = bt.bg->total_tiles, S = kFThreads * bt.bg->scan_ipt;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const uint32_t regions = kParts ? 2u : kFThreads / 32, units = kParts ? T * kFPer : T;
    __shared__ uint32_t s_feed[2];
    TileFeed feed(&bt.bg->tickets[kFeedWalks], s_feed, units);
    for (uint32_t u = feed.first(); u < units; u = feed.next()) {
        const uint32_t t = kParts ? u / kFPer : u;
        if (threadIdx.x < 3) s_tmp[threadIdx.x] = 0;
        stats_reset(s_cnt);
        ctx_tile(bt, bt.tile_base, t, T, c);
        // a copy: read again from shared memory after every store otherwise
        // (batch of 64: 307 us, 329; the same in the other phases gained nothing
        // or, in classify, cost registers: 407 us, 538)
        const Inst I = c.I;
        const uint32_t N = c.N, F = c.F, lt = c.lt;
        const uint32_t i0 = lt * kTileItems + (kParts ? 2u * kSubItems * (u % kFPer) : 0u);  // the unit's first item
        const uint32_t gate = c.fp.gate;
        // the bounds before the tile: the earlier groups of 32 tiles, then the
        // earlier tiles of its group
        unsigned long long before = 0;
        const unsigned long long* G = bound_groups(bt, c.b);
        for (uint32_t g = threadIdx.x; g < (lt >> 5); g += kFThreads) before += __ldcg(G + g);
        if (threadIdx.x < (lt & 31u)) before += __ldcg(bound_sums(bt) + t - 1u - threadIdx.x);
        if (threadIdx.x >= kFThreads - kFThreads / 32) {  // entries of warp k's items
            const uint32_t k = threadIdx.x - (kFThreads - kFThreads / 32);
            s_n[k] = k < regions && i0 + kSubItems * k < N ? *walk_region(I, i0 + kSubItems * k) : 0u;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(0xFFFFFFFFu, before, o);
        if (lane == 0) s_red[warp] = before;
        __syncthreads();
        before = 0;
        uint32_t n = 0;
#pragma unroll
        for (uint32_t w = 0; w < kFThreads / 32; ++w) {
            before += s_red[w];
            n += s_n[w];
        }
        const bool none = before > F;
        uint32_t smc = 0, ssc = 0;
        for (uint32_t q = threadIdx.x; q < n; q += kFThreads) {
            uint32_t w = 0, x = q;
#pragma unroll
            for (uint32_t k = 0; k + 1u < kFThreads / 32; ++k) {  // the warp's items that hold entry q
                const uint32_t m = s_n[k];
                const bool past = w == k && x >= m;
                x -= past ? m : 0u;
                w += past ? 1u : 0u;
            }
            const uint32_t e = reinterpret_cast<const uint16_t*>(walk_region(I, i0 + kSubItems * w) + 1)[x];
            const uint32_t i = i0 + kSubItems * w + (e & 127u);
            if (e & 128u) {
                if (none) continue;
                const uint32_t own = (e & 256u) ? 4u : 2u;
                uint32_t cost = own;
                if (before + own <= F) {
                    const uint32_t s = I.live[i];
                    uint4 rec;
                    cost = chain_walk(I, s, depth_of(I.heap[s], I.ch), false, &rec);
                    I.grp[i] = rec;
                }
                I.scan[i] = cost;
                ssc += cost;
            } else {
                const uint32_t s = I.live[i];
                Group g;
                if (group_if_mergeable(I, s, I.heap[s], g)) {
                    const uint32_t mc = gate == 1 ? 2u : (uint32_t)g.np;
                    I.grp[i] = make_uint4(g.m[0], g.m[1], g.m[2], g.m[3]);
                    atomicOr(cmd_ptr(I, s), kGrpMin);
                    I.scan[i] = mc << 24;
                    smc += mc;
                    atomicAdd(&s_cnt[0], 1u);
                }
            }
        }
        if (smc) atomicAdd(&s_tmp[0], smc);
        if (ssc) atomicAdd(&s_tmp[1], ssc);
        __syncthreads();
        if (threadIdx.x == 0 && (s_tmp[0] | s_tmp[1]))
            atomicAdd(bt.status + (bt.B == 1 ? 0u : bt.stile_base[c.b]) + i0 / S,
                      ((unsigned long long)s_tmp[0] << 32) | s_tmp[1]);
        stats_flush(s_cnt, I.g, kStMergeCand);
        __syncthreads();
    }
}

// Scan tiles: tile lt of an instance covers live indices [lt S, (lt+1) S)
// with S = kFThreads * ipt; thread x holds the ipt consecutive indices from
// lt S + x ipt (the order of the prefix sums).
__device__ __forceinline__ uint32_t stile_first(const FCtx& c, uint32_t ipt) {
    return c.lt * kFThreads * ipt + threadIdx.x * ipt;
}

// The items of a list that every instance of the batch has (count(I) of them),
// as one range walked evenly over the grid: body(b, I, q) -> uint32_t for
// item q of instance b, its results added to the instance's statistic `stat`.
// Lists cluster in a few instances; a block finds an item's instance in the
// prefix of the lists' lengths, built in shared memory.
template <typename Count, typename Body>
__device__ __forceinline__ void batch_list(const BatchDev& bt, FCtx& c, int stat, uint32_t* s_cnt, uint32_t* s_list,
                                           Pair* s_warp, Count count, Body body) {
    const uint32_t stride = gridDim.x * kFThreads;
    if (bt.B == 1) {
        stats_reset(s_cnt);
        ctx_tile(bt, bt.tile_base, 0, 1, c);  // instance 0 in shared memory
        const Inst& I = c.I;
        const uint32_t n = count(I);
        uint32_t sum = 0;
        for (uint32_t q = blockIdx.x * kFThreads + threadIdx.x; q < n; q += stride) sum += body(0u, I, q);
        if (sum) atomicAdd(&s_cnt[0], sum);
        __syncthreads();
        stats_flush(s_cnt, I.g, stat);
        __syncthreads();
        return;
    }
    const int lane = threadIdx.x & 31;
    const uint32_t wfirst = blockIdx.x * kFThreads + (threadIdx.x & ~31u);
    for (uint32_t cb = 0; cb < bt.B; cb += kFBuf) {  // kFBuf instances at a time
        const uint32_t nb = min(kFBuf, bt.B - cb);
        uint32_t total = 0;
        __syncthreads();
        for (uint32_t b0 = 0; b0 < nb; b0 += kFThreads) {
            const uint32_t b = b0 + threadIdx.x;
            const uint32_t n = b < nb ? count(bt.inst[cb + b]) : 0u;
            Pair tot;
            const Pair ex = block_scan(Pair{n, 0u}, tot, s_warp);
            if (b < nb) s_list[b] = total + ex.a;
            total += tot.a;
        }
        __syncthreads();
        for (uint32_t q0 = wfirst; q0 < total; q0 += stride) {  // warp-uniform trips
            const uint32_t q = q0 + (uint32_t)lane;
            uint32_t b = kNull, r = 0;
            if (q < total) {
                const uint32_t lb = find_inst(s_list, nb, q);
                b = cb + lb;
                // A copy: its fields stay in registers across the body's stores, after which
                // they would be loaded again (64 instances, 1.1M changed bisectors: 227 us, 262).
                const Inst I = bt.inst[b];
                r = body(b, I, q - s_list[lb]);
            }
            __syncwarp();
            const uint32_t same = __match_any_sync(0xFFFFFFFFu, b);
            const uint32_t sum = __reduce_add_sync(same, r);
            if (b != kNull && sum && lane == __ffs(same) - 1) atomicAdd(&bt.inst[b].g->stats[stat], sum);
        }
    }
}

// The ipt consecutive words from p + i0 (those at index >= n: `none`), as
// 16-byte loads when ipt and so i0 are multiples of 4.
__device__ __forceinline__ void load_items(const uint32_t* p, uint32_t i0, uint32_t ipt, uint32_t n, uint32_t none,
                                           uint32_t v[kMaxIpt]) {
    if ((ipt & 3u) == 0u) {
#pragma unroll
        for (uint32_t k = 0; k < kMaxIpt; k += 4u) {
            uint4 x = make_uint4(none, none, none, none);
            if (k < ipt && i0 + k < n) x = *reinterpret_cast<const uint4*>(p + i0 + k);
            v[k] = x.x;
            v[k + 1] = i0 + k + 1u < n ? x.y : none;
            v[k + 2] = i0 + k + 2u < n ? x.z : none;
            v[k + 3] = i0 + k + 3u < n ? x.w : none;
        }
        return;
    }
#pragma unroll
    for (uint32_t k = 0; k < kMaxIpt; ++k) v[k] = (k < ipt && i0 + k < n) ? p[i0 + k] : none;
}

// Granted merge total Mg when the merge requests of the instance overflow F:
// the largest inclusive merge prefix that fits (merges are granted first, in
// slot order). Only taken when the instance's merge sum exceeds F. The tile
// that crosses F is found by scans of the tile sums, 256 at a time: one
// thread adding them up one load after another made the gate of a full
// 2^23-slot pool (4,000 tiles) 563 us; so it is 71.
__device__ uint32_t crossing_mg(const BatchDev& bt, const FCtx& c, uint32_t F, uint32_t ipt, Pair* s_warp,
                                uint32_t* s_tmp) {
    uint32_t done = 0;
    for (uint32_t u0 = c.tb; u0 < c.te; u0 += blockDim.x) {  // block-uniform
        const uint32_t u = u0 + threadIdx.x;
        const uint32_t a = u < c.te ? unpack_pair(__ldcg(bt.status + u)).a : 0u;
        Pair all;
        const Pair ex = block_scan(Pair{a, 0u}, all, s_warp);
        const uint64_t before = (uint64_t)done + ex.a;
        if (before <= F && before + a > F) {  // one thread: the sums are not negative
            s_tmp[0] = u - c.tb;
            s_tmp[1] = s_tmp[2] = (uint32_t)before;
        }
        if ((uint64_t)done + all.a > F) break;
        done += all.a;
    }
    __syncthreads();
    const uint32_t lt = s_tmp[0], acc = s_tmp[1];
    const Inst& I = c.I;
    const uint32_t i0 = lt * kFThreads * ipt + threadIdx.x * ipt;
    uint32_t mc[kMaxIpt];
    uint32_t loc = 0;
#pragma unroll
    for (uint32_t k = 0; k < kMaxIpt; ++k) {
        mc[k] = (k < ipt && i0 + k < c.N) ? ((__ldcg(I.scan + i0 + k) >> 24) & kMergeCostMask) : 0u;
        loc += mc[k];
    }
    Pair tot;
    const Pair ex = block_scan(Pair{0, loc}, tot, s_warp);
    uint32_t run = acc + ex.b, best = acc;
#pragma unroll
    for (uint32_t k = 0; k < kMaxIpt; ++k) {
        run += mc[k];
        if (mc[k] && run <= F) best = max(best, run);
    }
    atomicMax(&s_tmp[2], best);
    __syncthreads();
    const uint32_t r = s_tmp[2];
    __syncthreads();
    return r;
}

// P3: tile prefix of the (merge, split) costs from the tile sums; merges are
// granted while their running total fits F, splits while Mg plus theirs
// does (R6 reading); granted splits mark their chains (command form of
// Alg. 3).
// kOne: the single-instance frame, whose descriptor is in the launch
// parameters (a copy in shared memory is reloaded after every store).
template <bool kOne = false>
__device__ void phase_gate(const BatchDev& bt, FCtx& c, uint32_t* s_cnt, uint32_t* s_red, Pair* s_warp,
                           uint32_t* s_tmp, uint32_t* s_n, uint2* s_list, bool always_recorded = false) {
    const uint32_t T = bt.bg->total_stiles, ipt = bt.bg->scan_ipt;
    __shared__ uint32_t s_feed[2];
    TileFeed feed(&bt.bg->tickets[kFeedGate], s_feed, T);
    for (uint32_t t = kOne ? blockIdx.x : feed.first(); t < T; t = kOne ? t + gridDim.x : feed.next()) {
        if (threadIdx.x == 0) *s_n = 0;
        stats_reset(s_cnt);
        ctx_tile(bt, bt.stile_base, t, T, c);
        const Inst& I = kOne ? bt.inst0 : c.I;
        const uint32_t N = c.N, F = c.F;
        // a tile without requests has nothing to grant (its sums are 0; the
        // instance's first tile also writes the totals)
        if (c.lt != 0u && __ldcg(bt.status + t) == 0ull) continue;  // block-uniform
        const uint32_t i0 = stile_first(c, ipt);
        uint32_t sl[kMaxIpt], w[kMaxIpt];
        load_items(I.live, i0, ipt, N, kNull, sl);  // before the tile sums, which do not need them
        load_items(I.scan, i0, ipt, N, 0u, w);
        Pair before, all;
        tile_sums(bt.status, c, before, all, s_red);
        const uint32_t Mg = all.a <= F ? all.a : crossing_mg(bt, c, F, ipt, s_warp, s_tmp);
        if (c.lt == 0 && threadIdx.x == 0) {
            I.g->Mg = Mg;
            I.g->Stot = all.b;
        }
        Pair loc{0, 0};
#pragma unroll
        for (uint32_t k = 0; k < kMaxIpt; ++k) loc = padd(loc, Pair{(w[k] >> 24) & kMergeCostMask, w[k] & 0xFFFFFFu});
        Pair tot;
        const Pair tex = block_scan(loc, tot, s_warp);
        Pair run = padd(before, tex);
        uint32_t gmask = 0, nmg = 0;  // the thread's granted splits (by k), granted merges
#pragma unroll
        for (uint32_t k = 0; k < kMaxIpt; ++k) {
            const uint32_t mc = (w[k] >> 24) & kMergeCostMask, sc = w[k] & 0xFFFFFFu;
            run = padd(run, Pair{mc, sc});
            if (sl[k] == kNull) continue;
            const bool mgrant = mc > 0u && run.a <= F;
            if (mc) atomicOr(cmd_ptr(I, sl[k]), mgrant ? (kCand | kMergeGrant) : kCand);
            nmg += mgrant ? 1u : 0u;
            // a split wish, and only a split wish, has a nonzero split cost
            if (sc > 0u && (uint64_t)Mg + (uint64_t)run.b <= F) gmask |= 1u << k;
        }
        // the granted splits listed in thread order (bit 31 of the list's
        // live index: its chain continues past the recorded members), the
        // counts added once per warp
        Pair ntot;
        const Pair gex = block_scan(Pair{(uint32_t)__popc(gmask), nmg}, ntot, s_warp);
        uint32_t q = gex.a;
#pragma unroll
        for (uint32_t k = 0; k < kMaxIpt; ++k)
            if ((gmask >> k) & 1u) s_list[q++] = make_uint2((i0 + k) | (w[k] & kScanMore), sl[k]);
        if (threadIdx.x == 0) {
            s_cnt[0] += ntot.b;
            s_cnt[1] += ntot.a;
        }
        __syncthreads();
        const uint32_t n = ntot.a;
        // the paper's gate charges 3d + 4 without a walk (the single-instance
        // frame walks, and records, every chain that can be granted); the
        // records of four grants are loaded before their marks go out
        const bool recorded = always_recorded || c.fp.gate != 1;
        for (uint32_t q0 = threadIdx.x; q0 < n; q0 += 4u * kFThreads) {
            uint2 e[4];
            uint4 r[4];
#pragma unroll
            for (uint32_t k = 0; k < 4; ++k) {
                const uint32_t q = q0 + k * kFThreads;
                e[k] = q < n ? s_list[q] : make_uint2(0u, kNull);
                r[k] = (q < n && recorded) ? I.grp[e[k].x & ~kScanMore] : make_uint4(kNull, kNull, kNull, kNull);
            }
#pragma unroll
            for (uint32_t k = 0; k < 4; ++k) {
                if (e[k].y == kNull) continue;
                if (r[k].x == kNull && r[k].w == kNull) {
                    chain_walk(I, e[k].y, 0, true);
                    continue;
                }
                atomicOr(cmd_ptr(I, e[k].y), kR);
                const uint32_t m[4] = {r[k].x, r[k].y, r[k].z, r[k].w};
#pragma unroll
                for (uint32_t q2 = 0; q2 < 4; ++q2)
                    if (m[q2] >> 30) atomicOr(cmd_ptr(I, m[q2] & 0x3FFFFFFFu), chain_code_bits(m[q2] >> 30));
                // a longer chain goes on from its fourth member (the walk
                // from there is the rest of the chain)
                if ((e[k].x & kScanMore) && (m[3] >> 30)) chain_walk(I, m[3] & 0x3FFFFFFFu, 0, true);
            }
        }
        __syncthreads();
        stats_flush(s_cnt, I.g, kStMergeGranted, kStSplitGranted);
        __syncthreads();
    }
}

__device__ void free_list(const BatchDev& bt, FCtx& c, uint32_t* s_w, bool all_granted,
                          const unsigned long long* tcounts = nullptr, uint32_t* list = nullptr);

// Exclusive prefix of one word per thread over the block, without saturation
// (sums over a whole batch may wrap; differences of prefixes are taken).
__device__ __forceinline__ uint32_t block_prefix_wrap(uint32_t x, uint32_t& total, uint32_t* s_w) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (int)(blockDim.x >> 5);
    uint32_t inc = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) s_w[warp] = inc;
    __syncthreads();
    uint32_t before = 0;
    total = 0;
    for (int q = 0; q < nw; ++q) {
        const uint32_t v = s_w[q];
        if (q < warp) before += v;
        total += v;
    }
    __syncthreads();
    return before + inc - x;
}

constexpr uint32_t kLocBits = 13, kLocMask = (1u << kLocBits) - 1u;  // offset of a new record within its scan tile
static_assert(kFThreads * kMaxIpt * 4u <= (1u << kLocBits), "a tile's allocations fit the offset");

// P4: per scan tile the fate of every item after the chains are marked
// (allocation count; granted merges validated from a list, their fates
// returned through shared memory), the tile-local prefix of the allocations,
// destination words (tile << kLocBits | offset), merged marks and the fill
// records, appended to the instance's list in any order (the records are
// independent). Then the free list (Alg. 8 for every rank at once, per word
// tile); and the last block to finish turns the tiles' allocation totals
// into prefixes (ReserveBlocks in ascending slot order, R7 reading) through
// which the fill resolves the destination words. This does in one pass over
// the live list what a pass for the sums, a barrier and a pass for the
// destinations did (364 us of a batch of 15M bisectors, now 278 us).
__device__ void phase_alloc(const BatchDev& bt, FCtx& c, uint32_t* s_cnt, Pair* s_warp, uint32_t* s_w, uint32_t* s_n,
                            uint32_t* s_tmp, uint32_t* s_buf) {
    const uint32_t T = bt.bg->total_stiles, ipt = bt.bg->scan_ipt, S = kFThreads * ipt;
    uint32_t* s_list = s_buf;              // local item indices to validate
    uint32_t* s_fate = s_buf + kFBuf / 2;  // their fates, by local item index
    __shared__ uint32_t s_feed[2];
    TileFeed feed(&bt.bg->tickets[kFeedAlloc], s_feed, T);
    for (uint32_t t = feed.first(); t < T; t = feed.next()) {
        if (threadIdx.x == 0) *s_n = 0;
        stats_reset(s_cnt);
        ctx_tile(bt, bt.stile_base, t, T, c);
        const Inst& I = c.I;
        const uint32_t N = c.N, ts = c.lt * S, e0 = threadIdx.x * ipt, i0 = ts + e0;
        uint32_t sl[kMaxIpt], cm[kMaxIpt], f[kMaxIpt];
        {  // slots and command words loaded coalesced (item ts + k 256 + tid)
           // through shared memory, then taken ipt consecutive per thread
            const uint32_t* const live = I.live;
            const uint2* const cd = I.cd;
            uint32_t a[kMaxIpt];
#pragma unroll
            for (uint32_t k = 0; k < kMaxIpt; ++k) {
                const uint32_t e = k * kFThreads + threadIdx.x;
                a[k] = (k < ipt && ts + e < N) ? live[ts + e] : kNull;
            }
#pragma unroll
            for (uint32_t k = 0; k < kMaxIpt; ++k) cm[k] = a[k] != kNull ? cd[a[k]].x : 0u;
#pragma unroll
            for (uint32_t k = 0; k < kMaxIpt; ++k)
                if (k < ipt) {
                    s_list[k * kFThreads + threadIdx.x] = a[k];
                    s_fate[k * kFThreads + threadIdx.x] = cm[k];
                }
            __syncthreads();
#pragma unroll
            for (uint32_t k = 0; k < kMaxIpt; ++k) {
                sl[k] = k < ipt ? s_list[e0 + k] : kNull;
                cm[k] = k < ipt ? s_fate[e0 + k] : 0u;
            }
            __syncthreads();
        }
        uint32_t lst = 0;  // granted merges without split bits, by k
#pragma unroll
        for (uint32_t k = 0; k < kMaxIpt; ++k) {
            f[k] = leaves_of(cm[k] & kSplitMask);
            if (!(cm[k] & kSplitMask) && (cm[k] & kCand) && (cm[k] & kMergeGrant)) {
                lst |= 1u << k;
                s_list[atomicAdd(s_n, 1u)] = e0 + k;
            }
        }
        __syncthreads();
        const uint32_t n = *s_n;
        for (uint32_t q = threadIdx.x; q < n; q += kFThreads) {
            const uint32_t e = s_list[q];
            s_fate[e] = alloc_fate(I, ts + e, kCand | kMergeGrant);
        }
        __syncthreads();
        Pair loc{0, 0};
#pragma unroll
        for (uint32_t k = 0; k < kMaxIpt; ++k) {
            if ((lst >> k) & 1u) f[k] = s_fate[e0 + k];
            const uint32_t na = f[k] & 7u;
            loc = padd(loc, Pair{na ? 1u : 0u, na});
        }
        Pair tot;
        const Pair ex = block_scan(loc, tot, s_warp);
        if (threadIdx.x == 0) {
            bt.status[bt.Titems + t] = tot.b;
            s_tmp[0] = tot.a ? atomicAdd(&I.g->C, tot.a) : 0u;
        }
        __syncthreads();
        uint32_t crun = s_tmp[0] + ex.a, arun = ex.b;
        uint4* const chgr = I.chgr;
#pragma unroll
        for (uint32_t k = 0; k < kMaxIpt; ++k) {
            const uint32_t na = f[k] & 7u;
            if (!na) continue;
            const uint32_t dw = (c.lt << kLocBits) | arun;
            // the fill's record: everything it needs before its first gather
            chgr[crun++] = make_uint4(i0 + k, sl[k], cm[k], dw);
            alloc_apply(I, i0 + k, f[k], dw, s_cnt);
            arun += na;
        }
        __syncthreads();
        stats_flush(s_cnt, I.g, kStSplitBis, kStMergeGroups, kStMergedBis);
        __syncthreads();
    }
    free_list(bt, c, s_w, false);
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        s_tmp[0] = atomicAdd(&bt.bg->tickets[kAllocDone], 1u) == gridDim.x - 1u ? 1u : 0u;
    }
    __syncthreads();
    if (!s_tmp[0]) return;
    __threadfence();
    uint32_t run = 0;
    unsigned long long* pre = bt.status;  // the gate's sums are done with
    for (uint32_t t0 = 0; t0 < T; t0 += 4u * kFThreads) {
        const uint32_t t = t0 + 4u * threadIdx.x;
        uint32_t v[4], sum = 0, tot;
#pragma unroll
        for (uint32_t k = 0; k < 4; ++k) {
            v[k] = t + k < T ? (uint32_t)__ldcg(bt.status + bt.Titems + t + k) : 0u;
            sum += v[k];
        }
        uint32_t r = run + block_prefix_wrap(sum, tot, s_w);
#pragma unroll
        for (uint32_t k = 0; k < 4; ++k) {
            if (t + k < T) pre[t + k] = r;
            r += v[k];
        }
        run += tot;
    }
    __syncthreads();
    for (uint32_t b = threadIdx.x; b < bt.B; b += kFThreads) {
        const uint32_t lo = bt.stile_base[b], hi = bt.stile_base[b + 1];
        Globals* g = bt.inst[b].g;
        const uint32_t end = hi < T ? (uint32_t)__ldcg(pre + hi) : run;
        const uint32_t A = hi > lo ? end - (uint32_t)__ldcg(pre + lo) : 0u;
        g->A = A;
        g->stats[kStAllocated] = A;
        if (A > (uint32_t)min((uint64_t)__ldcg(&g->F), (uint64_t)__ldcg(&g->Mg) + (uint64_t)__ldcg(&g->Stot)))
            set_err(g, kErrOverflow);
    }
}

// A destination word (local scan tile << kLocBits | offset) resolved through
// the prefixes of the instance's tiles.
struct DestBatch {
    const unsigned long long* pre;  // of the instance's first tile
    uint32_t base, last;            // its prefix, and the instance's last tile
    uint32_t A;
    __device__ __forceinline__ uint32_t operator()(uint32_t d) const {
        return (uint32_t)pre[min(d >> kLocBits, last)] - base + (d & kLocMask);
    }
    __device__ __forceinline__ const uint32_t* freel(const Inst& I) const { return I.freel; }
    __device__ __forceinline__ void set(const Inst& I, uint32_t s) const { set_bit(I, s); }
    __device__ __forceinline__ void clear(const Inst& I, uint32_t s) const { clear_bit(I, s); }
};

// The free list (Alg. 8 for every rank at once) per word tile: the frame's
// first `bound` zero bits of the frame-start bitfield, bound = the free
// slots or, when smaller, the granted merge cost plus the requested split
// cost (all requests with `all_granted`), an upper bound of the
// allocations.
// With `tcounts` (single instance, word tiles of the frame's tile counts)
// the ones before a word tile are summed over the block from those counts
// instead of read down the sum tree one level at a time.
// `list`: where it goes (the instance's first free list by default).
__device__ void free_list(const BatchDev& bt, FCtx& c, uint32_t* s_w, bool all_granted,
                          const unsigned long long* tcounts, uint32_t* list) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (uint32_t wt = blockIdx.x; wt < bt.Twords; wt += gridDim.x) {
        ctx_tile(bt, bt.wtile_base, wt, bt.Twords, c);
        const Inst& I = c.I;
        const uint32_t lt = c.lt;
        const uint64_t req = all_granted ? __ldcg(&I.g->rq_merge) + __ldcg(&I.g->rq_split)
                                         : (uint64_t)I.g->Mg + (uint64_t)I.g->Stot;
        const uint32_t bound = (uint32_t)min((uint64_t)c.F, req);
        const uint32_t TW = min(I.W, bt.tw);
        const uint32_t nt = I.W / TW;
        uint32_t ones_before = 0;
        if (tcounts) {
            uint32_t part = 0;
            for (uint32_t t = threadIdx.x; t < lt; t += blockDim.x) part += (uint32_t)(__ldcg(tcounts + t) >> 32);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xFFFFFFFFu, part, o);
            if (lane == 0) s_w[warp] = part;
            __syncthreads();
            for (int q = 0; q < nw; ++q) ones_before += s_w[q];
            __syncthreads();
        } else {
            for (uint32_t n = nt + lt; n > 1; n >>= 1)
                if (n & 1u) ones_before += I.sums[n - 1];
        }
        const uint64_t zeros_before = (uint64_t)lt * TW * 32u - ones_before;
        if (zeros_before < bound) {  // block-uniform
            const uint32_t w = lt * TW + threadIdx.x;
            uint32_t z = 0;
            if (threadIdx.x < TW) {
                const uint32_t valid = I.cap < 32u ? (1u << I.cap) - 1u : 0xFFFFFFFFu;
                z = ~I.bits[w] & valid;
            }
            const uint32_t mine = __popc(z);
            uint32_t inc = mine;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
                if (lane >= o) inc += y;
            }
            if (lane == 31) s_w[warp] = inc;
            __syncthreads();
            if (warp == 0) {
                const uint32_t x = lane < nw ? s_w[lane] : 0u;
                uint32_t xi = x;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, xi, o);
                    if (lane >= o) xi += y;
                }
                __syncwarp();
                if (lane < nw) s_w[lane] = xi - x;
            }
            __syncthreads();
            uint64_t r = zeros_before + s_w[warp] + (inc - mine);
            uint32_t* const freel = list ? list : I.freel;  // in a register across the stores
            while (z && r < bound) {
                freel[r] = w * 32u + (uint32_t)(__ffs(z) - 1);
                ++r;
                z &= z - 1u;
            }
        }
        __syncthreads();
    }
}

// One changed bisector: live index i, slot s, command word and free-list
// index of its first new record (a split, or a merge group's smallest
// member, whose command word carries no split bits). Returns the number of
// unchanged neighbours relinked.
template <typename DM>
__device__ __forceinline__ uint32_t fill_item_dm(const Inst& I, uint32_t i, uint32_t s, uint32_t cmd, uint32_t dest,
                                                 const DM& dm) {
    if (cmd & kSplitMask) {
        dm.clear(I, s);
        return fill_split(I, s, cmd, dest, dm);
    }
    const uint4 m = I.grp[i];
    const uint32_t ms[4] = {m.x, m.y, m.z, m.w};
#pragma unroll
    for (int q = 0; q < 4; ++q)
        if (ms[q] != kNull && !bad_slot(I, ms[q], kErrLink)) dm.clear(I, ms[q]);
    return fill_merge(I, dest, m, dm);
}

// P5: FillNewBlocks + UpdateNeighbors + UpdateBitfield for the changed items,
// from the fill records.
__device__ void phase_fill(const BatchDev& bt, FCtx& c, uint32_t* s_cnt, uint32_t* s_list, Pair* s_warp) {
    batch_list(bt, c, kStRelinked, s_cnt, s_list, s_warp, [](const Inst& I) { return __ldcg(&I.g->C); },
               [&](uint32_t b, const Inst& I, uint32_t q) {
                   const uint32_t t0 = bt.B == 1 ? 0u : bt.stile_base[b];
                   const unsigned long long* pre = bt.status + t0;
                   const Globals* g = I.g;
                   const DestBatch dm{pre, (uint32_t)pre[0], g->nstiles - 1u, g->A};
                   const uint4 r = I.chgr[q];
                   return fill_item_dm(I, r.x, r.y, r.z, dm(r.w), dm);
               });
}

// P6: SumReduction (Sec. 3.1) per word tile; the last tile of an instance to
// finish builds the levels above the tiles, in shared memory once a level
// has at most kFBuf / 2 nodes.
__device__ void phase_reduce(const BatchDev& bt, FCtx& c, uint32_t* s_buf, uint32_t* s_flag) {
    for (uint32_t wt = blockIdx.x; wt < bt.Twords; wt += gridDim.x) {
        ctx_tile(bt, bt.wtile_base, wt, bt.Twords, c);
        const Inst& I = c.I;
        const uint32_t lt = c.lt;
        const uint32_t W = I.W;
        const uint32_t TW = min(W, bt.tw);
        const uint32_t nt = W / TW;
        const uint32_t w = lt * TW + threadIdx.x;
        const bool mine = threadIdx.x < TW;
        const uint32_t pc = mine ? __popc(I.bits[w]) : 0u;
        if (mine) I.sums[W + w] = pc;
        s_buf[threadIdx.x] = pc;
        __syncthreads();
        uint32_t lvl = 1;
        for (uint32_t cnt = TW >> 1; cnt >= 1u; cnt >>= 1, ++lvl) {
            uint32_t v = 0;
            if (threadIdx.x < cnt) v = s_buf[2 * threadIdx.x] + s_buf[2 * threadIdx.x + 1];
            __syncthreads();
            if (threadIdx.x < cnt) {
                s_buf[threadIdx.x] = v;
                I.sums[((W + lt * TW) >> lvl) + threadIdx.x] = v;
            }
            __syncthreads();
        }
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) *s_flag = (atomicAdd(&I.g->done, 1u) == nt - 1u) ? 1u : 0u;
        __syncthreads();
        if (*s_flag) {
            __threadfence();
            uint32_t n = nt;  // nodes [n, 2n) hold the tile roots
            for (; n > kFBuf / 2u; n >>= 1) {
                for (uint32_t k = threadIdx.x; k < n / 2u; k += blockDim.x)
                    I.sums[n / 2u + k] = __ldcg(I.sums + n + 2u * k) + __ldcg(I.sums + n + 2u * k + 1u);
                __syncthreads();
            }
            if (n > 1u) {
                for (uint32_t k = threadIdx.x; k < n; k += blockDim.x) s_buf[n + k] = __ldcg(I.sums + n + k);
                __syncthreads();
                for (uint32_t m = n >> 1; m >= 1u; m >>= 1) {
                    for (uint32_t k = threadIdx.x; k < m; k += blockDim.x) {
                        const uint32_t p = m + k;
                        const uint32_t v = s_buf[2u * p] + s_buf[2u * p + 1u];
                        s_buf[p] = v;
                        I.sums[p] = v;
                    }
                    __syncthreads();
                }
            }
            if (threadIdx.x == 0) {
                I.g->stats[kStLiveAfter] = __ldcg(I.sums + 1);
                I.g->done = 0;
            }
        }
        __syncthreads();
    }
}

// P7: CachePointers (Alg. 7 for every rank at once) per word tile, and, in a
// batch, the FP32 vertices of the tile's live bisectors when the frame
// exports them.
template <int F>
__device__ void phase_compact(const BatchDev& bt, FCtx& c, const uint32_t* s_tab, uint32_t* s_buf,
                              uint32_t* s_w, float* s_stage) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    __shared__ uint32_t s_feed[2];
    TileFeed feed(&bt.bg->tickets[kFeedCompact], s_feed, bt.Twords);
    for (uint32_t wt = feed.first(); wt < bt.Twords; wt = feed.next()) {
        ctx_tile(bt, bt.wtile_base, wt, bt.Twords, c);
        const Inst& I = c.I;
        const FrameP& fp = c.fp;
        const uint32_t lt = c.lt;
        const uint32_t W = I.W;
        const uint32_t TW = min(W, bt.tw);
        const uint32_t nt = W / TW;
        if (32u * TW > kFBuf) {  // block-uniform: a tile's positions must fit the staging buffer
            if (threadIdx.x == 0) set_err(I.g, kErrOverflow);
            continue;
        }
        uint32_t before = 0;
        for (uint32_t n = nt + lt; n > 1; n >>= 1)
            if (n & 1u) before += __ldcg(I.sums + n - 1);
        const uint32_t w = lt * TW + threadIdx.x;
        const uint32_t wv = threadIdx.x < TW ? __ldcg(I.bits + w) : 0u;
        const uint32_t pc = __popc(wv);
        uint32_t inc = pc;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
            if (lane >= o) inc += y;
        }
        if (lane == 31) s_w[warp] = inc;
        __syncthreads();
        if (warp == 0) {
            const uint32_t x = lane < nw ? s_w[lane] : 0u;
            uint32_t xi = x;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, xi, o);
                if (lane >= o) xi += y;
            }
            __syncwarp();
            if (lane < nw) s_w[lane] = xi - x;
            if (lane == nw - 1) s_w[nw] = xi;
        }
        __syncthreads();
        uint32_t r = s_w[warp] + inc - pc;
        const uint32_t tot = s_w[nw];
        uint32_t m = wv;
        while (m) {
            s_buf[r++] = w * 32u + (uint32_t)(__ffs(m) - 1);
            m &= m - 1u;
        }
        __syncthreads();
        for (uint32_t k = threadIdx.x; k < tot; k += blockDim.x) I.live[before + k] = s_buf[k];
        if (fp.vout && bt.B > 1) {
            // rows of 32 consecutive live bisectors per warp, staged and stored
            // 16 bytes wide; the heap ID of the warp's next round loaded ahead
            const uint32_t n = before < fp.vcap ? min(tot, fp.vcap - before) : 0u;
            const uint64_t* const heap = I.heap;
            if (vc_form<F>(fp)) {
                for (uint32_t k = threadIdx.x; k < n; k += blockDim.x)
                    vertex_item_cached<F>(I, fp, before + k, s_buf[k], s_tab, fp.vout);
            } else {
                uint64_t j = threadIdx.x < n ? heap[s_buf[threadIdx.x]] : 0ull;
                for (uint32_t k0 = threadIdx.x & ~31u; k0 < n; k0 += blockDim.x) {  // warp-uniform
                    const uint32_t k = k0 + lane, kn = k + blockDim.x;
                    const uint64_t jn = kn < n ? heap[s_buf[kn]] : 0ull;
                    float r[9];
                    bool ok = true;
                    if (k < n) ok = vertex_eval<F>(I, fp, j, s_tab, r);
                    if (__all_sync(0xFFFFFFFFu, ok)) {
                        warp_rows_out(r, s_stage + 288u * warp, fp.vout, (uint64_t)before + k0, min(32u, n - k0));
                    } else if (k < n && ok) {  // a row the decode refused stays unwritten
                        float* o = fp.vout + 9ull * (before + k);
#pragma unroll
                        for (int q = 0; q < 9; ++q) o[q] = r[q];
                    }
                    j = jn;
                }
            }
        }
        __syncthreads();
    }
}

// Resident blocks per SM the register budget is sized for (the cooperative
// grid is that many blocks per SM).
#ifndef CBT_FRAME_MIN_BLOCKS
#define CBT_FRAME_MIN_BLOCKS 4
#endif

// P8 (single instance): the vertices of the new live list, strided over the
// whole grid (word tiles hold very different live counts). In the sphere and
// displaced forms the unchanged bisectors' vertices are copied from the
// cache P1 filled (each costs three FP64 projections or three noise sums to
// evaluate), and the new ones are listed and evaluated densely by the block
// (so that no warp idles beside one evaluating lane); otherwise the slot and
// heap ID of the next round are loaded while the current one is evaluated.
template <int F>
__device__ void vertices_of(const Inst& I, const FrameP& fp, const uint32_t* s_tab, uint32_t* s_list,
                            uint32_t* s_n) {
    if (!fp.vout) return;
    const uint32_t n = min(__ldcg(I.sums + 1), fp.vcap);
    const uint32_t stride = gridDim.x * kFThreads;
    if (vc_form<F>(fp)) {
        auto evaluate = [&](uint32_t cnt) {  // one point per thread: few rows, each three long evaluations
            for (uint32_t q = threadIdx.x; q < 3u * cnt; q += kFThreads) {
                const uint32_t i = s_list[q / 3u], v = q % 3u;
                vertex_point<F>(I, fp, I.heap[I.live[i]], (int)v, s_tab, fp.vout + 9ull * i + 3u * v);
            }
        };
        if (threadIdx.x == 0) *s_n = 0;
        __syncthreads();
        // the cached rows of a warp's 32 consecutive rows leave through the
        // warp's staging area (the list of uncached rows uses the front of
        // s_list, the staging its back) with one coalesced store per word
        const uint32_t lane = threadIdx.x & 31u;
        float* stage = reinterpret_cast<float*>(s_list) + (kFBuf - 288u * (kFThreads / 32)) + 288u * (threadIdx.x >> 5);
        // the list's length as every thread of the block counts it: *s_n itself
        // may already hold the next round's rows when a slow warp looks
        uint32_t cnt = 0;
        for (uint32_t base = blockIdx.x * kFThreads; base < n; base += stride) {
            const uint32_t i = base + threadIdx.x;
            bool cached = false;
            if (i < n) {
                const uint32_t s = I.live[i];
                if (*cmd_ptr(I, s) & kVcValid) {
                    const float* src = I.vc + 9ull * s;
#pragma unroll
                    for (int k = 0; k < 9; ++k) stage[9u * lane + (uint32_t)k] = src[k];
                    cached = true;
                } else {
                    s_list[atomicAdd(s_n, 1u)] = i;
                }
            }
            const uint32_t m = __ballot_sync(0xFFFFFFFFu, cached);
            __syncwarp();
            const uint32_t w0 = i - lane;
            float* dst = fp.vout + 9ull * w0;
            for (uint32_t w = lane; w < 288u; w += 32u)
                if ((m >> (w / 9u)) & 1u) dst[w] = stage[w];
            __syncwarp();
            cnt += (uint32_t)__syncthreads_count(i < n && !cached);
            if (cnt > kFBuf - 288u * (kFThreads / 32) - kFThreads) {  // block-uniform: keep clear of the staging
                evaluate(cnt);
                __syncthreads();
                cnt = 0;
                if (threadIdx.x == 0) *s_n = 0;
                __syncthreads();
            }
        }
        evaluate(cnt);
        return;
    }
    // warp-uniform rounds of 32 consecutive rows (warp-major over the grid,
    // so that rows of costly regions spread over the SMs), staged per warp in
    // s_list (8 warps x 288 floats) and stored 16 bytes wide
    const uint32_t lane = threadIdx.x & 31u;
    float* stage = reinterpret_cast<float*>(s_list) + 288u * (threadIdx.x >> 5);
    uint32_t w0 = ((threadIdx.x >> 5) * gridDim.x + blockIdx.x) * 32u;
    // the heap ID one round ahead and its slot two, so that no load waits on
    // one issued in the same round
    const uint32_t* const live = I.live;
    const uint64_t* const heap = I.heap;
    uint64_t j = w0 + lane < n ? heap[live[w0 + lane]] : 0ull;
    uint32_t sb = w0 + lane + stride < n ? live[w0 + lane + stride] : 0u;
    for (; w0 < n; w0 += stride) {
        const uint32_t i = w0 + lane;
        const uint32_t sc = i + 2u * stride < n ? live[i + 2u * stride] : 0u;
        const uint64_t jn = i + stride < n ? heap[sb] : 0ull;
        sb = sc;
        float r[9];
        bool ok = true;
        if (i < n) ok = vertex_eval<F>(I, fp, j, s_tab, r);
        if (__all_sync(0xFFFFFFFFu, ok)) {
            warp_rows_out(r, stage, fp.vout, w0, min(32u, n - w0));
        } else if (i < n && ok) {  // a row the decode refused stays unwritten
            float* o = fp.vout + 9ull * i;
#pragma unroll
            for (int k = 0; k < 9; ++k) o[k] = r[k];
        }
        j = jn;
    }
}
template <int F>
__device__ void phase_vertices(const BatchDev& bt, FCtx& c, const uint32_t* s_tab, uint32_t* s_list,
                               uint32_t* s_n) {
    ctx_tile(bt, bt.tile_base, 0, 1, c);
    vertices_of<F>(c.I, c.fp, s_tab, s_list, s_n);
}

template <int F, bool kOne>
__global__ void __launch_bounds__(kFThreads, CBT_FRAME_MIN_BLOCKS) k_frame(BatchDev bt) {
    __shared__ FCtx s_c;
    __shared__ __align__(16) uint32_t s_tab[kDecTabWords];
    __shared__ __align__(16) uint32_t s_buf[kFBuf];
    __shared__ Pair s_warp[kFThreads / 32 + 1];
    __shared__ uint32_t s_red[4 * (kFThreads / 32)];
    __shared__ uint32_t s_cnt[kBlockStats];
    __shared__ uint32_t s_w[kFThreads / 32 + 1];
    __shared__ uint32_t s_tmp[4];
    __shared__ uint32_t s_n;
    __shared__ __align__(16) float s_stage[288 * (kFThreads / 32)];  // per warp: 32 rows of 9 floats
    // every block reads the epoch before its first arrival; block 0 advances
    // it after the last barrier, when every block has read it
    const uint32_t epoch = ld_volatile(&bt.bg->bar_epoch);
    stamp(bt, 0);
    load_dec6(s_tab);
    if (threadIdx.x == 0) s_c.b = kNull;
    phase_prep(bt, s_warp, s_tmp);
    grid_sync(bt.bg, epoch, 1u);
    stamp(bt, 1);
    if (kOne && classify_in_parts<F>(bt.bg->total_tiles))
        phase_classify<F, true>(bt, s_c, s_tab, s_cnt);
    else
        phase_classify<F, false>(bt, s_c, s_tab, s_cnt);
    grid_sync(bt.bg, epoch, 2u);
    stamp(bt, 2);
    if (kOne && walks_in_parts(bt.bg->total_tiles))
        phase_walks<true>(bt, s_c, s_cnt, reinterpret_cast<unsigned long long*>(s_buf), s_tmp, s_w);
    else
        phase_walks<false>(bt, s_c, s_cnt, reinterpret_cast<unsigned long long*>(s_buf), s_tmp, s_w);
    grid_sync(bt.bg, epoch, 3u);
    stamp(bt, 3);
    phase_gate(bt, s_c, s_cnt, s_red, s_warp, s_tmp, &s_n, reinterpret_cast<uint2*>(s_buf));
    grid_sync(bt.bg, epoch, 4u);
    stamp(bt, 4);
    phase_alloc(bt, s_c, s_cnt, s_warp, s_w, &s_n, s_tmp, s_buf);
    grid_sync(bt.bg, epoch, 5u);
    stamp(bt, 5);
    phase_fill(bt, s_c, s_cnt, s_buf, s_warp);
    grid_sync(bt.bg, epoch, 6u);
    stamp(bt, 6);
    phase_reduce(bt, s_c, s_buf, &s_tmp[0]);
    grid_sync(bt.bg, epoch, 7u);
    stamp(bt, 7);
    phase_compact<F>(bt, s_c, s_tab, s_buf, s_w, s_stage);
    if (kOne) {
        grid_sync(bt.bg, epoch, 8u);
        stamp(bt, 8);
        phase_vertices<F>(bt, s_c, s_tab, s_buf, &s_n);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (bt.timing) atomicMax(&bt.bg->t[kFramePhases], global_ns());
        if (blockIdx.x == 0) {
            bt.bg->bar_epoch = epoch + (kOne ? kBarriers + 1u : kBarriers) * gridDim.x;
            if (ld_volatile(&bt.bg->abort))
                for (uint32_t b = 0; b < bt.B; ++b) set_err(bt.inst[b].g, kErrTimeout);
        }
    }
}

// Self-test of the bounded wait: one barrier that expects one more arrival
// than the grid has. Every wait runs out after `limit` polls, sets the abort
// word and returns; block 0 then moves the epoch past this launch's
// arrivals so that the counters stay consistent.
__global__ void __launch_bounds__(kFThreads) k_wait_selftest(BatchGlobals* bg, int limit) {
    const uint32_t epoch = ld_volatile(&bg->bar_epoch);
    grid_wait(bg, epoch + gridDim.x + 1u, limit);
    if (blockIdx.x == 0 && threadIdx.x == 0) bg->bar_epoch = epoch + gridDim.x;
}

// ===================================================== one instance, fewer phases
//
// k_frame1: the frame of a single instance (a batch of one), with the same
// results as k_frame in seven phases, without P3 when the frame's requests all
// fit the free slots, without P6 when nothing is exported. A grid barrier
// between every two of them (four to six), but for the one after P0 where that
// is not needed:
//   P0 prep      frame counters; the camera-relative roots; the word-tile
//                counts copied. When the last frame was not this kernel also
//                what that frame would have left: the chain-mark words of the
//                live slots, the wish counters and the walk list's length
//                cleared. When it was, and the mesh is small, every block fills
//                the whole root table and the phase ends without a barrier
//   P1 classify  wishes (Sec. 3.3 GenerateCommands), in 32-item chunks dealt
//                warp-major over the grid; the items that need a walk
//                appended to the frame's walk list; per scan tile the split
//                wishes' lower-bound costs
//   P2 walks     the walk list spread evenly over the grid. A split wish's
//                chain (command form of Alg. 3) is walked, recorded and
//                marked (into the chain-mark words) unless the split wishes
//                before its scan tile and itself already cost more than the
//                free slots at their lower bounds, so that the gate denies
//                it whatever its cost. A merge wish with an even heap ID
//                walks its Alg. 4 group while it can be a merge candidate
//                with this wish its smallest member, which then records it
//                with its merge cost. Per scan tile the (merge, split) cost
//                sums, per frame their totals.
//   P3 gate      (when the totals exceed the free slots F) grants in the
//                order of the R6 reading and chain marking into the command
//                words; otherwise every request is granted and the chain-mark
//                words hold the marks
//   P4 alloc     fates, their tile-local allocation prefix (a destination
//                word holds the tile and the offset within it), the fill
//                records per tile, the bits cleared per word tile; the free
//                list only when the last frame was not this kernel
//   P5 fill      on half of the blocks the tiles' record and allocation
//                offsets in shared memory, new records and links; on the
//                others every word tile's new count (frame-start count,
//                clears, and its share of the first A zero bits), hence the
//                sum tree, and per word tile (one warp) its new words, its
//                rows of the new live list and, from its zero bits, of the
//                next frame's free list (every zero bit in slot order)
//   P6 vertices  the export of the new list (FP32, fixed point, FP64
//                evaluated; sphere and displaced forms copied from the cache
//                of P1), 32 rows per warp, warp-major
// The instance descriptor and the frame parameters are read from the launch
// parameters (a copy in shared memory would be reloaded after every store
// through a generic pointer).
//
// From one frame to the next: while the instance's flag word freel_full says
// that its last frame was this kernel, a free list of every zero bit is kept
// (freel or freel2), the ones before each word tile (one half of tpre), and the
// chain marks (chg) of the live slots, the wish counters (wish), the cleared
// bits (clr) and the walk list's length (nwalk) are 0: P5's final part leaves
// them so. All of it lies in the instance's workspace, none in that of the
// handle that launches the frame; every other form of the frame clears the flag.

constexpr uint32_t kMaxTiles1 = kFBuf / 2;  // scan tiles and word tiles the shared tables hold
// Meshes up to kLocalRoots halfedges: every block fills the root table. With
// and without the barrier this saves, us a frame: 24 halfedges 46.8 and 45.3, 60
// 59.0 and 57.0 (with cached points 48.8 and 47.1), 96 47.4 and 47.4, 104 46.1 and
// 44.9, 208 46.0 and 46.8: the line lies where the gain is sure.
constexpr uint32_t kLocalRoots = 64;

// Exclusive prefix sums of n <= kMaxTiles1 pairs over the block: thread x
// takes the consecutive entries [x k, x k + k), k = ceil(n / threads), loads
// them all at once (load(i) -> Pair), and after one block scan hands each
// entry's exclusive prefix to store(i, Pair); returns the total.
template <typename Load, typename Store>
__device__ __forceinline__ Pair block_table(uint32_t n, Load load, Store store, Pair* s_warp) {
    constexpr uint32_t kPer = kMaxTiles1 / kFThreads;
    const uint32_t per = (n + kFThreads - 1u) / kFThreads;
    const uint32_t i0 = threadIdx.x * per;
    Pair v[kPer];
    Pair loc{0, 0};
#pragma unroll
    for (uint32_t k = 0; k < kPer; ++k) {
        v[k] = (k < per && i0 + k < n) ? load(i0 + k) : Pair{0, 0};
        loc = padd(loc, v[k]);
    }
    Pair tot;
    Pair run = block_scan(loc, tot, s_warp);
#pragma unroll
    for (uint32_t k = 0; k < kPer; ++k) {
        if (k < per && i0 + k < n) store(i0 + k, run);
        run = padd(run, v[k]);
    }
    __syncthreads();
    return tot;
}

// A destination word (tile << kLocBits | offset) resolved through the
// tiles' allocation offsets in shared memory.
struct DestTiles {
    const uint32_t* apre;
    const uint32_t* list;  // the frame's free list
    uint32_t A;
    __device__ __forceinline__ uint32_t operator()(uint32_t d) const {
        return apre[min(d >> kLocBits, kMaxTiles1 - 1u)] + (d & kLocMask);
    }
    __device__ __forceinline__ const uint32_t* freel(const Inst&) const { return list; }
    // the bitfield is rewritten from its frame-start words and the clear masks
    __device__ __forceinline__ void set(const Inst&, uint32_t) const {}
    __device__ __forceinline__ void clear(const Inst&, uint32_t) const {}
};

// What the last frame left, read from its flag word (freel_full) at the start:
// bit 0 that it was this kernel, bit 1 in which of their two buffers the free
// list and the ones before each word tile then are (0 without bit 0). The fill
// reads the one buffer while the next frame's is written beside it.
struct Carry {
    uint32_t w;
    __device__ __forceinline__ bool ok() const { return (w & 1u) != 0u; }
    __device__ __forceinline__ uint32_t buffer() const { return (w & 1u) ? (w >> 1) & 1u : 0u; }
};
// The free list of the current frame (ahead = 0) or the next one (ahead = 1).
__device__ __forceinline__ uint32_t* free_list1(const BatchDev& bt, Carry carry, uint32_t ahead) {
    return (carry.buffer() ^ ahead) ? bt.inst0.freel2 : bt.inst0.freel;
}

// Word-tile counts of the single-instance frame, one 64-bit word per word
// tile (2^tbits slots, its sum-tree node at nt + t): the node's frame-start
// value in the high half, the bits the frame clears in it in the low half.
// The bits it sets there follow from the allocation count A alone: the new
// records take the first A zero bits of the frame-start bitfield (Alg. 8).
__device__ __forceinline__ unsigned long long* tile_counts(const BatchDev& bt) {
    return bt.status + 2u * bt.Titems;
}
// Per scan tile: the split wishes' lower-bound costs (P1).
__device__ __forceinline__ unsigned long long* wish_counts(const BatchDev& bt) { return bt.wish; }
// The chain marks of P2 (one word per slot; the per-step frame's list of
// changed items uses the same array).
__device__ __forceinline__ uint32_t* chain_marks(const Inst& I) { return I.chg; }
// The frame's walk list, in the fill records' array (written only in P4):
// per entry {live index | split flag << 31, slot, heap ID low, high}.
__device__ __forceinline__ uint4* walk_list_of(const Inst& I) { return I.chgr; }
constexpr uint32_t kWalkCap1 = kFBuf / 4;  // uint4 entries of the block's list
// The x word of a walk entry: the live index, bit 31 for a split wish, bit
// 30 for a split wish under a root whose halfedge has a Twin, so that it has
// one too (its chain then costs at least 4: itself and the Twin's pair,
// Alg. 3); else the chain can cost 2.
constexpr uint32_t kWalkSplit = 0x80000000u, kWalkInterior = 0x40000000u, kWalkIndex = 0x3FFFFFFFu;

__device__ __forceinline__ uint32_t scan_ipt1(uint32_t N) {
    const uint32_t per_round = gridDim.x * kFThreads;
    return min(kMaxIpt, max(kMinIpt, (N + per_round - 1u) / per_round));
}

// The frame's counters and tile words that no other phase before the walks
// reads (N: the live count, which every block reads itself).
__device__ void frame_init1(const BatchDev& bt, uint32_t tbits, uint32_t N) {
    const Inst& I = bt.inst0;
    const uint32_t nt = I.cap >> tbits;
    const uint32_t ipt = scan_ipt1(N), S = ipt * kFThreads, T = (N + S - 1u) / S;
    const uint32_t gt = blockIdx.x * kFThreads + threadIdx.x, stride = gridDim.x * kFThreads;
    unsigned long long* tc = tile_counts(bt);
    for (uint32_t t = gt; t < nt; t += stride) tc[t] = (unsigned long long)__ldcg(I.sums + nt + t) << 32;
    for (uint32_t t = gt; t < T; t += stride) bt.status[t] = 0ull;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        Globals* g = I.g;
        g->N = N;
        g->F = I.cap - N;
        g->A = 0;
        g->Mg = 0;
        g->Stot = 0;
        g->C = 0;
        g->done = 0;
        g->ntiles = (N + kTileItems - 1u) / kTileItems;
        g->nstiles = T;
        for (int k = 0; k < kStCount; ++k) g->stats[k] = 0;
        g->stats[kStLiveBefore] = N;
        g->stats[kStFreeBefore] = I.cap - N;
        g->stats[kStFrame] = bt.fp0.frame;
        g->rq_merge = 0;
        g->rq_split = 0;
        if (bt.nout) bt.nout[0] = N;
        bt.tile_base[0] = 0;
        bt.tile_base[1] = g->ntiles;
        bt.stile_base[0] = 0;
        bt.stile_base[1] = T;
        bt.bg->total_tiles = g->ntiles;
        bt.bg->total_stiles = T;
        bt.bg->scan_ipt = ipt;
        bt.bg->live_total = N;
        bt.bg->t[kFramePhases] = 0;
    }
}

// P0 (single instance): the frame's counters, and what classify needs from
// other blocks: the camera-relative roots, the wish counters and the walk
// list's length cleared, and the chain-mark words of the live slots cleared
// unless the last frame (this kernel) left them 0.
__device__ void phase_prep1(const BatchDev& bt, uint32_t tbits, uint32_t N) {
    const Inst& I = bt.inst0;
    frame_init1(bt, tbits, N);
    const uint32_t gt = blockIdx.x * kFThreads + threadIdx.x, stride = gridDim.x * kFThreads;
    for (uint32_t t = gt; t < bt.Titems; t += stride) wish_counts(bt)[t] = 0ull;
    if (gt == 0u) I.g->nwalk = 0;
    const uint32_t nw = gridDim.x * (kFThreads / 32), wid = blockIdx.x * (kFThreads / 32) + threadIdx.x / 32u;
    const uint32_t per = min(kRelRange, ((bt.Trel + nw - 1u) / nw + 31u) & ~31u);
    for (uint32_t e = wid * per; e < bt.Trel; e += nw * per) rel_range(bt, e, min(bt.Trel, e + per));
    uint32_t* marks = chain_marks(I);
    if (__ldcg(&I.g->marks_clean)) return;  // the last frame left them 0
    for (uint32_t i0 = gt; i0 < N; i0 += 4u * stride) {
        uint32_t sl[4];
#pragma unroll
        for (uint32_t k = 0; k < 4; ++k) sl[k] = i0 + k * stride < N ? __ldcg(I.live + i0 + k * stride) : kNull;
#pragma unroll
        for (uint32_t k = 0; k < 4; ++k)
            if (sl[k] != kNull) marks[sl[k]] = 0u;
    }
}

// --- Points evaluated once per warp (displaced and projected forms)
//
// A bisector's LOD test reads four points, and a conforming triangulation has
// half a vertex per triangle, so most of a warp's 128 points are the same
// ones: siblings, diamond partners and finer neighbours lie close in slot
// order. Where a point is expensive (a noise sum of several octaves; an FP64
// projection on a chip with two FP64 lanes per SM) the warp finds the distinct
// ones with a hash table in shared memory and evaluates those alone, spread
// over its lanes. The results are those of evaluating each point, because a
// point is only shared when the inputs of its evaluation are equal bit for bit.
// The terrain's classify phase (877k leaves, six octaves) went from 126 to 106 us (98
// with two points per lane at a time, fbm2_pair), the wave planet's (117k) from
// 43 to 41, its frame from 109 to 102.
template <int F>
constexpr bool kSharedPoints = F == kFormF32Disp || F == kFormSphere;
constexpr uint32_t kPtSlots = 1024;  // hash slots (bytes) per warp, eight times its points
// Words per warp: the points' keys (world x, y in FP32; or the weights over
// 2^62 and the root), later their results, and the list of the distinct ones.
template <int F>
constexpr uint32_t kPtWords = !kSharedPoints<F> ? 0u : (F == kFormF32Disp ? 2u : 5u) * 128u + 32u;

// Finds the warp's distinct points among ids 32 k + lane (k = 0..3, those with
// has[k]), all lanes taking part: rep[k] = the id that stands for it; the
// standing ids listed; returns their number. Every point writes its id to the
// slot its key hashes to, and takes the id it then finds there if that has
// its key (same(k, id)); where two keys meet in a slot, the points of the one
// that lost stand for themselves, which costs an evaluation now and then and
// changes nothing else. (A table kept exact with compare-and-swap made
// classify slower than evaluating everything: 155 us against 126.)
template <typename Same>
__device__ __forceinline__ uint32_t warp_distinct(uint8_t* slots, uint8_t* list, const uint32_t hash[4],
                                                  const bool has[4], uint32_t rep[4], Same same) {
    const uint32_t lane = threadIdx.x & 31u;
#pragma unroll
    for (uint32_t k = 0; k < 4; ++k)
        if (has[k]) slots[hash[k] % kPtSlots] = (uint8_t)(32u * k + lane);
    __syncwarp();  // the keys, stored by the caller, too
#pragma unroll
    for (uint32_t k = 0; k < 4; ++k) {
        const uint32_t id = 32u * k + lane;
        rep[k] = id;
        if (has[k]) {
            const uint32_t other = slots[hash[k] % kPtSlots];
            if (same(k, other)) rep[k] = other;
        }
    }
    uint32_t n = 0;
#pragma unroll
    for (uint32_t k = 0; k < 4; ++k) {
        const uint32_t id = 32u * k + lane;
        const bool own = has[k] && rep[k] == id;
        const uint32_t m = __ballot_sync(0xFFFFFFFFu, own);
        if (own) list[n + __popc(m & ((1u << lane) - 1u))] = (uint8_t)id;
        n += __popc(m);
    }
    __syncwarp();
    return n;
}

// lod_wishes for the lanes with `ok`, the whole warp taking part.
template <int F>
__device__ __forceinline__ void lod_wishes_shared(const Inst& I, const FrameP& fp, bool ok, uint64_t j, int d,
                                                  uint32_t h, const uint32_t* tab, uint8_t* slots, uint32_t* pts,
                                                  bool& split, bool& merge, float* keep) {
    const uint32_t lane = threadIdx.x & 31u;
    uint8_t* list = reinterpret_cast<uint8_t*>(pts + kPtWords<F> - 32u);
    const bool has[4] = {ok, ok, ok, ok && d >= 1};
    uint32_t hash[4], rep[4];
    float r[12];
    if (F == kFormF32Disp) {
        u64* key = reinterpret_cast<u64*>(pts);
        if (ok) eval_rows<kFormF32>(fp, I.rel, j, d, h, tab, 15, r);
        const float ex = __double2float_rn(fp.eye[0]), ey = __double2float_rn(fp.eye[1]);
        u64 mine[4];
#pragma unroll
        for (uint32_t k = 0; k < 4; ++k) {
            const uint32_t x = __float_as_uint(__fadd_rn(r[3 * k], ex)), y = __float_as_uint(__fadd_rn(r[3 * k + 1], ey));
            mine[k] = (u64)x | ((u64)y << 32);
            hash[k] = (x * 0x9E3779B1u ^ y * 0x85EBCA77u) >> 20;
            key[32u * k + lane] = mine[k];
        }
        const uint32_t n = warp_distinct(slots, list, hash, has, rep, [&](uint32_t k, uint32_t id) {
            return *reinterpret_cast<volatile u64*>(key + id) == mine[k];
        });
#pragma unroll 1
        for (uint32_t base = 0; base < n; base += 64u) {
            const uint32_t q = base + lane;
            if (base + 32u < n) {  // two points per lane; the second may repeat the first
                const bool two = q + 32u < n;
                const uint32_t id = list[q], id2 = two ? list[q + 32u] : id;
                const u64 v = key[id], v2 = key[id2];
                const float2 f = fbm2_pair(make_float2(__uint_as_float((uint32_t)v), __uint_as_float((uint32_t)(v >> 32))),
                                           make_float2(__uint_as_float((uint32_t)v2), __uint_as_float((uint32_t)(v2 >> 32))),
                                           fp.dfreq, fp.doct, fp.dseed);
                // only this lane reads the keys of its listed points from here on
                pts[2u * id] = __float_as_uint(f.x);
                if (two) pts[2u * id2] = __float_as_uint(f.y);
            } else if (q < n) {
                const uint32_t id = list[q];
                const u64 v = key[id];
                pts[2u * id] = __float_as_uint(fbm2(__uint_as_float((uint32_t)v), __uint_as_float((uint32_t)(v >> 32)),
                                                    fp.dfreq, fp.doct, fp.dseed));
            }
        }
        __syncwarp();
#pragma unroll
        for (uint32_t k = 0; k < 4; ++k)
            r[3 * k + 2] = __fadd_rn(r[3 * k + 2], __fmul_rn(fp.damp, __uint_as_float(pts[2u * rep[k]])));
    } else {
        u64* key0 = reinterpret_cast<u64*>(pts);
        u64* key1 = key0 + 128;
        uint32_t* root = pts + 512;
        u64 m0[4] = {0, 0, 0, 0}, m1[4] = {0, 0, 0, 0};
        if (ok) {
            const bool odd = (j & 1ull) != 0ull;
            u64 a[6];
            decode_cols(j, d, tab, a);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                u64 w[3];
                if (k < 3)
                    weight_row<u64>(a, k, d, w);
                else
                    parent_row<u64>(a, odd, d, w);
                m0[k] = w[0] << (62 - d);
                m1[k] = w[1] << (62 - d);
            }
        }
#pragma unroll
        for (uint32_t k = 0; k < 4; ++k) {
            const u64 x = m0[k] * 0x9E3779B97F4A7C15ull + m1[k] * 0xC2B2AE3D27D4EB4Full;
            hash[k] = (uint32_t)(x >> 52) ^ (h * 0x85EBCA77u >> 22);
            key0[32u * k + lane] = m0[k];
            key1[32u * k + lane] = m1[k];
            root[32u * k + lane] = h;
        }
        const uint32_t n = warp_distinct(slots, list, hash, has, rep, [&](uint32_t k, uint32_t id) {
            return *reinterpret_cast<volatile u64*>(key0 + id) == m0[k] &&
                   *reinterpret_cast<volatile u64*>(key1 + id) == m1[k] &&
                   *reinterpret_cast<volatile uint32_t*>(root + id) == h;
        });
#pragma unroll 1
        for (uint32_t q = lane; q < n; q += 32u) {
            const uint32_t id = list[q];
            const u64 k0 = key0[id], k1 = key1[id];
            // the weights over 2^62 round to FP64 as those over 2^d do
            const double w[3] = {__dmul_rn(__ull2double_rn(k0), 0x1p-62), __dmul_rn(__ull2double_rn(k1), 0x1p-62),
                                 __dmul_rn(__ull2double_rn((1ull << 62) - k0 - k1), 0x1p-62)};
            double pf[4];
            float v[3];
            sphere_point(w, fp, static_cast<const double*>(I.rel) + 9u * root[id], pf);
            sphere_rel(pf[0], pf[1], pf[2], pf[3], fp, v);
            key0[id] = (u64)__float_as_uint(v[0]) | ((u64)__float_as_uint(v[1]) << 32);
            root[id] = __float_as_uint(v[2]);
        }
        __syncwarp();
#pragma unroll
        for (uint32_t k = 0; k < 4; ++k) {
            const u64 v = key0[rep[k]];
            r[3 * k] = __uint_as_float((uint32_t)v);
            r[3 * k + 1] = __uint_as_float((uint32_t)(v >> 32));
            r[3 * k + 2] = __uint_as_float(root[rep[k]]);
        }
    }
    __syncwarp();  // the next round reuses the table and the points
    split = merge = false;
    if (!ok) return;
    if (keep)
#pragma unroll
        for (int k = 0; k < 9; ++k) keep[k] = r[k];
    wishes_from(r, (j & 1ull) != 0ull, d, I.max_depth, fp,
                [&](float r2[3]) {
#pragma unroll
                    for (int k = 0; k < 3; ++k) r2[k] = r[6 + k];
                },
                [&](float nv[3]) {
#pragma unroll
                    for (int k = 0; k < 3; ++k) nv[k] = r[9 + k];
                },
                split, merge);
}

// classify_item for a round of a warp (lanes with `in`), by shared points.
template <int F>
__device__ __forceinline__ uint32_t classify_shared(const Inst& I, const FrameP& fp, bool in, uint32_t i, uint32_t s,
                                                    uint64_t j, const uint32_t* tab, uint32_t* s_cnt, uint8_t* slots,
                                                    uint32_t* pts, bool cache) {
    const int d = depth_of(j, I.ch);
    const uint32_t h = (uint32_t)((j >> (d & 63)) - (1ull << I.ch));
    const bool ok = in && d >= 0 && h < I.H;
    bool split, merge;
    lod_wishes_shared<F>(I, fp, ok, j, d, h, tab, slots, pts, split, merge, cache ? I.vc + 9ull * s : nullptr);
    if (!in) return 0u;
    if (!ok) {
        set_err(I.g, kErrLink);
        *cmd_ptr(I, s) = 0u;
        I.scan[i] = 0u;
        return 0u;
    }
    return store_command(I, fp, i, s, j, split, merge, cache, s_cnt);
}

// P1 (single instance): the live list strided over the whole grid, the slot
// and heap ID of the next rounds loaded while the current item is classified.
// Walk entries (live index | split flag << 31, slot, heap ID) are listed per
// warp and flushed to the frame's walk list; split wishes are counted per
// scan tile (warp-aggregated, consecutive live indices share a tile).
// A warp's walk buffer (kWarpWalks entries of the block's shared list) out
// to the frame's walk list: one atomic for the range, then a coalesced copy.
// With shared points, whose hash tables take the other half of the list.
template <int F>
constexpr uint32_t kWarpWalks = kWalkCap1 / (kFThreads / 32) / (kSharedPoints<F> ? 2u : 1u);
__device__ __forceinline__ void warp_walks_out(const Inst& I, const uint4* s_wl, uint32_t n) {
    if (n == 0u) return;  // warp-uniform
    uint32_t base = 0;
    if ((threadIdx.x & 31u) == 0u) base = atomicAdd(&I.g->nwalk, n);
    base = __shfl_sync(0xFFFFFFFFu, base, 0);
    uint4* wl = walk_list_of(I);
    for (uint32_t q = threadIdx.x & 31u; q < n; q += 32u) wl[base + q] = s_wl[q];
    __syncwarp();
}

template <int F>
__device__ void phase_classify1(const BatchDev& bt, FCtx& c, uint32_t* s_tab, uint32_t* s_cnt, uint4* s_list,
                                uint32_t* s_pts, unsigned long long gen) {
    stats_reset(s_cnt);
    ctx_tile(bt, bt.tile_base, 0, 1, c);
    const Inst& I = bt.inst0;
    const FrameP& fp = bt.fp0;
    const uint32_t N = c.N;
    const uint32_t S = kFThreads * scan_ipt1(N);
    unsigned long long* wc = wish_counts(bt);
    const uint64_t key = splitmix64(((uint64_t)fp.seed << 32) | (uint64_t)fp.frame);
    const bool cache = vc_form<F>(fp) && fp.vout;
    // points evaluated once per warp, unless the slots' point cache holds them
    const bool shared = kSharedPoints<F> && fp.mode == 0u && !(F == kFormSphere && I.pc);
    uint8_t* slots = reinterpret_cast<uint8_t*>(reinterpret_cast<uint32_t*>(s_list) + kFBuf / 2u) + kPtSlots * (threadIdx.x >> 5);
    uint32_t* pts = s_pts + kPtWords<F> * (threadIdx.x >> 5);
    const uint32_t lane = threadIdx.x & 31u;
    uint4* s_wl = s_list + kWarpWalks<F> * (threadIdx.x >> 5);  // the warp's walk buffer
    uint32_t nwl = 0;                                           // its entries (warp-uniform)
    // 32-item chunks, warp-major (chunk c to warp c mod (warps of the grid),
    // warps numbered across the blocks first), so that the costly parts of
    // the list (in slot order, i.e. clustered in space) spread over the SMs;
    // the warps run independently (no block barrier in the loop)
    const uint32_t stride = gridDim.x * kFThreads;
    uint32_t i = ((threadIdx.x >> 5) * gridDim.x + blockIdx.x) * 32u + lane;
    uint32_t sa = i < N ? I.live[i] : 0u;
    uint64_t ja = i < N ? I.heap[sa] : 0ull;
    uint32_t sb = i + stride < N ? I.live[i + stride] : 0u;
    for (; i - lane < N; i += stride) {  // warp-uniform
        const uint32_t sc = i + 2u * stride < N ? I.live[i + 2u * stride] : 0u;
        const uint64_t jb = i + stride < N ? I.heap[sb] : 0ull;
        bool split = false, walk = false, interior = false;
        uint32_t cmd = 0u;
        if (kSharedPoints<F> && shared)
            cmd = classify_shared<F>(I, fp, i < N, i, sa, ja, s_tab, s_cnt, slots, pts, cache);
        else if (i < N)
            cmd = classify_item<F>(I, fp, key, i, sa, ja, s_tab, s_cnt, cache, gen);
        if (i < N) {
            split = (cmd & kSplitWish) != 0u;
            walk = split || ((cmd & kMergeWish) && !(cmd & kHeapOdd));
            interior = split && has_twin_bound(I, ja);
        }
        const unsigned wm = __ballot_sync(0xFFFFFFFFu, walk), sm = __ballot_sync(0xFFFFFFFFu, split);
        if (walk)
            s_wl[nwl + __popc(wm & ((1u << lane) - 1u))] =
                make_uint4(i | (split ? kWalkSplit : 0u) | (interior ? kWalkInterior : 0u), sa, (uint32_t)ja,
                           (uint32_t)(ja >> 32));
        nwl += __popc(wm);
        if (sm) {  // the split wishes' lower-bound costs per scan tile (S is a multiple of 32: one tile per round)
            const uint32_t lb = 2u * (__popc(sm) + __popc(__ballot_sync(0xFFFFFFFFu, interior)));
            if (lane == 0u) atomicAdd(&wc[(i - lane) / S], (unsigned long long)lb);
        }
        sa = sb;
        ja = jb;
        sb = sc;
        __syncwarp();
        if (nwl > kWarpWalks<F> - 32u) {  // warp-uniform: room for the next round
            warp_walks_out(I, s_wl, nwl);
            nwl = 0;
        }
    }
    __syncwarp();
    warp_walks_out(I, s_wl, nwl);
    __syncthreads();  // the split wishes counted in s_cnt[0] go out with the walks' counts
}

// P2 (single instance): the frame's walk list over the whole grid. s_wpre
// (shared) gets the split wishes' lower-bound costs before each scan tile
// (4 with a Twin, else 2). A block first takes
// its share of the entries and settles the splits past the bound below; the
// walks left are queued and spread evenly over the block's threads. Per
// entry:
//   - a split wish: unless those costs plus its own bound exceed F, its
//     chain is walked on the frame-start links, checked, its first members
//     recorded in grp[i] and marked in the chain-mark words; its scan word
//     the chain's allocation count (or 3d + 4 under the paper's gate, set by
//     classify); past that bound the gate denies it whatever its cost, and
//     its bound stands in;
//   - a merge wish with an even heap ID: its Alg. 4 group, walked while the
//     wish can be its smallest member and every member wishes to merge (a
//     merge candidate); then it records the members and kGrpMin, and the
//     merge cost (parents, or 2 under the paper's gate) in the top byte of
//     its scan word. A group that is no candidate can never merge.
// The costs go to their scan tile's (merge, split) sums in status[t] and to
// the frame's totals.
__device__ void phase_walks1(const BatchDev& bt, FCtx& c, uint32_t* s_cnt, uint32_t* s_buf, Pair* s_warp,
                             uint32_t* s_tmp, uint32_t* s_n1) {
    if (threadIdx.x == 0) {
        s_cnt[3] = s_cnt[0];
        s_cnt[0] = 0;
    }
    ctx_tile(bt, bt.tile_base, 0, 1, c);
    const Inst& I = bt.inst0;
    if (blockIdx.x == 0 && threadIdx.x == 0) pc_generation(I.g, bt.fp0);
    const FrameP& fp = bt.fp0;
    const uint32_t T = bt.bg->total_stiles, S = kFThreads * bt.bg->scan_ipt;
    if (threadIdx.x == 0) s_tmp[0] = s_tmp[1] = s_tmp[2] = 0;
    if (T > kMaxTiles1) {  // the host keeps pools within the tables
        if (blockIdx.x == 0 && threadIdx.x == 0) set_err(I.g, kErrOverflow);
        __syncthreads();
        return;
    }
    uint32_t* s_wpre = s_buf;
    const unsigned long long* wc = wish_counts(bt);
    const uint32_t n = __ldcg(&I.g->nwalk), F = c.F;
    const uint4* wl = walk_list_of(I);
    // a warp takes 32 consecutive entries per round (neighbouring entries
    // walk neighbouring records, which its L1 then holds), warp-major over
    // the grid so that every SM gets its share of a short list; a thread
    // loads the entries of four rounds together, the first four before the
    // table of split wishes below is built
    const uint32_t stride = gridDim.x * kFThreads;
    const uint32_t mine = ((threadIdx.x >> 5) * gridDim.x + blockIdx.x) * 32u + (threadIdx.x & 31u);
    uint32_t qq[4];
    uint4 e[4];
    auto fetch = [&](uint32_t c0) {
#pragma unroll
        for (uint32_t k = 0; k < 4; ++k) {
            const uint32_t q = c0 + k * stride + mine;
            qq[k] = q < n ? q : kNull;
            e[k] = qq[k] != kNull ? wl[qq[k]] : make_uint4(0u, 0u, 0u, 0u);
        }
    };
    fetch(0u);
    block_table(T, [&](uint32_t t) { return Pair{(uint32_t)__ldcg(wc + t), 0u}; },
                [&](uint32_t t, Pair ex) { s_wpre[t] = ex.a; }, s_warp);
    uint32_t* marks = chain_marks(I);
    uint32_t* s_q = s_buf + kMaxTiles1;  // list indices of the block's walks to do
    constexpr uint32_t kQCap = kFBuf - kMaxTiles1;
    // a split's cost and a group's merge cost, added to their scan tile's
    // sums (one atomic per tile present among the active lanes)
    auto account = [&](uint32_t t, uint32_t mc, uint32_t sc) {
        const unsigned act = __activemask();
        const unsigned m = __match_any_sync(act, t);
        const uint32_t smc = __reduce_add_sync(m, mc), ssc = __reduce_add_sync(m, sc);
        if (t != kNull && (threadIdx.x & 31u) == (uint32_t)(__ffs(m) - 1) && (smc | ssc))
            atomicAdd(&bt.status[min(t, T - 1u)], ((unsigned long long)smc << 32) | ssc);
        if (mc) atomicAdd(&s_tmp[0], mc);
        if (sc) atomicAdd(&s_tmp[1], sc);
        count_stat(s_cnt, 0, mc != 0u);
    };
    // the queued walks over the block's threads, each taking the next one
    // when its last is done (chain lengths differ; s_tmp[2] counts them out)
    auto walk_queue = [&](uint32_t cnt) {
        for (uint32_t k = atomicAdd(&s_tmp[2], 1u); k < cnt; k = atomicAdd(&s_tmp[2], 1u)) {
            const uint32_t q = s_q[k];
            const uint4 e = wl[q];
            const uint32_t i = e.x & kWalkIndex, s = e.y;
            const uint64_t j = (uint64_t)e.z | ((uint64_t)e.w << 32);
            uint32_t mc = 0, sc = 0;
            if (e.x & kWalkSplit) {
                const int d = depth_of(j, I.ch);
                uint4 rec;
                bool more;
                const uint32_t cost = chain_walk(I, s, d, true, &rec, true, marks, &more);
                I.grp[i] = rec;
                sc = fp.gate == 1 ? 3u * (uint32_t)d + 4u : cost;
                I.scan[i] = sc | (more ? kScanMore : 0u);
            } else {
                Group g;
                if (group_if_mergeable(I, s, j, g)) {
                    I.grp[i] = make_uint4(g.m[0], g.m[1], g.m[2], g.m[3]);
                    atomicOr(cmd_ptr(I, s), kGrpMin);
                    mc = fp.gate == 1 ? 2u : (uint32_t)g.np;
                    I.scan[i] = mc << 24;
                }
            }
            account(i / S, mc, sc);
        }
    };
    if (threadIdx.x == 0) *s_n1 = 0;
    __syncthreads();
    for (uint32_t c0 = 0; c0 + blockIdx.x * 32u < n; c0 += 4u * stride) {  // block-uniform
        if (c0) fetch(c0);
#pragma unroll
        for (uint32_t k = 0; k < 4; ++k) {
            if (qq[k] == kNull) continue;
            const uint32_t i = e[k].x & kWalkIndex;
            const uint32_t t = i / S;
            // a split is denied whatever its cost when the lower bounds of
            // the split wishes before its scan tile and of its own exceed F
            const bool skip =
                (e[k].x & kWalkSplit) && (unsigned long long)s_wpre[min(t, T - 1u)] +
                                                 ((e[k].x & kWalkInterior) ? 4ull : 2ull) > (unsigned long long)F;
            if (skip) {
                // its bound stands in for its cost: every split after it in
                // the gate's order is then denied on these costs as on the
                // true ones, and the requested total still exceeds F
                const uint64_t j = (uint64_t)e[k].z | ((uint64_t)e[k].w << 32);
                const uint32_t sc = fp.gate == 1 ? 3u * (uint32_t)depth_of(j, I.ch) + 4u
                                                 : ((e[k].x & kWalkInterior) ? 4u : 2u);
                if (fp.gate != 1) I.scan[i] = sc;
                account(t, 0u, sc);
            } else {
                s_q[atomicAdd(s_n1, 1u)] = qq[k];
            }
        }
        __syncthreads();
        const uint32_t cnt = *s_n1;
        __syncthreads();
        if (cnt > kQCap - 4u * kFThreads) {  // block-uniform
            walk_queue(cnt);
            __syncthreads();
            if (threadIdx.x == 0) *s_n1 = s_tmp[2] = 0;
            __syncthreads();
        }
    }
    walk_queue(*s_n1);
    __syncthreads();
    stats_flush(s_cnt, I.g, kStMergeCand, -1, -1, kStSplitWishes);
    if (threadIdx.x == 0) {
        if (s_tmp[0]) atomicAdd(&I.g->rq_merge, (unsigned long long)s_tmp[0]);
        if (s_tmp[1]) atomicAdd(&I.g->rq_split, (unsigned long long)s_tmp[1]);
    }
    __syncthreads();
}

// Fate of live index i that charges its group (kGrpMin) when every request
// is granted: the group's parent count (1 or 2) and bit 3 when every member
// wishes to merge and none is marked by a chain (marks in the command words
// or, with `marks`, in those words).
__device__ __forceinline__ uint32_t fate_group_granted(const Inst& I, uint32_t i, const uint32_t* marks) {
    const uint4 m = I.grp[i];
    const uint32_t ms[3] = {m.y, m.z, m.w};
    uint32_t c[3];
    bool bad = false;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const bool b = ms[q] != kNull && bad_slot(I, ms[q], kErrLink);
        bad = bad || b;
        c[q] = (ms[q] != kNull && !b) ? (*cmd_ptr(I, ms[q]) | marks[ms[q]]) : kMergeWish;
    }
    const bool all = !bad && (c[0] & c[1] & c[2] & kMergeWish);
    const bool ok = all && !((c[0] | c[1] | c[2]) & kSplitMask);
    return ok ? ((m.z == kNull ? 1u : 2u) | 8u) : 0u;
}

// The most this frame can allocate: the free slots, or the requests granted.
__device__ __forceinline__ uint32_t alloc_bound1(const BatchDev& bt, const FCtx& c, bool all_granted) {
    const Globals* g = bt.inst0.g;
    const uint64_t req = all_granted ? __ldcg(&g->rq_merge) + __ldcg(&g->rq_split)
                                     : (uint64_t)__ldcg(&g->Mg) + (uint64_t)__ldcg(&g->Stot);
    return (uint32_t)min((uint64_t)c.F, req);
}

// P4 (single instance): per scan tile the fate of every item (allocation
// count, bit 3 for a merging group), the tile-local exclusive prefix of
// (changed, allocations), the fill records in the tile's region of chgr
// (tile t at t S), destination words (t << kLocBits | offset) and merged
// marks; the tile's totals go to status[Titems + t] for the fill. When every
// request was granted, the chain marks are ORed into the command words (the
// fill reads them there). Then the free list. Group validations run from a
// list (dependent loads), their fates returned through shared memory.
__device__ void phase_alloc1(const BatchDev& bt, FCtx& c, bool all_granted, Carry carry, uint32_t tbits,
                             uint32_t* s_cnt, Pair* s_warp, uint32_t* s_w, uint32_t* s_n, uint32_t* s_buf) {
    const uint32_t T = bt.bg->total_stiles, ipt = bt.bg->scan_ipt;
    const uint32_t S = kFThreads * ipt;
    uint32_t* s_list = s_buf;          // local item indices to validate
    uint32_t* s_fate = s_buf + kFBuf / 2;  // their fates, by local item index
    __shared__ uint32_t s_first;
    if (T > kMaxTiles1 || S > kFBuf / 2) {  // the host keeps pools within the tables
        if (blockIdx.x == 0 && threadIdx.x == 0) set_err(bt.inst0.g, kErrOverflow);
        return;
    }
    if (all_granted && blockIdx.x == 0 && threadIdx.x == 0) {
        Globals* g = bt.inst0.g;
        g->stats[kStSplitGranted] = __ldcg(&g->stats[kStSplitWishes]);
        g->stats[kStMergeGranted] = __ldcg(&g->stats[kStMergeCand]);
    }
    for (uint32_t t = blockIdx.x; t < T; t += gridDim.x) {
        if (threadIdx.x == 0) *s_n = 0;
        stats_reset(s_cnt);
        ctx_tile(bt, bt.stile_base, t, T, c);
        const Inst& I = bt.inst0;
        const uint32_t N = c.N;
        const uint32_t* marks = chain_marks(I);
        const uint32_t ts = c.lt * S;  // the tile's first live index
        const uint32_t e0 = threadIdx.x * ipt, i0 = ts + e0;
        uint32_t sl[kMaxIpt], cm[kMaxIpt], f[kMaxIpt];
        {  // slots and command words loaded coalesced (item ts + k 256 + tid)
           // through shared memory, then taken ipt consecutive per thread
            uint32_t* s_sl = s_buf;
            uint32_t* s_cm = s_buf + kFBuf / 2;
            uint32_t a[kMaxIpt];
#pragma unroll
            for (uint32_t k = 0; k < kMaxIpt; ++k) {
                const uint32_t e = k * kFThreads + threadIdx.x;
                a[k] = (k < ipt && ts + e < N) ? I.live[ts + e] : kNull;
            }
#pragma unroll
            for (uint32_t k = 0; k < kMaxIpt; ++k) {
                if (k >= ipt) continue;
                uint32_t m = a[k] != kNull ? *cmd_ptr(I, a[k]) : 0u;
                if (all_granted && a[k] != kNull) {
                    const uint32_t mk = marks[a[k]];
                    if (mk) {
                        m |= mk;
                        atomicOr(cmd_ptr(I, a[k]), mk);
                    }
                }
                s_sl[k * kFThreads + threadIdx.x] = a[k];
                s_cm[k * kFThreads + threadIdx.x] = m;
            }
            __syncthreads();
#pragma unroll
            for (uint32_t k = 0; k < kMaxIpt; ++k) {
                sl[k] = k < ipt ? s_sl[e0 + k] : kNull;
                cm[k] = k < ipt ? s_cm[e0 + k] : 0u;
            }
            if (threadIdx.x == 0) s_first = s_sl[0];  // the tile's first slot
            __syncthreads();  // s_buf is the lists' below
        }
        // groups to validate: when every request is granted, every recorded
        // group without split bits at its charged member; else the granted
        // candidates without split bits
        bool lst[kMaxIpt];
#pragma unroll
        for (uint32_t k = 0; k < kMaxIpt; ++k) {
            f[k] = leaves_of(cm[k] & kSplitMask);
            lst[k] = sl[k] != kNull && !(cm[k] & kSplitMask) &&
                     (all_granted ? (cm[k] & kGrpMin) != 0u : ((cm[k] & kCand) && (cm[k] & kMergeGrant)));
            if (lst[k]) s_list[atomicAdd(s_n, 1u)] = e0 + k;
        }
        __syncthreads();
        const uint32_t n = *s_n;
        for (uint32_t q = threadIdx.x; q < n; q += kFThreads) {
            const uint32_t e = s_list[q];
            const uint32_t i = c.lt * S + e;
            s_fate[e] = all_granted ? fate_group_granted(I, i, marks) : alloc_fate(I, i, kCand | kMergeGrant);
        }
        __syncthreads();
#pragma unroll
        for (uint32_t k = 0; k < kMaxIpt; ++k)
            if (lst[k]) f[k] = s_fate[e0 + k];
        Pair loc{0, 0};
#pragma unroll
        for (uint32_t k = 0; k < kMaxIpt; ++k) {
            const uint32_t na = f[k] & 7u;
            loc = padd(loc, Pair{na ? 1u : 0u, na});
        }
        Pair tot;
        const Pair ex = block_scan(loc, tot, s_warp);
        if (threadIdx.x == 0) bt.status[bt.Titems + t] = pack_pair(tot);
        // the bits this tile's changed items clear, per word tile: a block
        // histogram over the word tiles from the one holding the tile's first
        // slot (slots ascend with the live index); others go straight out
        uint32_t* s_hist = s_buf + kFBuf / 2;
        uint32_t* s_ml = s_buf;  // the tile's merges: local index << 13 | allocation offset
        const uint32_t hbase = (I.cap + s_first) >> tbits, nt = I.cap >> tbits;
        unsigned long long* tc = tile_counts(bt);
        s_hist[threadIdx.x] = 0u;
        if (threadIdx.x == 0) *s_n = 0;
        __syncthreads();
        uint32_t* const clr = I.clr;
        auto cleared = [&](uint32_t slot) {
            if (slot >= I.cap) return;  // never: the callers have checked it
            atomicOr(clr + (slot >> 5), 1u << (slot & 31u));
            const uint32_t node = (I.cap + slot) >> tbits;
            if (node - hbase < (uint32_t)kFThreads)
                atomicAdd(&s_hist[node - hbase], 1u);
            else if (node - nt < nt)
                atomicAdd(&tc[node - nt], 1ull);
        };
        uint32_t crun = ex.a, arun = ex.b;
#pragma unroll
        for (uint32_t k = 0; k < kMaxIpt; ++k) {
            const uint32_t na = f[k] & 7u;
            if (!na) continue;
            const uint32_t dw = (t << kLocBits) | arun;
            I.chgr[t * S + crun] = make_uint4(i0 + k, sl[k], cm[k], dw);
            // alloc_apply, with the clears counted; a merge is listed and
            // applied below, one per thread
            if (!(f[k] & 8u)) {
                *dest_ptr(I, sl[k]) = dw;
                count_stat(s_cnt, 0, true);
                cleared(sl[k]);
            } else {
                s_ml[atomicAdd(s_n, 1u)] = ((e0 + k) << kLocBits) | arun;
            }
            ++crun;
            arun += na;
        }
        __syncthreads();
        const uint32_t nm = *s_n;
        for (uint32_t q = threadIdx.x; q < nm; q += kFThreads) {
            const uint32_t e = s_ml[q] >> kLocBits, dw = (t << kLocBits) | (s_ml[q] & kLocMask);
            const uint4 m = I.grp[ts + e];
            const uint32_t ms[4] = {m.x, m.y, m.z, m.w};
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                if (ms[r] == kNull || bad_slot(I, ms[r], kErrLink)) continue;
                atomicOr(cmd_ptr(I, ms[r]), kMerged);
                *dest_ptr(I, ms[r]) = dw + (r < 2 ? 0u : 1u);
                cleared(ms[r]);
            }
            atomicAdd(&s_cnt[2], m.z == kNull ? 2u : 4u);
            count_stat(s_cnt, 1, true);
        }
        __syncthreads();
        if (s_hist[threadIdx.x] && hbase + threadIdx.x - nt < nt)
            atomicAdd(&tc[hbase + threadIdx.x - nt], (unsigned long long)s_hist[threadIdx.x]);
        stats_flush(s_cnt, I.g, kStSplitBis, kStMergeGroups, kStMergedBis);
        __syncthreads();
    }
    // the last frame's final phase listed every zero bit of this frame's
    // starting bitfield, unless another form of the frame ran since
    if (!carry.ok()) free_list(bt, c, s_w, all_granted, tile_counts(bt), free_list1(bt, carry, 0u));
}

// P5 (single instance) has two parts that share nothing they write, each on
// half of the blocks, so that the one's dependent loads overlap the other's
// (one after the other, with a barrier between, they took 15.4 and 9.9 us of
// the 124 us grid frame; together 18.8 us).
//
// The fill: every block scans the tiles' (changed, allocation) totals into
// shared memory; the changed records of the frame, one range strided evenly
// over the part's blocks, are then filled with their destinations resolved
// through the allocation offsets: FillNewBlocks + UpdateNeighbors. (`fb` of
// `nfb`: the block's place in the part.)
__device__ void phase_fill1(const BatchDev& bt, FCtx& c, bool all_granted, Carry carry, uint32_t fb, uint32_t nfb, uint32_t* s_cnt,
                            uint32_t* s_buf, Pair* s_warp) {
    stats_reset(s_cnt);
    ctx_tile(bt, bt.tile_base, 0, 1, c);
    const Inst& I = bt.inst0;
    const uint32_t T = bt.bg->total_stiles, S = kFThreads * bt.bg->scan_ipt;
    uint32_t* s_cpre = s_buf;
    uint32_t* s_apre = s_buf + kMaxTiles1;
    if (T > kMaxTiles1) {  // alloc has set the error word
        __syncthreads();
        return;
    }
    const Pair all = block_table(
        T, [&](uint32_t t) { return unpack_pair(__ldcg(bt.status + bt.Titems + t)); },
        [&](uint32_t t, Pair ex) {
            s_cpre[t] = ex.a;
            s_apre[t] = ex.b;
        },
        s_warp);
    const uint32_t C = all.a;
    const uint32_t bound = alloc_bound1(bt, c, all_granted);
    if (fb == 0 && threadIdx.x == 0) {
        I.g->A = all.b;
        I.g->C = C;
        I.g->stats[kStAllocated] = all.b;
        if (all.b > bound) set_err(I.g, kErrOverflow);
    }
    const DestTiles dm{s_apre, free_list1(bt, carry, 0u), min(all.b, bound)};
    uint32_t relinked = 0;
    // 32 records per warp, warp-major over the blocks: with fewer records than
    // threads, every SM still gets its share
    for (uint32_t q = ((threadIdx.x >> 5) * nfb + fb) * 32u + (threadIdx.x & 31u); q < C; q += nfb * kFThreads) {
        uint32_t lo = 0, hi = T;  // the last tile whose first record is at or before q
        while (lo < hi) {
            const uint32_t mid = (lo + hi) >> 1;
            if (s_cpre[mid] <= q)
                lo = mid + 1u;
            else
                hi = mid;
        }
        const uint32_t t = lo - 1u;
        const uint4 r = I.chgr[t * S + (q - s_cpre[t])];
        relinked += fill_item_dm(I, r.x, r.y, r.z, dm(r.w), dm);
    }
    if (relinked) atomicAdd(&s_cnt[0], relinked);
    __syncthreads();
    stats_flush(s_cnt, I.g, kStRelinked);
    __syncthreads();
}

// The lowest k of the set bits of z.
__device__ __forceinline__ uint32_t lowest_set(uint32_t z, int k) {
    if (k <= 0) return 0u;
    if (k >= __popc(z)) return z;
    uint32_t t = z;
    for (; k > 0; --k) t &= t - 1u;
    return z ^ t;
}

// The final part: UpdateBitfield, SumReduction and CachePointers, from what
// the allocation left: the frame-start bitfield, the bits cleared (clr) and
// the count A of new records, which take the first A zero bits (Alg. 8).
// Every block of it computes each word tile's new count and scans them into
// shared memory: the new live count and each tile's first row. The first
// block writes the sum tree's nodes above the tiles as differences of that
// scan; a warp per word tile rewrites the tile's words, the nodes from the
// tile down (the count checked against the scan), and the tile's rows of the
// new live list and, from the zero bits, of the next frame's free list.
__device__ void phase_final1(const BatchDev& bt, FCtx& c, bool all_granted, uint32_t rb, uint32_t nrb, uint32_t* s_buf,
                             Pair* s_warp, uint32_t* s_red, uint32_t tbits, Carry carry) {
    ctx_tile(bt, bt.tile_base, 0, 1, c);
    const Inst& I = bt.inst0;
    const uint32_t W = I.W, TW = min(W, bt.tw), nt = I.cap >> tbits;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    uint32_t* s_tpre = s_buf;               // ones before each tile in the new bitfield
    uint32_t* s_old = s_buf + kMaxTiles1;   // and in the frame-start one
    if (nt > kMaxTiles1 || TW > 64u) {  // the host keeps pools within the tables
        if (rb == 0 && threadIdx.x == 0) set_err(I.g, kErrOverflow);
        return;
    }
    const uint32_t T = min(bt.bg->total_stiles, kMaxTiles1);
    Pair sum{0, 0}, none{0, 0};
    for (uint32_t t = threadIdx.x; t < T; t += kFThreads)
        sum.b += unpack_pair(__ldcg(bt.status + bt.Titems + t)).b;
    block_sum2(sum, none, s_red);
    const uint32_t A = min(sum.b, alloc_bound1(bt, c, all_granted)), TS = 1u << tbits;
    // the ones before each tile at frame start: kept by the last frame's
    // final part when that was this kernel, else scanned here from the tile
    // counts; then the new counts from them, scanned, and kept for the next
    // frame in the other buffer
    const unsigned long long* tc = tile_counts(bt);
    const uint32_t cur = carry.buffer();
    const uint32_t* tpre_in = bt.tpre + cur * bt.Twords;
    uint32_t* tpre_out = bt.tpre + (cur ^ 1u) * bt.Twords;
    if (carry.ok()) {
        for (uint32_t t = threadIdx.x; t < nt; t += kFThreads) s_old[t] = __ldcg(tpre_in + t);
        __syncthreads();
    } else {
        block_table(nt, [&](uint32_t t) { return Pair{(uint32_t)(__ldcg(tc + t) >> 32), 0u}; },
                    [&](uint32_t t, Pair ex) { s_old[t] = ex.a; }, s_warp);
    }
    const Pair tot = block_table(
        nt,
        [&](uint32_t t) {
            const unsigned long long w = __ldcg(tc + t);
            const uint32_t old = (uint32_t)(w >> 32), clr = (uint32_t)w;
            const long long zb = (long long)t * TS - s_old[t];  // zero bits before the tile at frame start
            const long long set = min(max((long long)A - zb, 0ll), (long long)(TS - old));
            return Pair{old - clr + (uint32_t)set, 0u};
        },
        [&](uint32_t t, Pair ex) { s_tpre[t] = ex.a; }, s_warp);
    for (uint32_t t = rb + threadIdx.x * nrb; t < nt; t += kFThreads * nrb) tpre_out[t] = s_tpre[t];
    for (uint32_t t = rb * kFThreads + threadIdx.x; t < bt.Titems; t += kFThreads * nrb) wish_counts(bt)[t] = 0ull;
    const uint32_t Nn = tot.a;
    if (rb == 0) {
        // node m (1 <= m < nt) covers tile nodes [m 2^k, (m + 1) 2^k) at 2^k
        // tiles per node of its level
        const int lnt = 31 - __clz((int)nt);
        for (uint32_t m = 1u + threadIdx.x; m < nt; m += kFThreads) {
            const int k = lnt - (31 - __clz((int)m));
            const uint32_t a = (m << k) - nt, b = ((m + 1u) << k) - nt;
            I.sums[m] = (b < nt ? s_tpre[b] : Nn) - s_tpre[a];
        }
        if (threadIdx.x == 0) {
            I.g->stats[kStLiveAfter] = Nn;
            if (nt == 1u) I.sums[1] = Nn;
            I.g->marks_clean = 1u;  // read by the next frame
            I.g->nwalk = 0u;
            I.g->freel_full = 1u | ((cur ^ 1u) << 1);
        }
    }
    // the instance's fields in registers
    uint32_t* const marks = chain_marks(I);
    uint32_t* const live = I.live;
    uint32_t* const freel = free_list1(bt, carry, 1u);
    uint32_t* const sums = I.sums;
    uint32_t* const bits = I.bits;
    uint32_t* const clr = I.clr;
    const uint32_t cap = I.cap;
    const uint32_t vmask = cap < 32u ? (1u << cap) - 1u : 0xFFFFFFFFu;  // the slots of a word
    const uint32_t nwarps = nrb * (kFThreads / 32u);
    const uint32_t lt_mask = (1u << lane) - 1u;
    // a word tile (TW <= 64 words) per warp: lane holds words lane and 32 + lane
    for (uint32_t wt = warp * nrb + rb; wt < nt; wt += nwarps) {
        const uint32_t w0 = wt * TW + lane, w1 = w0 + 32u;
        const bool h0 = lane < TW, h1 = 32u + lane < TW;
        uint32_t x0 = h0 ? __ldcg(bits + w0) : 0u, x1 = h1 ? __ldcg(bits + w1) : 0u;
        const uint32_t c0 = h0 ? __ldcg(clr + w0) : 0u, c1 = h1 ? __ldcg(clr + w1) : 0u;
        const uint32_t r0 = s_tpre[wt];
        {  // the tile's share of the first A zero bits, by the zeros before each word
            const uint32_t z0 = h0 ? ~x0 & vmask : 0u, z1 = h1 ? ~x1 & vmask : 0u;
            uint32_t e0 = __popc(z0), e1 = __popc(z1);
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y0 = __shfl_up_sync(0xFFFFFFFFu, e0, o), y1 = __shfl_up_sync(0xFFFFFFFFu, e1, o);
                if ((int)lane >= o) {
                    e0 += y0;
                    e1 += y1;
                }
            }
            e1 += __shfl_sync(0xFFFFFFFFu, e0, 31);
            const int left = (int)min((long long)A - ((long long)wt * TS - s_old[wt]), 4096ll);  // A less the zeros before the tile
            x0 = (x0 & ~c0) | lowest_set(z0, left - (int)(e0 - __popc(z0)));
            x1 = (x1 & ~c1) | lowest_set(z1, left - (int)(e1 - __popc(z1)));
        }
        if (h0) bits[w0] = x0;
        if (h1) bits[w1] = x1;
        if (c0) clr[w0] = 0u;
        if (c1) clr[w1] = 0u;
        uint32_t v0 = __popc(x0), v1 = __popc(x1);
        if (TW > 1u) {
            if (h0) sums[W + w0] = v0;
            if (h1) sums[W + w1] = v1;
        }
#pragma unroll
        for (uint32_t L = 1; L <= 5; ++L) {
            v0 += __shfl_down_sync(0xFFFFFFFFu, v0, 1u << (L - 1u));
            v1 += __shfl_down_sync(0xFFFFFFFFu, v1, 1u << (L - 1u));
            if ((1u << L) < TW && (lane & ((1u << L) - 1u)) == 0u) {
                if (h0) sums[(W + w0) >> L] = v0;
                if (h1) sums[(W + w1) >> L] = v1;
            }
        }
        const uint32_t half0 = __shfl_sync(0xFFFFFFFFu, v0, 0), half1 = __shfl_sync(0xFFFFFFFFu, v1, 0);
        const uint32_t node = (wt + 1u < nt ? s_tpre[wt + 1u] : Nn) - r0;
        if (lane == 0) {
            if (half0 + half1 != node) set_err(I.g, kErrLink);
            if (nt > 1u) sums[nt + wt] = node;  // (a single tile's node is the root, written above)
        }
        // the tile's rows of the live list (Alg. 7 for every index) and, from
        // its zero bits, of the next frame's free list (Alg. 8 for every rank;
        // every earlier tile holds 2^tbits slots): word by word, lane b tests
        // bit b and the set ones take consecutive rows, so every store is one
        // contiguous run
        uint32_t row = r0, zrow = wt * TS - r0;
#pragma unroll 4
        for (uint32_t i = 0; i < TW; ++i) {
            const uint32_t x = __shfl_sync(0xFFFFFFFFu, i < 32u ? x0 : x1, i & 31u);
            const uint32_t z = ~x & vmask;
            const uint32_t sl = (wt * TW + i) * 32u + lane;
            const uint32_t r = row + __popc(x & lt_mask), zr = zrow + __popc(z & lt_mask);
            if (((x >> lane) & 1u) && r < cap) {
                live[r] = sl;
                marks[sl] = 0u;  // for the next frame's chain marks
            } else if (((z >> lane) & 1u) && zr < cap) {
                freel[zr] = sl;
            }
            row += __popc(x);
            zrow += __popc(z);
        }
    }
}

template <int F>
__global__ void __launch_bounds__(kFThreads, CBT_FRAME_MIN_BLOCKS) k_frame1(BatchDev bt, uint32_t tbits) {
    __shared__ FCtx s_c;
    __shared__ __align__(16) uint32_t s_tab[kDecTabWords];
    __shared__ __align__(16) uint32_t s_buf[kFBuf];
    __shared__ Pair s_warp[kFThreads / 32 + 1];
    __shared__ uint32_t s_red[4 * (kFThreads / 32)];
    __shared__ uint32_t s_cnt[kBlockStats];
    __shared__ uint32_t s_w[kFThreads / 32 + 1];
    __shared__ uint32_t s_tmp[4];
    __shared__ uint32_t s_n;
    __shared__ __align__(16) uint32_t s_pts[kSharedPoints<F> ? kPtWords<F> * (kFThreads / 32) : 4u];
    const uint32_t epoch = ld_volatile(&bt.bg->bar_epoch);
    uint32_t nbar = 0;
    auto sync = [&]() {
        ++nbar;
        grid_sync(bt.bg, epoch, nbar);
    };
    stamp(bt, 0);
    // read before any block can reach the phases that set them
    const Carry carry{__ldcg(&bt.inst0.g->freel_full)};
    const uint32_t N = __ldcg(bt.inst0.sums + 1);
    const unsigned long long gen = F == kFormSphere ? pc_generation_of(bt.inst0.g, bt.fp0) : 0ull;
    // the decode tables are fetched now and stored after prep's own loads
    // have gone out
    static_assert(kFThreads == 256, "dec_fetch splits the table over 256 threads");
    uint4 tab[kDecVecs];
    dec_fetch(tab);
    // the block's context is instance 0 throughout
    for (uint32_t k = threadIdx.x; k < sizeof(Inst) / 4u; k += kFThreads)
        reinterpret_cast<uint32_t*>(&s_c.I)[k] = reinterpret_cast<const uint32_t*>(&bt.inst0)[k];
    for (uint32_t k = threadIdx.x; k < sizeof(FrameP) / 4u; k += kFThreads)
        reinterpret_cast<uint32_t*>(&s_c.fp)[k] = reinterpret_cast<const uint32_t*>(&bt.fp0)[k];
    if (threadIdx.x == 0) {
        s_c.b = 0;
        s_c.N = N;
        s_c.F = bt.inst0.cap - N;
    }
    // After a frame of this kernel classify needs only the roots from other
    // blocks; of a small mesh every block writes the whole table (the same
    // values) and reads its own, and the phase ends without a grid barrier:
    // prep and classify of a cube 8.6 -> 5.7 us, of the dodecahedron planet 22.5 -> 19.9.
    if (carry.ok() && bt.inst0.H <= kLocalRoots) {
        const Inst& I = bt.inst0;
        const FrameP& fp = bt.fp0;
        constexpr uint32_t kPer = (9u * kLocalRoots + kFThreads - 1u) / kFThreads;
        double v[kPer];
#pragma unroll
        for (uint32_t k = 0; k < kPer; ++k) {  // all loads out before the first store
            const uint32_t e = threadIdx.x + k * kFThreads;
            v[k] = e < 9u * I.H ? I.root64[e] : 0.0;
        }
#pragma unroll
        for (uint32_t k = 0; k < kPer; ++k) {
            const uint32_t e = threadIdx.x + k * kFThreads;
            if (e < 9u * I.H) rel_put(v[k], I.rel, I.g, fp.eye, fp.precision, fp.shift, e);
        }
        frame_init1(bt, tbits, N);
        dec_store(s_tab, tab);
        __syncthreads();
    } else {
        phase_prep1(bt, tbits, N);
        dec_store(s_tab, tab);
        sync();
    }
    stamp(bt, 1);
    phase_classify1<F>(bt, s_c, s_tab, s_cnt, reinterpret_cast<uint4*>(s_buf), s_pts, gen);
    sync();
    stamp(bt, 2);
    phase_walks1(bt, s_c, s_cnt, s_buf, s_warp, s_tmp, &s_n);
    sync();
    stamp(bt, 3);
    const Globals* g = bt.inst0.g;
    const bool all_granted = __ldcg(&g->rq_merge) + __ldcg(&g->rq_split) <= (unsigned long long)s_c.F;
    if (!all_granted) {
        phase_gate<true>(bt, s_c, s_cnt, s_red, s_warp, s_tmp, &s_n, reinterpret_cast<uint2*>(s_buf), true);
        sync();
    }
    stamp(bt, 4);
    phase_alloc1(bt, s_c, all_granted, carry, tbits, s_cnt, s_warp, s_w, &s_n, s_buf);
    sync();
    stamp(bt, 5);
    const uint32_t half = gridDim.x / 2u, nfb = gridDim.x - half;  // half of the blocks for the final part
    if (blockIdx.x < nfb) phase_fill1(bt, s_c, all_granted, carry, blockIdx.x, nfb, s_cnt, s_buf, s_warp);
    if (half == 0u || blockIdx.x >= nfb)
        phase_final1(bt, s_c, all_granted, half ? blockIdx.x - nfb : 0u, half ? half : 1u, s_buf, s_warp, s_red, tbits,
                     carry);
    if (bt.fp0.vout) {
        sync();
        stamp(bt, 6);
        vertices_of<F>(bt.inst0, bt.fp0, s_tab, s_buf, &s_n);
    } else {
        stamp(bt, 6);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (bt.timing) atomicMax(&bt.bg->t[kFramePhases], global_ns());
        if (blockIdx.x == 0) {
            bt.bg->bar_epoch = epoch + nbar * gridDim.x;
            if (ld_volatile(&bt.bg->abort)) set_err(bt.inst0.g, kErrTimeout);
        }
    }
}

}  // namespace

template <typename... A>
cudaError_t launch_coop(void (*kernel)(A...), int grid, cudaStream_t s, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(grid));
    cfg.blockDim = dim3(kFThreads);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <int F>
cudaError_t launch_frame_form(const BatchDev& bt, int grid, cudaStream_t s) {
    if constexpr (F != kFormAny)
        if (bt.B == 1) return launch_coop<BatchDev>(k_frame<F, true>, grid, s, bt);
    return launch_coop<BatchDev>(k_frame<F, false>, grid, s, bt);
}
template <int F>
cudaError_t launch_frame1_form(const BatchDev& bt, int grid, uint32_t tbits, cudaStream_t s) {
    return launch_coop<BatchDev, uint32_t>(k_frame1<F>, grid, s, bt, tbits);
}
template <int F>
int frame_blocks_form() {
    int n = 0, m = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_frame<F, false>, kFThreads, 0) != cudaSuccess) return 0;
    if constexpr (F != kFormAny) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&m, k_frame<F, true>, kFThreads, 0) != cudaSuccess) return 0;
        return n < m ? n : m;
    }
    return n;
}
template <int F>
int frame1_blocks_form() {
    int n = 0;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_frame1<F>, kFThreads, 0) == cudaSuccess ? n : 0;
}

}  // namespace cbtgpu
