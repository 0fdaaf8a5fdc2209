// Device-side data layout and helpers of the CBT bisection update.
//
// Per instance (one halfedge mesh, one pool of 2^D slots) the workspace holds:
//   heap[cap]  u64   bisector heap ID j (Sec. 2.3; root of h = 2^ch + h)
//   nb[cap]    uint4 {Twin, Next, Prev, rev}: neighbour slots across the edges
//                    (v0,v1), (v1,v2), (v2,v0); rev holds, per link, which edge
//                    of the neighbour points back (2 bits each, 3 = none)
//   cd[cap]    uint2 {cmd, dest}: per-frame command word and the index into
//                    the free list of the bisector's first new record
//   bits[W]    u32   CBT bitfield, W = max(1, cap / 32) words
//   sums[2W]   u32   CBT sum tree above the words in heap order: sums[1] is the
//                    root, sums[W + w] = popc(bits[w]) (Sec. 3.1)
//   live[cap]  u32   slots of the live bisectors, ascending (Alg. 7 for all i)
//   freel[cap] u32   the first A zero bits of the frame-start bitfield (Alg. 8)
//   freel2[cap] u32  single-instance frame: the other free list (this frame's and
//                    the next one's change places every frame)
//   clr[W]     u32   single-instance frame: bits cleared this frame; 0 between frames
//   tpre[2 W/64] u32 single-instance frame: ones before each word tile, this
//                    frame's and the next one's
//   wish[cap/1024] u64 single-instance frame: lower-bound split costs per scan
//                    tile; 0 between frames
//   scan[cap]  u32   per live index: split cost, then its running total
//   grp[cap]   uint4 per live index: the members of the merge group whose
//                    smallest member it is, or of a split wish's chain
//   chg[cap]   u32   live indices of the frame's changed bisectors, ascending
//   chgr[cap]  uint4 the same as records {live index, slot, cmd, dest}
//   vc[cap]    9 x f32 in the sphere and displaced forms, the vertices the LOD test
//                    evaluated this frame (valid while the slot's cmd has
//                    kVcValid), copied by the vertex export
// and, when a point cache is attached (caller memory of its own):
//   pc[16][cap] f64  sphere form: per slot the frame-independent part of the
//                    LOD test's four vertices (its three and the parent's new
//                    one), {p_x, p_y, p_z, f} each (component-major: entry k
//                    of slot s at pc[k cap + s])
//   pct[cap]   u64x2 the tag of pc[.][s]: {heap ID, cache generation}
//   root64[H*9], rel[H*9]: root vertices (FP64) and their per-frame offsets
//                    from the camera (FP32, fixed point or FP64)
//   corner[H*3] u32  global points of the root corners (mesh vertex ids, and
//                    V + face id for the face centroid), for the indexed export
// and, per batch (a single instance carries a batch of one), the instance
// table, per-instance frame parameters, tile prefixes and the look-back
// tile descriptors of the two scans and the reduction.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace cbtgpu {

constexpr uint32_t kNull = 0xFFFFFFFFu;

// cmd word bits.
constexpr uint32_t kR = 1u, kN = 2u, kP = 4u;  // split bits (R5 reading)
constexpr uint32_t kSplitMask = 7u;
constexpr uint32_t kMerged = 1u << 3;
constexpr uint32_t kSplitWish = 1u << 4;
constexpr uint32_t kMergeWish = 1u << 5;
constexpr uint32_t kMergeGrant = 1u << 6;
constexpr uint32_t kDepthOdd = 1u << 7;
constexpr uint32_t kHeapOdd = 1u << 8;
constexpr uint32_t kCand = 1u << 9;    // smallest member of a mergeable group (members in grp[i])
constexpr uint32_t kGrpMin = 1u << 10; // smallest member of a merge group whose members are in grp[i]
constexpr uint32_t kVcValid = 1u << 11; // vc[slot] holds this frame's vertices (sphere or displaced form, one-launch frame)
// scan word of a live index: split cost in bits 0-23, merge cost in bits
// 24-30, and (single-instance frame) bit 31 when the split's chain has more
// members than its record keeps
constexpr uint32_t kScanMore = 1u << 31;
constexpr uint32_t kMergeCostMask = 0x7Fu;

// Edge indices of a bisector: Twin (v0,v1), Next (v1,v2), Prev (v2,v0).
constexpr int kT = 0, kNe = 1, kPe = 2;
// Portion of an old edge covered by a new edge: whole, the half at the
// edge's first vertex, the half at its second vertex (in the bisector's own
// vertex order: Twin v0->v1, Next v1->v2, Prev v2->v0).
constexpr int kWhole = 0, kFirst = 1, kSecond = 2;

// Device error bits (mirrors CBT_DERR_*).
constexpr uint32_t kErrChain = 1u, kErrLink = 2u, kErrTimeout = 4u, kErrRange = 8u,
                   kErrOverflow = 16u;

enum StatIdx {
    kStLiveBefore = 0, kStLiveAfter, kStFreeBefore, kStSplitWishes, kStMergeCand,
    kStSplitGranted, kStMergeGranted, kStSplitBis, kStMergedBis, kStMergeGroups,
    kStAllocated, kStRelinked, kStFrame, kStCount
};

// Per-instance counters (256 bytes at the start of the instance workspace).
struct Globals {
    uint32_t N;         // live bisectors at frame start (CBT root)
    uint32_t F;         // free slots at frame start
    uint32_t A;         // allocations of this frame
    uint32_t Mg;        // granted merge cost of this frame
    uint32_t err;       // sticky error bits
    uint32_t done;      // finished word tiles of the reduction
    uint32_t ntiles;    // item tiles of this frame: ceil(N / kTileItems)
    uint32_t C;         // changed bisectors of this frame (split, or smallest member of a merge)
    uint32_t nstiles;   // scan tiles of this frame: ceil(N / kScanItems)
    uint32_t Stot;      // total split cost requested this frame (one-launch frame)
    uint32_t stats[kStCount];
    uint32_t pc_pad;
    unsigned long long pc_gen;     // sphere-point cache generation (0: none made yet)
    unsigned long long pc_radius;  // the shape it was made with: radius (FP64 bits),
    uint32_t pc_damp, pc_dfreq, pc_doct, pc_dseed;  // displacement (FP32 bits)
    // single-instance frame: the frame's merge cost (groups whose members all
    // wish to merge) and requested split cost, summed by the walks; when their
    // sum fits the free slots every request is granted without the prefix gate
    unsigned long long rq_merge, rq_split;
    uint32_t nwalk;  // single-instance frame: entries of the frame's walk list (0 between its frames)
    uint32_t marks_clean;  // 1 when the chain-mark words (chg) of the live slots are 0 (the
                           // single-instance frame leaves them so; the other frames clear this)
    uint32_t freel_full;   // bit 0: a free list of every zero bit of the bitfield in slot order is kept, in
                           // freel or (bit 1) freel2, and the word tiles' prefix in the same one of its two
                           // buffers (the single-instance frame leaves it so; the other frames clear this)
    uint32_t pad[64 - 39];
};
static_assert(sizeof(Globals) == 256, "Globals must be 256 bytes");
static_assert(10 + kStCount + 1 == 24, "pc_gen must sit at byte 96");

// Per-instance device arrays and sizes.
struct Inst {
    uint64_t* heap;
    uint4* nb;
    uint2* cd;
    uint32_t* bits;
    uint32_t* sums;
    uint32_t* live;
    uint32_t* freel;
    uint32_t* scan;
    uint4* grp;  // per live index: members of the group whose smallest member it is
    uint32_t* chg;  // live indices of the changed bisectors, in ascending slot order
    uint4* chgr;    // one-launch frame: per changed bisector {live index, slot, cmd, dest}
    float* vc;      // per slot, the frame's FP32 vertices [3][3] (sphere form, one-launch frame)
    double* pc;     // optional point cache (sphere form): per slot {p, f} of the LOD test's four vertices, [16][cap]
    ulonglong2* pct;  // tag of pc[.][s]: {heap ID, generation}; both null without a cache
    double* root64;
    void* rel;
    Globals* g;
    uint32_t cap, W, D, H, ch, max_depth;
    uint32_t ntiles_items;  // ceil(cap / kTileItems)
    uint32_t pad_;
    uint32_t* freel2;       // single-instance frame: the other free list
    uint32_t* clr;          // single-instance frame: the frame's cleared bits, 0 between frames
    const uint32_t* rbnd;   // bit h: halfedge h has no Twin (mesh boundary), [ceil(H / 32)]
};

struct FrameP {
    double eye[3];
    float planes[15];
    float q;
    uint32_t nplanes, mode, seed, precision;
    int32_t shift;
    uint32_t gate;
    const uint64_t* split_list;
    uint32_t n_split;
    const uint64_t* merge_list;
    uint32_t n_merge;
    uint32_t frame;  // frame counter (RANDOM mode key)
    float* vout;     // optional vertex export, vcap rows of 9 floats
    uint32_t vcap;
    double radius;   // precision 3: radius of the sphere about the world origin
    float damp;      // displacement amplitude (0: none), precisions 0 and 3
    float dfreq;     // displacement base frequency (lattice cells per unit)
    uint32_t doct;   // displacement octaves (1..8)
    uint32_t dseed;  // displacement lattice seed
};

// The vertex form a kernel is compiled for: the precision of the frame's
// vertices and, in FP32, whether they are displaced (kFormAny: read from the
// frame's parameters, for a batch whose frames differ). One form per kernel
// keeps the others' code and registers out of it: the single-instance frame
// of the FP32 grid is 129 us a pass against 156 us with every form in one kernel.
enum Form : int { kFormAny = 0, kFormF32, kFormF32Disp, kFormFixed, kFormF64, kFormSphere, kForms };
__host__ __device__ inline Form form_of(const FrameP& fp) {
    return fp.precision == 0u ? (fp.damp != 0.0f ? kFormF32Disp : kFormF32)
                              : fp.precision == 1u ? kFormFixed : fp.precision == 2u ? kFormF64 : kFormSphere;
}
template <int F>
__device__ __forceinline__ uint32_t precision_in(const FrameP& fp) {
    return F == kFormAny ? fp.precision : F == kFormFixed ? 1u : F == kFormF64 ? 2u : F == kFormSphere ? 3u : 0u;
}
template <int F>
__device__ __forceinline__ bool displaced_in(const FrameP& fp) {
    return F == kFormF32Disp || ((F == kFormAny || F == kFormSphere) && fp.damp != 0.0f);
}

constexpr int kFramePhases = 9;  // phases of the one-launch frame (a batch skips the last)

// Launch-wide counters of one batch (256 bytes).
struct BatchGlobals {
    uint32_t tickets[8];
    uint32_t total_tiles;   // item tiles of this frame over all instances
    uint32_t total_ctiles;  // tiles of changed bisectors (kThreads each) over all instances
    uint32_t total_stiles;  // scan tiles (kScanItems each) over all instances
    uint32_t bar_count;     // grid barrier of the one-launch frame: arrivals (monotonic),
    uint32_t bar_epoch;     // and their count when the current launch started
    uint32_t abort;         // a bounded wait ran out: later waits return at once
    uint32_t scan_ipt;      // one-launch frame: items per thread of its scan tiles
    uint32_t live_total;    // live bisectors of the batch at frame start (saturating)
    unsigned long long t[16];  // phase boundaries (ns) of the one-launch frame
    uint32_t pad[64 - 16 - 32];
};
static_assert(sizeof(BatchGlobals) == 256, "BatchGlobals must be 256 bytes");

// A batch of independent instances updated by one launch per kernel. Item
// tiles of instance b are the global tiles [tile_base[b], tile_base[b+1])
// (recomputed on the device every frame from the live counts); word tiles
// and vertex tiles use static prefixes. A single instance is a batch of one.
struct BatchDev {
    const Inst* inst;     // [B]
    const FrameP* fps;    // [B] in device memory, or null: fp0 for every instance
    FrameP fp0;
    Inst inst0;           // B == 1: a copy of inst[0] (read from the launch's parameters)
    uint32_t B;
    uint32_t tw;          // word-tile size of the reduction and free-list kernels
    uint32_t* tile_base;  // [B+1]
    uint32_t* ctile_base; // [B+1] tiles of kThreads changed bisectors, per frame
    uint32_t* stile_base; // [B+1] scan tiles of kScanItems live bisectors, per frame
    const uint32_t* wtile_base;  // [B+1] word tiles, min(W_b, tw) words each
    const uint32_t* vtile_base;  // [B+1] ceil(cap_b / kTileItems)
    const uint32_t* rel_base;    // [B+1] 9 * H_b
    BatchGlobals* bg;
    unsigned long long* status;  // [2 * Titems + Twords] look-back descriptors
    uint32_t Titems, Twords, Trel;
    uint32_t* nout;              // optional [B]: live count at frame start per instance
    uint32_t* vcount;            // the export on its own (B == 1): the live count goes here, in mapped
                                 // host memory, and nothing else is written when it exceeds vcap
    uint32_t timing;             // one-launch frame: record phase boundaries
    // B == 1, what the instance's freel_full vouches for: in the instance's workspace, not in the batch's,
    // since cbt_update and a batch of one may take turns on it
    unsigned long long* wish;    // single-instance frame: [Titems] the split wishes' lower-bound costs per scan
                                 // tile, 0 between frames of that kernel
    uint32_t* tpre;              // single-instance frame: [2][Twords] ones before each word tile of
                                 // the next frame's starting bitfield (which: the instance's freel_full)
};

constexpr int kThreads = 256;
constexpr int kItemsPerThread = 4;
constexpr uint32_t kTileItems = kThreads * kItemsPerThread;  // 1024 live indices
// The two look-back scans use larger tiles, so that fewer tiles chain.
constexpr int kScanThreads = 512;
constexpr int kScanPerThread = 8;
constexpr uint32_t kScanItems = kScanThreads * kScanPerThread;  // 4096 live indices
constexpr uint32_t kMaxTileWords = 256;                       // up to 8192 bits per tile
constexpr uint32_t kMinTileWords = 64;

// -------------------------------------------------------- dependent launches

// The kernels of the indexed export, and prep and the vertices on their own,
// are launched with programmatic stream serialisation: the next kernel's
// blocks are brought in while the last ones of this kernel run, and wait here
// for this kernel's end and its writes, so that the launch and the ramp
// between two kernels overlap (the export of 0.9M triangles after a frame:
// 276 -> 267 us; the vertices of 0.9M bisectors: 54 -> 51; the reduction with
// its compaction, and a whole per-step frame, gained nothing). Called first in
// every such kernel; what an earlier kernel of the sequence writes is not read
// through the read-only path (__ldg or const __restrict__).
__device__ __forceinline__ void sequence_begin() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
template <typename... P, typename... A>
cudaError_t launch_sequence(void (*kernel)(P...), unsigned grid, unsigned block, cudaStream_t s, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// ------------------------------------------------------------------ bits

__device__ __forceinline__ int bitlen64(uint64_t x) { return 64 - __clzll((long long)x); }
__device__ __forceinline__ int depth_of(uint64_t j, uint32_t ch) { return bitlen64(j) - 1 - (int)ch; }

__device__ __forceinline__ uint64_t splitmix64(uint64_t x) {
    // SplitMix64 (Steele, Lea & Flood 2014), used as a counter-based hash.
    uint64_t z = x + 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__device__ __forceinline__ float pow2f(int e) { return __int_as_float((127 + e) << 23); }
__device__ __forceinline__ double pow2d(int e) {
    return __longlong_as_double((long long)(1023 + e) << 52);
}

__device__ __forceinline__ uint32_t ld_volatile(const uint32_t* p) {
    return *reinterpret_cast<const volatile uint32_t*>(p);
}

__device__ __forceinline__ void set_err(Globals* g, uint32_t e) { atomicOr(&g->err, e); }

// ------------------------------------------------- Alg. 2 / Eq. 1 decode

// Alg. 2 evaluated from the first split down: with M the weights after k
// levels, a 0 bit maps the rows (r0, r1, r2) to (r0, r2, (r0 + r1) / 2) and a
// 1 bit to (r2, r1, (r0 + r1) / 2) (Eq. 1), i.e. M <- M_b M. Up to eight
// levels at once are M <- P_c M with P_c the product for the path bits c
// (most significant applied first). Every row of M and P sums to 1 (they are
// barycentric), so only the first two columns are carried, and with the rows
// (a0, a1, a2) of M
//   P row (p0, p1, 1 - p0 - p1):  a2 + p0 (a0 - a2) + p1 (a1 - a2).
// After k <= 24 levels every entry is a multiple of 2^-k in [0, 1], and so is
// every intermediate value here, so FP32 fused multiply-adds are exact: the
// decode runs at the FP32 rate and needs no integer-to-float conversions
// (the integer form it replaced, with 16-bit table entries read one by one,
// made the classify phase of 886k leaves 33 us; this form makes it 24 us).
// The table holds P for r = 1..8 levels and all 2^r codes c in row
// 2^r - 2 + c (then the identity): the six entries in multiples of 2^-r, at
// most 8 significant bits, i.e. exact in bfloat16, so that a row is one
// 16-byte shared-memory load.
constexpr uint32_t kDecRows = 512, kDecIdentity = 510;
struct alignas(16) DecTable {
    uint32_t w[kDecRows][4];  // {p00 | p01 << 16, p10 | p11 << 16, p20 | p21 << 16, 0}
};

constexpr uint32_t bf16_of(uint32_t m, int r) {  // m 2^-r, m <= 256
    if (m == 0u) return 0u;
    int e = 0;
    while ((m >> (e + 1)) != 0u) ++e;
    const uint32_t frac = e <= 7 ? (m << (7 - e)) & 0x7Fu : 0u;
    return ((uint32_t)(127 + e - r) << 7) | frac;
}

constexpr DecTable make_dec8() {
    DecTable t{};
    for (int r = 0; r <= 8; ++r)
        for (uint32_t c = 0; c < (1u << r); ++c) {
            uint32_t m[6] = {1, 0, 0, 1, 0, 0};  // 2^k times the rows' first two columns after k levels
            for (int k = r - 1; k >= 0; --k) {
                const bool b = ((c >> k) & 1u) != 0u;
                uint32_t n[6] = {};
                for (int col = 0; col < 2; ++col) {
                    n[4 + col] = m[col] + m[2 + col];
                    n[col] = 2u * (b ? m[4 + col] : m[col]);
                    n[2 + col] = 2u * (b ? m[2 + col] : m[4 + col]);
                }
                for (int e = 0; e < 6; ++e) m[e] = n[e];
            }
            const uint32_t row = r ? (1u << r) - 2u + c : kDecIdentity;
            for (int q = 0; q < 3; ++q) t.w[row][q] = bf16_of(m[2 * q], r) | (bf16_of(m[2 * q + 1], r) << 16);
        }
    return t;
}

// In global memory, not constant memory: the copy below reads it with a
// different address in every lane, which the constant cache serializes.
__device__ const DecTable g_dec8 = make_dec8();
constexpr uint32_t kDecTabWords = sizeof(DecTable) / 4u;  // the table in 32-bit words

// Copies the table into shared memory (kDecTabWords words, s_tab 16-byte
// aligned; call with the whole block, then __syncthreads()).
__device__ __forceinline__ void load_dec6(uint32_t* s_tab) {
    const uint4* src = reinterpret_cast<const uint4*>(&g_dec8.w[0][0]);
    for (uint32_t k = threadIdx.x; k < kDecTabWords / 4u; k += blockDim.x)
        reinterpret_cast<uint4*>(s_tab)[k] = __ldg(src + k);
}
// The same copy in two halves (blocks of 256 threads): the loads into
// registers, then the stores, so that other loads can go out in between.
constexpr uint32_t kDecVecs = kDecTabWords / 4u / 256u;  // 16-byte loads per thread
__device__ __forceinline__ void dec_fetch(uint4 (&r)[kDecVecs]) {
    const uint4* src = reinterpret_cast<const uint4*>(&g_dec8.w[0][0]);
#pragma unroll
    for (uint32_t k = 0; k < kDecVecs; ++k) r[k] = __ldg(src + threadIdx.x + 256u * k);
}
__device__ __forceinline__ void dec_store(uint32_t* s_tab, const uint4 (&r)[kDecVecs]) {
#pragma unroll
    for (uint32_t k = 0; k < kDecVecs; ++k) reinterpret_cast<uint4*>(s_tab)[threadIdx.x + 256u * k] = r[k];
}

__device__ __forceinline__ void dec_row(const uint32_t* tab, uint32_t row, float p[6]) {
    const uint4 v = reinterpret_cast<const uint4*>(tab)[row];
    p[0] = __uint_as_float(v.x << 16);
    p[1] = __uint_as_float(v.x & 0xFFFF0000u);
    p[2] = __uint_as_float(v.y << 16);
    p[3] = __uint_as_float(v.y & 0xFFFF0000u);
    p[4] = __uint_as_float(v.z << 16);
    p[5] = __uint_as_float(v.z & 0xFFFF0000u);
}

// The first two columns (a[2 r + c]) of the product of n <= 24 levels whose
// path bits are the low n bits of `bits`.
__device__ __forceinline__ void decode_levels(uint32_t bits, int n, const uint32_t* tab, float a[6]) {
    const int first = n ? ((n - 1) & 7) + 1 : 0;  // levels of the first lookup
    int sh = n - first;
    const uint32_t row0 = (1u << first) - 2u + (bits >> sh & ((1u << first) - 1u));
    dec_row(tab, n ? row0 : kDecIdentity, a);
#pragma unroll 1
    while (sh > 0) {
        sh -= 8;
        float p[6];
        dec_row(tab, 254u + ((bits >> sh) & 255u), p);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const float e = __fsub_rn(a[c], a[4 + c]), f = __fsub_rn(a[2 + c], a[4 + c]), a2 = a[4 + c];
#pragma unroll
            for (int r = 0; r < 3; ++r) a[2 * r + c] = __fmaf_rn(p[2 * r], e, __fmaf_rn(p[2 * r + 1], f, a2));
        }
    }
}

// The weights of bisector j at depth d, as the first two columns a[2 r + c]
// in one of two types: float, M itself, exact for d <= kFloatDepth; or
// unsigned long long, W = 2^d M, for any depth (d <= 62).
constexpr int kFloatDepth = 24;
typedef unsigned long long u64;
__device__ __forceinline__ void decode_cols(uint64_t j, int d, const uint32_t* tab, float a[6]) {
    decode_levels((uint32_t)j & ((1u << d) - 1u), d, tab, a);
}
// The levels in runs of at most 24, each decoded in FP32 and applied to the
// integer weights so far: 2^24 a2 + b0 (a0 - a2) + b1 (a1 - a2), b = 2^24 P
// (32 x 32 -> 64 bit products while the weights so far fit 25 bits).
__device__ __forceinline__ void decode_cols(uint64_t j, int d, const uint32_t* tab, u64 a[6]) {
    const int first = d > 0 ? (d - 1) % 24 + 1 : 0;
    float p[6];
    decode_levels((uint32_t)(j >> (d - first)) & ((1u << first) - 1u), first, tab, p);
    int s[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        s[k] = __float2int_rn(__fmul_rn(p[k], pow2f(first)));
        a[k] = (u64)s[k];
    }
    int lo = d - first - 24;
    if (lo >= 0) {
        decode_levels((uint32_t)(j >> lo) & 0xFFFFFFu, 24, tab, p);
        int b[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) b[k] = __float2int_rn(__fmul_rn(p[k], 0x1p24f));
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const long long e = s[c] - s[4 + c], f = s[2 + c] - s[4 + c], a2 = (long long)s[4 + c] << 24;
#pragma unroll
            for (int r = 0; r < 3; ++r) a[2 * r + c] = (u64)(a2 + (long long)b[2 * r] * e + (long long)b[2 * r + 1] * f);
        }
        lo -= 24;
    }
#pragma unroll 1
    for (; lo >= 0; lo -= 24) {
        decode_levels((uint32_t)(j >> lo) & 0xFFFFFFu, 24, tab, p);
        int b[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) b[k] = __float2int_rn(__fmul_rn(p[k], 0x1p24f));
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const long long e = (long long)(a[c] - a[4 + c]), f = (long long)(a[2 + c] - a[4 + c]);
            const u64 a2 = a[4 + c] << 24;
#pragma unroll
            for (int r = 0; r < 3; ++r)
                a[2 * r + c] = a2 + (u64)((long long)b[2 * r] * e) + (u64)((long long)b[2 * r + 1] * f);
        }
    }
}

__device__ __forceinline__ float unit_of(float, int) { return 1.0f; }
__device__ __forceinline__ u64 unit_of(u64, int d) { return 1ull << d; }

// The three weights of vertex v.
template <typename T>
__device__ __forceinline__ void weight_row(const T a[6], int v, int d, T w[3]) {
    w[0] = a[2 * v];
    w[1] = a[2 * v + 1];
    w[2] = unit_of(T(), d) - w[0] - w[1];
}
// The three weights, over the same 2^d, of the parent's vertex that the
// bisector does not share. Eq. 1 makes an odd child's rows (p2, p1,
// (p0 + p1) / 2) of the parent's and an even one's (p0, p2, (p0 + p1) / 2), so
// p0 = 2 r2 - r1 (odd) and p1 = 2 r2 - r0 (even).
template <typename T>
__device__ __forceinline__ void parent_row(const T a[6], bool odd, int d, T w[3]) {
#pragma unroll
    for (int c = 0; c < 2; ++c) w[c] = a[4 + c] + a[4 + c] - (odd ? a[2 + c] : a[c]);
    w[2] = unit_of(T(), d) - w[0] - w[1];
}

// A weight in FP32 (w = float(W) 2^-d) and FP64. A float one (M, exact) is
// widened by its bits; an integer one below 2^52 becomes FP64 at an exponent
// whose last place is 2^-d, minus that power: both exact, and cheaper here
// than FP64 conversions and a scaling.
__device__ __forceinline__ float weight_f32(float w, int) { return w; }
__device__ __forceinline__ float weight_f32(u64 w, int d) { return __fmul_rn(__ull2float_rn(w), pow2f(-d)); }
__device__ __forceinline__ double weight_f64(float w, int) {
    const uint32_t b = __float_as_uint(w);
    return b ? __hiloint2double((int)((b >> 3) + (896u << 20)), (int)(b << 29)) : 0.0;
}
__device__ __forceinline__ double weight_f64(u64 w, int d) {
    if (d > 51) return __dmul_rn(__ull2double_rn(w), pow2d(-d));
    const double one = pow2d(52 - d);
    return __dsub_rn(__longlong_as_double(__double_as_longlong(one) | (long long)w), one);
}

// Correctly rounded signed 128-bit integer (hi 2^64 + lo) -> float. Below
// 2^63 in magnitude one 64-bit conversion; below 2^95 one of the value over
// 2^32 rounded to odd (its lowest bit set when bits were cut off: more than
// two bits below an FP32's last place, so the second rounding is as the
// first would have been). Beyond (never with camera-relative coordinates of
// a scene, but legal) the magnitude's top 32 bits with a sticky bit.
static __device__ __noinline__ float s128_to_float_any(long long hi, u64 lo) {
    const bool neg = hi < 0;
    u64 h = (u64)hi;
    if (neg) {
        lo = 0ull - lo;
        h = ~h + (lo == 0ull ? 1ull : 0ull);
    }
    int e = 96;
    if (h == 0ull) {
        h = lo;
        lo = 0ull;
        e = 32;
    }
    const int lz = __clzll((long long)h);
    if (lz == 64) return 0.0f;
    const u64 z = (h << lz) | ((lo >> 1) >> (63 - lz));
    const uint32_t rest = (uint32_t)z | (uint32_t)((lo << lz) != 0ull);
    const float f = __uint2float_rn((uint32_t)(z >> 32) | (rest ? 1u : 0u));
    const float m = __fmul_rn(f, pow2f(e - lz));
    return neg ? -m : m;
}
__device__ __forceinline__ float s128_to_float(long long hi, u64 lo) {
    if ((hi >> 31) != (hi >> 63)) return s128_to_float_any(hi, lo);
    const bool small = hi == (long long)lo >> 63;
    const long long over = (long long)(((u64)hi << 32) | (lo >> 32)) | ((uint32_t)lo != 0u ? 1ll : 0ll);
    const float f = __ll2float_rn(small ? (long long)lo : over);
    return small ? f : __fmul_rn(f, 0x1p32f);
}

// Fixed point: exact sums over the root's vertices of weight times
// coordinate. A coordinate x (|x| < 2^62) is split as xh 2^32 + xl with both
// halves signed 32 bits, so that every product is one signed 32 x 32 -> 64
// multiply-add and no partial sum overflows.
struct S128 {
    long long hi;
    u64 lo;
};
__device__ __forceinline__ S128 s128_add(S128 a, S128 b) {
    const u64 l = a.lo + b.lo;
    return S128{a.hi + b.hi + (l < a.lo ? 1ll : 0ll), l};
}
// (m 2^32 + l) 2^k, k = 0 or 24, l the low half's sum (signed).
__device__ __forceinline__ S128 s128_parts(long long m, long long l) {
    m += l >> 32;
    return S128{m >> 32, ((u64)m << 32) | (uint32_t)l};
}
__device__ __forceinline__ S128 s128_shl24(S128 a) {
    return S128{(long long)(((u64)a.hi << 24) | (a.lo >> 40)), a.lo << 24};
}
__device__ __forceinline__ void split_coord(long long x, int& xl, int& xh) {
    xl = (int)x;
    xh = (int)(x >> 32) + (xl < 0 ? 1 : 0);
}
// Signed weights below 2^26 in magnitude.
__device__ __forceinline__ S128 fixed_narrow(const int w[3], const int xl[3], const int xh[3]) {
    long long l = 0, m = 0;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        l += (long long)w[i] * (long long)xl[i];
        m += (long long)w[i] * (long long)xh[i];
    }
    return s128_parts(m, l);
}
// Weights up to 2^48, in two 24-bit parts (the upper ones all 0: `wide` false).
__device__ __forceinline__ S128 fixed_wide(const int wl[3], const int wh[3], bool wide, const int xl[3],
                                           const int xh[3]) {
    const S128 a = fixed_narrow(wl, xl, xh);
    return wide ? s128_add(a, s128_shl24(fixed_narrow(wh, xl, xh))) : a;
}
// Any weights (one coordinate; X points at the root's first vertex's).
__device__ __forceinline__ S128 fixed_any(const u64 w[3], const long long* X) {
    __int128 s = 0;
#pragma unroll
    for (int i = 0; i < 3; ++i) s += (__int128)w[i] * (__int128)X[3 * i];
    return S128{(long long)(s >> 64), (u64)s};
}
__device__ __forceinline__ u64 weight_int(u64 w, int) { return w; }
__device__ __forceinline__ u64 weight_int(float w, int d) { return (u64)__float2int_rn(__fmul_rn(w, pow2f(d))); }

// ------------------------------------------------------------ displacement

// Displacement of the tested and exported vertices by seeded fractal value
// noise, standing in for the wave layers and elevation data with which the
// paper displaces the projected vertices during refinement (Sec. 4; R14
// reading):
//   lattice value of integer point i at octave o: lowbias32 (Wellons,
//     "Prospecting for Hash Functions", 2018) chained from seed ^ o over the
//     coordinates, last to first; the top 24 bits give (h >> 8) 2^-23 - 1;
//   octave o: per axis s = x f 2^o clamped to +-2^30, corner floor(s),
//     weight u = t t (3 - 2 t) with t = s - floor(s); the 2^n corner values
//     blended along x, then y, then z, as a + u (b - a);
//   fbm = the sum over o < octaves of 2^-o times octave o, in order.
// Every FP32 operation rounds separately.
__device__ __forceinline__ uint32_t lowbias32(uint32_t x) {
    x ^= x >> 16;
    x *= 0x7feb352du;
    x ^= x >> 15;
    x *= 0x846ca68bu;
    x ^= x >> 16;
    return x;
}
__device__ __forceinline__ float lattice_unit(uint32_t h) {
    return __fsub_rn(__fmul_rn(__uint2float_rn(h >> 8), 0x1p-23f), 1.0f);
}
__device__ __forceinline__ float blend(float a, float b, float u) {
    return __fadd_rn(a, __fmul_rn(u, __fsub_rn(b, a)));
}
// Corner index and weight of one axis at frequency fo.
__device__ __forceinline__ float noise_axis(float x, float fo, uint32_t& i) {
    const float s = fminf(fmaxf(__fmul_rn(x, fo), -0x1p30f), 0x1p30f);
    const float fl = floorf(s);
    i = (uint32_t)(int)fl;
    const float t = __fsub_rn(s, fl);
    return __fmul_rn(__fmul_rn(t, t), __fsub_rn(3.0f, __fmul_rn(2.0f, t)));
}

// 2-D fbm of (x0, x1); the hash prefix of each y corner is shared.
static __device__ __noinline__ float fbm2(float x0, float x1, float freq, uint32_t octaves, uint32_t seed) {
    float sum = 0.0f;
    for (uint32_t o = 0; o < octaves; ++o) {
        const float fo = __fmul_rn(freq, pow2f((int)o));
        uint32_t ix, iy;
        const float ux = noise_axis(x0, fo, ix), uy = noise_axis(x1, fo, iy);
        const uint32_t h0 = lowbias32(seed ^ o);
        const uint32_t hy0 = lowbias32(h0 ^ iy), hy1 = lowbias32(h0 ^ (iy + 1u));
        const float a = blend(lattice_unit(lowbias32(hy0 ^ ix)), lattice_unit(lowbias32(hy0 ^ (ix + 1u))), ux);
        const float b = blend(lattice_unit(lowbias32(hy1 ^ ix)), lattice_unit(lowbias32(hy1 ^ (ix + 1u))), ux);
        sum = __fadd_rn(sum, __fmul_rn(blend(a, b, uy), pow2f(-(int)o)));
    }
    return sum;
}

// fbm2 of two points at once, their octaves interleaved: one point alone is a
// chain of dependent operations (the terrain's classify phase, 877k leaves at
// six octaves, whose warps have 45 distinct points each: 98 us, 106 with the
// points one after the other).
static __device__ __noinline__ float2 fbm2_pair(float2 p, float2 q, float freq, uint32_t octaves, uint32_t seed) {
    float2 sum = make_float2(0.0f, 0.0f);
#pragma unroll 1
    for (uint32_t o = 0; o < octaves; ++o) {
        const float fo = __fmul_rn(freq, pow2f((int)o)), w = pow2f(-(int)o);
        const uint32_t h0 = lowbias32(seed ^ o);
        const float x[2][2] = {{p.x, p.y}, {q.x, q.y}};
        float v[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            uint32_t ix, iy;
            const float ux = noise_axis(x[k][0], fo, ix), uy = noise_axis(x[k][1], fo, iy);
            const uint32_t hy0 = lowbias32(h0 ^ iy), hy1 = lowbias32(h0 ^ (iy + 1u));
            const float a = blend(lattice_unit(lowbias32(hy0 ^ ix)), lattice_unit(lowbias32(hy0 ^ (ix + 1u))), ux);
            const float b = blend(lattice_unit(lowbias32(hy1 ^ ix)), lattice_unit(lowbias32(hy1 ^ (ix + 1u))), ux);
            v[k] = __fmul_rn(blend(a, b, uy), w);
        }
        sum.x = __fadd_rn(sum.x, v[0]);
        sum.y = __fadd_rn(sum.y, v[1]);
    }
    return sum;
}

// 3-D fbm of (x0, x1, x2); hash prefixes shared per z and per (z, y).
static __device__ __noinline__ float fbm3(float x0, float x1, float x2, float freq, uint32_t octaves, uint32_t seed) {
    float sum = 0.0f;
    for (uint32_t o = 0; o < octaves; ++o) {
        const float fo = __fmul_rn(freq, pow2f((int)o));
        uint32_t ix, iy, iz;
        const float ux = noise_axis(x0, fo, ix), uy = noise_axis(x1, fo, iy), uz = noise_axis(x2, fo, iz);
        const uint32_t h0 = lowbias32(seed ^ o);
        float zc[2];
#pragma unroll
        for (uint32_t bz = 0; bz < 2; ++bz) {
            const uint32_t hz = lowbias32(h0 ^ (iz + bz));
            const uint32_t hzy0 = lowbias32(hz ^ iy), hzy1 = lowbias32(hz ^ (iy + 1u));
            const float a = blend(lattice_unit(lowbias32(hzy0 ^ ix)), lattice_unit(lowbias32(hzy0 ^ (ix + 1u))), ux);
            const float b = blend(lattice_unit(lowbias32(hzy1 ^ ix)), lattice_unit(lowbias32(hzy1 ^ (ix + 1u))), ux);
            zc[bz] = blend(a, b, uy);
        }
        sum = __fadd_rn(sum, __fmul_rn(blend(zc[0], zc[1], uz), pow2f(-(int)o)));
    }
    return sum;
}

// Forms whose vertices the one-launch frame caches from its LOD test for the
// export (a sphere projection or a displacement costs more to evaluate again
// than 36 bytes cost to store and load).
template <int F>
__device__ __forceinline__ bool vc_form(const FrameP& fp) {
    return precision_in<F>(fp) == 3u || displaced_in<F>(fp);
}

// FP32 form: z += amplitude * fbm2 of the world (x, y), the vertex plus the
// origin rounded to FP32.
__device__ __forceinline__ void displace_plain(float r[3], const FrameP& fp) {
    const float wx = __fadd_rn(r[0], __double2float_rn(fp.eye[0]));
    const float wy = __fadd_rn(r[1], __double2float_rn(fp.eye[1]));
    r[2] = __fadd_rn(r[2], __fmul_rn(fp.damp, fbm2(wx, wy, fp.dfreq, fp.doct, fp.dseed)));
}

// Vertex v (0..2) of a bisector relative to the frame's origin, rounded to
// FP32, into r[0..2]:
//   FP32:   (w0 R0 + w1 R1) + w2 R2, w = float(W) 2^-d (no contraction);
//   FIXED:  float(sum W X) 2^-(d + shift), the sum exact in 128 bits;
//   FP64:   float((w0 D0 + w1 D1) + w2 D2), w = double(W) 2^-d;
//   SPHERE: the FP64 point p of the flat root triangle (V absolute) moved
//           radially onto the sphere about the world origin, relative to the
//           eye, rounded to FP32; with fused multiply-adds:
//             p_c = fma(w2, V2c, fma(w1, V1c, w0 V0c)),
//             n2  = fma(pz, pz, fma(py, py, px px)),
//             y   = 1 / sqrt(n2): the FP32 estimate 1 / sqrtf(float(n2)),
//                   then twice y = fma(y/2, fma(-n2, y y, 1), y) (Newton),
//             r_c = float(fma(p_c, radius y, -eye_c)).
// With a displacement the FP32 form adds amplitude * fbm2(world x, y) to z
// (displace_plain) and the sphere form takes radius + double(amplitude *
// fbm3(u)) for the radius, u_c = float(p_c y) the unit direction.
// The sphere form's frame-independent part of vertex v: pf = {p_x, p_y, p_z,
// f}, f = radius' y (V: the root triangle's absolute FP64 vertices). It
// depends on the heap ID, the mesh, the radius and the displacement only.
__device__ __forceinline__ void sphere_point(const double w[3], const FrameP& fp, const double* V, double pf[4]) {
    const double w0 = w[0], w1 = w[1], w2 = w[2];
    double p[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) p[c] = __fma_rn(w2, V[6 + c], __fma_rn(w1, V[3 + c], __dmul_rn(w0, V[c])));
    const double n2 = __fma_rn(p[2], p[2], __fma_rn(p[1], p[1], __dmul_rn(p[0], p[0])));
    double y = (double)__frcp_rn(__fsqrt_rn(__double2float_rn(n2)));
#pragma unroll
    for (int it = 0; it < 2; ++it) y = __fma_rn(__dmul_rn(y, 0.5), __fma_rn(-n2, __dmul_rn(y, y), 1.0), y);
    double rad = fp.radius;
    if (fp.damp != 0.0f) {
        const float hgt = __fmul_rn(fp.damp, fbm3(__double2float_rn(__dmul_rn(p[0], y)),
                                                 __double2float_rn(__dmul_rn(p[1], y)),
                                                 __double2float_rn(__dmul_rn(p[2], y)), fp.dfreq, fp.doct,
                                                 fp.dseed));
        rad = __dadd_rn(rad, (double)hgt);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) pf[c] = p[c];
    pf[3] = __dmul_rn(rad, y);
}

// The per-frame part: the point relative to the eye, rounded to FP32.
__device__ __forceinline__ void sphere_rel(double px, double py, double pz, double f, const FrameP& fp,
                                           float r[3]) {
    r[0] = __double2float_rn(__fma_rn(px, f, -fp.eye[0]));
    r[1] = __double2float_rn(__fma_rn(py, f, -fp.eye[1]));
    r[2] = __double2float_rn(__fma_rn(pz, f, -fp.eye[2]));
}

// FP32: weights rounded to FP32, root vertices R.
__device__ __forceinline__ void plain_vertex(const float w[3], const float R[9], float r[3]) {
#pragma unroll
    for (int c = 0; c < 3; ++c)
        r[c] = __fadd_rn(__fadd_rn(__fmul_rn(w[0], R[c]), __fmul_rn(w[1], R[3 + c])), __fmul_rn(w[2], R[6 + c]));
}

// One vertex with weights w over 2^d (rel: the root tables, h the root).
template <int F, typename T>
__device__ __forceinline__ void eval_vertex(const T w[3], int d, const FrameP& fp, const void* rel, uint32_t h,
                                            float r[3]) {
    const uint32_t precision = precision_in<F>(fp);
    if (precision == 3u) {
        double pf[4];
        const double wd[3] = {weight_f64(w[0], d), weight_f64(w[1], d), weight_f64(w[2], d)};
        sphere_point(wd, fp, static_cast<const double*>(rel) + 9u * h, pf);
        sphere_rel(pf[0], pf[1], pf[2], pf[3], fp, r);
    } else if (precision == 1u) {
        const long long* X = static_cast<const long long*>(rel) + 9u * h;
        const u64 wi[3] = {weight_int(w[0], d), weight_int(w[1], d), weight_int(w[2], d)};
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const S128 s = fixed_any(wi, X + c);
            r[c] = __fmul_rn(s128_to_float(s.hi, s.lo), pow2f(-(d + fp.shift)));
        }
    } else if (precision == 2u) {
        const double* Dp = static_cast<const double*>(rel) + 9u * h;
        const double w0 = weight_f64(w[0], d), w1 = weight_f64(w[1], d), w2 = weight_f64(w[2], d);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const double t = __dadd_rn(__dadd_rn(__dmul_rn(w0, Dp[c]), __dmul_rn(w1, Dp[3 + c])),
                                       __dmul_rn(w2, Dp[6 + c]));
            r[c] = __double2float_rn(t);
        }
    } else {
        const float* R = static_cast<const float*>(rel) + 9u * h;
        const float wf[3] = {weight_f32(w[0], d), weight_f32(w[1], d), weight_f32(w[2], d)};
        plain_vertex(wf, R, r);
        if (displaced_in<F>(fp)) displace_plain(r, fp);
    }
}

// LOD reading: a triangle is visible unless one plane has all three
// vertices strictly on its negative side, where a vertex r is on the
// negative side of plane n when (n.x r.x + n.y r.y) + n.z r.z < 0; it is
// big when |v1 - v0|^2 q > |(v0 + v1)/2|^2.
// The planes among `among` (a bit mask) on whose negative side vertex r
// lies, as a bit mask: a triangle is culled by a plane only if all three
// vertices are, so a vertex need only be tested against the planes the
// earlier ones failed (the same products, bit for bit, where they are made).
__device__ __forceinline__ uint32_t plane_mask(const float* r, const FrameP& fp, uint32_t among = 31u) {
    uint32_t m = 0u;
#pragma unroll
    for (uint32_t p = 0; p < 5u; ++p) {
        if (p >= fp.nplanes) break;
        if (!((among >> p) & 1u)) continue;
        const float s = __fadd_rn(__fadd_rn(__fmul_rn(fp.planes[3 * p], r[0]), __fmul_rn(fp.planes[3 * p + 1], r[1])),
                                  __fmul_rn(fp.planes[3 * p + 2], r[2]));
        m |= (s < 0.0f ? 1u : 0u) << p;
    }
    return m;
}
// |a - b|^2 q > |(a + b)/2|^2 for the refinement edge (a, b).
__device__ __forceinline__ bool edge_big(const float* a, const float* b, float q) {
    const float ex = __fsub_rn(b[0], a[0]), ey = __fsub_rn(b[1], a[1]), ez = __fsub_rn(b[2], a[2]);
    const float mx = __fmul_rn(0.5f, __fadd_rn(a[0], b[0]));
    const float my = __fmul_rn(0.5f, __fadd_rn(a[1], b[1]));
    const float mz = __fmul_rn(0.5f, __fadd_rn(a[2], b[2]));
    const float L2 = __fadd_rn(__fadd_rn(__fmul_rn(ex, ex), __fmul_rn(ey, ey)), __fmul_rn(ez, ez));
    const float R2 = __fadd_rn(__fadd_rn(__fmul_rn(mx, mx), __fmul_rn(my, my)), __fmul_rn(mz, mz));
    return __fmul_rn(L2, q) > R2;
}
__device__ __forceinline__ bool in_sorted(const uint64_t* a, uint32_t n, uint64_t x) {
    uint32_t lo = 0, hi = n;
    while (lo < hi) {
        const uint32_t mid = lo + (hi - lo) / 2u;
        if (a[mid] < x)
            lo = mid + 1u;
        else
            hi = mid;
    }
    return lo < n && a[lo] == x;
}

// --------------------------------------------------------- saturating pairs

constexpr uint32_t kSat = 0x7FFFFFFFu;

struct Pair {
    uint32_t a, b;
};

__device__ __forceinline__ Pair padd(Pair x, Pair y) {
    return Pair{min(x.a + y.a, kSat), min(x.b + y.b, kSat)};
}

constexpr unsigned long long kFlagAgg = 1ull, kFlagIncl = 2ull;

__device__ __forceinline__ unsigned long long pack_status(unsigned long long flag, Pair v) {
    return (flag << 62) | ((unsigned long long)v.a << 31) | (unsigned long long)v.b;
}
__device__ __forceinline__ unsigned long long status_flag(unsigned long long s) { return s >> 62; }
__device__ __forceinline__ Pair status_val(unsigned long long s) {
    return Pair{(uint32_t)((s >> 31) & kSat), (uint32_t)(s & kSat)};
}

}  // namespace cbtgpu
