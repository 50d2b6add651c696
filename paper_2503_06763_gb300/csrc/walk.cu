// The walk of the chunks (arXiv 2503.06763, Eqs. reacher and builder; see
// walk.cuh): one run per chunk and direction, from where the chunk's
// speculative runs had met to its far edge and on through the next chunk's
// head.  With OUT every column's state goes to FS / BS.
//
// A step is the lookup of the byte's class and of the transition, the latter a
// chain of about 35 cycles per byte that some 20 warps per SM cover.  With 32
// copies of the table (LaneTab) neither lookup conflicts: 2 wavefronts per byte
// where one byte-indexed table took 4.2.  A tile of text is 32 chunks x 32
// bytes (32-byte TMA rows) and its states replace it in place, so a warp needs
// two 1 KB tiles: one walked, the other sending its states and then loading.
// Moving a lane's 32 bytes straight between registers and global memory needs
// no tiles and no barriers, but costs a wavefront per lane and access, 0.27 ms
// at 256 MiB of log text.
//
// Measured (heads and walk together, log text): 11 MiB 45 us, 256 MiB 0.27 ms,
// 1 GiB 0.94 ms (autotuned chunk length) = 3.4 TB/s of text read once and states
// written, where one kernel of byte-indexed tables that held a chunk's runs in
// registers and local memory took 140 us, 0.37 ms and 1.10 ms and left the chunk
// heads to another.  What bounds it: issue slots (69 % busy, 11 instructions per
// byte step) and the shared-memory pipe (70 %) together (256 MiB, the rule's
// chunk length).
#include <algorithm>
#include <type_traits>

#include "walk.cuh"

namespace slpf {
namespace {

constexpr uint32_t kWalkWarps = 24;          // warps of a block at most: leaves 80 registers a thread
constexpr size_t kWalkSmemMax = 227 * 1024;

constexpr uint32_t kWalkTile = 32 * kUnit;
struct WalkRing {
    uint8_t *tiles;       // [2][kWalkTile], 1024-byte aligned
    uint32_t bars;        // shared address of 2 mbarriers
    uint32_t phase;       // bit s: parity of the next completion of stage s
};

// TMA copies of one tile by the lane with `on` set.  Predicated rather than
// branched: with divergent branches the walk of 1 GiB of log text took 4 %
// longer.
__device__ __forceinline__ void tile_load(bool on, uint32_t dst, const CUtensorMap *map, int32_t x, int32_t y, uint32_t bar) {
    asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %0, 0;\n"
                 " @p mbarrier.arrive.expect_tx.shared::cta.b64 _, [%5], %6;\n"
                 " @p cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%1], [%2, {%3, %4}], [%5];\n}"
                 :: "r"((uint32_t)on), "r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar),
                    "n"(kWalkTile) : "memory");
}
__device__ __forceinline__ void tile_store(bool on, uint32_t src, const CUtensorMap *map, int32_t x, int32_t y) {
    asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %0, 0;\n"
                 " @p cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%1, {%2, %3}], [%4];\n"
                 " cp.async.bulk.commit_group;\n}"
                 :: "r"((uint32_t)on), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(src) : "memory");
}

// Units [0, nb) of a full 32-chunk tile, unit u at column x0 + 32 u (forward)
// or x0 - 32 (u + 1) (backward) of every chunk: text in by TMA, states out by
// TMA from the same tile.  Unit u uses stage u % 2; half way through it, its
// states of a unit ago sent, the other stage starts loading unit u + 1.  False
// when a TMA completion was lost.
template <int LOGR, bool FWD, bool OUT>
__device__ bool walk_units(const Params &p, const LaneTab &T, WalkRing &ring, const CUtensorMap *map,
                           const CUtensorMap *smap, uint32_t i0, uint32_t x0, uint32_t nb, uint32_t &s) {
    const uint32_t lane = threadIdx.x & 31, swz = (lane >> 2) & 1;
    const uint32_t tiles = smem_u32(ring.tiles);
    uint8_t *row = ring.tiles + lane * kUnit;
    uint4 *const qa = reinterpret_cast<uint4 *>(row + (swz << 4)), *const qb = reinterpret_cast<uint4 *>(row + ((swz ^ 1u) << 4));
    const int32_t step = FWD ? (int32_t)kUnit : -(int32_t)kUnit;
    int32_t x = FWD ? (int32_t)x0 : (int32_t)x0 - (int32_t)kUnit;   // column of the unit being walked
    const uint8_t *ahead = p.x + (uint64_t)(i0 + lane) * p.k + x;
    uint32_t st = 0;
    if (OUT) bulk_wait_read_all();
    tile_load(lane == 0 && nb, tiles, map, x, (int32_t)i0, ring.bars);
    // rolled (a unit, and its two halves): 972 us at 1 GiB, 990 with two units unrolled
#pragma unroll 1
    for (uint32_t u = 0; u < nb; ++u) {
        // text lines (128 bytes) come into L2 a line ahead of the unit that
        // loads from them: the ring covers an L2 access, not one to HBM.
        // Further ahead the lines of all rows in flight no longer stay in L2
        // until they are read: three lines ahead, the text was read 1.5 times.
        if ((u & 3) == 0 && u + 4 < nb) prefetch_l2(ahead + (int64_t)(u + 4) * step);
        if (!__all_sync(0xFFFFFFFFu, mbar_try_wait(ring.bars + 8 * st, (ring.phase >> st) & 1u))) {
            bool ok = false;
            for (uint32_t it = 0; it < kWaitLimit && !ok; ++it)
                ok = mbar_try_wait(ring.bars + 8 * st, (ring.phase >> st) & 1u);
            if (!__all_sync(0xFFFFFFFFu, ok)) return false;
        }
        ring.phase ^= 1u << st;
        uint4 *const a = qa + st * (kWalkTile / 16), *const b = qb + st * (kWalkTile / 16);
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
            uint4 *const q = (h == 0) == FWD ? a : b;
            const uint4 tx = *q;
            uint4 ox;
            s = walk16<LOGR, FWD>(T, s, tx, ox);
            if (OUT) *q = ox;
            if (h == 0) {
                if (OUT) bulk_wait_read_all();
                tile_load(lane == 0 && u + 1 < nb, tiles + (st ^ 1u) * kWalkTile, map, x + step, (int32_t)i0, ring.bars + 8 * (st ^ 1u));
            }
        }
        if (OUT) fence_async_smem();
        __syncwarp();                                         // states written, or the text read
        if (OUT) tile_store(lane == 0, tiles + st * kWalkTile, smap, x, (int32_t)i0);
        x += step;
        st ^= 1u;
    }
    return true;
}

// The chunk of this lane (a warp's 32 consecutive chunks): its own columns,
// then the head of the chunk its run goes on into.
template <int LOGR, bool FWD, bool OUT>
__device__ bool walk_chunk(const Params &p, const LaneTab &T, uint32_t ns, uint64_t tile, bool wide,
                           const CUtensorMap *map, const CUtensorMap *smap, WalkRing &ring) {
    const uint32_t lane = threadIdx.x & 31, i0 = (uint32_t)(tile * 32), i = i0 + lane;
    const bool valid = i < p.c;
    const uint32_t *convs = FWD ? p.w.fconv : p.w.bconv, *kinds = FWD ? p.w.fkind : p.w.bkind;
    const uint32_t *states = FWD ? p.w.fnrec : p.w.bnrec;
    uint8_t *S = OUT ? (FWD ? p.w.FS : p.w.BS) : nullptr;
    const uint64_t base = (uint64_t)i * p.k;
    const uint32_t len = valid ? chunk_len(p, i) : 0, o = FWD ? i + 1 : i - 1;
    const bool known = valid && kinds[i] == 0;
    uint32_t s = 0, edge = 0, skip;
    if (known) {
        s = states[i];
        if (s >= ns) s = 0;                                   // no state of the classic DFA: the text is rejected
        edge = min(kUnit * convs[i], len);
    }
    // columns of the next chunk's head
    auto head_of = [&]() -> uint32_t {
        if (!known || p.rall || !(FWD ? i + 1 < p.c : i > 0)) return 0;
        if (!OUT && kinds[o] != 0) return 0;                  // no columns, and no state to check
        const uint32_t nlen = chunk_len(p, o), e = min(kUnit * convs[o], nlen);
        return FWD ? e : nlen - e;
    };
    uint32_t mid = 0, e = 0, head;
    const uint64_t m = FWD ? base + len : base;               // this chunk's far edge
    if (p.text_tma && i0 + 32 <= p.c_full && __all_sync(0xFFFFFFFFu, known)) {
        // lanes whose runs met earlier walk up to the last one's start, then all move together
        const uint32_t from = FWD ? __reduce_max_sync(0xFFFFFFFFu, edge) : __reduce_min_sync(0xFFFFFFFFu, edge);
        s = walk_cols<LOGR, FWD, OUT>(T, p.x, S, base + (FWD ? edge : from), base + (FWD ? from : edge),
                                      base + (FWD ? from : edge), s, wide, skip);
        __syncwarp();
        if (!walk_units<LOGR, FWD, OUT>(p, T, ring, map, smap, i0, from, (FWD ? p.k - from : from) / kUnit, s))
            return false;
        mid = s;
        head = head_of();
        e = walk_cols<LOGR, FWD, OUT>(T, p.x, S, FWD ? m : m - head, FWD ? m + head : m, m, s, wide, skip);
    } else {
        head = head_of();
        if (known)
            e = walk_cols<LOGR, FWD, OUT>(T, p.x, S, FWD ? base + edge : m - head, FWD ? m + head : base + edge, m, s, wide,
                                          mid);
    }
    if (!valid) return true;
    if (p.rall) {                                             // slice maps: every slot's end state
        const uint32_t ms = FWD ? p.t.msf : p.t.msb;
        uint32_t *R = (FWD ? p.w.Rf : p.w.Rb) + (size_t)i * ms;
        const uint32_t live = (FWD ? p.w.fhit : p.w.bhit)[i];
        if (known)
            for (uint32_t j = 0; j < ms; ++j) R[j] = (live >> j) & 1u ? mid : 0u;
        return true;
    }
    uint32_t *J = FWD ? p.w.FJ : p.w.BJ;
    if (FWD ? i == 0 : i == p.c - 1) {
        J[FWD ? 0 : p.c] = FWD ? p.t.fI : p.t.bF;
        if (OUT && !FWD) S[p.n] = (uint8_t)p.t.bF;
    }
    if (!known) {                                             // the join evaluates this chunk
        atomicAdd(p.w.scan + kScanGeneral, 1u);
        return true;
    }
    J[FWD ? i + 1 : i] = mid;
    if (FWD && OUT && i == p.c - 1) S[p.n] = (uint8_t)mid;
    // the state where the next chunk's runs had met must be theirs
    const bool check = (FWD ? i + 1 < p.c : i > 0) && kinds[o] == 0;
    if (mid == 0 || (check && (e == 0 || e != states[o]))) atomicMin(&p.w.flags[FWD ? FLAG_FFAIL : FLAG_BFAIL], (int32_t)i);
    return true;
}

// Dynamic shared memory: [pad to 1024][two tiles per warp][the table's
// copies][two mbarriers per warp].
template <int LOGR>
__host__ __device__ inline size_t lane_table_bytes(const DevTables &t) {
    const size_t ns = (t.nfd > t.nbd ? t.nfd : t.nbd) + 1;
    return (((ns * class_words(t) * 4) << LOGR) + 127) & ~(size_t)127;
}

constexpr size_t kWalkFixed = 1024 + 256, kWalkWarpSmem = 2 * (kWalkTile + 8);
template <int LOGR>
inline uint32_t walk_wpb(const DevTables &t) {               // warps a block's shared memory holds
    const size_t fixed = kWalkFixed + lane_table_bytes<LOGR>(t);
    return fixed >= kWalkSmemMax ? 0u : (uint32_t)std::min<size_t>(kWalkWarps, (kWalkSmemMax - fixed) / kWalkWarpSmem);
}

// A block's tables, tiles and barriers.
struct WalkBlock {
    LaneTab T;
    WalkRing ring;
    uint32_t ns;
};
template <int LOGR>
__device__ __forceinline__ WalkBlock walk_setup(const DevTables &t, bool backward, uint32_t wpb, uint8_t *sm, uint8_t *cls) {
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, cw = class_words(t);
    WalkBlock w;
    w.ns = (backward ? t.nbd : t.nfd) + 1;
    uint8_t *tiles = sm + ((1024 - (smem_u32(sm) & 1023)) & 1023);
    uint8_t *tab = tiles + wpb * 2 * kWalkTile;
    w.ring = WalkRing{tiles + warp * 2 * kWalkTile, smem_u32(tab + lane_table_bytes<LOGR>(t)) + warp * 16, 0};
    if (lane == 0 && warp < wpb) {
        mbar_init(w.ring.bars, 1);
        mbar_init(w.ring.bars + 8, 1);
        mbar_init_fence();
    }
    w.T.cls = cls;
    w.T.tab = smem_u32(tab) + (lane & ((1u << LOGR) - 1)) * 4;
    w.T.rowb = (cw * 4) << LOGR;
    stage_classes(t, cls);
    stage_lane_table<LOGR>(backward ? t.bc8 : t.fc8, w.ns * cw, tab);
    __syncthreads();
    return w;
}

// One 32-chunk tile of a text; false: a lost TMA completion, after which the
// loads in flight are given a bounded wait more.
template <int LOGR, bool OUT>
__device__ __forceinline__ bool walk_tile(const Params &p, WalkBlock &w, bool backward, uint64_t tile, const CUtensorMap *map,
                                          const CUtensorMap *fmap, const CUtensorMap *bmap) {
    const bool wide = (reinterpret_cast<uintptr_t>(p.x) & 31) == 0;
    const bool ok = backward ? walk_chunk<LOGR, false, OUT>(p, w.T, w.ns, tile, wide, map, bmap, w.ring)
                             : walk_chunk<LOGR, true, OUT>(p, w.T, w.ns, tile, wide, map, fmap, w.ring);
    __syncwarp();
    if (ok) return true;
    atomicExch(&p.w.flags[FLAG_INTERNAL], 1);
    for (uint32_t st = 0; st < 2; ++st) {
        bool done = false;
        for (uint32_t it = 0; it < kWaitLimit && !done; ++it)
            done = mbar_try_wait(w.ring.bars + 8 * st, (w.ring.phase >> st) & 1u);
    }
    return false;
}

template <int LOGR, bool OUT>
__global__ void __launch_bounds__(kWalkWarps * 32, 1)
    walk_kernel(const __grid_constant__ Params p, const __grid_constant__ CUtensorMap map,
                const __grid_constant__ StateMaps smaps) {
    extern __shared__ __align__(16) uint8_t sm[];
    __shared__ __align__(128) uint8_t cls[256];              // a fixed address: the lookups' offset is an immediate
    const bool pairs = !p.recognize, backward = pairs && (blockIdx.x & 1);
    const uint32_t warp = threadIdx.x >> 5, wpb = blockDim.x / 32;
    WalkBlock w = walk_setup<LOGR>(p.t, backward, wpb, sm, cls);
    pdl_wait();
    pdl_trigger();
    const uint64_t gblk = pairs ? blockIdx.x >> 1 : blockIdx.x, nblk = pairs ? gridDim.x >> 1 : gridDim.x;
    for (uint64_t t = (uint64_t)warp * nblk + gblk; t * 32 < p.c; t += nblk * wpb)
        if (!walk_tile<LOGR, OUT>(p, w, backward, t, &map, &smaps.f, &smaps.b)) break;
    if (OUT) bulk_wait_all();                                 // states written before the grid ends
}

// Every lane-walk group of a batch: a block takes tiles of one group's texts,
// its warps from the group's queue of its direction (the tiles differ in
// length and come longest first; dealt round-robin instead, 768 texts of 1 KiB
// to 4 MiB took 0.52 ms; from the queue, and with whole tiles, 0.39 ms).
template <int LOGR, bool OUT>
__device__ void walk_group(const WalkBatch &b, const WalkGroup &g, bool backward, uint8_t *sm, uint8_t *cls) {
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const size_t fixed = 1024 + lane_table_bytes<LOGR>(g.t);  // warps this group's tables leave room for
    const uint32_t wpb = min(blockDim.x / 32, (uint32_t)((b.walk_smem - fixed) / kWalkWarpSmem));
    WalkBlock w = walk_setup<LOGR>(g.t, backward, wpb, sm, cls);
    if (warp >= wpb) return;
    for (;;) {
        uint32_t t = 0;
        if (lane == 0) t = atomicAdd(g.queue + (backward ? 1 : 0), 1u);
        t = __shfl_sync(0xFFFFFFFFu, t, 0);
        if (t >= g.tiles) break;
        const uint32_t ti = text_of(g.rtile_base, g.nt, t);
        const Params &p = g.texts[ti];
        if (p.text_tma && lane == 0) {                        // maps in the descriptor area
            tensormap_acquire(p.tmaps);
            if (OUT) tensormap_acquire(p.tmaps + (backward ? 2 : 1));
        }
        __syncwarp();
        if (!walk_tile<LOGR, OUT>(p, w, backward, t - __ldg(g.rtile_base + ti), p.tmaps, p.tmaps + 1, p.tmaps + 2)) break;
    }
    if (OUT) bulk_wait_all();
}

template <bool OUT>
__global__ void __launch_bounds__(kWalkWarps * 32, 1) walk_batch_kernel(const __grid_constant__ WalkBatch b) {
    extern __shared__ __align__(16) uint8_t sm[];
    __shared__ __align__(128) uint8_t cls[256];
    const bool pairs = !b.recognize, backward = pairs && (blockIdx.x & 1);
    const WalkSpan sp = b.walk[pairs ? blockIdx.x >> 1 : blockIdx.x];
    const WalkGroup &g = b.groups[sp.group];
    switch (g.logr) {
        case 5: walk_group<5, OUT>(b, g, backward, sm, cls); break;
        case 4: walk_group<4, OUT>(b, g, backward, sm, cls); break;
        case 2: walk_group<2, OUT>(b, g, backward, sm, cls); break;
        default: walk_group<0, OUT>(b, g, backward, sm, cls); break;
    }
}

// Table copies: as many of 32, 16 or 4 as leave room for kWalkMinWarps warps.
// With few tiles per block the walk is one chain's latency, and copying the
// table costs more than its conflicts: one copy (heads and walk of log text: 64 KiB
// 30 us with one copy and 49 with 32, 1 MiB 30 and 55; above the line 4 MiB 35 and
// 40, 11 MiB and more by 32).  Random REs whose 32 copies leave 16 to 24 warps, 64
// MiB: 84 to 88 us with 32 copies, 90 with 16, 103 with 4.
constexpr uint32_t kWalkMinWarps = 12;
int walk_logr(const DevTables &t, uint64_t tiles, uint64_t blocks) {
    if (tiles <= 2 * blocks) return 0;
    return walk_wpb<5>(t) >= kWalkMinWarps ? 5 : walk_wpb<4>(t) >= kWalkMinWarps ? 4 : walk_wpb<2>(t) >= kWalkMinWarps ? 2 : 0;
}
template <int LOGR, bool OUT>
void walk_one(const Params &p, const CUtensorMap &map, const StateMaps &smaps, cudaStream_t s, int sm_count) {
    const uint64_t dirs = p.recognize ? 1 : 2, tiles = ((uint64_t)p.c + 31) / 32;
    const uint64_t per_dir = std::max<uint64_t>(1, std::min<uint64_t>(tiles, sm_count / dirs));
    const uint32_t wpb = (uint32_t)std::min<uint64_t>(walk_wpb<LOGR>(p.t), (tiles + per_dir - 1) / per_dir);
    static uint64_t attr_done = 0;
    allow_smem(walk_kernel<LOGR, OUT>, &attr_done, (int)kWalkSmemMax - 256);
    launch_dependent(walk_kernel<LOGR, OUT>, (uint32_t)(per_dir * dirs), wpb * 32,
                     1024 + lane_table_bytes<LOGR>(p.t) + wpb * kWalkWarpSmem, s, p, map, smaps);
}

template <bool OUT>
void walk_any(const Params &p, const CUtensorMap &map, const StateMaps &smaps, cudaStream_t s, int sm_count) {
    const uint64_t tiles = ((uint64_t)p.c + 31) / 32, blocks = sm_count / (p.recognize ? 1 : 2);
    switch (walk_logr(p.t, tiles, blocks)) {
        case 5: walk_one<5, OUT>(p, map, smaps, s, sm_count); break;
        case 4: walk_one<4, OUT>(p, map, smaps, s, sm_count); break;
        case 2: walk_one<2, OUT>(p, map, smaps, s, sm_count); break;
        default: walk_one<0, OUT>(p, map, smaps, s, sm_count); break;
    }
}

}  // namespace

int walk_copies(const DevTables &t, uint64_t tiles, uint64_t blocks) { return walk_logr(t, tiles, blocks); }
size_t walk_smem_bytes(const DevTables &t, int logr) {
    const size_t tab = logr == 5 ? lane_table_bytes<5>(t) : logr == 4 ? lane_table_bytes<4>(t)
                     : logr == 2 ? lane_table_bytes<2>(t) : lane_table_bytes<0>(t);
    return std::min<size_t>(kWalkSmemMax - 256, 1024 + tab + kWalkWarps * kWalkWarpSmem);
}
void launch_walk_batch(const WalkBatch &b, cudaStream_t s) {
    if (!b.n_walk) return;
    const uint32_t blocks = b.n_walk * (b.recognize ? 1 : 2);
    static uint64_t attr_out = 0, attr_rec = 0;
    if (b.recognize) {
        allow_smem(walk_batch_kernel<false>, &attr_rec, (int)kWalkSmemMax - 256);
        walk_batch_kernel<false><<<blocks, kWalkWarps * 32, b.walk_smem, s>>>(b);
    } else {
        allow_smem(walk_batch_kernel<true>, &attr_out, (int)kWalkSmemMax - 256);
        walk_batch_kernel<true><<<blocks, kWalkWarps * 32, b.walk_smem, s>>>(b);
    }
}

void launch_walk(const Params &p, const CUtensorMap &map, const StateMaps &smaps, cudaStream_t s, int sm_count) {
    if (p.mat) walk_any<true>(p, map, smaps, s, sm_count);
    else walk_any<false>(p, map, smaps, s, sm_count);
}

// Chunks the walk takes at once per direction (a lane each) on a full device.
uint64_t walk_lanes(const DevTables &t, bool recognize, int sm_count) {
    const uint64_t blocks = sm_count / (recognize ? 1 : 2);
    const int logr = walk_logr(t, ~0ull, blocks);
    return 32 * blocks * (logr == 5 ? walk_wpb<5>(t) : logr == 4 ? walk_wpb<4>(t) : logr == 2 ? walk_wpb<2>(t) : walk_wpb<0>(t));
}

}  // namespace slpf
