// Match extraction (arXiv 2503.06763, Sect. 4.2, "Match extraction",
// getMatches): the spans (i, j) of a group k -- pairs such that some syntax
// tree has the node k( ... )k over text[i:j] -- read off the clean SLPF.
//
// A segment is the parentheses and leaves before an end letter.  Column r's
// segments that hold a whole "k( ... )k" give (r, r).  Those whose last
// k-parenthesis is k( leave group k open; the visit then follows FolSeg arcs
// (Eq. folsegdef) column by column: segments without a k-parenthesis keep it
// open, and a segment whose first k-parenthesis is )k at column j closes it,
// giving (i, j).  The SLPF is clean, so each such path lies on a whole tree.
//
// A warp takes tiles of kTile start columns, kSubTile at a time, their columns
// staged in shared memory beside the block's copy of the tables (column
// dictionary, FolSeg).  Most columns open no group, so the lanes first mark
// the starts of the kSubTile columns by a flag per column id (or the masks
// themselves) and pack them into a list, and then a lane visits a start of the
// list.  A warp that visits 32 consecutive columns in step waits for the few
// of them that are starts (DNA stop codons: 1 column in 21).  A count pass, an
// exclusive scan of the per-tile counts and a write pass put the pairs in
// (i, j) order with no atomics; the total is reported even when the caller's
// buffer is smaller.  The count pass leaves a tile's spans as 32-bit records
// (start in the tile, length), up to kRecs of them, so the write pass only
// expands them; a tile with more spans, or longer ones, is visited again.
#include <algorithm>

#include "kernels.cuh"

namespace slpf {

constexpr uint32_t kScanBlock = 1024;

namespace {

constexpr uint32_t kTile = 2048;             // start columns per warp and count
constexpr uint32_t kSubTile = 512;           // staged and packed at once, kLane per lane
constexpr uint32_t kLane = kSubTile / 32;
constexpr uint32_t kAhead = 64;              // columns staged past them: most visits end within
constexpr uint32_t kMatchThreads = 256;
constexpr uint32_t kRecs = 256;              // records per tile: one span per 8 columns
constexpr uint32_t kRecLen = 21;             // bits of a record's length; the start above them
constexpr uint32_t kNoRecs = 0xFFFFFFFFu;    // in place of the first record: the tile has none
constexpr size_t kMatchDictMax = 48 * 1024, kMatchFolMax = 32 * 1024, kMatchFlagsMax = 16 * 1024;

// Tables of a block: in shared memory where they fit, else in global memory.
struct MatchTabs {
    const uint64_t *dict, *fol;
    const uint8_t *flags;                     // [dict_size + 1] 1: the column opens or holds the group; null: test the masks
    const uint8_t *tile;                      // this warp's staged columns
    uint64_t t0;                              // the first of them
    uint32_t cnt;                             // how many
};

// Segment set of the column with the stored value raw.
template <int W>
__device__ __forceinline__ void column_bits(const MatchArgs &a, const MatchTabs &T, uint64_t raw, uint64_t (&v)[W]) {
    if (a.kind == RE_SLPF_PAIRS) {                          // C_r = B_r ∩ B̂_r from the two state ids
        const uint64_t f = a.col_bytes == 4 ? raw & 0xFFFFu : raw & 0xFFFFFFFFull, b = a.col_bytes == 4 ? raw >> 16 : raw >> 32;
#pragma unroll
        for (int w = 0; w < W; ++w)
            v[w] = w < (int)a.W ? __ldg(a.fbits + f * a.W + w) & __ldg(a.bbits + b * a.W + w) : 0ull;
    } else if (a.kind == RE_SLPF_DICT) {
#pragma unroll
        for (int w = 0; w < W; ++w)                          // W rounds a.W up: the rows have stride a.W
            v[w] = (w < (int)a.W && raw && raw <= a.dict_size) ? T.dict[(size_t)(raw - 1) * a.W + w] : 0ull;
    } else {
        v[0] = raw;
#pragma unroll
        for (int w = 1; w < W; ++w) v[w] = 0;
    }
}

template <int CB> struct ColumnOf;
template <> struct ColumnOf<1> { using type = uint8_t; };
template <> struct ColumnOf<2> { using type = uint16_t; };
template <> struct ColumnOf<4> { using type = uint32_t; };
template <> struct ColumnOf<8> { using type = unsigned long long; };
// One step of a visit: the open set S moves over a column with stored value
// raw; true when the group closes there.  live: the set is not empty after.
template <int W>
__device__ __forceinline__ bool visit_step(const MatchArgs &a, const MatchTabs &T, uint64_t raw, uint64_t (&S)[W], bool &live) {
    uint64_t N[W], C[W];
#pragma unroll
    for (int w = 0; w < W; ++w) N[w] = 0;
#pragma unroll
    for (int w = 0; w < W; ++w) {
        uint64_t m = S[w];
        while (m) {
            const uint32_t q = 64 * w + (uint32_t)__ffsll((long long)m) - 1;
            m &= m - 1;
#pragma unroll
            for (int w2 = 0; w2 < W; ++w2)
                if (w2 < (int)a.W) N[w2] |= T.fol[q * a.W + w2];
        }
    }
    column_bits<W>(a, T, raw, C);
    bool close = false;
    live = false;
#pragma unroll
    for (int w = 0; w < W; ++w) {
        N[w] &= C[w];
        close |= (N[w] & a.close_first[w]) != 0;
        S[w] = N[w] & a.none[w];
        live |= S[w] != 0;
    }
    return close;
}

// A visit past the staged columns: from column r on, with the load of a
// step's column ahead of the step before it.
template <int W, int CB, typename F>
__device__ __forceinline__ void visit_on(const MatchArgs &a, const MatchTabs &T, uint64_t r, uint64_t (&S)[W], F &emit) {
    using C = typename ColumnOf<CB>::type;
    const C *cols = static_cast<const C *>(a.cols);
    uint64_t next = r < a.n ? __ldg(cols + r + 1) : 0;
    bool live = true;
#pragma unroll 1
    while (live && r < a.n) {
        const uint64_t raw = next;
        ++r;
        if (r < a.n) next = __ldg(cols + r + 1);
        if (visit_step<W>(a, T, raw, S, live)) emit(r);
    }
}

// The visit from the staged column d: emit(j - t0) for its matches (t0 + d, j)
// in j order.
template <int W, int CB, typename F>
__device__ __forceinline__ void visit(const MatchArgs &a, const MatchTabs &T, uint32_t d, F emit) {
    using C = typename ColumnOf<CB>::type;
    const C *tile = reinterpret_cast<const C *>(T.tile);
    uint64_t S[W];
    column_bits<W>(a, T, tile[d], S);
    bool whole = false, live = false;
#pragma unroll
    for (int w = 0; w < W; ++w) {
        whole |= (S[w] & a.whole[w]) != 0;
        S[w] &= a.open[w];
        live |= S[w] != 0;
    }
    if (whole) emit((uint64_t)d);
    while (live && d + 1 < T.cnt) {
        ++d;
        if (visit_step<W>(a, T, tile[d], S, live)) emit((uint64_t)d);
    }
    if (live && T.t0 + d < a.n) {
        auto on = [&](uint64_t r) { emit(r - T.t0); };
        visit_on<W, CB>(a, T, T.t0 + d, S, on);
    }
}

// Exclusive scan over the warp; total gets the sum.
template <typename V>
__device__ __forceinline__ V warp_exclusive(V c, V &total) {
    const uint32_t lane = threadIdx.x & 31;
    V s = c;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const V y = __shfl_up_sync(0xFFFFFFFFu, s, d);
        if ((int)lane >= d) s += y;
    }
    total = __shfl_sync(0xFFFFFFFFu, s, 31);
    return s - c;
}

// Bytes of shared memory a block's tables and its warps' columns take.
struct MatchLayout {
    uint32_t dict, fol, flags, tile, total;   // offsets; 0xFFFFFFFF: not staged
    uint32_t warp;                            // bytes per warp: columns, then the list of starts
};
__host__ __device__ inline MatchLayout match_layout(const MatchArgs &a) {
    MatchLayout L;
    uint32_t o = 0;
    const size_t dict = a.kind == RE_SLPF_DICT ? (size_t)a.dict_size * a.W * 8 : 0, fol = (size_t)a.ell * a.W * 8;
    const size_t flags = a.kind == RE_SLPF_DICT ? (size_t)a.dict_size + 1 : 0;
    L.dict = dict && dict <= kMatchDictMax ? o : 0xFFFFFFFFu;
    if (L.dict != 0xFFFFFFFFu) o += (uint32_t)dict;
    L.fol = fol <= kMatchFolMax ? o : 0xFFFFFFFFu;
    if (L.fol != 0xFFFFFFFFu) o += (uint32_t)fol;
    L.tile = (o + 15) & ~15u;
    L.warp = (kSubTile + kAhead) * a.col_bytes + kSubTile * 2;
    o = L.tile + (kMatchThreads / 32) * L.warp;
    L.flags = flags && flags <= kMatchFlagsMax ? o : 0xFFFFFFFFu;
    if (L.flags != 0xFFFFFFFFu) o += (uint32_t)flags;
    L.total = o;
    return L;
}

// The starts among this warp's kSubTile columns, packed in order into list;
// returns their number.  Lane l holds columns kLane * l .. of the subtile.
template <int W, int CB>
__device__ __forceinline__ uint32_t pack_starts(const MatchArgs &a, const MatchTabs &T, uint16_t *list) {
    using C = typename ColumnOf<CB>::type;
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t here = (uint32_t)min((uint64_t)kSubTile, a.n + 1 - T.t0);   // columns of the subtile
    const uint32_t mine = here > kLane * lane ? min(kLane, here - kLane * lane) : 0u;
    uint32_t starts = 0;                                      // bit j: column kLane * lane + j
    constexpr int V = 16 / CB;                                // columns per 16-byte vector
#pragma unroll
    for (int v = 0; v < (int)kLane / V; ++v) {
        union { uint4 q; C c[V]; } u;
        u.q = *reinterpret_cast<const uint4 *>(T.tile + (kLane * lane + V * v) * CB);
#pragma unroll
        for (int j = 0; j < V; ++j) {
            const uint64_t raw = u.c[j];
            bool on = false;
            if (T.flags) {
                on = raw <= a.dict_size && T.flags[raw];
            } else {
                uint64_t bits[W];
                if ((uint32_t)(V * v + j) < mine) {
                    column_bits<W>(a, T, raw, bits);
#pragma unroll
                    for (int w = 0; w < W; ++w) on |= (bits[w] & (a.open[w] | a.whole[w])) != 0;
                }
            }
            if (on) starts |= 1u << (V * v + j);
        }
    }
    starts &= mine >= 32 ? ~0u : (1u << mine) - 1;            // past the last column: stale bytes of the tile
    uint32_t n;
    uint32_t at = warp_exclusive<uint32_t>(__popc(starts), n);
    for (uint32_t m = starts; m; m &= m - 1) list[at++] = (uint16_t)(kLane * lane + __ffs(m) - 1);
    __syncwarp();
    return n;
}

// Count (WRITE = false): matches per tile into a.cnt, their records into
// a.recs.  Write: the pairs, each tile from its offset on.
template <int W, int CB, bool WRITE>
__global__ void __launch_bounds__(kMatchThreads) match_kernel(const __grid_constant__ MatchArgs a) {
    extern __shared__ __align__(16) uint8_t sm[];
    const MatchLayout L = match_layout(a);
    const bool ok = *a.status == RE_OK;
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    MatchTabs T;
    T.dict = L.dict == 0xFFFFFFFFu ? a.dict : reinterpret_cast<const uint64_t *>(sm + L.dict);
    T.fol = L.fol == 0xFFFFFFFFu ? a.folseg : reinterpret_cast<const uint64_t *>(sm + L.fol);
    T.flags = L.flags == 0xFFFFFFFFu ? nullptr : sm + L.flags;
    uint8_t *tile = sm + L.tile + warp * L.warp;
    uint16_t *list = reinterpret_cast<uint16_t *>(tile + (kSubTile + kAhead) * CB);
    T.tile = tile;
    if (ok) {
        if (L.dict != 0xFFFFFFFFu)
            for (uint32_t q = threadIdx.x; q < a.dict_size * a.W; q += blockDim.x)
                reinterpret_cast<uint64_t *>(sm + L.dict)[q] = __ldg(a.dict + q);
        if (L.fol != 0xFFFFFFFFu)
            for (uint32_t q = threadIdx.x; q < a.ell * a.W; q += blockDim.x)
                reinterpret_cast<uint64_t *>(sm + L.fol)[q] = __ldg(a.folseg + q);
        if (L.flags != 0xFFFFFFFFu)
            for (uint32_t q = threadIdx.x; q <= a.dict_size; q += blockDim.x) {
                uint64_t any = 0;
                for (uint32_t w = 0; q && w < a.W; ++w)
                    any |= __ldg(a.dict + (size_t)(q - 1) * a.W + w) & (a.open[w] | a.whole[w]);
                sm[L.flags + q] = any ? 1 : 0;
            }
    }
    __syncthreads();
    const bool vec = (reinterpret_cast<uintptr_t>(a.cols) & 15) == 0;
    const uint64_t warps = (uint64_t)gridDim.x * (kMatchThreads / 32);
    for (uint64_t g = (uint64_t)blockIdx.x * (kMatchThreads / 32) + warp; g < a.G; g += warps) {
        uint32_t *recs = a.recs ? a.recs + g * kRecs : nullptr;
        uint64_t off = 0;                                     // the tile's matches so far
        bool fit = recs != nullptr;                           // ... are all in its records
        const uint64_t first = WRITE ? a.cnt[g] + a.bsum[g / kScanBlock] : 0;   // matches before the tile
        if (WRITE) {
            const uint64_t after = g + 1 == a.G ? a.count[0] : a.cnt[g + 1] + a.bsum[(g + 1) / kScanBlock];
            off = after - first;
            if (off == 0 || first >= a.cap) continue;
            if (recs && off <= kRecs && recs[0] != kNoRecs) {
                const uint32_t m = (uint32_t)min(off, a.cap - first);
                for (uint32_t q = lane; q < m; q += 32) {
                    const uint32_t r = recs[q];
                    const uint64_t i = g * kTile + (r >> kRecLen);
                    a.pairs[2 * (first + q)] = i;
                    a.pairs[2 * (first + q) + 1] = i + (r & ((1u << kRecLen) - 1));
                }
                continue;
            }
            off = 0;
        }
        for (uint32_t sub = 0; ok && sub < kTile / kSubTile; ++sub) {
            T.t0 = g * kTile + sub * kSubTile;
            if (T.t0 > a.n) break;                            // warp-uniform
            T.cnt = (uint32_t)min((uint64_t)(kSubTile + kAhead), a.n + 1 - T.t0);
            __syncwarp();                                     // the last subtile's visits are over
            const uint8_t *src = static_cast<const uint8_t *>(a.cols) + T.t0 * CB;
            const uint32_t bytes = T.cnt * CB, from = vec ? bytes & ~15u : 0u;
            for (uint32_t q = 16 * lane; q < from; q += 512)
                *reinterpret_cast<uint4 *>(tile + q) = __ldg(reinterpret_cast<const uint4 *>(src + q));
            for (uint32_t q = from + lane; q < bytes; q += 32) tile[q] = __ldg(src + q);
            __syncwarp();
            const uint32_t n = pack_starts<W, CB>(a, T, list);
            for (uint32_t q0 = 0; q0 < n; q0 += 32) {
                const uint32_t q = q0 + lane;
                const uint32_t d = q < n ? list[q] : 0u;
                uint64_t c = 0, len0 = 0;                     // matches of this start, the first one's length
                bool big = false;
                if (q < n)
                    visit<W, CB>(a, T, d, [&](uint64_t j) {
                        if (c == 0) len0 = j - d;
                        big |= j - d >= (1u << kRecLen) - 1;
                        ++c;
                    });
                uint64_t o = off;
                if (__any_sync(0xFFFFFFFFu, c >> 24)) {
                    uint64_t t;
                    o += warp_exclusive<uint64_t>(c, t);
                    off += t;
                } else {
                    uint32_t t;
                    o += warp_exclusive<uint32_t>((uint32_t)c, t);
                    off += t;
                }
                if (!WRITE) {
                    fit = fit && off <= kRecs && !__any_sync(0xFFFFFFFFu, big);
                    const uint32_t key = (sub * kSubTile + d) << kRecLen;
                    if (!fit) {
                    } else if (c == 1) {
                        recs[o] = key | (uint32_t)len0;
                    } else if (c) {
                        visit<W, CB>(a, T, d, [&](uint64_t j) { recs[o++] = key | (uint32_t)(j - d); });
                    }
                } else if (c) {
                    const uint64_t i = T.t0 + d;
                    visit<W, CB>(a, T, d, [&](uint64_t j) {
                        if (first + o < a.cap) { a.pairs[2 * (first + o)] = i; a.pairs[2 * (first + o) + 1] = T.t0 + j; }
                        ++o;
                    });
                }
            }
        }
        if (!WRITE && lane == 0) {
            a.cnt[g] = off;
            if (recs && !fit) recs[0] = kNoRecs;
        }
    }
}

// Exclusive scan of kScanBlock values per block (in place); block totals to out.
__global__ void scan_block_kernel(uint64_t *v, uint64_t n, uint64_t *out) {
    __shared__ uint64_t warp_tot[kScanBlock / 32];
    const uint64_t j = (uint64_t)blockIdx.x * kScanBlock + threadIdx.x;
    const uint64_t x = j < n ? v[j] : 0;
    const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint64_t s = x;                                          // inclusive within the warp
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint64_t y = __shfl_up_sync(0xFFFFFFFFu, s, d);
        if ((int)lane >= d) s += y;
    }
    if (lane == 31) warp_tot[wid] = s;
    __syncthreads();
    if (wid == 0) {
        uint64_t t = warp_tot[lane];
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint64_t y = __shfl_up_sync(0xFFFFFFFFu, t, d);
            if ((int)lane >= d) t += y;
        }
        warp_tot[lane] = t;                                  // inclusive warp totals
    }
    __syncthreads();
    const uint64_t before = (wid ? warp_tot[wid - 1] : 0) + s - x;
    if (j < n) v[j] = before;
    if (threadIdx.x == kScanBlock - 1) out[blockIdx.x] = warp_tot[31];
}

// Exclusive scan of the block totals by one block, kScanBlock at a time, and their sum.
__global__ void scan_totals_kernel(uint64_t *v, uint64_t n, uint64_t *total) {
    __shared__ uint64_t carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (uint64_t base = 0; base < n; base += kScanBlock) {
        const uint64_t j = base + threadIdx.x;
        const uint64_t x = j < n ? v[j] : 0;
        uint64_t s = x;
        for (uint32_t d = 1; d < kScanBlock; d <<= 1) {     // simple Hillis-Steele in shared memory
            __shared__ uint64_t buf[kScanBlock];
            buf[threadIdx.x] = s;
            __syncthreads();
            if (threadIdx.x >= d) s += buf[threadIdx.x - d];
            __syncthreads();
        }
        const uint64_t c0 = carry;
        if (j < n) v[j] = c0 + s - x;
        __syncthreads();
        if (threadIdx.x == kScanBlock - 1) carry = c0 + s;
        __syncthreads();
    }
    if (threadIdx.x == 0) *total = carry;
}

}  // namespace

namespace {
// Workspace: per-tile counts, block sums of the scan, the records.  Without room
// for the records the write pass visits every tile again.
struct MatchWorkspace {
    uint64_t G, nb;
    size_t bsum, recs, bytes;
    explicit MatchWorkspace(uint64_t n) {
        auto up = [](size_t v) { return (v + 255) & ~(size_t)255; };
        G = n / kTile + 1;                                    // tiles of kTile start columns, a warp each
        nb = (G + kScanBlock - 1) / kScanBlock;
        bsum = up(G * 8);
        recs = bsum + up(nb * 8);
        bytes = recs + up(G * kRecs * 4);
    }
};
}  // namespace

size_t match_workspace_bytes(uint64_t n, bool records) {
    const MatchWorkspace w(n);
    return records ? w.bytes : w.recs;
}

template <int W, int CB>
static void run_matches(const MatchArgs &a, uint64_t nb, cudaStream_t s, int sm_count) {
    const size_t smem = match_layout(a).total;
    static uint64_t attr_count = 0, attr_write = 0;
    allow_smem(match_kernel<W, CB, false>, &attr_count);
    allow_smem(match_kernel<W, CB, true>, &attr_write);
    int pc = 1, pw = 1;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&pc, match_kernel<W, CB, false>, kMatchThreads, smem);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&pw, match_kernel<W, CB, true>, kMatchThreads, smem);
    const uint64_t want = (a.G + kMatchThreads / 32 - 1) / (kMatchThreads / 32);
    const uint64_t gc = std::min<uint64_t>(want, (uint64_t)std::max(pc, 1) * sm_count);
    const uint64_t gw = std::min<uint64_t>(want, (uint64_t)std::max(pw, 1) * sm_count);
    match_kernel<W, CB, false><<<(uint32_t)gc, kMatchThreads, smem, s>>>(a);
    scan_block_kernel<<<(uint32_t)nb, kScanBlock, 0, s>>>(a.cnt, a.G, a.bsum);
    scan_totals_kernel<<<1, kScanBlock, 0, s>>>(a.bsum, nb, a.count);
    match_kernel<W, CB, true><<<(uint32_t)gw, kMatchThreads, smem, s>>>(a);
}

template <int W>
static void matches_of_width(const MatchArgs &a, uint64_t nb, cudaStream_t s, int sm_count) {
    switch (a.col_bytes) {
        case 1: run_matches<W, 1>(a, nb, s, sm_count); break;
        case 2: run_matches<W, 2>(a, nb, s, sm_count); break;
        case 4: run_matches<W, 4>(a, nb, s, sm_count); break;
        default: run_matches<W, 8>(a, nb, s, sm_count); break;
    }
}

// DNA 64 MiB, the stop codon group (3.1 M spans): count pass 112 us, scan 6,
// write pass 27 us, where a lane per column in both passes took 0.79 and 1.42
// ms.  The count pass is bound by instruction issue (74 % of the slots; 740
// instructions per warp and 512 columns), the write pass by its 50 MB of pairs.
void launch_matches(MatchArgs a, void *ws, size_t ws_bytes, cudaStream_t s, int sm_count) {
    const MatchWorkspace w(a.n);
    uint8_t *p = static_cast<uint8_t *>(ws);
    const uint64_t nb = w.nb;
    a.G = w.G;
    a.cnt = reinterpret_cast<uint64_t *>(p);
    a.bsum = reinterpret_cast<uint64_t *>(p + w.bsum);
    a.recs = ws_bytes >= w.bytes ? reinterpret_cast<uint32_t *>(p + w.recs) : nullptr;
    if (a.W <= 1) matches_of_width<1>(a, nb, s, sm_count);
    else if (a.W <= 2) matches_of_width<2>(a, nb, s, sm_count);
    else if (a.W <= 4) matches_of_width<4>(a, nb, s, sm_count);
    else matches_of_width<8>(a, nb, s, sm_count);
}

}  // namespace slpf
