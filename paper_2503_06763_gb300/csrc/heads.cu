// Speculative chunk heads (arXiv 2503.06763, Eq. reacher and Sect. 4.3; see
// walk.cuh).
//
// For every chunk and direction the speculative runs are walked from the
// chunk's edge until the live ones are in one state, checked every kUnit
// bytes; the state, the unit boundary it holds at and the slots alive there
// are recorded.  The chunk's slots are those of the class pair around its edge
// (the start sets after the boundary byte, the last-character filter of Sect.
// 6).  A chunk whose runs never meet (kind 1) is walked to its end here and
// leaves every slot's end state to the join.
//
// A block takes up to kHeadChunks chunks of one direction.  Their first bytes
// come into shared memory together (the walk itself then waits for no text:
// on most chunks it ends within them).  A chunk with more slots than a lane
// holds in registers (kRuns) is first taken by a whole warp, a lane per slot,
// until few enough states are left: on log text 8 slots on average (at most
// 23) are 2.4 states after 4 bytes and 1.6 after 32, so that is a few bytes.
// Then a lane walks the chunk's runs.  The loops are rolled, a word of text a
// turn: unrolled over a unit the kernel spent a third of its time fetching
// instructions.
#include <algorithm>
#include <type_traits>

#include "walk.cuh"

namespace slpf {
namespace {

constexpr uint32_t kHeadThreads = 256;
constexpr uint32_t kHeadChunks = 64;        // chunks a block takes at once, at most
constexpr uint32_t kHeadWindow = 144;       // bytes of a chunk staged, from its edge (a multiple of 16)
constexpr uint32_t kHeadStride = 148;       // their stride: an odd number of words, so lanes hit different banks
constexpr int kRuns = 4;
constexpr uint32_t kWideBytes = 32;         // bytes a warp walks a chunk's slots
constexpr uint32_t kWideRuns = 8;           // runs a lane takes on from there

// Drop dead runs and merge runs in equal states (their slot sets are joined);
// unused runs hold the empty state.
__device__ __forceinline__ void merge_runs(uint32_t (&s)[kRuns], uint32_t (&k)[kRuns], uint32_t &cnt) {
    uint32_t ns[kRuns] = {}, nk[kRuns] = {};
    cnt = 0;
#pragma unroll
    for (int j = 0; j < kRuns; ++j) {
        if (!s[j]) continue;
        bool merged = false;
#pragma unroll
        for (int q = 0; q < j; ++q)
            if (q < (int)cnt && ns[q] == s[j]) { nk[q] |= k[j]; merged = true; }
        if (merged) continue;
#pragma unroll
        for (int q = 0; q <= j; ++q)
            if (q == (int)cnt) { ns[q] = s[j]; nk[q] = k[j]; }
        ++cnt;
    }
#pragma unroll
    for (int j = 0; j < kRuns; ++j) { s[j] = ns[j]; k[j] = nk[j]; }
}

// The chunks of a kernel: one text's, or those of every text of a batch group.
struct OneText {
    const Params &p;
    __device__ const DevTables &tables() const { return p.t; }
    __device__ const Params &text(uint32_t) const { return p; }
    __device__ uint32_t index(uint64_t first, uint32_t q, uint32_t) const { return (uint32_t)(first + q); }
    __device__ uint32_t find(uint64_t) const { return 0; }
};
struct GroupTexts {
    const WalkGroup &g;
    __device__ const DevTables &tables() const { return g.t; }
    __device__ const Params &text(uint32_t ti) const { return g.texts[ti]; }
    __device__ uint32_t index(uint64_t first, uint32_t q, uint32_t ti) const { return (uint32_t)(first + q - __ldg(g.chunk_base + ti)); }
    __device__ uint32_t find(uint64_t chunk) const { return text_of(g.chunk_base, g.nt, chunk); }
};

struct HeadShared {
    uint32_t ti[kHeadChunks];                // the text of each chunk of the round
    uint8_t text[kHeadChunks * kHeadStride];
    uint32_t s[kRuns][kHeadChunks], k[kWideRuns][kHeadChunks], cnt[kHeadChunks], col[kHeadChunks];
    uint8_t s8[kWideRuns][kHeadChunks];      // states of a chunk with more than kRuns runs, their slot sets in k
    uint16_t wide[kHeadChunks];              // chunks of this round with more than kRuns slots: slots << 8 | chunk
    uint32_t pr[kHeadChunks], nwide;
};

// The chunk of slot q of a round, and where its staged window starts.
template <bool FWD> struct HeadChunk {
    uint64_t base;
    uint32_t i, len, win;                    // window: bytes [win, win + kHeadWindow) of the chunk, inside it
    __device__ HeadChunk(const Params &p, uint32_t chunk) {
        i = chunk;
        base = (uint64_t)i * p.k;
        len = chunk_len(p, i);
        win = FWD || len <= kHeadWindow - 15 ? 0u : (len - (kHeadWindow - 15)) & ~15u;
    }
};

// One byte, then four bytes of text, for the first W of a lane's runs.
template <int W>
__device__ __forceinline__ void head_byte(const LaneTab &T, uint32_t byte, uint32_t (&s)[kRuns]) {
    const uint32_t col = lane_col<0>(T, byte);
#pragma unroll
    for (int j = 0; j < W; ++j) s[j] = lds8(s[j] * T.rowb + col);
}
template <bool FWD, int W>
__device__ __forceinline__ void head_word(const LaneTab &T, uint32_t w, uint32_t (&s)[kRuns]) {
#pragma unroll
    for (int q = 0; q < 4; ++q) head_byte<W>(T, __byte_perm(w, 0u, 0x4440u | (uint32_t)(FWD ? q : 3 - q)), s);
}

// Eight runs of a lane over columns [c, to) (right to left where not FWD): a state
// is a byte, and the eight are kept in two words.
template <bool FWD>
__device__ __forceinline__ void walk_eight(const LaneTab &T, const uint8_t *x, uint32_t len, uint32_t &c, uint32_t to,
                                           uint32_t (&s)[2]) {
    auto step = [&](uint32_t byte) {
        const uint32_t col = lane_col<0>(T, byte);
        uint32_t v[8];
#pragma unroll
        for (uint32_t u = 0; u < 8; ++u) v[u] = lds8(__byte_perm(s[u >> 2], 0u, 0x4440u | (u & 3)) * T.rowb + col);
#pragma unroll
        for (uint32_t h = 0; h < 2; ++h)
            s[h] = __byte_perm(__byte_perm(v[4 * h], v[4 * h + 1], 0x0040u), __byte_perm(v[4 * h + 2], v[4 * h + 3], 0x0040u), 0x5410u);
    };
#pragma unroll 1
    while (c != to && (s[0] | s[1])) {
        const uint32_t left = FWD ? to - c : c - to;
        if ((c & 3) == 0 && left >= 4) {
            const uint32_t a4 = FWD ? c : c - 4;
            if ((c & 127) == 0 && (FWD ? len - c : c) > 256) prefetch_l2(x + (FWD ? c + 128 : c - 256));
            const uint32_t w = __ldg(reinterpret_cast<const uint32_t *>(x + a4));
#pragma unroll
            for (int q = 0; q < 4; ++q) step(__byte_perm(w, 0u, 0x4440u | (uint32_t)(FWD ? q : 3 - q)));
            c = FWD ? c + 4 : c - 4;
        } else {
            step(__ldg(x + (FWD ? c : c - 1)));
            c = FWD ? c + 1 : c - 1;
        }
    }
    c = to;                                                   // no run was left
}
__device__ __forceinline__ uint32_t state_of(const uint32_t (&s)[2], uint32_t u) { return (s[u >> 2] >> (8 * (u & 3))) & 0xFFu; }

// A chunk with more than kRuns and at most kWideRuns runs after kWideBytes: a lane
// goes on with them, equal ones joined after every unit, until kRuns are left
// (returned in S) or the chunk ends (every slot's end state written).  A warp per
// chunk going on to that point, most of its lanes idle, made the heads of 64 MiB of
// a's under twenty (c{6}) 3.4 ms (0.45 now); the genome RE, whose runs meet after some
// 450 bytes, has 5 to 8 of them for a while (256 MiB by the lane walk 778 us, and 1554
// with every such chunk walked to its end).
template <bool FWD>
__device__ void eight_runs(const LaneTab &T, HeadShared &S, const uint8_t *x, uint32_t len, uint32_t q, uint32_t ms, uint32_t *R) {
    uint32_t s[2], c = S.col[q], n = kWideRuns;
#pragma unroll
    for (uint32_t u = 0; u < 8; ++u) s[u >> 2] = (u & 3 ? s[u >> 2] : 0u) | (uint32_t)S.s8[u][q] << (8 * (u & 3));
    while ((FWD ? c < len : c > 0) && n > (uint32_t)kRuns) {
        walk_eight<FWD>(T, x, len, c, FWD ? min((c / kUnit + 1) * kUnit, len) : (c - 1) / kUnit * kUnit, s);
        n = 0;
#pragma unroll
        for (uint32_t u = 0; u < 8; ++u) {
            const uint32_t v = state_of(s, u);
            bool own = v != 0;
#pragma unroll
            for (uint32_t e = 0; e < u; ++e)
                if (v && state_of(s, e) == v) {
                    S.k[e][q] |= S.k[u][q];
                    s[u >> 2] &= ~(0xFFu << (8 * (u & 3)));
                    own = false;
                    break;
                }
            n += own;
        }
    }
    S.col[q] = c;
    S.cnt[q] = min(n, (uint32_t)kRuns + 1);
    uint32_t at = 0;
    if (n <= (uint32_t)kRuns) {
#pragma unroll
        for (uint32_t u = 0; u < 8; ++u)
            if (state_of(s, u)) { S.s[at][q] = state_of(s, u); S.k[at][q] = S.k[u][q]; ++at; }
        for (; at < (uint32_t)kRuns; ++at) S.s[at][q] = S.k[at][q] = 0;
    } else {
        for (uint32_t j = 0; j < ms; ++j) {
            uint32_t v = 0;
#pragma unroll
            for (uint32_t u = 0; u < 8; ++u)
                if (state_of(s, u) && (S.k[u][q] >> j & 1u)) v = state_of(s, u);
            R[j] = v;
        }
    }
}

// The end states of a chunk's slots, eight at a time from its edge, by a lane: where
// even more runs are apart after kWideBytes.
template <bool FWD>
__device__ void slots_to_end(const LaneTab &T, const uint8_t *x, uint32_t len, const uint32_t *starts, uint32_t m,
                             uint32_t ms, uint32_t *R) {
#pragma unroll 1
    for (uint32_t j = 0; j < ms; j += 8) {
        uint32_t s[2] = {0, 0}, c = FWD ? 1u : len - 1;
#pragma unroll
        for (uint32_t u = 0; u < 8; ++u)
            if (j + u < m) s[u >> 2] |= __ldg(starts + j + u) << (8 * (u & 3));
        walk_eight<FWD>(T, x, len, c, FWD ? len : 0u, s);
#pragma unroll
        for (uint32_t u = 0; u < 8; ++u)
            if (j + u < ms) R[j + u] = state_of(s, u);
    }
}

// A round of a block: chunks first .. first + cnt - 1 (cnt <= per).
template <bool FWD, typename Src>
__device__ void head_round(const Src &src, const LaneTab &T, HeadShared &S, uint64_t first, uint32_t cnt) {
    const DevTables &t = src.tables();
    const uint32_t ms = FWD ? t.msf : t.msb;
    const uint32_t *starts = FWD ? t.fSlotStart : t.bSlotStart;
    if (threadIdx.x == 0) S.nwide = 0;
    if (threadIdx.x < cnt) S.ti[threadIdx.x] = src.find(first + threadIdx.x);
    __syncthreads();
    auto text_at = [&](uint32_t q) -> const Params & { return src.text(S.ti[q]); };
    auto chunk_at = [&](uint32_t q) { return HeadChunk<FWD>(text_at(q), src.index(first, q, S.ti[q])); };
    // text windows, 16 bytes a thread
    for (uint32_t q = threadIdx.x; q < cnt * (kHeadWindow / 16); q += blockDim.x) {
        const Params &p = text_at(q / (kHeadWindow / 16));
        const HeadChunk<FWD> c = chunk_at(q / (kHeadWindow / 16));
        const uint32_t at = 16 * (q % (kHeadWindow / 16));
        if (c.win + at < c.len) {
            const uint4 v = load16(p.x, p.n, c.base + c.win + at);
            uint32_t *d = reinterpret_cast<uint32_t *>(S.text + (q / (kHeadWindow / 16)) * kHeadStride + at);
            d[0] = v.x; d[1] = v.y; d[2] = v.z; d[3] = v.w;
        }
    }
    __syncthreads();
    // slots of each chunk
    bool exact = false;
    if (threadIdx.x < cnt) {
        const uint32_t q = threadIdx.x;
        const Params &p = text_at(q);
        const HeadChunk<FWD> c = chunk_at(q);
        exact = FWD ? (c.i == 0 && !(p.shard & SHARD_PREV)) : (c.i == p.c - 1 && !(p.shard & SHARD_NEXT));
        uint32_t m = 0;
        if (!exact) {
            const uint64_t e = FWD ? c.base : c.base + c.len;    // the edge
            const uint32_t pr = __ldg(t.cls + __ldg(p.x + e - 1)) * t.ncls + __ldg(t.cls + __ldg(p.x + e));
            m = __ldg((FWD ? t.fSlotCount : t.bSlotCount) + pr);
            S.pr[q] = pr;
            if (m > (uint32_t)kRuns) S.wide[atomicAdd(&S.nwide, 1u)] = (uint16_t)(m << 8 | q);
            else
                for (uint32_t j = 0; j < (uint32_t)kRuns; ++j) {
                    S.s[j][q] = j < m ? __ldg(starts + (size_t)pr * ms + j) : 0u;
                    S.k[j][q] = 1u << j;
                }
        }
        S.cnt[q] = m > (uint32_t)kRuns ? 0u : m;
        S.col[q] = FWD ? 1u : c.len - 1;                      // the slots' states include the edge byte
    }
    __syncthreads();
    const uint32_t lane = threadIdx.x & 31;
    // chunks with more slots than a lane holds: a warp each, a lane per slot
    for (uint32_t r = threadIdx.x >> 5; r < S.nwide; r += blockDim.x / 32) {
        const uint32_t q = S.wide[r] & 0xFFu, m = S.wide[r] >> 8;
        const Params &p = text_at(q);
        const HeadChunk<FWD> ch = chunk_at(q);
        uint32_t v = lane < m ? __ldg(starts + (size_t)S.pr[q] * ms + lane) : 0u, c = FWD ? 1u : ch.len - 1;
        for (;;) {
            // to a multiple of four bytes, or the chunk's end; a chunk of one byte starts at its end
            // (backward c is 0 then), its slots' states are its end states
            const uint32_t to = FWD ? min((c + 4) & ~3u, ch.len) : (max(c, 1u) - 1) & ~3u;
            while (c != to) {
                const uint32_t at = FWD ? c : c - 1, w = at - ch.win;
                v = lane_step<0>(T, v, w < kHeadWindow ? S.text[q * kHeadStride + w] : __ldg(p.x + ch.base + at));
                c = FWD ? c + 1 : c - 1;
            }
            const unsigned same = __match_any_sync(0xFFFFFFFFu, v);
            const bool is_lead = v != 0 && lane == (uint32_t)__ffs(same) - 1;
            const unsigned lead = __ballot_sync(0xFFFFFFFFu, is_lead);
            const uint32_t n = __popc(lead);
            if (n <= (uint32_t)kRuns) {
                const uint32_t at = __popc(lead & ((1u << lane) - 1));
                if (is_lead) { S.s[at][q] = v; S.k[at][q] = same; }
                if (lane >= n && lane < (uint32_t)kRuns) { S.s[lane][q] = 0; S.k[lane][q] = 0; }
                if (lane == 0) { S.cnt[q] = n; S.col[q] = c; }
                break;
            }
            if (FWD ? c >= ch.len : c == 0) {                 // never met: every slot's end state
                if (lane < ms) ((FWD ? p.w.Rf : p.w.Rb) + (size_t)ch.i * ms)[lane] = v;
                if (lane == 0) { S.cnt[q] = kRuns + 1; S.col[q] = c; }
                break;
            }
            if ((FWD ? c : ch.len - c) >= kWideBytes) {       // a lane takes the runs, or all slots from the edge
                if (n <= kWideRuns) {
                    const uint32_t at = __popc(lead & ((1u << lane) - 1));
                    if (is_lead) { S.s8[at][q] = (uint8_t)v; S.k[at][q] = same; }
                    if (lane >= n && lane < kWideRuns) { S.s8[lane][q] = 0; S.k[lane][q] = 0; }
                }
                if (lane == 0) { S.cnt[q] = n <= kWideRuns ? kRuns + 3 : kRuns + 2; S.col[q] = c; }
                break;
            }
        }
    }
    __syncthreads();
    // a lane per chunk
    if (threadIdx.x < ((cnt + 31) & ~31u)) {
        const uint32_t q = threadIdx.x;
        const bool valid = q < cnt;
        const Params &p = text_at(valid ? q : 0);
        const HeadChunk<FWD> ch = chunk_at(valid ? q : 0);
        const uint32_t nU = (ch.len + kUnit - 1) / kUnit;
        uint32_t s[kRuns], k[kRuns], n = 0, c = 0, conv = FWD ? 0 : nU, kind = 0;
        bool open = false, all = false;                       // all: every slot's end state is written already
#pragma unroll
        for (int j = 0; j < kRuns; ++j) s[j] = k[j] = 0;
        if (valid && exact) {                                 // J_0 = I, or F past the last chunk
            s[0] = FWD ? t.fI : t.bF;
            k[0] = 1;
        } else if (valid) {
            n = S.cnt[q];
            c = S.col[q];
            if (n > (uint32_t)kRuns + 1) {
                uint32_t *R = (FWD ? p.w.Rf : p.w.Rb) + (size_t)ch.i * ms;
                if (n == kRuns + 3) {
                    eight_runs<FWD>(T, S, p.x + ch.base, ch.len, q, ms, R);
                    n = S.cnt[q];
                    c = S.col[q];
                } else {
                    slots_to_end<FWD>(T, p.x + ch.base, ch.len, starts + (size_t)S.pr[q] * ms,
                                      __ldg((FWD ? t.fSlotCount : t.bSlotCount) + S.pr[q]), ms, R);
                }
            }
            all = n > (uint32_t)kRuns;
            open = !all && (FWD ? c < ch.len : c > 0);
#pragma unroll
            for (int j = 0; j < kRuns; ++j)
                if (!all) { s[j] = S.s[j][q]; k[j] = S.k[j][q]; }
            if (!open) {                                      // walked to the chunk's end
                conv = FWD ? nU : 0;
                kind = n > 1 ? 1u : 0u;
            }
        }
        const uint8_t *text = S.text + q * kHeadStride;
        while (__any_sync(0xFFFFFFFFu, open)) {
            const uint32_t wm = __reduce_max_sync(0xFFFFFFFFu, open ? n : 0u);
            if (open) {                                       // one unit, or what is left of it
                const uint32_t to = FWD ? min((c / kUnit + 1) * kUnit, ch.len) : (c - 1) / kUnit * kUnit;
                auto go = [&](auto width) {
                    constexpr int Wd = decltype(width)::value;
#pragma unroll 1
                    while (c != to) {
                        const uint32_t left = FWD ? to - c : c - to, at = FWD ? c : c - 1;
                        if ((c & 3) == 0 && left >= 4) {      // four bytes
                            const uint32_t a4 = FWD ? c : c - 4, w = a4 - ch.win;
                            const uint32_t x = w < kHeadWindow ? *reinterpret_cast<const uint32_t *>(text + w)
                                                               : __ldg(reinterpret_cast<const uint32_t *>(p.x + ch.base + a4));
                            head_word<FWD, Wd>(T, x, s);
                            c = FWD ? c + 4 : c - 4;
                        } else {
                            const uint32_t w = at - ch.win;
                            head_byte<Wd>(T, w < kHeadWindow ? text[w] : __ldg(p.x + ch.base + at), s);
                            c = FWD ? c + 1 : c - 1;
                        }
                    }
                };
                if (wm <= 1) go(std::integral_constant<int, 1>{});
                else if (wm <= 2) go(std::integral_constant<int, 2>{});
                else go(std::integral_constant<int, kRuns>{});
                merge_runs(s, k, n);
                const bool end = FWD ? c >= ch.len : c == 0;
                if (n <= 1 || end) {
                    open = false;
                    conv = FWD ? (c + kUnit - 1) / kUnit : c / kUnit;
                    kind = n > 1 ? 1u : 0u;
                }
            }
        }
        if (valid) {
            if (kind && !all) {
                uint32_t *R = (FWD ? p.w.Rf : p.w.Rb) + (size_t)ch.i * ms;
                for (uint32_t j = 0; j < ms; ++j) {
                    uint32_t v = 0;
#pragma unroll
                    for (int r = 0; r < kRuns; ++r)
                        if ((k[r] >> j) & 1u) v = s[r];
                    R[j] = v;
                }
            }
            (FWD ? p.w.fconv : p.w.bconv)[ch.i] = conv;
            (FWD ? p.w.fnrec : p.w.bnrec)[ch.i] = s[0];
            (FWD ? p.w.fhit : p.w.bhit)[ch.i] = k[0];
            (FWD ? p.w.fkind : p.w.bkind)[ch.i] = kind;
        }
    }
    __syncthreads();                                          // S is refilled next
}

// Even blocks walk heads forward, odd ones backward (all forward for the
// recognizer); a block stages its direction's table.
__global__ void __launch_bounds__(kHeadThreads) heads_kernel(const __grid_constant__ Params p, uint32_t per) {
    extern __shared__ __align__(16) uint8_t sm[];
    __shared__ __align__(128) uint8_t cls[256];
    __shared__ HeadShared S;
    pdl_trigger();
    if (blockIdx.x == 0) {                                    // the join's flags: read by the kernels after this one
        if (threadIdx.x < FLAG_COUNT) p.w.flags[threadIdx.x] = threadIdx.x < 2 ? (int32_t)p.c : 0;
        if (threadIdx.x >= 32 && threadIdx.x < 32 + kScanWords) p.w.scan[threadIdx.x - 32] = 0;
    }
    const bool pairs = !p.recognize, backward = pairs && (blockIdx.x & 1);
    const uint32_t cw = class_words(p.t);
    const LaneTab T{smem_u32(sm), cls, cw * 4};
    stage_classes(p.t, cls);
    stage_lane_table<0>(backward ? p.t.bc8 : p.t.fc8, (backward ? p.t.nb : p.t.nf) * cw, sm);
    const uint64_t blk = pairs ? blockIdx.x >> 1 : blockIdx.x, nblk = pairs ? gridDim.x >> 1 : gridDim.x;
    const OneText src{p};
    for (uint64_t first = blk * per; first < p.c; first += nblk * per) {   // head_round's first barrier: the tables are staged
        const uint32_t cnt = (uint32_t)min((uint64_t)per, p.c - first);
        if (backward) head_round<false>(src, T, S, first, cnt);
        else head_round<true>(src, T, S, first, cnt);
    }
}

// Every lane-walk group of a batch: a block takes rounds of one group's chunks.
__global__ void __launch_bounds__(kHeadThreads, 8) heads_batch_kernel(const __grid_constant__ WalkBatch b) {
    extern __shared__ __align__(16) uint8_t sm[];
    __shared__ __align__(128) uint8_t cls[256];
    __shared__ HeadShared S;
    const bool pairs = !b.recognize, backward = pairs && (blockIdx.x & 1);
    const WalkSpan w = b.heads[pairs ? blockIdx.x >> 1 : blockIdx.x];
    const WalkGroup &g = b.groups[w.group];
    const uint32_t cw = class_words(g.t);
    const LaneTab T{smem_u32(sm), cls, cw * 4};
    stage_classes(g.t, cls);
    stage_lane_table<0>(backward ? g.t.bc8 : g.t.fc8, (backward ? g.t.nb : g.t.nf) * cw, sm);
    const GroupTexts src{g};
    for (uint64_t first = (uint64_t)w.idx * g.per; first < g.chunks; first += (uint64_t)w.cnt * g.per) {
        const uint32_t cnt = (uint32_t)min((uint64_t)g.per, g.chunks - first);
        if (backward) head_round<false>(src, T, S, first, cnt);
        else head_round<true>(src, T, S, first, cnt);
    }
}

}  // namespace

size_t heads_smem(const DevTables &t) { return (size_t)std::max(t.nf, t.nb) * class_words(t) * 4; }
int heads_blocks_per_sm(size_t smem) {
    static uint64_t attr_done = 0;
    allow_smem(heads_batch_kernel, &attr_done);
    int per_sm = 1;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, heads_batch_kernel, kHeadThreads, smem);
    return std::max(per_sm, 1);
}
void launch_heads_batch(const WalkBatch &b, cudaStream_t s) {
    if (b.n_heads) heads_batch_kernel<<<b.n_heads * (b.recognize ? 1 : 2), kHeadThreads, b.heads_smem, s>>>(b);
}

// Chunks per block and round: kHeadChunks, fewer while that leaves the device
// short of blocks (a warp takes about 1 us per chunk with many slots): log text of
// 64 KiB to 1 MiB, heads and walk, 32 us with 64, 29.5 to 30.5 with 16 or 8; 4 MiB 40
// and 57.
void launch_heads(const Params &p, cudaStream_t s, int sm_count) {
    const size_t smem = heads_smem(p.t);
    static uint64_t attr_done = 0;
    allow_smem(heads_kernel, &attr_done);
    int per_sm = 1;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, heads_kernel, kHeadThreads, smem);
    const uint64_t dirs = p.recognize ? 1 : 2;
    uint32_t per = kHeadChunks;
    while (per > 8 && dirs * p.c / per < (uint64_t)sm_count * 2) per >>= 1;
    const uint64_t want = (p.c + per - 1) / per, slots = (uint64_t)std::max(per_sm, 1) * sm_count / dirs;
    heads_kernel<<<(uint32_t)(std::max<uint64_t>(1, std::min(want, slots)) * dirs), kHeadThreads, smem, s>>>(p, per);
}

}  // namespace slpf
