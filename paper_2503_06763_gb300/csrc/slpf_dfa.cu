// SLPF compression (arXiv 2503.06763, App. C, "SLPF compression").
//
// App. C keeps the SLPF of a text as its initial column and a lookup table
// delta(C_{r-1}, x_r) = C_r over the columns that occur, and rebuilds the
// columns by running the table over the text.  A clean column also depends on
// bytes after r (only segments on a complete LST survive), so the table alone
// does not always give C_r; the archive here adds the positions where it does
// not (exceptions), and a checkpoint column every K positions so that the
// rebuild runs in independent pieces on the device (the evenly spaced
// columns App. C proposes for a parallel rebuild).
//
// Columns are column ids (DICT indices, or DENSE values below 65536).  The
// table row of id v and byte a holds the column that followed the first
// occurrence of (v, a) in the text.
//
// Encoding runs on the host (once per text, for storage); decoding is a
// kernel with one thread per K-column piece for short pieces, else a warp per
// piece (slpf_dfa_warp_kernel).
#include <algorithm>
#include <cstring>
#include <string>
#include <new>
#include <vector>

#include "kernels.cuh"
#include "re_internal.h"

namespace slpf {
namespace {

constexpr uint32_t kDfaMagic = 0x46504C53u;   // "SLPF"
constexpr uint32_t kDfaVersion = 2;
constexpr uint32_t kNoEntry = 0xFFFFu;          // a table entry no (column, byte) pair filled
constexpr uint32_t kMaxIds = 65535;            // ids fit u16 beside kNoEntry (tables of at most 32 MiB)
constexpr uint32_t kDecodeTableThread = 200 * 1024;   // table bytes a thread-per-piece block stages at most
constexpr uint32_t kMaxInterval = 65536;       // exception offsets within a piece fit u16

size_t align16(size_t v) { return (v + 15) & ~(size_t)15; }

struct Sections {
    size_t table, checkpoints, starts, exceptions, total;
};

Sections sections_of(uint32_t n_ids, uint64_t n_checkpoints, uint64_t n_exceptions) {
    Sections s{};
    s.table = align16(sizeof(re_slpf_dfa_header));
    s.checkpoints = s.table + align16((size_t)n_ids * 256 * 2);
    s.starts = s.checkpoints + align16(n_checkpoints * 2);
    s.exceptions = s.starts + align16((n_checkpoints + 1) * 8);
    s.total = s.exceptions + align16(n_exceptions * 4);
    return s;
}

// What an archive holds of host columns of one id width.
struct Encoded {
    uint32_t n_ids = 0;
    std::vector<uint16_t> table, checkpoints;
    std::vector<uint64_t> starts;
    std::vector<uint32_t> exceptions;                          // offset in its piece << 16 | id
};

// One pass over the columns, piece by piece: the id width is a type, the
// previous id stays in a register and no position is divided by the interval
// (an archive of 3 MiB of log text: 9.0 ms in two calls,
// one to learn the size, of a pass that did; 3.6 ms in one call of this one).  False: an id is too large.
template <typename Id>
bool encode_columns(const Id *cols, const uint8_t *text, uint64_t len, uint32_t interval, Encoded &e) {
    uint32_t max_id = 0;
    for (uint64_t r = 0; r <= len; ++r) max_id = std::max<uint32_t>(max_id, cols[r]);
    if (max_id >= kMaxIds) return false;
    e.n_ids = max_id + 1;
    e.table.assign((size_t)e.n_ids * 256, (uint16_t)kNoEntry);
    uint16_t *table = e.table.data();
    const uint64_t n_cp = len / interval + 1;
    e.starts.assign(n_cp + 1, 0);
    e.checkpoints.resize(n_cp);
    for (uint64_t s = 0; s < n_cp; ++s) {
        const uint64_t r0 = s * interval, end = std::min(len, r0 + interval - 1);
        uint32_t prev = cols[r0];
        e.checkpoints[s] = (uint16_t)prev;
        if (r0) {                                              // a checkpoint column needs no exception
            uint16_t &slot = table[(size_t)cols[r0 - 1] * 256 + text[r0 - 1]];
            if (slot == kNoEntry) slot = (uint16_t)prev;
        }
        for (uint64_t r = r0 + 1; r <= end; ++r) {
            const uint32_t cur = cols[r];
            uint16_t &slot = table[(size_t)prev * 256 + text[r - 1]];
            if (slot != cur) {
                if (slot == kNoEntry) slot = (uint16_t)cur;
                else e.exceptions.push_back((uint32_t)(r - r0) << 16 | cur);
            }
            prev = cur;
        }
        e.starts[s + 1] = e.exceptions.size();                 // exceptions before the next piece
    }
    return true;
}

struct DecodeArgs {
    const uint16_t *table;       // [n_ids][256]
    const uint16_t *checkpoints; // [n_checkpoints]
    const uint64_t *starts;      // [n_checkpoints + 1]: first exception of each piece
    const uint32_t *exceptions;  // [n_exceptions]: offset in its piece << 16 | id, ascending
    const uint8_t *x;
    uint64_t n, n_checkpoints, n_exceptions;
    uint32_t n_ids, interval, col_bytes, table_in_smem;
    uint32_t vector;             // 16-byte text loads and column stores (aligned buffers, interval % 16 == 0)
    void *out;
    int32_t *status;
};

__device__ __forceinline__ void put(const DecodeArgs &a, uint64_t r, uint32_t v) {
    if (a.col_bytes == 1) static_cast<uint8_t *>(a.out)[r] = (uint8_t)v;
    else if (a.col_bytes == 2) static_cast<uint16_t *>(a.out)[r] = (uint16_t)v;
    else static_cast<uint32_t *>(a.out)[r] = v;
}

// One thread per piece of K columns: the checkpoint, then the table (or the
// exception at that position) column after column.
__global__ void __launch_bounds__(256) slpf_dfa_decode_kernel(const __grid_constant__ DecodeArgs a) {
    extern __shared__ __align__(16) uint16_t stab[];
    const uint16_t *table = a.table;
    if (a.table_in_smem) {
        const size_t entries = (size_t)a.n_ids * 256;
        for (size_t q = threadIdx.x; q < entries; q += blockDim.x) stab[q] = __ldg(a.table + q);
        __syncthreads();
        table = stab;
    }
    bool bad = false;
    for (uint64_t s = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; s < a.n_checkpoints;
         s += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t r0 = s * a.interval;
        const uint64_t r1 = min(r0 + a.interval, a.n + 1);
        uint32_t cur = __ldg(a.checkpoints + s);
        uint64_t e = __ldg(a.starts + s);
        const uint64_t e_end = min(__ldg(a.starts + s + 1), a.n_exceptions);
        uint32_t ev = e < e_end ? __ldg(a.exceptions + e) : 0u;
        while (e < e_end && (ev >> 16) == 0) {                 // none at the checkpoint column (a bad archive)
            ++e;
            ev = e < e_end ? __ldg(a.exceptions + e) : 0u;
        }
        uint64_t next = e < e_end ? r0 + (ev >> 16) : ~0ull;
        auto step = [&](uint64_t r, uint32_t byte) {             // column r from column r - 1 and byte x[r-1]
            if (r == next) {
                cur = ev & 0xFFFFu;
                ++e;
                ev = e < e_end ? __ldg(a.exceptions + e) : 0u;
                next = e < e_end ? r0 + (ev >> 16) : ~0ull;
            } else {
                const uint32_t v = cur < a.n_ids ? table[(size_t)cur * 256 + byte] : kNoEntry;
                if (v == kNoEntry) { bad = true; cur = 0; }   // not an archive of this text
                else cur = v;
            }
        };
        if (a.vector) {
            // 16 columns at a time: one 16-byte text load (bytes g .. g+15 serve
            // columns g+1 .. g+16) and the ids packed into 16-byte stores
            uint32_t prev = 0;                                   // x[g - 1]
            for (uint64_t g = r0; g < r1; g += 16) {
                const uint4 xv = load16(a.x, a.n, g);
                const uint32_t xw[4] = {xv.x, xv.y, xv.z, xv.w};
                uint32_t ow[16];                                 // up to 16 ids of 4 bytes
#pragma unroll
                for (int q = 0; q < 16; ++q) ow[q] = 0;
                const uint64_t end = min(g + 16, r1);
#pragma unroll
                for (int u = 0; u < 16; ++u) {
                    const uint64_t r = g + u;
                    if (r < end) {
                        if (r > r0) step(r, u == 0 ? prev : (xw[(u - 1) >> 2] >> (8 * ((u - 1) & 3))) & 0xFFu);
                        if (a.col_bytes == 1) ow[u >> 2] |= (cur & 0xFFu) << (8 * (u & 3));
                        else if (a.col_bytes == 2) ow[u >> 1] |= (cur & 0xFFFFu) << (16 * (u & 1));
                        else ow[u] = cur;
                    }
                }
                prev = xw[3] >> 24;
                uint4 *dst = reinterpret_cast<uint4 *>(static_cast<uint8_t *>(a.out) + g * a.col_bytes);
                if (end == g + 16) {                             // a full group: col_bytes stores of 16 bytes
                    dst[0] = make_uint4(ow[0], ow[1], ow[2], ow[3]);
                    if (a.col_bytes >= 2) dst[1] = make_uint4(ow[4], ow[5], ow[6], ow[7]);
                    if (a.col_bytes == 4) {
                        dst[2] = make_uint4(ow[8], ow[9], ow[10], ow[11]);
                        dst[3] = make_uint4(ow[12], ow[13], ow[14], ow[15]);
                    }
                } else {                                         // the piece's last columns, one at a time
                    for (uint64_t q = g; q < end; ++q) {
                        const uint32_t u = (uint32_t)(q - g);
                        const uint32_t v = a.col_bytes == 1 ? (ow[u >> 2] >> (8 * (u & 3))) & 0xFFu
                                         : a.col_bytes == 2 ? (ow[u >> 1] >> (16 * (u & 1))) & 0xFFFFu
                                                            : ow[u];
                        put(a, q, v);
                    }
                }
            }
        } else {
            put(a, r0, cur);
            for (uint64_t r = r0 + 1; r < r1; ++r) {
                step(r, __ldg(a.x + r - 1));
                put(a, r, cur);
            }
        }
    }
    if (bad) atomicExch(a.status, RE_E_INTERNAL);
}

// Long pieces.  An exception is an exact column, so it is as good a place to
// start from as a checkpoint: a warp takes a window of up to kWindow columns of
// a piece and its lanes share it, lane j from the first exception at or after
// column j * seg to the one where the next lane starts (the checkpoint for the
// first).  Columns stand at 0.05 to 0.25 exceptions each, so the lanes' shares
// are near seg, and a chain of dependent lookups is some 150 columns long
// instead of K: for 48 MiB of log columns and K = 4096, where a thread per
// piece left 12 289 chains of 4096 steps, the kernel went from 1371 to 138 us.
//
// In shared memory: the table, only the byte columns that occur (used bytes
// renumbered; one byte per entry while ids and the mark of a missing entry
// fit), the piece's exceptions, and a tile that holds each column's text byte
// until the column replaces it.  The tile is padded by a word every 128 bytes,
// as the lanes walk about 128 columns apart.  Bound by latency (the chains of
// the longest share of each window) and issue: 16 warps a block 212 us, the 28
// that the shared memory holds 138 us.
constexpr uint32_t kWindow = 4096;
template <int CB> constexpr uint32_t decode_warps() { return CB == 1 ? 28u : CB == 2 ? 16u : 8u; }   // what the shared memory holds
constexpr uint32_t kDecodeExc = 512;           // exceptions staged per window; the rest are read from the archive
constexpr uint32_t kDecodeTable = 48 * 1024;   // table bytes staged at most
constexpr uint32_t kDecodeRows = 192;          // rows looked through for staging, or in long texts
constexpr uint32_t kDecodeRowsLong = 400;      // as many as a thread-per-piece block stages
constexpr uint32_t kDecodeMinInterval = 256;   // shorter pieces: a thread each
// Below kDecodeShort a thread each, too, from kDecodePieces * K pieces on: a warp's lanes then
// have 8 to 16 columns each, and copying the tile weighs more than the chains.  Log text, K = 256:
// 1 MiB 37 us by warps, 85 by threads; 8 MiB 127 and 87; 48 MiB 589 and 268.
constexpr uint32_t kDecodeShort = 512;
constexpr uint64_t kDecodePieces = 64;

template <int CB> struct IdOf;
template <> struct IdOf<1> { using type = uint8_t; };
template <> struct IdOf<2> { using type = uint16_t; };
template <> struct IdOf<4> { using type = uint32_t; };

template <int CB> __host__ __device__ constexpr uint32_t tile_at(uint32_t a) { return a * CB + (a * CB / 128) * 4; }
template <int CB> __host__ __device__ constexpr uint32_t tile_bytes() { return (tile_at<CB>(kWindow) + 15) / 16 * 16; }

template <int CB, bool BYTE>                   // BYTE: table entries of one byte (ids below 255)
__global__ void __launch_bounds__(decode_warps<CB>() * 32, 1) slpf_dfa_warp_kernel(const __grid_constant__ DecodeArgs a,
                                                                          uint32_t table_bytes, uint32_t windows) {
    using Id = typename IdOf<CB>::type;
    using Entry = typename IdOf<BYTE ? 1 : 2>::type;
    constexpr uint32_t none = BYTE ? 0xFFu : kNoEntry;
    extern __shared__ __align__(16) uint8_t sm[];
    __shared__ uint32_t used[256];
    __shared__ uint8_t cls[256];               // byte -> column of the staged table
    __shared__ uint32_t ncol;
    // Used byte columns: one entry of a row that occurs.  Every block looks the table through,
    // which pays only where it is small for the columns that follow; else the walk reads it
    // where it is.  DNA (349 ids, K = 4096): 1 MiB 97 us staged, 66 not; 48 MiB 291 and 328.
    // 5000 ids, 4 MiB: 472 and 116; 65 534 ids: 3250 and 381.
    const uint32_t rows = a.n_ids;
    const bool small = rows <= kDecodeRows || (rows <= kDecodeRowsLong && a.n >= (uint64_t)rows << 16);
    for (uint32_t q = threadIdx.x; q < 256; q += blockDim.x) used[q] = 0;
    __syncthreads();
    for (uint32_t q = threadIdx.x; small && q < rows * 128; q += blockDim.x) {
        const uint32_t v = __ldg(reinterpret_cast<const uint32_t *>(a.table) + q);
        if ((v & 0xFFFFu) != kNoEntry) used[2 * (q & 127)] = 1;
        if (v >> 16 != kNoEntry) used[2 * (q & 127) + 1] = 1;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        uint32_t n = 0;
        for (uint32_t g = 0; g < 8; ++g) {
            const uint32_t b = 32 * g + threadIdx.x;
            const unsigned m = __ballot_sync(0xFFFFFFFFu, used[b] != 0);
            cls[b] = (uint8_t)(n + __popc(m & ((1u << threadIdx.x) - 1)));
            n += __popc(m);
        }
        if (threadIdx.x == 0) ncol = n;
    }
    __syncthreads();
    // row stride: an odd number of words, so equal bytes of different rows are in different banks; the
    // last column is that of every byte that does not occur
    const uint32_t nc = ncol + 1;
    const uint32_t rowe = ((nc * sizeof(Entry) + 3) / 4 | 1) * 4 / sizeof(Entry);
    const bool staged = small && (uint64_t)rows * rowe * sizeof(Entry) <= table_bytes;
    Entry *tab = reinterpret_cast<Entry *>(sm);
    if (staged) {
        for (uint32_t q = threadIdx.x; q < rows * 256; q += blockDim.x) {
            const uint32_t b = q & 255, v = __ldg(a.table + q);
            if (used[b]) tab[(q >> 8) * rowe + cls[b]] = v >= rows ? (Entry)none : (Entry)v;   // kNoEntry, or no id
        }
        for (uint32_t q = threadIdx.x; q < rows; q += blockDim.x) tab[q * rowe + nc - 1] = (Entry)none;
    }
    __syncthreads();
    if (threadIdx.x < 256 && !used[threadIdx.x]) cls[threadIdx.x] = (uint8_t)min(nc - 1, 255u);   // 256 used: no other byte
    __syncthreads();
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint8_t *tile = sm + table_bytes + warp * (tile_bytes<CB>() + kDecodeExc * 4);
    uint32_t *exc = reinterpret_cast<uint32_t *>(tile + tile_bytes<CB>());
    Id *out = static_cast<Id *>(a.out);
    auto next_of = [&](uint32_t cur, uint32_t byte) -> uint32_t {   // none: no such pair in the archived text
        if (staged) return tab[cur * rowe + cls[byte]];
        const uint32_t v = __ldg(a.table + (size_t)cur * 256 + byte);
        return v >= rows ? none : v;
    };
    bool bad = false;
    for (uint64_t w = (uint64_t)blockIdx.x * decode_warps<CB>() + warp; w < a.n_checkpoints * windows;
         w += (uint64_t)gridDim.x * decode_warps<CB>()) {
        const uint64_t piece = w / windows, r0 = piece * a.interval;
        const uint32_t len = (uint32_t)min((uint64_t)a.interval, a.n + 1 - r0), w0 = (uint32_t)(w % windows) * kWindow;
        if (w0 >= len) continue;                              // the text's last piece is shorter
        const uint32_t wl = min(kWindow, len - w0), seg = max(32u, (wl + 31) / 32);
        const uint64_t e0 = __ldg(a.starts + piece), e1 = min(__ldg(a.starts + piece + 1), a.n_exceptions);
        // first exception of [lo, hi) at or after column o of the piece
        auto lower = [&](auto get, uint64_t lo, uint64_t hi, uint32_t o) -> uint64_t {
            while (lo < hi) {
                const uint64_t mid = (lo + hi) / 2;
                if ((get(mid) >> 16) < o) lo = mid + 1; else hi = mid;
            }
            return lo;
        };
        auto global = [&](uint64_t e) -> uint32_t { return __ldg(a.exceptions + e); };
        // none stands at the checkpoint column (a bad archive): the piece's start is the checkpoint
        const uint64_t es = e0 < e1 ? lower(global, e0, e1, max(w0, 1u)) : e1;
        __syncwarp();                                         // the last window's tile has left
        for (uint32_t q = lane; q < kDecodeExc && es + q < e1; q += 32) exc[q] = __ldg(a.exceptions + es + q);
        // text byte before each column: column c takes x[c - 1]
        const bool vec = ((r0 + w0) & 15) == 0 && (reinterpret_cast<uintptr_t>(a.x) & 15) == 0;
        const uint32_t wv = vec ? wl & ~15u : 0u;             // 16 columns a lane and turn
        for (uint32_t q = 16 * lane; q < wv; q += 512) {
            const uint8_t *at = a.x + r0 + w0 + q;
            const uint4 v = load16(a.x, a.n, r0 + w0 + q);    // the text may end before the last column
            const uint32_t before = r0 + w0 + q > 0 ? (uint32_t)__ldg(at - 1) : 0u;
            const uint32_t w[5] = {before << 24, v.x, v.y, v.z, v.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint32_t four = __funnelshift_l(w[u], w[u + 1], 8);
                uint32_t *d = reinterpret_cast<uint32_t *>(tile + tile_at<CB>(q + 4 * u));
                if constexpr (CB == 1) {
                    d[0] = four;
                } else if constexpr (CB == 2) {
                    d[0] = __byte_perm(four, 0u, 0x4140u);
                    d[1] = __byte_perm(four, 0u, 0x4342u);
                } else {
#pragma unroll
                    for (int b = 0; b < 4; ++b) d[b] = __byte_perm(four, 0u, 0x4440u | (uint32_t)b);
                }
            }
        }
        for (uint32_t q = wv + lane; q < wl; q += 32)
            if (r0 + w0 + q > 0) *reinterpret_cast<Id *>(tile + tile_at<CB>(q)) = (Id)__ldg(a.x + r0 + w0 + q - 1);
        __syncwarp();
        auto get = [&](uint64_t e) -> uint32_t { return e - es < kDecodeExc ? exc[e - es] : __ldg(a.exceptions + e); };
        // this lane's columns [from, to) of the piece
        uint64_t e = lane == 0 && w0 == 0 ? es : lower(get, es, e1, w0 + lane * seg);
        const uint64_t last = lower(global, es, e1, w0 + wl);
        uint32_t ev = e < e1 ? get(e) : 0u;
        uint32_t from = lane == 0 && w0 == 0 ? 0u : e < e1 ? ev >> 16 : len;
        uint32_t to = __shfl_down_sync(0xFFFFFFFFu, from, 1);
        if (lane == 31) to = last < e1 ? global(last) >> 16 : len;
        from = min(from, len);
        to = min(to, len);
        const uint32_t first = __shfl_sync(0xFFFFFFFFu, from, 0);   // columns before it are the last window's
        if (from < to) {
            uint32_t cur;
            if (lane == 0 && w0 == 0) {
                cur = __ldg(a.checkpoints + piece);
            } else {
                cur = ev & 0xFFFFu;
                ++e;
                ev = e < e1 ? get(e) : 0u;
            }
            uint32_t next = e < e1 ? ev >> 16 : 0xFFFFFFFFu;
            auto step = [&](uint32_t o, uint32_t byte) {      // column o of the piece from the one before
                if (o == next) {
                    cur = ev & 0xFFFFu;
                    ++e;
                    ev = e < e1 ? get(e) : 0u;
                    next = e < e1 ? ev >> 16 : 0xFFFFFFFFu;
                } else {
                    const uint32_t v = cur < rows ? next_of(cur, byte) : none;
                    bad |= v == none;                          // not an archive of this text
                    cur = v == none ? 0u : v;
                }
            };
            const uint32_t in = min(to, w0 + wl);             // columns inside the tile
            uint32_t o = from;
            if (o < in) { *reinterpret_cast<Id *>(tile + tile_at<CB>(o - w0)) = (Id)cur; ++o; }
            else { out[r0 + o] = (Id)cur; ++o; }              // the share starts after the window
            if (staged && e1 - es <= kDecodeExc) {            // the common case, on shared memory alone
                uint32_t ei = (uint32_t)(e - es);
                const uint32_t en = (uint32_t)(e1 - es);
#pragma unroll 2
                for (; o < in; ++o) {
                    Id *t = reinterpret_cast<Id *>(tile + tile_at<CB>(o - w0));
                    const uint32_t v = cur < rows ? (uint32_t)tab[cur * rowe + cls[(uint32_t)*t & 0xFFu]] : none;
                    if (o == next) {
                        cur = ev & 0xFFFFu;
                        ++ei;
                        ev = exc[min(ei, kDecodeExc - 1)];
                        next = ei < en ? ev >> 16 : 0xFFFFFFFFu;
                    } else {
                        bad |= v == none;
                        cur = v == none ? 0u : v;
                    }
                    *t = (Id)cur;
                }
                e = es + ei;
            }
            for (; o < in; ++o) {
                Id *t = reinterpret_cast<Id *>(tile + tile_at<CB>(o - w0));
                step(o, (uint32_t)*t & 0xFFu);
                *t = (Id)cur;
            }
            for (; o < to; ++o) {
                step(o, __ldg(a.x + r0 + o - 1));
                out[r0 + o] = (Id)cur;
            }
        }
        __syncwarp();
        // the tile's columns out, from `first` on
        constexpr uint32_t V = 4 / CB;                        // columns per word
        const uint64_t c0 = r0 + w0;
        const uint32_t skip = first > w0 ? min(first - w0, wl) : 0u;
        constexpr uint32_t C16 = 4 * V;                       // columns per 16 bytes
        if ((c0 % C16) == 0 && (reinterpret_cast<uintptr_t>(a.out) & 15) == 0) {
            for (uint32_t q = C16 * lane; q < wl; q += 32 * C16) {
                if (q >= skip && q + C16 <= wl) {             // inside a 128-byte row of the tile
                    const uint32_t *t = reinterpret_cast<const uint32_t *>(tile + tile_at<CB>(q));
                    reinterpret_cast<uint4 *>(out)[(c0 + q) / C16] = make_uint4(t[0], t[1], t[2], t[3]);
                } else {
                    for (uint32_t u = 0; u < C16; ++u)
                        if (q + u >= skip && q + u < wl) out[c0 + q + u] = *reinterpret_cast<const Id *>(tile + tile_at<CB>(q + u));
                }
            }
        } else {
            for (uint32_t q = skip + lane; q < wl; q += 32) out[c0 + q] = *reinterpret_cast<const Id *>(tile + tile_at<CB>(q));
        }
    }
    if (bad) atomicExch(a.status, RE_E_INTERNAL);
}

// The shared-memory limit of each kernel is raised once, to the most any archive
// takes: a limit per call would be another thread's limit between its launch
// and the call that set it.
template <int CB, bool BYTE>
cudaError_t launch_decode_warp(const DecodeArgs &a, cudaStream_t s, int sms) {
    constexpr uint32_t warps = decode_warps<CB>(), warp_smem = tile_bytes<CB>() + kDecodeExc * 4;
    const uint32_t windows = (a.interval + kWindow - 1) / kWindow;
    const uint32_t table = std::min<uint32_t>(kDecodeTable, (uint32_t)(((size_t)a.n_ids * (260 + 4) * (BYTE ? 1 : 2) + 15) / 16 * 16));
    const size_t smem = table + warps * warp_smem;
    static uint64_t attr_done = 0;
    allow_smem(slpf_dfa_warp_kernel<CB, BYTE>, &attr_done, kDecodeTable + warps * warp_smem);
    int per_sm = 1;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, slpf_dfa_warp_kernel<CB, BYTE>, warps * 32, smem);
    const uint64_t want = (a.n_checkpoints * windows + warps - 1) / warps;
    const uint32_t blocks = (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>(want, (uint64_t)sms * std::max(per_sm, 1)));
    slpf_dfa_warp_kernel<CB, BYTE><<<blocks, warps * 32, smem, s>>>(a, table, windows);
    return cudaGetLastError();
}

__global__ void slpf_dfa_status_kernel(int32_t *status) { *status = RE_OK; }

}  // namespace
}  // namespace slpf

using namespace slpf;

extern "C" re_status re_slpf_dfa_encode(const void *cols, uint32_t col_bytes, const uint8_t *text, uint64_t len,
                                        uint32_t interval, void *archive, uint64_t cap, uint64_t *size) {
    if (!cols || !size || (len && !text) || (cap && !archive)) { set_error("null argument"); return RE_E_INVALID_ARG; }
    if (col_bytes != 1 && col_bytes != 2 && col_bytes != 4) { set_error("col_bytes must be 1, 2 or 4"); return RE_E_INVALID_ARG; }
    if (interval == 0) { set_error("interval must be positive"); return RE_E_INVALID_ARG; }
    if (interval > kMaxInterval) { set_error("interval above 65536"); return RE_E_INVALID_ARG; }
    Encoded e;
    bool fits = false;
    try {
        fits = col_bytes == 1   ? encode_columns(static_cast<const uint8_t *>(cols), text, len, interval, e)
               : col_bytes == 2 ? encode_columns(static_cast<const uint16_t *>(cols), text, len, interval, e)
                                : encode_columns(static_cast<const uint32_t *>(cols), text, len, interval, e);
    } catch (const std::bad_alloc &) {
        set_error("out of host memory while encoding");
        return RE_E_NOMEM;
    }
    if (!fits) { set_error("column ids must be below 65535"); return RE_E_CAPACITY; }
    const Sections sec = sections_of(e.n_ids, e.checkpoints.size(), e.exceptions.size());
    *size = sec.total;
    if (cap < sec.total) { set_error("archive buffer too small (size reported)"); return RE_E_CAPACITY; }
    uint8_t *b = static_cast<uint8_t *>(archive);
    re_slpf_dfa_header hdr{};
    hdr.magic = kDfaMagic;
    hdr.version = kDfaVersion;
    hdr.n = len;
    hdr.n_ids = e.n_ids;
    hdr.interval = interval;
    hdr.n_exceptions = e.exceptions.size();
    hdr.n_checkpoints = e.checkpoints.size();
    // each section, and zeros up to the next one
    auto section = [b](size_t at, const void *src, size_t bytes, size_t next) {
        if (bytes) std::memcpy(b + at, src, bytes);
        std::memset(b + at + bytes, 0, next - at - bytes);
    };
    section(0, &hdr, sizeof(hdr), sec.table);
    section(sec.table, e.table.data(), e.table.size() * 2, sec.checkpoints);
    section(sec.checkpoints, e.checkpoints.data(), e.checkpoints.size() * 2, sec.starts);
    section(sec.starts, e.starts.data(), e.starts.size() * 8, sec.exceptions);
    section(sec.exceptions, e.exceptions.data(), e.exceptions.size() * 4, sec.total);
    return RE_OK;
}

extern "C" re_status re_slpf_dfa_decode(const re_slpf_dfa_header *hdr, const void *d_archive, uint64_t archive_bytes,
                                        const uint8_t *d_text, void *d_cols, uint64_t cols_cap_bytes,
                                        uint32_t col_bytes, int32_t *d_status, re_stream stream) {
    if (!hdr || !d_archive || !d_cols || !d_status || (hdr->n && !d_text)) { set_error("null argument"); return RE_E_INVALID_ARG; }
    if (hdr->magic != kDfaMagic || hdr->version != kDfaVersion) { set_error("not an SLPF archive of this version"); return RE_E_INVALID_ARG; }
    if (col_bytes != 1 && col_bytes != 2 && col_bytes != 4) { set_error("col_bytes must be 1, 2 or 4"); return RE_E_INVALID_ARG; }
    if (hdr->n_ids == 0 || hdr->n_ids > kMaxIds || hdr->interval == 0 || hdr->interval > kMaxInterval ||
        hdr->n_checkpoints != hdr->n / hdr->interval + 1 || hdr->n_exceptions > hdr->n) {
        set_error("inconsistent archive header");
        return RE_E_INVALID_ARG;
    }
    if (col_bytes < 4 && hdr->n_ids > (1ull << (8 * col_bytes))) { set_error("column ids do not fit col_bytes"); return RE_E_INVALID_ARG; }
    const Sections sec = sections_of(hdr->n_ids, hdr->n_checkpoints, hdr->n_exceptions);
    if (archive_bytes < sec.total) { set_error("archive shorter than its header says"); return RE_E_INVALID_ARG; }
    if (cols_cap_bytes < (hdr->n + 1) * col_bytes) { set_error("column buffer too small"); return RE_E_CAPACITY; }
    if (((uintptr_t)d_archive & 15)) { set_error("archive must be 16-byte aligned"); return RE_E_INVALID_ARG; }
    const uint8_t *b = static_cast<const uint8_t *>(d_archive);
    DecodeArgs a{};
    a.table = reinterpret_cast<const uint16_t *>(b + sec.table);
    a.checkpoints = reinterpret_cast<const uint16_t *>(b + sec.checkpoints);
    a.starts = reinterpret_cast<const uint64_t *>(b + sec.starts);
    a.exceptions = reinterpret_cast<const uint32_t *>(b + sec.exceptions);
    a.x = d_text;
    a.n = hdr->n;
    a.n_checkpoints = hdr->n_checkpoints;
    a.n_exceptions = hdr->n_exceptions;
    a.n_ids = hdr->n_ids;
    a.interval = hdr->interval;
    a.col_bytes = col_bytes;
    a.out = d_cols;
    a.status = d_status;
    const size_t tab_bytes = (size_t)hdr->n_ids * 256 * 2;
    a.table_in_smem = tab_bytes <= kDecodeTableThread ? 1u : 0u;
    a.vector = (hdr->interval % 16 == 0 && ((uintptr_t)d_text & 15) == 0 && ((uintptr_t)d_cols & 15) == 0) ? 1u : 0u;
    const size_t smem = a.table_in_smem ? tab_bytes : 0;
    cudaStream_t s = (cudaStream_t)stream;
    slpf_dfa_status_kernel<<<1, 1, 0, s>>>(d_status);
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const bool thread_each = hdr->interval < kDecodeMinInterval ||
                             (hdr->interval < kDecodeShort && a.vector && hdr->n_checkpoints > kDecodePieces * hdr->interval);
    if (!thread_each) {                                        // a warp per piece
        cudaError_t e;
        if (col_bytes == 1) e = hdr->n_ids < 255 ? launch_decode_warp<1, true>(a, s, sms) : launch_decode_warp<1, false>(a, s, sms);
        else if (col_bytes == 2) e = hdr->n_ids < 255 ? launch_decode_warp<2, true>(a, s, sms) : launch_decode_warp<2, false>(a, s, sms);
        else e = hdr->n_ids < 255 ? launch_decode_warp<4, true>(a, s, sms) : launch_decode_warp<4, false>(a, s, sms);
        if (e != cudaSuccess) { set_error(std::string("decode launch: ") + cudaGetErrorString(e)); return RE_E_CUDA; }
        return RE_OK;
    }
    static uint64_t attr_done = 0;
    allow_smem(slpf_dfa_decode_kernel, &attr_done, kDecodeTableThread);
    const uint64_t want = (hdr->n_checkpoints + 255) / 256;
    const uint32_t blocks = (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>(want, (uint64_t)sms * 4));
    slpf_dfa_decode_kernel<<<blocks, 256, smem, s>>>(a);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) { set_error(std::string("decode launch: ") + cudaGetErrorString(e)); return RE_E_CUDA; }
    return RE_OK;
}
