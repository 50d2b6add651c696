// The lane walk: device code shared by heads.cu (speculative chunk heads) and
// walk.cu (the walk of the chunks), for automata of at most 256 states per
// direction (shape 1 of RE_PARSE_REACH).
//
// Eq. (reacher) runs every speculative start of a chunk to the chunk's end.
// Runs meet within the first bytes of most chunks (Sect. 4.3), and from there
// on a chunk is one run of the classic DFA.  So the two parts are separate
// kernels with a layout each:
//   heads  walks every speculative start, a lane per run, until the chunk's
//          live runs are in one state (at a multiple of kUnit bytes);
//   walk   takes one run per chunk and direction from there to the chunk's
//          far edge, a lane per chunk, and goes on through the head of the
//          next chunk.  Those columns are exact once the run is (Eq. builder),
//          and the state it reaches where the next chunk's runs had met must
//          be theirs: the check that Eq. (joiner) makes with the slots' keys.
#pragma once

#include "kernels.cuh"

namespace slpf {

constexpr uint32_t kUnit = 32;              // bytes of a chunk per step of the walk: one 32-byte load and store

// Class-indexed transition rows of one direction: bytes per row (classes
// rounded up to whole words).
__host__ __device__ inline uint32_t class_words(const DevTables &t) { return (t.ncls + 3) / 4; }

// Transition table of one direction in shared memory, 2^LOGR copies word by
// word: word (state, class / 4) of copy r lies at word (state * cw + class / 4)
// * 2^LOGR + r.  With 32 copies a warp's lookup touches 32 different banks
// whatever the states and bytes are: one wavefront, where one table costs
// about 3.5 (the fullest of 32 banks under 32 random words).  The class map's
// first 128 bytes are one word per bank, so looking ASCII bytes up in it never
// conflicts either.  Addresses are shared-window offsets: one 32-bit
// multiply-add per lookup.
struct LaneTab {
    uint32_t tab;            // this lane's copy
    const uint8_t *cls;      // [256] byte -> class (shared memory)
    uint32_t rowb;           // bytes from one state's row to the next
};

// A byte of an immutable shared-memory table (staged before a barrier).
__device__ __forceinline__ uint32_t lds8(uint32_t at) {
    uint32_t v;
    asm volatile("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"(at));
    return v;
}

// Offset of a byte's class in a row of this lane's copy.
template <int LOGR>
__device__ __forceinline__ uint32_t lane_col(const LaneTab &T, uint32_t byte) {
    const uint32_t c = T.cls[byte];
    // 2^LOGR * (c - c % 4) + c % 4, as two multiply-adds
    return LOGR == 0 ? T.tab + c : (c << LOGR) + (T.tab - ((1u << LOGR) - 1) * (c & 3u));
}

template <int LOGR>
__device__ __forceinline__ uint32_t lane_step(const LaneTab &T, uint32_t s, uint32_t byte) {
    return lds8(s * T.rowb + lane_col<LOGR>(T, byte));
}

// States of 16 consecutive bytes.  Forward: o[u] is the state before byte u;
// backward: the state after consuming byte u, from byte 15 down to 0.  The
// next four columns are looked up while the current four steps wait for one
// another.
template <int LOGR, bool FWD>
__device__ __forceinline__ uint32_t walk16(const LaneTab &T, uint32_t s, const uint4 &x, uint4 &o) {
    const uint32_t w[4] = {x.x, x.y, x.z, x.w};
    uint32_t ow[4], col[4];
#pragma unroll
    for (int h = 0; h < 4; ++h)
        col[h] = lane_col<LOGR>(T, __byte_perm(w[FWD ? 0 : 3], 0u, 0x4440u | (uint32_t)(FWD ? h : 3 - h)));
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        const int g = FWD ? v : 3 - v, gn = FWD ? v + 1 : 2 - v;
        uint32_t st[4], nx[4];
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            const int b = FWD ? h : 3 - h;
            if (FWD) st[b] = s;
            s = lds8(s * T.rowb + col[h]);
            if (!FWD) st[b] = s;
            if (v < 3) nx[h] = lane_col<LOGR>(T, __byte_perm(w[gn], 0u, 0x4440u | (uint32_t)b));
        }
        ow[g] = __byte_perm(__byte_perm(st[0], st[1], 0x0040u), __byte_perm(st[2], st[3], 0x0040u), 0x5410u);
#pragma unroll
        for (int h = 0; h < 4; ++h) col[h] = v < 3 ? nx[h] : 0u;
    }
    o = make_uint4(ow[0], ow[1], ow[2], ow[3]);
    return s;
}

// A unit of text (32 bytes), with the rest of its 128-byte line brought into
// L2; `wide`: the text is 32-byte aligned.
struct Unit {
    uint4 a, b;
};
__device__ __forceinline__ Unit load_unit(const uint8_t *x, bool wide) {
    Unit u;
    if (wide) {
        asm volatile("ld.global.nc.L2::128B.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=r"(u.a.x), "=r"(u.a.y), "=r"(u.a.z), "=r"(u.a.w), "=r"(u.b.x), "=r"(u.b.y), "=r"(u.b.z), "=r"(u.b.w)
                     : "l"(x));
    } else {
        u.a = __ldg(reinterpret_cast<const uint4 *>(x));
        u.b = __ldg(reinterpret_cast<const uint4 *>(x) + 1);
    }
    return u;
}
__device__ __forceinline__ void store_unit(uint8_t *out, const Unit &u) {   // 32-byte aligned
    asm volatile("st.global.v8.b32 [%8], {%0, %1, %2, %3, %4, %5, %6, %7};"
                 :: "r"(u.a.x), "r"(u.a.y), "r"(u.a.z), "r"(u.a.w), "r"(u.b.x), "r"(u.b.y), "r"(u.b.z), "r"(u.b.w), "l"(out)
                 : "memory");
}

// Fewer bytes than a unit, the text's end: bytes [0, cnt).
template <int LOGR, bool FWD, bool OUT>
__device__ uint32_t walk_part(const LaneTab &T, uint32_t s, const uint8_t *x, uint8_t *out, uint32_t cnt) {
#pragma unroll 1
    for (uint32_t q = 0; q < cnt; ++q) {
        const uint32_t u = FWD ? q : cnt - 1 - q;
        if (OUT && FWD) out[u] = (uint8_t)s;
        s = lane_step<LOGR>(T, s, __ldg(x + u));
        if (OUT && !FWD) out[u] = (uint8_t)s;
    }
    return s;
}

// One lane's walk of the columns [lo, hi) of x, left to right or right to
// left, states into out; `mid` gets the state at column m on the way (lo <= m
// <= hi).  Unit boundaries are multiples of kUnit of lo; m lies on one, and
// only the text's end makes hi anything else (m == hi then, or m == lo).
template <int LOGR, bool FWD, bool OUT>
__device__ uint32_t walk_cols(const LaneTab &T, const uint8_t *x, uint8_t *out, uint64_t lo, uint64_t hi, uint64_t m,
                              uint32_t s, bool wide, uint32_t &mid) {
    if (lo >= hi) { mid = s; return s; }
    const uint32_t part = (uint32_t)(hi - lo) & (kUnit - 1), nu = (uint32_t)((hi - lo) / kUnit);
    const uint64_t top = hi - part;
    if (!FWD && part) {
        if (m == hi) mid = s;
        s = walk_part<LOGR, FWD, OUT>(T, s, x + top, OUT ? out + top : nullptr, part);
    }
    // units walked before column m; the state there is kept when it is reached
    const uint32_t um = FWD ? (uint32_t)((m - lo) / kUnit) : (m >= top ? 0u : (uint32_t)((top - m) / kUnit));
    const bool mid_part = !FWD && part && m == hi;
    if (um == 0 && !mid_part) mid = s;
    const int64_t step = FWD ? (int64_t)kUnit : -(int64_t)kUnit;
    const uint8_t *px = x + (FWD ? lo : top - kUnit);
    uint8_t *po = OUT ? out + (FWD ? lo : top - kUnit) : nullptr;
    auto walk = [&](const Unit &t) {
        Unit o;
        s = walk16<LOGR, FWD>(T, s, FWD ? t.a : t.b, FWD ? o.a : o.b);
        s = walk16<LOGR, FWD>(T, s, FWD ? t.b : t.a, FWD ? o.b : o.a);
        if (OUT) { store_unit(po, o); po += step; }
    };
    if (nu) {
        Unit t0 = load_unit(px, wide), t1 = t0;
#pragma unroll 1
        for (uint32_t u = 0;;) {                              // two units a turn: each in registers of its own
            if (u + 1 < nu) t1 = load_unit(px + step, wide);
            walk(t0);
            if (++u == um && !mid_part) mid = s;
            if (u >= nu) break;
            px += 2 * step;
            if (u + 1 < nu) t0 = load_unit(px, wide);
            walk(t1);
            if (++u == um && !mid_part) mid = s;
            if (u >= nu) break;
        }
    }
    if (FWD && part) {
        s = walk_part<LOGR, FWD, OUT>(T, s, x + top, OUT ? out + top : nullptr, part);
        if (m == hi) mid = s;
    }
    return s;
}

// Copy ns rows of a class-indexed table into shared memory, 2^LOGR copies
// (block-wide, no barrier).
template <int LOGR>
__device__ void stage_lane_table(const uint8_t *src, uint32_t words, uint8_t *dst) {
    const uint32_t *s32 = reinterpret_cast<const uint32_t *>(src);
    if (LOGR >= 2) {
        uint4 *d = reinterpret_cast<uint4 *>(dst);
        const uint32_t cnt = words << (LOGR >= 2 ? LOGR - 2 : 0);
#pragma unroll 4
        for (uint32_t q = threadIdx.x; q < cnt; q += blockDim.x) {
            const uint32_t v = __ldg(s32 + (q >> (LOGR >= 2 ? LOGR - 2 : 0)));
            d[q] = make_uint4(v, v, v, v);
        }
    } else {
        uint32_t *d = reinterpret_cast<uint32_t *>(dst);
#pragma unroll 4
        for (uint32_t q = threadIdx.x; q < words; q += blockDim.x) d[q] = __ldg(s32 + q);
    }
}

__device__ inline void stage_classes(const DevTables &t, uint8_t *dst) {
    for (uint32_t q = threadIdx.x; q < 64; q += blockDim.x)
        reinterpret_cast<uint32_t *>(dst)[q] = __ldg(reinterpret_cast<const uint32_t *>(t.cls) + q);
}

}  // namespace slpf
