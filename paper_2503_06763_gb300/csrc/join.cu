// Join phase (arXiv 2503.06763, Eq. joiner): FJ[i] = J_i, the forward state at
// the boundary before chunk i (J_0 = I), and BJ[i] = Ĵ at that boundary
// (BJ[c] = F).
//
// Every chunk maps an input state S to the union, over its slots whose keys
// S contains, of the slot's end state.  When all live slots of a chunk end in
// one state (the common case: speculative runs meet within a few hundred
// bytes, Sect. 4.3) the chunk's output is that state for every input that
// enters a live slot, so it is known without its neighbour.  The remaining
// chunks form chains that are evaluated in order from the nearest known
// neighbour.  A verify pass checks each guessed output against its actual
// input; the first chunk where the text cannot continue makes the whole text
// rejected (no accepting run: every clean column is empty).
#include <algorithm>

#include "walk.cuh"

namespace slpf {
namespace {

__device__ uint32_t probe(const uint32_t *hash, uint32_t mask, const uint64_t *bits, uint32_t W,
                          const uint64_t *key) {
    uint64_t h = bits_hash(key, W) & mask;
    for (uint32_t step = 0; step <= mask; ++step) {
        const uint32_t id = __ldg(hash + h);
        if (id == 0) return 0;
        bool eq = true;
        for (uint32_t w = 0; w < W; ++w)
            if (__ldg(bits + (size_t)id * W + w) != key[w]) { eq = false; break; }
        if (eq) return id;
        h = (h + 1) & mask;
    }
    return 0;
}

__device__ __forceinline__ uint32_t pair_fwd(const Params &p, uint32_t i) {
    const uint64_t base = (uint64_t)i * p.k;
    return __ldg(p.t.cls + __ldg(p.x + base - 1)) * p.t.ncls + __ldg(p.t.cls + __ldg(p.x + base));
}
__device__ __forceinline__ uint32_t pair_bwd(const Params &p, uint32_t i) {
    const uint64_t end = (uint64_t)i * p.k + chunk_len(p, i);
    return __ldg(p.t.cls + __ldg(p.x + end - 1)) * p.t.ncls + __ldg(p.t.cls + __ldg(p.x + end));
}

// State after chunk i for input state S: union over the slots S enters.
__device__ uint32_t eval_chunk(const Params &p, bool fwd, uint32_t i, uint32_t S, bool &bad) {
    const DevTables &t = p.t;
    if (S == 0) return 0;
    const uint32_t W = t.W;
    uint32_t pr, m, ms;
    const uint32_t *R;
    const uint64_t *mask, *bits;
    if (fwd) {
        pr = pair_fwd(p, i); m = __ldg(t.fSlotCount + pr); ms = t.msf; R = p.w.Rf + (size_t)i * ms;
        mask = t.fSlotMask + (size_t)pr * ms * W; bits = t.fBits;
    } else {
        pr = pair_bwd(p, i); m = __ldg(t.bSlotCount + pr); ms = t.msb; R = p.w.Rb + (size_t)i * ms;
        mask = t.bSlotMask + (size_t)pr * ms * W; bits = t.bBits;
    }
    const uint8_t *of = fwd ? t.fSlotOf : t.bSlotOf;
    if (of) {                                    // starts from every DFA state: exact lookup
        const uint32_t n = fwd ? t.nf : t.nb;
        const uint32_t j = S < n ? __ldg(of + (size_t)pr * n + S) : 0xFFu;
        return j == 0xFFu ? 0u : R[j];
    }
    const uint64_t *sb = bits + (size_t)S * W;
    uint32_t single = 0;
    bool multi = false;
    uint64_t acc[kMaxW];
    for (uint32_t w = 0; w < W; ++w) acc[w] = 0;
    for (uint32_t s = 0; s < m; ++s) {
        const uint32_t e = R[s];
        if (!e || !any_and(sb, mask + (size_t)s * W, W)) continue;
        if (!single) single = e;
        else if (e != single) multi = true;
        for (uint32_t w = 0; w < W; ++w) acc[w] |= __ldg(bits + (size_t)e * W + w);
    }
    if (!multi) return single;
    const uint32_t id = fwd ? probe(t.fHash, t.fHashMask, t.fBits, W, acc)
                            : probe(t.bHash, t.bHashMask, t.bBits, W, acc);
    if (!id) bad = true;
    return id;
}

// One live end state (or none) for every chunk?  Record it as the guess.
__device__ void classify(const Params &p, bool fwd, uint32_t i) {
    const DevTables &t = p.t;
    const uint32_t pr = fwd ? pair_fwd(p, i) : pair_bwd(p, i);
    const uint32_t m = __ldg((fwd ? t.fSlotCount : t.bSlotCount) + pr);
    const uint32_t ms = fwd ? t.msf : t.msb;
    const uint32_t *R = (fwd ? p.w.Rf : p.w.Rb) + (size_t)i * ms;
    uint32_t rep = 0;
    bool gen = false;
    for (uint32_t s = 0; s < m; ++s) {
        const uint32_t e = R[s];
        if (e) { if (!rep) rep = e; else if (e != rep) gen = true; }
    }
    if (fwd) {
        p.w.fkind[i] = gen ? 1u : 0u;
        if (!gen) p.w.FJ[i + 1] = rep;
    } else {
        p.w.bkind[i] = gen ? 1u : 0u;
        if (!gen) p.w.BJ[i] = rep;
    }
    if (gen && p.scan) atomicAdd(p.w.scan + kScanGeneral, 1u);   // the scan has work
}

__device__ void classify_at(const Params &p, uint32_t i) {
    if (i == 0 && !(p.shard & SHARD_PREV)) {
        p.w.FJ[0] = p.t.fI;
        p.w.FJ[1] = p.w.Rf[0];
        p.w.fkind[0] = 0;
    } else {
        classify(p, true, i);
    }
    if (p.recognize) return;
    if (i == p.c - 1 && !(p.shard & SHARD_NEXT)) {
        p.w.BJ[p.c] = p.t.bF;
        p.w.BJ[i] = p.w.Rb[(size_t)i * p.t.msb];
        p.w.bkind[i] = 0;
    } else {
        classify(p, false, i);
    }
}

// Chains of general chunks, evaluated in order from their known neighbour
// (started by the chunk just after / before the neighbour).
template <bool FWD>
__device__ void chain_from(const Params &p, uint32_t i) {
    bool bad = false;
    if (FWD && p.w.fkind[i] == 1 && p.w.fkind[i - 1] == 0) {     // i >= 1: fkind[0] == 0
        uint32_t cur = p.w.FJ[i];
        for (uint32_t j = i; j < p.c && p.w.fkind[j] == 1; ++j) {
            cur = eval_chunk(p, true, j, cur, bad);
            p.w.FJ[j + 1] = cur;
        }
    }
    if (!FWD && p.w.bkind[i] == 1 && p.w.bkind[i + 1] == 0) {    // i <= c-2: bkind[c-1] == 0
        uint32_t cur = p.w.BJ[i + 1];
        for (int64_t j = i; j >= 0 && p.w.bkind[j] == 1; --j) {
            cur = eval_chunk(p, false, (uint32_t)j, cur, bad);
            p.w.BJ[j] = cur;
        }
    }
    if (bad) atomicExch(&p.w.flags[FLAG_INTERNAL], 1);
}
__device__ void chain_at(const Params &p, uint32_t i) {
    chain_from<true>(p, i);
    if (!p.recognize) chain_from<false>(p, i);
}

__global__ void join_classify_kernel(const __grid_constant__ Params p) {
    pdl_wait();
    pdl_trigger();
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < p.c) classify_at(p, i);
}

__global__ void join_chain_kernel(const __grid_constant__ Params p) {
    pdl_wait();
    pdl_trigger();
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < p.c) chain_at(p, i);
}

__device__ bool grid_barrier(uint32_t *w);

// ------------------------------------------------------------------ slice maps
// A slice of a longer text (sharded parse): its forward map sends the
// forward state S at the slice's start to the state at its end, the
// composition of its chunk maps (Eq. joiner) in order; its backward map sends
// the backward state at the slice's end to the state at its start.  Every
// chunk's map over the classic-DFA states is a byte table (eval_chunk; the
// first chunk of the text's first slice starts from I, so its map is
// constant, and the last chunk of the last slice from F), and the tables are
// composed by a tree reduction: in round r, the table of chunk i (i a
// multiple of 2^{r+1}) absorbs that of chunk i + 2^r.  Cooperative launch,
// the rounds separated by the bounded grid barrier.
template <uint32_t LANES>
__device__ void shard_map(const Params &p, uint8_t *maps) {
    const uint32_t lane = LANES == 1 ? 0u : (threadIdx.x & 31), upb = blockDim.x / LANES;
    const uint64_t gw = (uint64_t)blockIdx.x * upb + threadIdx.x / LANES, nw = (uint64_t)gridDim.x * upb;
    const uint32_t nsf = p.t.nfd + 1, nsb = p.t.nbd + 1, c = p.c;
    bool bad = false;
    for (uint64_t i = gw; i < c; i += nw) {
        uint8_t *T = p.w.fTab + i * nsf;
        const bool first = i == 0 && !(p.shard & SHARD_PREV);           // runs from I: one output
        for (uint32_t S = lane; S < nsf; S += LANES)
            T[S] = (uint8_t)(first ? (S ? p.w.Rf[0] : 0u) : eval_chunk(p, true, (uint32_t)i, S, bad));
        uint8_t *B = p.w.bTab + i * nsb;
        const bool last = i == c - 1 && !(p.shard & SHARD_NEXT);         // runs from F: one output
        for (uint32_t S = lane; S < nsb; S += LANES)
            B[S] = (uint8_t)(last ? (S ? p.w.Rb[(size_t)i * p.t.msb] : 0u) : eval_chunk(p, false, (uint32_t)i, S, bad));
    }
    if (bad) atomicExch(&p.w.flags[FLAG_INTERNAL], 1);
    for (uint32_t r = 0; (1ull << r) < c; ++r) {
        if (!grid_barrier(p.w.scan)) { atomicExch(&p.w.flags[FLAG_TIMEOUT], 1); return; }
        const uint64_t step = 1ull << r, pairs = (c + 2 * step - 1) / (2 * step);
        for (uint64_t q = gw; q < pairs; q += nw) {
            const uint64_t i = q * 2 * step, j = i + step;
            if (j >= c) continue;
            uint8_t *Ti = p.w.fTab + i * nsf;                          // [i, j) then [j, j + step)
            const uint8_t *Tj = p.w.fTab + j * nsf;
            for (uint32_t S = lane; S < nsf; S += LANES) Ti[S] = __ldcg(Tj + __ldcg(Ti + S));
            uint8_t *Bi = p.w.bTab + i * nsb;                          // the later range first
            const uint8_t *Bj = p.w.bTab + j * nsb;
            uint8_t v[kScanStates / (LANES == 1 ? 1 : 32)];
            uint32_t nv = 0;
            for (uint32_t S = lane; S < nsb; S += LANES) v[nv++] = __ldcg(Bi + __ldcg(Bj + S));
            if (LANES == 32) __syncwarp();
            nv = 0;
            for (uint32_t S = lane; S < nsb; S += LANES) Bi[S] = v[nv++];
        }
    }
    if (!grid_barrier(p.w.scan)) { atomicExch(&p.w.flags[FLAG_TIMEOUT], 1); return; }
    if (blockIdx.x == 0) {                                            // the slice's maps
        for (uint32_t S = threadIdx.x; S < nsf; S += blockDim.x) maps[S] = __ldcg(p.w.fTab + S);
        for (uint32_t S = threadIdx.x; S < nsb; S += blockDim.x) maps[nsf + S] = __ldcg(p.w.bTab + S);
        if (threadIdx.x == 0) {
            const int32_t fl = __ldcg(&p.w.flags[FLAG_INTERNAL]), to = __ldcg(&p.w.flags[FLAG_TIMEOUT]);
            *p.status = to ? RE_E_TIMEOUT : fl ? RE_E_INTERNAL : RE_OK;
        }
    }
}

__global__ void __launch_bounds__(kBlockThreads) join_map_kernel(const __grid_constant__ Params p, uint8_t *maps) {
    if (p.t.nfd < 16 && p.t.nbd < 16) shard_map<1>(p, maps);
    else shard_map<32>(p, maps);
}

// Live slots of chunk i (their end state is not the empty set).
__device__ uint32_t live_slots(const Params &p, bool fwd, uint32_t i, uint32_t pr) {
    const DevTables &t = p.t;
    const uint32_t m = __ldg((fwd ? t.fSlotCount : t.bSlotCount) + pr);
    const uint32_t ms = fwd ? t.msf : t.msb;
    const uint32_t *R = (fwd ? p.w.Rf : p.w.Rb) + (size_t)i * ms;
    uint32_t L = 0;
    for (uint32_t s = 0; s < m; ++s)
        if (R[s]) L |= 1u << s;
    return L;
}

// Check each chunk's guessed output against its (now known) input and keep
// the slots that input enters for the fix-up.
__device__ void verify_at(const Params &p, uint32_t i) {
    {   // forward: input FJ[i] -> output FJ[i+1]
        const uint32_t in = p.w.FJ[i], out = p.w.FJ[i + 1];
        bool fail = in == 0 || out == 0;
        uint32_t H = 0;
        if (i > 0 && in != 0) {
            const uint32_t pr = pair_fwd(p, i);
            H = slot_hits(p.t, true, pr, in);
            if (!fail && p.w.fkind[i] == 0) fail = (H & live_slots(p, true, i, pr)) == 0;
        }
        p.w.fhit[i] = H;
        if (fail) atomicMin(&p.w.flags[FLAG_FFAIL], (int32_t)i);
        p.w.FC[(uint64_t)i * p.S] = in;                              // position i*k
        if (i == p.c - 1 && (p.n & 63) == 0) p.w.FC[p.n >> 6] = p.w.FJ[p.c];   // position n
    }
    if (p.recognize) return;
    {   // backward: input BJ[i+1] -> output BJ[i]
        const uint32_t in = p.w.BJ[i + 1], out = p.w.BJ[i];
        bool fail = in == 0 || out == 0;
        uint32_t H = 0;
        if (i < p.c - 1 && in != 0) {
            const uint32_t pr = pair_bwd(p, i);
            H = slot_hits(p.t, false, pr, in);
            if (!fail && p.w.bkind[i] == 0) fail = (H & live_slots(p, false, i, pr)) == 0;
        }
        p.w.bhit[i] = H;
        if (fail) atomicMin(&p.w.flags[FLAG_BFAIL], (int32_t)i);
        if (i + 1 < p.c) {
            p.w.BC[(uint64_t)(i + 1) * p.S - 1] = in;                // position (i+1)*k
        } else {                                                     // groups whose end is clipped to n
            for (uint64_t g = (p.n + 63) / 64 - 1; g < p.Gc; ++g) p.w.BC[g] = in;
        }
    }
}

// verify_at with a warp per chunk: lane j tests slot j (whether the input
// enters it, whether its run is live) and a ballot gathers the masks; lane 0
// does the rest.  Slot counts are at most 32.
__device__ __forceinline__ uint32_t hits_warp(const Params &p, bool fwd, uint32_t i, uint32_t pr, uint32_t S,
                                              uint32_t &live) {
    const DevTables &t = p.t;
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t m = __ldg((fwd ? t.fSlotCount : t.bSlotCount) + pr);
    const uint32_t ms = fwd ? t.msf : t.msb;
    const uint32_t *R = (fwd ? p.w.Rf : p.w.Rb) + (size_t)i * ms;
    live = __ballot_sync(0xFFFFFFFFu, lane < m && R[lane] != 0);
    const uint8_t *of = fwd ? t.fSlotOf : t.bSlotOf;
    if (of) {                                    // starts from every DFA state: S enters its own slot only
        const uint32_t n = fwd ? t.nf : t.nb;
        const uint32_t j = S < n ? __ldg(of + (size_t)pr * n + S) : 0xFFu;
        return j == 0xFFu ? 0u : 1u << j;
    }
    const uint32_t W = t.W;
    const uint64_t *mask = (fwd ? t.fSlotMask : t.bSlotMask) + (size_t)pr * ms * W;
    const uint64_t *sb = (fwd ? t.fBits : t.bBits) + (size_t)S * W;
    return __ballot_sync(0xFFFFFFFFu, lane < m && any_and(sb, mask + (size_t)lane * W, W));
}

// Both directions' loads come before any store (a store could alias a later
// load, so the compiler would keep them in order), so the two dependent load
// chains of a chunk overlap.
__device__ void verify_warp(const Params &p, uint32_t i) {
    const uint32_t lane = threadIdx.x & 31;
    const bool both = !p.recognize;
    // forward: input FJ[i] -> output FJ[i+1]; backward: input BJ[i+1] -> output BJ[i]
    const uint32_t fin = p.w.FJ[i], fout = p.w.FJ[i + 1];
    const uint32_t bin = both ? p.w.BJ[i + 1] : 0u, bout = both ? p.w.BJ[i] : 0u;
    const uint32_t fkind = p.w.fkind[i], bkind = both ? p.w.bkind[i] : 1u;
    const uint32_t fend = (i == p.c - 1 && (p.n & 63) == 0) ? p.w.FJ[p.c] : 0u;
    bool ffail = fin == 0 || fout == 0, bfail = both && (bin == 0 || bout == 0);
    uint32_t fH = 0, bH = 0;
    if (i > 0 && fin != 0) {
        uint32_t L;
        fH = hits_warp(p, true, i, pair_fwd(p, i), fin, L);
        if (!ffail && fkind == 0) ffail = (fH & L) == 0;
    }
    if (both && i < p.c - 1 && bin != 0) {
        uint32_t L;
        bH = hits_warp(p, false, i, pair_bwd(p, i), bin, L);
        if (!bfail && bkind == 0) bfail = (bH & L) == 0;
    }
    if (lane != 0) return;
    p.w.fhit[i] = fH;
    if (ffail) atomicMin(&p.w.flags[FLAG_FFAIL], (int32_t)i);
    p.w.FC[(uint64_t)i * p.S] = fin;                                     // position i*k
    if (i == p.c - 1 && (p.n & 63) == 0) p.w.FC[p.n >> 6] = fend;       // position n
    if (!both) return;
    p.w.bhit[i] = bH;
    if (bfail) atomicMin(&p.w.flags[FLAG_BFAIL], (int32_t)i);
    if (i + 1 < p.c) {
        p.w.BC[(uint64_t)(i + 1) * p.S - 1] = bin;                       // position (i+1)*k
    } else {                                                             // groups whose end is clipped to n
        for (uint64_t g = (p.n + 63) / 64 - 1; g < p.Gc; ++g) p.w.BC[g] = bin;
    }
}

// Accept iff both joins ran through and C_0 = I ∩ Ĵ_1 is not empty
// (recognizer: iff the forward join ran through and J_c ∩ F is not empty).
__device__ void status_of(const Params &p) {
    const DevTables &t = p.t;
    int32_t st = RE_OK;
    // flags are updated by atomics of the verify blocks: read them from L2
    const int32_t ffail = __ldcg(&p.w.flags[FLAG_FFAIL]), bfail = __ldcg(&p.w.flags[FLAG_BFAIL]);
    if (ffail < (int32_t)p.c || (!p.recognize && bfail < (int32_t)p.c)) {
        st = RE_REJECTED;
    } else if (p.recognize) {
        const uint32_t jc = __ldcg(p.w.FJ + p.c);
        if (!any_and(t.fBits + (size_t)jc * t.W, t.bBits + (size_t)t.bF * t.W, t.W)) st = RE_REJECTED;
    } else {
        const uint32_t b0 = __ldcg(p.w.BJ);
        if (!(b0 && any_and(t.fBits + (size_t)t.fI * t.W, t.bBits + (size_t)b0 * t.W, t.W))) st = RE_REJECTED;
    }
    if (__ldcg(&p.w.flags[FLAG_INTERNAL])) st = RE_E_INTERNAL;
    if (__ldcg(&p.w.flags[FLAG_TIMEOUT])) st = RE_E_TIMEOUT;
    *p.status = st;
}

// Verify every chunk; the last block to finish then sets the status word,
// once every block's writes are visible (each block fences its writes before
// it takes a ticket; the last ticket holder fences again before reading).
__global__ void join_verify_kernel(const __grid_constant__ Params p) {
    pdl_wait();
    pdl_trigger();
    const uint64_t i = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;   // a warp per chunk
    if (i < p.c) verify_warp(p, (uint32_t)i);
    __shared__ int last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&p.w.flags[FLAG_DONE], 1) == (int32_t)gridDim.x - 1;
    __syncthreads();
    if (last && threadIdx.x == 0) {
        __threadfence();
        status_of(p);
    }
}

__global__ void flags_init_kernel(const __grid_constant__ Params p) {
    if (threadIdx.x < FLAG_COUNT) p.w.flags[threadIdx.x] = threadIdx.x < 2 ? (int32_t)p.c : 0;
    if (p.scan)
        for (uint32_t q = threadIdx.x; q < kScanWords; q += blockDim.x) p.w.scan[q] = 0;
}

// ------------------------------------------------------------------ scan join
// Eq. (joiner) as a scan.  Chunk i maps its input state J_i to J_{i+1}; a
// chunk whose live slots all end in one state maps every input that can
// continue to that state (classify resolves it at once).  Every other chunk
// gets its map over the classic-DFA states (a byte table; the union of the
// slot end states the input enters, as eval_chunk computes it), and the
// chunks are resolved by pointer jumping: chunk i holds the map of the
// chunk range (l_i, i] and the link l_i; in each round, if chunk l_i is
// resolved, J_{i+1} = map(J_{l_i + 1}), else the range doubles: map becomes
// map_i o map_{l_i} and l_i becomes l_{l_i}.  A chain of L chunks resolves in
// ceil(log2 L) + 1 rounds instead of L dependent steps.  Backward (Ĵ) the same
// with the chunks taken right to left.  The rounds are separated by a grid
// barrier of this cooperative launch; each barrier wait is bounded, and a
// wait that runs out sets the status RE_E_TIMEOUT.
constexpr uint32_t kResolved = 0xFFFFFFFFu;
static_assert(kScanGeneral < kScanWords, "scan words");

// All blocks of the grid meet here; false when this block's wait ran out.
__device__ bool grid_barrier(uint32_t *w) {
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        ok = 1;
        volatile uint32_t *gen = w + 1;
        const uint32_t g = *gen;
        __threadfence();
        if (atomicAdd(w, 1u) == gridDim.x - 1) {
            w[0] = 0;                                   // every other block waits on gen: reset first
            __threadfence();
            atomicAdd(w + 1, 1u);
        } else {
            uint32_t it = 0;
            while (*gen == g)
                if (++it > kWaitLimit) { ok = 0; break; }
        }
        __threadfence();
    }
    __syncthreads();
    return ok != 0;
}

// The scan's units are groups of p.scan consecutive chunks (at most 32): a warp
// composes a group's maps, its lanes over the states, and once the scan has every
// group's output, a thread per group takes the state through its chunks.  In a
// round a unit costs its barrier's share and two dependent reads whatever it
// stands for, so tens of thousands of single chunks were most of the join: 64 MiB in
// one line under the log RE 1360 us with a unit per chunk, 679 with one per 8.
template <bool FWD> struct ScanGroup {
    uint32_t a, n;                                     // its first chunk in the text, and how many
    __device__ ScanGroup(const Params &p, uint32_t g) : a(g * p.scan), n(min(p.scan, p.c - g * p.scan)) {}
    __device__ uint32_t chunk(uint32_t q) const { return FWD ? a + q : a + n - 1 - q; }   // in walking order
    __device__ uint32_t in() const { return FWD ? a : a + n; }      // J indices of its input and output
    __device__ uint32_t out() const { return FWD ? a + n : a; }
};

// A group whose output some chunk of its own determines is resolved at once;
// the others get their map over the classic-DFA states.
template <bool FWD>
__device__ void scan_map(const Params &p, uint32_t g, bool &bad) {
    const uint32_t lane = threadIdx.x & 31, ns = (FWD ? p.t.nfd : p.t.nbd) + 1;
    const ScanGroup<FWD> G(p, g);
    uint32_t *J = FWD ? p.w.FJ : p.w.BJ, *link = FWD ? p.w.fLink : p.w.bLink;
    const uint32_t *kinds = FWD ? p.w.fkind : p.w.bkind;
    const unsigned known = __ballot_sync(0xFFFFFFFFu, lane < G.n && kinds[G.chunk(lane < G.n ? lane : 0)] == 0);
    if (known) {
        if (lane == 0) {
            uint32_t q = 31 - __clz(known);            // the last of them
            if (q + 1 < G.n) {
                uint32_t cur = J[FWD ? G.chunk(q) + 1 : G.chunk(q)];
                while (++q < G.n) cur = eval_chunk(p, FWD, G.chunk(q), cur, bad);
                J[G.out()] = cur;
            }
            link[g] = kResolved;
        }
        return;
    }
    uint8_t *T = (FWD ? p.w.fTab : p.w.bTab) + (size_t)g * ns;
    for (uint32_t S = lane; S < ns; S += 32) {
        uint32_t cur = S;
        for (uint32_t q = 0; q < G.n; ++q) cur = eval_chunk(p, FWD, G.chunk(q), cur, bad);
        T[S] = (uint8_t)cur;
    }
    if (lane == 0) link[g] = FWD ? g - 1 : g + 1;      // the text's first (last) chunk has one output
}

// One direction of one group in a round, by a warp.
template <bool FWD>
__device__ uint32_t scan_step(const Params &p, uint32_t g, uint32_t ng, uint32_t cur) {
    const uint32_t lane = threadIdx.x & 31, ns = (FWD ? p.t.nfd : p.t.nbd) + 1;
    uint32_t *link = FWD ? p.w.fLink : p.w.bLink;
    uint8_t *tab = FWD ? p.w.fTab : p.w.bTab;
    uint32_t *J = FWD ? p.w.FJ : p.w.BJ;
    const uint32_t nxt = cur ^ 1u;
    const uint32_t l = __ldcg(link + (size_t)cur * ng + g);
    if (l == kResolved) {
        if (lane == 0) link[(size_t)nxt * ng + g] = kResolved;
        return 0;
    }
    const uint8_t *Tg = tab + ((size_t)cur * ng + g) * ns;
    const uint32_t ll = __ldcg(link + (size_t)cur * ng + l);
    if (ll == kResolved) {                             // the range's input is known
        if (lane == 0) {
            const uint32_t v = __ldcg(J + ScanGroup<FWD>(p, l).out());
            J[ScanGroup<FWD>(p, g).out()] = v < ns ? (uint32_t)__ldcg(Tg + v) : 0u;   // v >= ns: no DFA state, rejected
            link[(size_t)nxt * ng + g] = kResolved;
        }
        return 0;
    }
    const uint8_t *Tl = tab + ((size_t)cur * ng + l) * ns;
    uint8_t *Tn = tab + ((size_t)nxt * ng + g) * ns;
    for (uint32_t S = lane; S < ns; S += 32) Tn[S] = __ldcg(Tg + __ldcg(Tl + S));
    if (lane == 0) link[(size_t)nxt * ng + g] = ll;
    return 1;
}

// The states between a group's chunks from its input, by a thread.
template <bool FWD>
__device__ void scan_fill(const Params &p, uint32_t g, bool &bad) {
    const ScanGroup<FWD> G(p, g);
    uint32_t *J = FWD ? p.w.FJ : p.w.BJ;
    const uint32_t *kinds = FWD ? p.w.fkind : p.w.bkind;
    uint32_t cur = __ldcg(J + G.in());
    for (uint32_t q = 0; q < G.n; ++q) {
        const uint32_t i = G.chunk(q);
        uint32_t *o = J + (FWD ? i + 1 : i);
        if (kinds[i]) *o = cur = eval_chunk(p, FWD, i, cur, bad);
        else cur = __ldcg(o);
    }
}

// False when a barrier wait ran out.
__device__ bool join_scan(const Params &p) {
    const uint32_t wpb = blockDim.x / 32, ng = (p.c + p.scan - 1) / p.scan;
    const uint64_t gw = (uint64_t)blockIdx.x * wpb + threadIdx.x / 32, nw = (uint64_t)gridDim.x * wpb;
    const bool bwd = !p.recognize;
    bool bad = false;
    for (uint64_t g = gw; g < ng; g += nw) {
        scan_map<true>(p, (uint32_t)g, bad);
        if (bwd) scan_map<false>(p, (uint32_t)g, bad);
    }
    if (p.scan_stall && blockIdx.x == 0) return false;   // test hook: the other blocks' waits run out
    if (!grid_barrier(p.w.scan)) { atomicExch(&p.w.flags[FLAG_TIMEOUT], 1); return false; }
    for (uint32_t r = 0; r < kScanRounds; ++r) {
        uint32_t open = 0;
        for (uint64_t g = gw; g < ng; g += nw) {
            open += scan_step<true>(p, (uint32_t)g, ng, r & 1);
            if (bwd) open += scan_step<false>(p, (uint32_t)g, ng, r & 1);
        }
        if ((threadIdx.x & 31) == 0 && open) atomicAdd(p.w.scan + 2 + r, open);
        if (!grid_barrier(p.w.scan)) { atomicExch(&p.w.flags[FLAG_TIMEOUT], 1); return false; }
        if (__ldcg(p.w.scan + 2 + r) == 0) break;     // every group resolved (same value in every block)
    }
    if (bad) atomicExch(&p.w.flags[FLAG_INTERNAL], 1);
    if (p.scan == 1) return true;                     // a group's output is its chunk's
    for (uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; j < (bwd ? 2ull : 1ull) * ng;
         j += (uint64_t)gridDim.x * blockDim.x) {
        if (j < ng) scan_fill<true>(p, (uint32_t)j, bad);
        else scan_fill<false>(p, (uint32_t)(j - ng), bad);
    }
    if (bad) atomicExch(&p.w.flags[FLAG_INTERNAL], 1);
    if (!grid_barrier(p.w.scan)) { atomicExch(&p.w.flags[FLAG_TIMEOUT], 1); return false; }
    return true;
}

__global__ void __launch_bounds__(kBlockThreads) join_scan_kernel(const __grid_constant__ Params p) {
    // every chunk has one output for every input (the common case): classify
    // has resolved them all
    if (__ldcg(p.w.scan + kScanGeneral) == 0 && !p.scan_stall) return;
    join_scan(p);
}

// ------------------------------------------------------------------ after the lane walk
// A general chunk (kind 1: its runs never met) of the lane walk, once the scan
// has its output: the walk had no state to go on with, so the head of the
// chunk its run enters is walked here, with the check the walk makes.
constexpr uint32_t kFixThreads = 64;           // a batch's: as many as a heads round has chunks
template <bool FWD, bool OUT>
__device__ void join_walk_fix(const Params &p, const LaneTab &T, uint32_t ns, uint32_t i) {
    const uint32_t *kinds = FWD ? p.w.fkind : p.w.bkind, *J = FWD ? p.w.FJ : p.w.BJ;
    if (!kinds[i]) return;
    uint8_t *S = FWD ? p.w.FS : p.w.BS;
    const uint32_t in = __ldcg(J + (FWD ? i : i + 1)), out = __ldcg(J + (FWD ? i + 1 : i));
    bool fail = in == 0 || out == 0 || out >= ns;
    if (OUT && FWD && i == p.c - 1) S[p.n] = (uint8_t)out;
    const uint32_t o = FWD ? i + 1 : i - 1;
    if (!fail && (FWD ? i + 1 < p.c : i > 0) && (OUT || kinds[o] == 0)) {   // else no columns, and no state to check
        const uint64_t nbase = (uint64_t)o * p.k;
        const uint32_t nlen = chunk_len(p, o), edge = min(kUnit * (FWD ? p.w.fconv : p.w.bconv)[o], nlen);
        uint32_t mid;
        const uint32_t e = walk_cols<0, FWD, OUT>(T, p.x, S, nbase + (FWD ? 0 : edge), nbase + (FWD ? edge : nlen),
                                                  nbase + (FWD ? 0 : nlen), out,
                                                  (reinterpret_cast<uintptr_t>(p.x) & 31) == 0, mid);
        if (kinds[o] == 0) fail = e == 0 || e != (FWD ? p.w.fnrec : p.w.bnrec)[o];
    }
    if (fail) atomicMin(&p.w.flags[FWD ? FLAG_FFAIL : FLAG_BFAIL], (int32_t)i);
}

// The status after the lane walk.  The walk has checked every chunk whose
// runs met (J_i is the state before it, and it enters live slots exactly when
// the walk through the head reaches their state), so without general chunks
// nothing is left but the verdict; with them, the scan over their maps, the
// heads after them and then the verdict, separated by the bounded grid
// barrier (cooperative launch).
__global__ void __launch_bounds__(kBlockThreads) join_walk_kernel(const __grid_constant__ Params p) {
    extern __shared__ __align__(16) uint8_t sm[];
    if (__ldcg(p.w.scan + kScanGeneral) == 0 && !p.scan_stall) {
        if (blockIdx.x == 0 && threadIdx.x == 0) status_of(p);
        return;
    }
    if (!join_scan(p)) {
        if (threadIdx.x == 0) atomicExch(p.status, RE_E_TIMEOUT);
        return;
    }
    const uint32_t cw = class_words(p.t), nsf = p.t.nfd + 1, nsb = p.t.nbd + 1;
    stage_classes(p.t, sm);
    stage_lane_table<0>(p.t.fc8, nsf * cw, sm + 256);
    stage_lane_table<0>(p.t.bc8, nsb * cw, sm + 256 + nsf * cw * 4);
    __syncthreads();
    const LaneTab F{smem_u32(sm + 256), sm, cw * 4}, B{smem_u32(sm + 256 + nsf * cw * 4), sm, cw * 4};
    const uint64_t items = (p.recognize ? 1ull : 2ull) * p.c;     // a thread per chunk and direction
    for (uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; j < items; j += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t i = (uint32_t)(j < p.c ? j : j - p.c);
        if (j < p.c) {
            if (p.mat) join_walk_fix<true, true>(p, F, nsf, i);
            else join_walk_fix<true, false>(p, F, nsf, i);
        } else {
            if (p.mat) join_walk_fix<false, true>(p, B, nsb, i);
            else join_walk_fix<false, false>(p, B, nsb, i);
        }
    }
    if (!grid_barrier(p.w.scan)) {
        if (threadIdx.x == 0) atomicExch(p.status, RE_E_TIMEOUT);
        return;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) status_of(p);
}

// The same for every text of a batch's lane-walk groups, a block per text, its
// lower half forward and its upper half backward: chunks whose runs never met are
// evaluated in chains.  Longer texts with such chunks are left to join_long_kernel.
constexpr uint32_t kJoinThreads = 128;
__global__ void __launch_bounds__(kJoinThreads) join_walk_batch_kernel(const __grid_constant__ WalkBatch b) {
    extern __shared__ __align__(16) uint8_t sm[];
    const Params &p = b.texts[blockIdx.x];
    if (!p.rvar) return;                                      // a group of the other kernels
    if (p.n == 0) {
        if (threadIdx.x == 0) empty_text(p);
        return;
    }
    if (p.w.scan[kScanGeneral]) {
        if (p.c > kJoinChunks) {
            if (threadIdx.x == 0) *b.general = 1;
            return;
        }
        const uint32_t half = b.recognize ? blockDim.x : blockDim.x / 2, t = threadIdx.x % half;
        const bool fwd = threadIdx.x < half;
        for (uint32_t i = t; i < p.c; i += half) {
            if (fwd) chain_from<true>(p, i);
            else chain_from<false>(p, i);
        }
        __threadfence();
        const uint32_t cw = class_words(p.t), nsf = p.t.nfd + 1, nsb = p.t.nbd + 1;
        stage_classes(p.t, sm);
        stage_lane_table<0>(p.t.fc8, nsf * cw, sm + 256);
        stage_lane_table<0>(p.t.bc8, nsb * cw, sm + 256 + nsf * cw * 4);
        __syncthreads();
        const LaneTab F{smem_u32(sm + 256), sm, cw * 4}, B{smem_u32(sm + 256 + nsf * cw * 4), sm, cw * 4};
        for (uint32_t i = t; i < p.c; i += half) {
            if (b.recognize) join_walk_fix<true, false>(p, F, nsf, i);
            else if (fwd) join_walk_fix<true, true>(p, F, nsf, i);
            else join_walk_fix<false, true>(p, B, nsb, i);
        }
        __threadfence();
        __syncthreads();
    }
    if (threadIdx.x == 0) status_of(p);
}

// Texts of more than kJoinChunks chunks some of whose runs never met: the
// chains, then (HEADS) the heads after such chunks, over the spans of the heads
// kernel, a thread per chunk and direction of all groups.  By a block per text one
// genome text of 64 MiB took 38 ms.  The last item of a text sets its status.
// Launched only for batches with such long texts.
template <bool HEADS>
__global__ void __launch_bounds__(kFixThreads) join_long_kernel(const __grid_constant__ WalkBatch b) {
    extern __shared__ __align__(16) uint8_t sm[];
    pdl_wait();
    if (!__ldcg(b.general)) return;
    const bool pairs = !b.recognize, backward = pairs && (blockIdx.x & 1);
    const WalkSpan w = b.heads[pairs ? blockIdx.x >> 1 : blockIdx.x];
    const WalkGroup &g = b.groups[w.group];
    const uint32_t cw = class_words(g.t), ns = (backward ? g.t.nbd : g.t.nfd) + 1;
    const LaneTab T{smem_u32(sm + 256), sm, cw * 4};
    bool staged = false;
    for (uint64_t first = (uint64_t)w.idx * kFixThreads; first < g.chunks; first += (uint64_t)w.cnt * kFixThreads) {
        const uint64_t j = first + threadIdx.x;
        const uint32_t ti = j < g.chunks ? text_of(g.chunk_base, g.nt, j) : 0u;
        const Params &p = g.texts[ti];
        const uint32_t i = (uint32_t)(j - __ldg(g.chunk_base + ti));
        const bool mine = j < g.chunks && p.c > kJoinChunks && p.w.scan[kScanGeneral] != 0;
        if (!HEADS) {
            if (mine && backward) chain_from<false>(p, i);
            else if (mine) chain_from<true>(p, i);
            continue;
        }
        if (__syncthreads_or(mine) && !staged) {
            stage_classes(g.t, sm);
            stage_lane_table<0>(backward ? g.t.bc8 : g.t.fc8, ns * cw, sm + 256);
            __syncthreads();
            staged = true;
        }
        if (!mine) continue;
        if (b.recognize) join_walk_fix<true, false>(p, T, ns, i);
        else if (backward) join_walk_fix<false, true>(p, T, ns, i);
        else join_walk_fix<true, true>(p, T, ns, i);
        __threadfence();
        if ((uint32_t)atomicAdd(&p.w.flags[FLAG_DONE], 1) + 1 == (pairs ? 2u : 1u) * p.c) {
            __threadfence();
            status_of(p);
        }
    }
}

// ------------------------------------------------------------------ batch
// The same steps over every chunk of every text of a group: thread j takes
// flat chunk j (its text by binary search on the chunk prefix sums).
enum BatchStep { B_CLASSIFY = 0, B_CHAIN = 1, B_VERIFY = 2 };

template <int STEP>
__global__ void join_batch_kernel(const __grid_constant__ BatchGroup b) {
    const uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= b.chunks) return;
    const uint32_t ti = text_of(b.chunk_base, b.nt, j);
    const Params &p = b.texts[ti];
    const uint32_t i = (uint32_t)(j - b.chunk_base[ti]);
    if (STEP == B_CLASSIFY) classify_at(p, i);
    else if (STEP == B_CHAIN) chain_at(p, i);
    else verify_at(p, i);
}

// Status of every text; an empty text has the single column C_0 = I ∩ F.
__global__ void status_batch_kernel(const __grid_constant__ BatchGroup b) {
    const uint32_t ti = blockIdx.x * blockDim.x + threadIdx.x;
    if (ti >= b.nt) return;
    const Params &p = b.texts[ti];
    if (p.n == 0) empty_text(p);
    else status_of(p);
}

// Work counters of every group and the join flags of every text.
__global__ void batch_init_kernel(const Params *texts, uint32_t nt, uint32_t *queues, uint32_t nq) {
    const uint32_t j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < nq) queues[j] = 0;
    if (j < nt && texts[j].n) {
        int32_t *f = texts[j].w.flags;
        for (uint32_t q = 0; q < FLAG_COUNT; ++q) f[q] = q < 2 ? (int32_t)texts[j].c : 0;
        if (texts[j].rvar) texts[j].w.scan[kScanGeneral] = 0;
    }
}

}  // namespace

// Cooperative launch of kernel with a warp per unit, at most the blocks the
// device holds at once.
template <typename... KArgs, typename... Args>
static bool launch_coop(void (*kernel)(KArgs...), size_t smem, uint64_t units, cudaStream_t s, int sm_count,
                        Args &&...args) {
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kBlockThreads, smem);
    const uint64_t want = (units + kBlockThreads / 32 - 1) / (kBlockThreads / 32);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>(want, (uint64_t)std::max(per_sm, 1) * sm_count));
    cfg.blockDim = kBlockThreads;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...) == cudaSuccess;
}

// A warp per group of the scan, and a second block where there are chunks for
// one (the bounded waits are tested between blocks).
static uint64_t scan_units(const Params &p) { return std::max(p.c / p.scan + 1, std::min(p.c, 16u)); }

// Classify, then the scan (a cooperative launch: its blocks meet at grid
// barriers, so they must all be resident) or the chains, then verify.
bool launch_join(const Params &p, cudaStream_t s, int sm_count) {
    const uint32_t blocks = (p.c + kBlockThreads - 1) / kBlockThreads;
    launch_dependent(join_classify_kernel, blocks, kBlockThreads, 0, s, p);
    if (p.scan) {
        if (!launch_coop(join_scan_kernel, 0, scan_units(p), s, sm_count, p)) return false;
    } else {
        launch_dependent(join_chain_kernel, blocks, kBlockThreads, 0, s, p);
    }
    const uint32_t vblocks = (uint32_t)(((uint64_t)p.c * 32 + kBlockThreads - 1) / kBlockThreads);
    launch_dependent(join_verify_kernel, vblocks, kBlockThreads, 0, s, p);
    return true;
}

void launch_flags_init(const Params &p, cudaStream_t s) { flags_init_kernel<<<1, 32, 0, s>>>(p); }

void launch_batch_init(const Params *texts, uint32_t nt, uint32_t *queues, uint32_t nq, cudaStream_t s) {
    const uint32_t n = nt > nq ? nt : nq;
    batch_init_kernel<<<(n + kBlockThreads - 1) / kBlockThreads, kBlockThreads, 0, s>>>(texts, nt, queues, nq);
}

size_t join_walk_smem(const DevTables &t) { return 256 + (size_t)(t.nfd + t.nbd + 2) * class_words(t) * 4; }

void launch_join_walk_batch(const WalkBatch &b, cudaStream_t s) {
    if (!b.nt) return;
    static uint64_t attr_walk = 0, attr_long = 0;
    allow_smem(join_walk_batch_kernel, &attr_walk);
    allow_smem(join_long_kernel<true>, &attr_long);
    join_walk_batch_kernel<<<b.nt, kJoinThreads, b.join_smem, s>>>(b);
    if (b.n_heads && b.long_texts) {
        const uint32_t blocks = b.n_heads * (b.recognize ? 1 : 2);
        launch_dependent(join_long_kernel<false>, blocks, kFixThreads, 0, s, b);
        launch_dependent(join_long_kernel<true>, blocks, kFixThreads, b.join_smem, s, b);
    }
}

bool launch_join_walk(const Params &p, cudaStream_t s, int sm_count) {
    const size_t smem = join_walk_smem(p.t);
    static uint64_t attr_done = 0;
    allow_smem(join_walk_kernel, &attr_done);
    return launch_coop(join_walk_kernel, smem, scan_units(p), s, sm_count, p);
}

// A slice's maps after the lane walk (every slot's end state, p.rall) or the
// other reach shapes.
bool launch_shard_map(const Params &p, uint8_t *d_maps, cudaStream_t s, int sm_count) {
    return launch_coop(join_map_kernel, 0, p.c, s, sm_count, p, d_maps);
}

void launch_join_batch(const BatchGroup &b, cudaStream_t s) {
    if (b.chunks) {
        const uint32_t blocks = (uint32_t)((b.chunks + kBlockThreads - 1) / kBlockThreads);
        join_batch_kernel<B_CLASSIFY><<<blocks, kBlockThreads, 0, s>>>(b);
        join_batch_kernel<B_CHAIN><<<blocks, kBlockThreads, 0, s>>>(b);
        join_batch_kernel<B_VERIFY><<<blocks, kBlockThreads, 0, s>>>(b);
    }
    status_batch_kernel<<<(b.nt + kBlockThreads - 1) / kBlockThreads, kBlockThreads, 0, s>>>(b);
}

}  // namespace slpf
