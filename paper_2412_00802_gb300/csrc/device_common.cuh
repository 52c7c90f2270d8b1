// Device building blocks shared by the batched interpreter (exec.cu) and the
// one-operation-per-launch path (plain.cu).
//
// Layout: a set of individuals is a row of uint32 words, bit i of word w =
// individual 32*w + i.  A warp works on 32*WPL consecutive words; lane l holds
// words wb + l*WPL .. wb + l*WPL + WPL-1 (so WPL = 4 gives 128-bit loads).
#pragma once

#include <cstdint>

#include "hedl_internal.h"

namespace hedl {

constexpr unsigned FULL = 0xFFFFFFFFu;

__device__ __forceinline__ uint32_t tail_mask(uint32_t w, uint32_t n_words, uint32_t n) {
    if (w + 1 < n_words) return FULL;
    if (w + 1 == n_words) {
        uint32_t r = n & 31u;
        return r ? ((1u << r) - 1u) : FULL;
    }
    return 0u;
}

// bits lo..hi-1 set (0 <= lo <= hi <= 32)
__device__ __forceinline__ uint32_t range_mask(uint32_t lo, uint32_t hi) {
    uint32_t up = hi >= 32 ? FULL : ((1u << hi) - 1u);
    uint32_t dn = lo >= 32 ? FULL : ((1u << lo) - 1u);
    return up & ~dn;
}

template <int WPL>
__device__ __forceinline__ void load_row_ro(const uint32_t *__restrict__ row, uint32_t wb, uint32_t lane,
                                            uint32_t wp, uint32_t (&v)[WPL]) {
    uint32_t w0 = wb + lane * WPL;
    if constexpr (WPL == 4) {
        if (w0 < wp) {
            uint4 q = __ldg(reinterpret_cast<const uint4 *>(row + w0));
            v[0] = q.x, v[1] = q.y, v[2] = q.z, v[3] = q.w;
        } else {
            v[0] = v[1] = v[2] = v[3] = 0u;
        }
    } else {
#pragma unroll
        for (int s = 0; s < WPL; ++s) v[s] = (w0 + s < wp) ? __ldg(row + w0 + s) : 0u;
    }
}

// Rows written earlier in the same kernel (slots) are read with plain loads,
// never through the read-only path.
template <int WPL>
__device__ __forceinline__ void load_row_rw(const uint32_t *row, uint32_t wb, uint32_t lane, uint32_t wp,
                                            uint32_t (&v)[WPL]) {
    uint32_t w0 = wb + lane * WPL;
    if constexpr (WPL == 4) {
        if (w0 < wp) {
            uint4 q = *reinterpret_cast<const uint4 *>(row + w0);
            v[0] = q.x, v[1] = q.y, v[2] = q.z, v[3] = q.w;
        } else {
            v[0] = v[1] = v[2] = v[3] = 0u;
        }
    } else {
#pragma unroll
        for (int s = 0; s < WPL; ++s) v[s] = (w0 + s < wp) ? row[w0 + s] : 0u;
    }
}

template <int WPL>
__device__ __forceinline__ void store_row(uint32_t *row, uint32_t wb, uint32_t lane, uint32_t wp,
                                          const uint32_t (&v)[WPL]) {
    uint32_t w0 = wb + lane * WPL;
    if constexpr (WPL == 4) {
        if (w0 < wp) *reinterpret_cast<uint4 *>(row + w0) = make_uint4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
        for (int s = 0; s < WPL; ++s)
            if (w0 + s < wp) row[w0 + s] = v[s];
    }
}

// Does count `cnt` decide the restriction?  Returns the threshold at which the
// answer can no longer change (the walk over a row may stop there).
__device__ __forceinline__ uint64_t decide_cap(uint32_t kind, uint32_t n) {
    switch (kind) {
    case HEDL_OP_EXISTS: return 1;             // one C-successor
    case HEDL_OP_FORALL: return 1;             // one successor outside C
    case HEDL_OP_ATLEAST: return n;
    default: return (uint64_t)n + 1;           // ATMOST / EXACTLY: n+1 of them
    }
}

__device__ __forceinline__ bool role_pred(uint32_t kind, uint32_t cnt, uint32_t n) {
    switch (kind) {
    case HEDL_OP_EXISTS: return cnt >= 1;
    case HEDL_OP_FORALL: return cnt == 0;      // cnt counts successors NOT in C
    case HEDL_OP_ATLEAST: return cnt >= n;
    case HEDL_OP_ATMOST: return cnt <= n;
    default: return cnt == n;                  // EXACTLY
    }
}

// Streaming read of KB arrays (CSR): read-only for the kernel's lifetime and
// used once per pass, so they do not take L1 lines from the filler bitsets.
__device__ __forceinline__ uint32_t ld_stream(const uint32_t *p) {
    uint32_t v;
    asm("ld.global.nc.L1::no_allocate.u32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}

// A hint to bring bytes [p, p + bytes) into L2 (p 16-byte aligned, bytes a
// multiple of 16, the range inside one allocation); no register waits on it.
__device__ __forceinline__ void prefetch_l2(const void *p, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// L2 prefetch of a[lo, hi) by lane 0 (a 16-byte aligned): the start is
// rounded down and the size down to whole 16-byte units, so the hint stays
// inside [0, hi).
__device__ __forceinline__ void prefetch_range(const uint32_t *a, uint32_t lo, uint32_t hi, uint32_t lane) {
    if (lane != 0u || lo >= hi) return;
    lo &= ~3u;
    const uint32_t bytes = ((hi - lo) * 4u) & ~15u;
    if (bytes) prefetch_l2(a + lo, bytes);
}

// Role restriction over the warp's 32*WPL words (Algorithms 3-8 of the
// paper, recast).  For each word (32 individuals) the warp walks the word's
// CSR edge range, a block of BLK (<= 32) chunks of 32 edges at a time: lane e
// loads edge e of each chunk (coalesced), tests the filler bit of its object,
// and a ballot packs each chunk's tests into a mask that lane c keeps for
// chunk c.  A warp scan turns the masks' popcounts into prefix counts, so
// lane i counts the hits inside its own row [lo, hi) with two rank lookups,
// however many chunks the row spans.  Counts stay in registers (no atomics,
// no counter matrix), and the walk stops once every lane's answer is decided.
// FORALL counts successors outside the filler.
// filler_inverted: the caller already complemented a FORALL filler.
template <int WPL, int BLK>
__device__ __forceinline__ void role_words(const DevCSR g, const uint32_t *filler, uint32_t kind, uint32_t n_arg,
                                           uint32_t n, uint32_t n_words, uint32_t wb, uint32_t lane,
                                           uint32_t (&v)[WPL], bool filler_inverted = false) {
    static_assert(BLK >= 1 && BLK <= 32, "a block holds 1..32 chunks");
    constexpr int ROLE_BLOCK = BLK;
    constexpr uint32_t BE = 32u * ROLE_BLOCK;     // edges per block
    const uint32_t neg = (kind == HEDL_OP_FORALL && !filler_inverted) ? 1u : 0u;
    const uint64_t cap = decide_cap(kind, n_arg);
    const uint32_t *__restrict__ rp = g.rp;
    const uint32_t *__restrict__ col = g.col;
    uint32_t nlo = 0, nhi = 0;   // row pointers of the next word, fetched ahead
    {
        const uint32_t i = wb * 32u + lane;
        if (wb < n_words && i < n) {
            nlo = ld_stream(rp + i);
            nhi = ld_stream(rp + i + 1);
        }
    }
#pragma unroll 1
    for (int j = 0; j < 32; ++j) {
#pragma unroll
        for (int s = 0; s < WPL; ++s) {
            const uint32_t w = wb + (uint32_t)j * WPL + s;
            uint32_t word = 0;
            if (w < n_words) {
                const uint32_t i = w * 32u + lane;
                const bool valid = i < n;
                const uint32_t lo = nlo, hi = nhi;
                {
                    const uint32_t i2 = i + 32u;
                    if (w + 1 < n_words && i2 < n) {
                        nlo = ld_stream(rp + i2);
                        nhi = ld_stream(rp + i2 + 1);
                    }
                }
                const uint32_t nv = min(32u, n - w * 32u);
                const uint32_t e0 = __shfl_sync(FULL, lo, 0);
                const uint32_t e1 = __shfl_sync(FULL, hi, nv - 1);
                // my row relative to the word's first edge (empty for lanes past n)
                const uint32_t r0 = valid ? lo - e0 : 0u, r1 = valid ? hi - e0 : 0u;
                uint32_t cnt = 0;
                if (cap > 0) {
#pragma unroll 1
                    for (uint32_t rb = 0; rb < e1 - e0; rb += BE) {
                        const uint32_t base = e0 + rb;
                        // Edge index clamped to the word's last edge: lanes past the end reload
                        // a valid edge, and their bits lie beyond every row so no rank counts them.
                        uint32_t hit[ROLE_BLOCK];
#pragma unroll
                        for (int u = 0; u < ROLE_BLOCK; ++u)
                            hit[u] = ld_stream(col + min(base + 32u * u + lane, e1 - 1u));
#pragma unroll
                        for (int u = 0; u < ROLE_BLOCK; ++u)
                            hit[u] = (__funnelshift_r(filler[hit[u] >> 5], 0u, hit[u]) & 1u) ^ neg;
                        uint32_t mc = 0;   // lane c < ROLE_BLOCK: mask of chunk c
#pragma unroll
                        for (int u = 0; u < ROLE_BLOCK; ++u) {
                            const uint32_t m = __ballot_sync(FULL, hit[u]);
                            if (lane == (uint32_t)u) mc = m;
                        }
                        // exclusive prefix of the chunks' popcounts over lanes 0..ROLE_BLOCK-1
                        const uint32_t pc = __popc(mc);
                        uint32_t incl = pc;
#pragma unroll
                        for (int o = 1; o < ROLE_BLOCK; o <<= 1) {
                            const uint32_t t = __shfl_up_sync(FULL, incl, o);
                            if (lane >= (uint32_t)o) incl += t;
                        }
                        const uint32_t excl = incl - pc;
                        // hits before block-relative position x in [0, BE]
                        auto rank = [&](uint32_t x) -> uint32_t {
                            const uint32_t c = min(x >> 5, (uint32_t)ROLE_BLOCK - 1);
                            const uint32_t e = __shfl_sync(FULL, excl, c);
                            const uint32_t m = __shfl_sync(FULL, mc, c);
                            const uint32_t sh = x - 32u * c;   // 0..32
                            return e + __popc(sh >= 32u ? m : (m & ((1u << sh) - 1u)));
                        };
                        const uint32_t a = r0 > rb ? min(r0 - rb, BE) : 0u;
                        const uint32_t z = r1 > rb ? min(r1 - rb, BE) : 0u;
                        cnt += rank(z) - rank(a);
                        const bool done = !valid || r1 <= rb + BE || (uint64_t)cnt >= cap;
                        if (__all_sync(FULL, done)) break;
                    }
                }
                word = __ballot_sync(FULL, valid && role_pred(kind, cnt, n_arg));
            }
            if (lane == (uint32_t)j) v[s] = word;
        }
    }
}

// Role restriction over the warp's words as ONE edge stream (the interpreter's
// walk).  The words wb .. wb+K-1 are consecutive individuals, so their CSR
// rows form one contiguous edge range [E0, E1).  The warp reads that range in
// blocks of BLK 32-edge chunks, always loading the next block while it tests
// the current one (the gather's DRAM latency overlaps the filler lookups) and
// asking L2 for the blocks after it (prefetch hints that hold no registers),
// and attributes each block's hits to the words whose rows it covers: lane i
// of word k counts the hits inside its row with two rank lookups, as in
// role_words, and a word is emitted (ballot) once its last edge has passed.
// A word whose every lane is decided (cap reached or row ended) makes the
// stream jump to the next word's first edge.  Word k of the warp goes to lane
// k / WPL, slot k % WPL.  n_words bounds the warp's words; lanes of
// individuals >= n hold empty rows and emit 0.  GLOBAL: the filler row is said
// to lie in global memory (else it may be staged in shared memory).  A function
// of its own, with registers of its own: inlined, the stack machine around it
// spilled.
//
// Bound: latency and the filler's gathers.  Which block is faster depends on
// the rows, which the plan does not know: on heavy-tailed ones a block of 8
// chunks keeps more in flight (a lone hypothesis on 10^7 individuals, Zipf
// degrees of mean 8: 1,416 us with 4, 1,369 with 8; on 10^6: 265 and 218), on
// even ones its emptier blocks cost more (Poisson degrees of mean 4, 10^6
// individuals: 127 and 134).  So it is part of the launch shape (role_block),
// 4 unless the tuner has timed it.
template <int WPL>
struct RowWords {
    uint32_t v[WPL];
};
template <int WPL, uint32_t BLK, bool GLOBAL>
__device__ __noinline__ RowWords<WPL> role_stream(const uint32_t *rp, const uint32_t *col, const uint32_t *filler,
                                                  uint32_t kind, uint32_t n_arg, uint32_t n, uint32_t n_words,
                                                  uint32_t wb, bool filler_inverted) {
    if constexpr (GLOBAL) __builtin_assume(__isGlobal(filler));
    constexpr uint32_t BE = 32u * BLK;              // edges per block
    const uint32_t lane = threadIdx.x & 31u;
    RowWords<WPL> out;
    uint32_t (&v)[WPL] = out.v;
    const uint32_t neg = (kind == HEDL_OP_FORALL && !filler_inverted) ? 1u : 0u;
    const uint64_t cap = decide_cap(kind, n_arg);
#pragma unroll
    for (int s = 0; s < WPL; ++s) v[s] = 0u;
    if (wb >= n_words) return out;
    const uint32_t K = min(32u * WPL, n_words - wb);
    auto put = [&](uint32_t k, uint32_t word) {
#pragma unroll
        for (int s = 0; s < WPL; ++s)
            if (lane == k / WPL && k % WPL == (uint32_t)s) v[s] = word;
    };
    auto lane_valid = [&](uint32_t k) { return (wb + k) * 32u + lane < n; };
    if (cap == 0) {   // decided before any edge (at least 0): every individual
        for (uint32_t k = 0; k < K; ++k) put(k, __ballot_sync(FULL, lane_valid(k)));
        return out;
    }
    // row pointers of words k, k+1, k+2 (empty rows for lanes past n or words past K)
    auto ld_rows = [&](uint32_t k, uint32_t &lo, uint32_t &hi) {
        const uint32_t i = (wb + k) * 32u + lane;
        if (k < K && i < n) {
            lo = ld_stream(rp + i);
            hi = ld_stream(rp + i + 1);
        } else {
            lo = 0u;
            hi = 0u;
        }
    };
    // last edge (exclusive) of word k, from its last valid lane
    auto word_end = [&](uint32_t k, uint32_t hi) {
        const uint32_t nv = min(32u, n - (wb + k) * 32u);
        return __shfl_sync(FULL, hi, nv - 1u);
    };
    uint32_t lo0, hi0, lo1, hi1, lo2, hi2;
    ld_rows(0, lo0, hi0);
    ld_rows(1, lo1, hi1);
    ld_rows(2, lo2, hi2);
    const uint32_t E0 = __shfl_sync(FULL, lo0, 0);
    const uint32_t E1 = ld_stream(rp + min(n, (wb + K) * 32u));
    uint32_t k = 0, cnt = 0;
    uint32_t ew1 = word_end(0, hi0);
    auto next_word = [&]() {
        lo0 = lo1, hi0 = hi1, lo1 = lo2, hi1 = hi2;
        ld_rows(k + 2, lo2, hi2);
        ew1 = word_end(k, hi0);
        cnt = 0;
    };
    uint32_t pf[BLK];
    auto fetch = [&](uint32_t at) {
#pragma unroll
        for (uint32_t u = 0; u < BLK; ++u) pf[u] = ld_stream(col + min(at + 32u * u + lane, E1 - 1u));
    };
    // L2 hints (no registers held): the warp's row pointers, and the edge
    // blocks two to four ahead of the one loading into registers
    const bool cvec = (reinterpret_cast<uintptr_t>(col) & 15u) == 0;
    if ((reinterpret_cast<uintptr_t>(rp) & 15u) == 0) prefetch_range(rp, wb * 32u, min(n, (wb + K) * 32u) + 1u, lane);
    auto ahead = [&](uint32_t from, uint32_t blocks) {
        if (cvec && from < E1) prefetch_range(col, from, min(E1, from + blocks * BE), lane);
    };
    uint32_t base = E0;
    if (base < E1) fetch(base);
    ahead(E0 + BE, 3u);
#pragma unroll 1
    while (base < E1) {
        uint32_t hit[BLK];
#pragma unroll
        for (uint32_t u = 0; u < BLK; ++u) hit[u] = pf[u];
        const uint32_t nb = base + BE;
        if (nb < E1) fetch(nb);
        ahead(base + 4u * BE, 1u);
        // Positions past E1 reloaded edge E1-1; they lie beyond every row, so no rank counts them.
#pragma unroll
        for (uint32_t u = 0; u < BLK; ++u) hit[u] = (__funnelshift_r(filler[hit[u] >> 5], 0u, hit[u]) & 1u) ^ neg;
        uint32_t mc = 0;   // lane c < BLK: mask of chunk c
#pragma unroll
        for (uint32_t u = 0; u < BLK; ++u) {
            const uint32_t m = __ballot_sync(FULL, hit[u]);
            if (lane == u) mc = m;
        }
        const uint32_t pc = __popc(mc);
        uint32_t incl = pc;
#pragma unroll
        for (uint32_t o = 1; o < BLK; o <<= 1) {
            const uint32_t t = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += t;
        }
        const uint32_t excl = incl - pc;
        // hits before block-relative position x in [0, BE]
        auto rank = [&](uint32_t x) -> uint32_t {
            const uint32_t c = min(x >> 5, BLK - 1u);
            const uint32_t e = __shfl_sync(FULL, excl, c);
            const uint32_t m = __shfl_sync(FULL, mc, c);
            const uint32_t sh = x - 32u * c;   // 0..32
            return e + __popc(sh >= 32u ? m : (m & ((1u << sh) - 1u)));
        };
        // the words whose rows meet this block, in order
        bool finished = false;
#pragma unroll 1
        for (;;) {
            const uint32_t a = lo0 > base ? min(lo0 - base, BE) : 0u;
            const uint32_t z = hi0 > base ? min(hi0 - base, BE) : 0u;
            cnt += rank(z) - rank(a);
            if (ew1 > nb) break;                       // word k goes on in the next block
            put(k, __ballot_sync(FULL, lane_valid(k) && role_pred(kind, cnt, n_arg)));
            if (++k == K) {
                finished = true;
                break;
            }
            next_word();
        }
        if (finished) return out;
        // word k spans past this block: skip the rest of it once every lane is decided
        const bool decided = !lane_valid(k) || hi0 <= nb || (uint64_t)cnt >= cap;
        if (__all_sync(FULL, decided)) {
            put(k, __ballot_sync(FULL, lane_valid(k) && role_pred(kind, cnt, n_arg)));
            if (++k == K) return out;
            const uint32_t nxt = ew1;                  // the next word's first edge
            next_word();
            if (nxt != nb && nxt < E1) {
                fetch(nxt);
                ahead(nxt + BE, 3u);
            }
            base = nxt;
        } else {
            base = nb;
        }
    }
    // the stream ended (or was empty): the remaining words have no edges left
    for (; k < K; ++k) {
        put(k, __ballot_sync(FULL, lane_valid(k) && role_pred(kind, cnt, n_arg)));
        cnt = 0;
    }
    return out;
}

__device__ __forceinline__ bool data_cmp(uint32_t cmp, float x, float t);

// Numeric data-range restriction (Algorithms 9-10): one float compare per
// individual.  Lane l builds its own words wb + l*WPL + s from the 32
// contiguous values of each (eight 16-byte loads, all in flight at once, when
// the row is 16-byte aligned and the word is whole; scalar loads otherwise).
// NaN (missing) compares false.
template <int WPL>
__device__ __forceinline__ void data_words(const float *__restrict__ vals, uint32_t cmp, float t, uint32_t n,
                                           uint32_t n_words, uint32_t wb, uint32_t lane, uint32_t (&v)[WPL]) {
    const bool vec = (reinterpret_cast<uintptr_t>(vals) & 15u) == 0;
#pragma unroll
    for (int s = 0; s < WPL; ++s) {
        const uint32_t w = wb + lane * WPL + s;
        uint32_t word = 0;
        if (w < n_words) {
            const uint32_t i0 = w * 32u;
            if (vec && i0 + 32u <= n) {
                float4 q[8];
                const float4 *p4 = reinterpret_cast<const float4 *>(vals + i0);
#pragma unroll
                for (int k = 0; k < 8; ++k) q[k] = __ldg(p4 + k);
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    word |= (uint32_t)data_cmp(cmp, q[k].x, t) << (4 * k);
                    word |= (uint32_t)data_cmp(cmp, q[k].y, t) << (4 * k + 1);
                    word |= (uint32_t)data_cmp(cmp, q[k].z, t) << (4 * k + 2);
                    word |= (uint32_t)data_cmp(cmp, q[k].w, t) << (4 * k + 3);
                }
            } else {
                for (uint32_t k = 0; k < 32u && i0 + k < n; ++k)
                    word |= (uint32_t)data_cmp(cmp, __ldg(vals + i0 + k), t) << k;
            }
        }
        v[s] = word;
    }
}

__device__ __forceinline__ bool data_cmp(uint32_t cmp, float x, float t) {
    return cmp == HEDL_OP_DGE ? (x >= t) : cmp == HEDL_OP_DLE ? (x <= t) : (x == t);
}

// The test a concrete-role restriction applies to each asserted value (the
// 32-bit word of a float value or of a string id): a float compare (numeric
// roles, Algorithms 9-10), id equality (string EQUAL, Algorithms 11-12) or a
// bit of the pattern's containment row (string CONTAIN, Algorithms 13-14).
struct ValueTest {
    enum : uint32_t { GE = 0, LE = 1, EQ = 2, ID_EQ = 3, ID_BIT = 4 };
    uint32_t kind;
    uint32_t arg;           // the threshold's bits or the string id
    const uint32_t *bits;   // ID_BIT: the containment row
};

// Existential restriction on a concrete role with several values per
// subject (Section III-B): individual i belongs iff one of its values
// vals[rp[i] .. rp[i+1]) passes the test.  The warp's 32*WPL words are
// 1024*WPL consecutive individuals, so their values form one contiguous run,
// which the warp streams once, in windows of EX_WIN values that asynchronous
// 16-byte copies bring into one of two places in shared memory, the next
// window while one is tested (no registers hold what is in flight).  Lane l tests
// value 32u + l of a window, and a ballot packs 32 tests into a mask word in
// the order of the values, which lane 0 puts into a ring of masks.  The row
// pointers come the same way, a batch of four words (128 individuals) ahead.  A
// batch needs the masks of its run; each lane then looks its rows up with two
// reads and a funnel shift each (rows over 32 values go on word by word).
//
// A batch whose run does not fit the mask ring (a heavy subject) is walked word
// by word in pieces of EX_STAGES windows, each only as long as a row that has
// not passed yet reaches into it, jumping to the first such row (the paper's
// early exit): a heavy subject costs its values up to the piece of its first
// pass.
//
// Bound: instruction issue, 83 % of the cycles for 12 restrictions on 4 numeric
// roles of four values a subject at 10^7 individuals (593 us, 160 instructions a
// word of 32 individuals and restriction, the stack machine's included).  With
// the values loaded into registers and packed into masks by shuffles it was 142
// instructions, but issue at 51 %: warps waited for their loads (864 us).  A
// function for each kind of test made warps wait for instructions.  24
// restrictions on 8 roles (3.8 GB by the model, each role read three times):
// 1.96 ms -> 1.26 ms, with rings half as large 1.10 ms.
static_assert(EX_RING % EX_LOADS == 0 && EX_LOADS % 4 == 0, "a window's masks are whole 16-byte stores");

// Asynchronous copy of src[at .. at + COUNT) to dst, the elements below end
// only: 16 bytes a lane where they are aligned and all wanted, else 4.
template <uint32_t COUNT>
__device__ __forceinline__ void ex_copy(uint32_t *dst, const uint32_t *src, uint32_t at, uint32_t end, bool vec,
                                        uint32_t lane) {
    const uint32_t to = (uint32_t)__cvta_generic_to_shared(dst);
    if (vec && at + COUNT <= end) {   // warp-uniform
#pragma unroll
        for (uint32_t u = 0; u < COUNT; u += 128u)
            if (COUNT >= 128u || 4u * lane < COUNT)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to + 4u * u + 16u * lane),
                             "l"(src + at + u + 4u * lane)
                             : "memory");
    } else {
#pragma unroll 1
        for (uint32_t u = lane; u < COUNT; u += 32u)
            if (at + u < end)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(to + 4u * u), "l"(src + at + u)
                             : "memory");
    }
}

// Waits until at most `after` of this thread's groups of asynchronous copies
// are pending (warp-uniform), then for the warp.
__device__ __forceinline__ void ex_wait(uint32_t after) {
    if (after == 0u) asm volatile("cp.async.wait_group 0;" ::: "memory");
    else if (after == 1u) asm volatile("cp.async.wait_group 1;" ::: "memory");
    else if (after == 2u) asm volatile("cp.async.wait_group 2;" ::: "memory");
    else asm volatile("cp.async.wait_group 3;" ::: "memory");
    __syncwarp();
}

// The masks of the window x (value c on; those at and past end fail) to ring[0 .. EX_LOADS).
__device__ __forceinline__ void ex_masks(const uint32_t *x, uint32_t c, uint32_t end, uint32_t lane, const ValueTest &t,
                                         uint32_t *ring) {
    uint32_t v[EX_LOADS], m[EX_LOADS];
#pragma unroll
    for (uint32_t u = 0; u < EX_LOADS; ++u) v[u] = x[32u * u + lane];
    const float f = __uint_as_float(t.arg);
    switch (t.kind) {   // warp-uniform
    case ValueTest::GE:
#pragma unroll
        for (uint32_t u = 0; u < EX_LOADS; ++u) m[u] = __ballot_sync(FULL, __uint_as_float(v[u]) >= f);
        break;
    case ValueTest::LE:
#pragma unroll
        for (uint32_t u = 0; u < EX_LOADS; ++u) m[u] = __ballot_sync(FULL, __uint_as_float(v[u]) <= f);
        break;
    case ValueTest::EQ:
#pragma unroll
        for (uint32_t u = 0; u < EX_LOADS; ++u) m[u] = __ballot_sync(FULL, __uint_as_float(v[u]) == f);
        break;
    case ValueTest::ID_EQ:
#pragma unroll
        for (uint32_t u = 0; u < EX_LOADS; ++u) m[u] = __ballot_sync(FULL, v[u] == t.arg);
        break;
    default: {
        uint32_t w[EX_LOADS];
#pragma unroll
        for (uint32_t u = 0; u < EX_LOADS; ++u)   // past the end the ring holds no id
            w[u] = c + 32u * u + lane < end ? __ldg(t.bits + (v[u] >> 5)) >> (v[u] & 31u) : 0u;
#pragma unroll
        for (uint32_t u = 0; u < EX_LOADS; ++u) m[u] = __ballot_sync(FULL, w[u] & 1u);
        break;
    }
    }
    if (c + EX_WIN > end) {   // the run's last window
#pragma unroll
        for (uint32_t u = 0; u < EX_LOADS; ++u) m[u] &= range_mask(0u, end > c + 32u * u ? min(end - c - 32u * u, 32u) : 0u);
    }
    if (lane == 0u) {
#pragma unroll
        for (uint32_t u = 0; u < EX_LOADS; u += 4u)
            *reinterpret_cast<uint4 *>(ring + u) = make_uint4(m[u], m[u + 1], m[u + 2], m[u + 3]);
    }
}

// how many values of [lo, hi) pass (hi > lo), by the ring's masks, of the first 32
__device__ __forceinline__ uint32_t ex_count(const uint32_t *ring, uint32_t lo, uint32_t hi) {
    const uint32_t k = lo >> 5;
    const uint32_t f = __funnelshift_r(ring[k % EX_RING], ring[(k + 1u) % EX_RING], lo);   // 32 tests from lo on
    return __popc(f & (FULL >> (32u - min(hi - lo, 32u))));
}

// ring: EX_SMEM_WORDS of shared memory of this warp, 16-byte aligned (mask
// words, row pointers, windows).  The warp's words are wb .. of n_words, n
// individuals.  A function of its own, so that its registers do not raise the
// spills of the whole stack machine; a call costs little beside the words that
// it walks.
template <int WPL>
__device__ __noinline__ RowWords<WPL> exist_run(const uint32_t *rp, const uint32_t *vals, const ValueTest test,
                                                uint32_t n, uint32_t n_words, uint32_t wb, uint32_t *ring) {
    const uint32_t lane = threadIdx.x & 31u;
    RowWords<WPL> out;
#pragma unroll
    for (int s = 0; s < WPL; ++s) out.v[s] = 0u;
    const uint32_t w_end = min(wb + 32u * WPL, n_words);   // the warp's words [wb, w_end)
    if (wb >= w_end) return out;
    uint32_t *rows = ring + EX_RING, *stages = rows + 2u * EX_ROWS;
    const bool rvec = (reinterpret_cast<uintptr_t>(rp) & 15u) == 0, vec = (reinterpret_cast<uintptr_t>(vals) & 15u) == 0;
    const uint32_t i1 = min(32u * w_end, n);                   // past the warp's last individual
    uint32_t c = ld_stream(rp + 32u * wb) & ~(EX_WIN - 1u);     // the next window to test
    const uint32_t end = ld_stream(rp + i1);                    // the end of the warp's run
    // Copy groups, numbered in the order of their commits (empty ones past the
    // last batch or the run): a batch's row pointers, a window of elements.
    uint32_t groups = 0;
    auto commit = [&]() {
        asm volatile("cp.async.commit_group;" ::: "memory");
        return groups++;
    };
    // row pointers 32w .. 32w + 128 (the last one ends the batch's last row) to their half of rows
    auto copy_rows = [&](uint32_t w, uint32_t half) {
        const uint32_t i = 32u * w;
        if (i < i1) {
            ex_copy<128>(rows + half * EX_ROWS, rp, i, i1 + 1u, rvec, lane);
            if (lane == 0u && i + 128u <= i1)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                                 (uint32_t)__cvta_generic_to_shared(rows + half * EX_ROWS + 128u)),
                             "l"(rp + i + 128u)
                             : "memory");
        }
        return commit();
    };
    uint32_t slot = 0;   // window c's place of the two
    auto copy_window = [&](uint32_t at, uint32_t to) {
        if (at < end) ex_copy<EX_WIN>(stages + to * EX_WIN, vals, at, end, vec, lane);
        return commit();
    };
    static_assert(EX_STAGES == 2, "the window that is read and the next one");
    if (rvec) prefetch_range(rp, 32u * wb, i1 + 1u, lane);
    uint32_t half = 0, r = copy_rows(wb, 0u);                            // the next batch's group
    uint32_t v0 = copy_window(c, 0u), v1 = copy_window(c + EX_WIN, 1u);   // window c's and the next one's
#pragma unroll 1
    for (uint32_t w0 = wb; w0 < w_end; w0 += 4u, half ^= 1u) {
        ex_wait(groups - 1u - r);
        r = copy_rows(w0 + 4u, half ^ 1u);
        // this lane's rows [lo, hi); individuals past n have none
        const uint32_t *p = rows + half * EX_ROWS + lane;
        uint32_t lo[4], hi[4], longest = 0;
#pragma unroll
        for (uint32_t q = 0; q < 4u; ++q) {
            lo[q] = p[32u * q];
            hi[q] = p[32u * q + 1u];
        }
        if (32u * w0 + 128u > i1) {   // the last batch
#pragma unroll
            for (uint32_t q = 0; q < 4u; ++q)
                if (32u * (w0 + q) + lane >= i1) lo[q] = hi[q] = end;
        }
#pragma unroll
        for (uint32_t q = 0; q < 4u; ++q) longest = max(longest, hi[q] - lo[q]);
        longest = __reduce_max_sync(FULL, longest);
        const uint32_t e0 = __shfl_sync(FULL, lo[0], 0);
        const uint32_t e1 = __reduce_max_sync(FULL, max(max(hi[0], hi[1]), max(hi[2], hi[3])));
        uint32_t hit[4] = {0u, 0u, 0u, 0u};
        if (e1 <= (e0 & ~(EX_WIN - 1u)) + 32u * EX_RING) {
            while (c < e1) {
                ex_wait(groups - 1u - v0);
                ex_masks(stages + slot * EX_WIN, c, end, lane, test, ring + (c >> 5) % EX_RING);
                __syncwarp();   // the window has been read, its masks are there
                v0 = v1, v1 = copy_window(c + 2u * EX_WIN, slot);   // into the place of window c
                slot ^= 1u;
                c += EX_WIN;
            }
#pragma unroll
            for (uint32_t q = 0; q < 4u; ++q)
                if (hi[q] > lo[q]) hit[q] = ex_count(ring, lo[q], hi[q]);
            if (longest > 32u) {   // warp-uniform
#pragma unroll
                for (uint32_t q = 0; q < 4u; ++q)
#pragma unroll 1
                    for (uint32_t at = lo[q] + 32u; at < hi[q] && !hit[q]; at += 32u) hit[q] = ex_count(ring, at, hi[q]);
            }
        } else {
#pragma unroll
            for (uint32_t q = 0; q < 4u; ++q) {
                uint32_t at = lo[q];   // the row's next untested element
#pragma unroll 1
                for (;;) {
                    const uint32_t first = __reduce_min_sync(FULL, !hit[q] && at < hi[q] ? at : FULL);
                    if (first == FULL) break;
                    const uint32_t p0 = first & ~(EX_WIN - 1u), p1 = min(p0 + EX_STAGES * EX_WIN, end);
                    asm volatile("cp.async.wait_all;" ::: "memory");
                    __syncwarp();
                    for (uint32_t x = 0; p0 + x < p1; x += EX_WIN) ex_copy<EX_WIN>(stages + x, vals, p0 + x, end, vec, lane);
                    asm volatile("cp.async.wait_all;" ::: "memory");
                    __syncwarp();
#pragma unroll 1
                    for (uint32_t x = 0; p0 + x < p1; x += EX_WIN)
                        ex_masks(stages + x, p0 + x, end, lane, test, ring + ((p0 + x) >> 5) % EX_RING);
                    __syncwarp();
                    const uint32_t stop = min(hi[q], p1);
                    for (; at < stop && !hit[q]; at = min(stop, at + 32u)) hit[q] = ex_count(ring, at, stop);
                    __syncwarp();
                }
            }
            // the rings no longer hold what is before c: go on from this batch's end
            c = e1 & ~(EX_WIN - 1u);
            slot = 0;
            v0 = copy_window(c, 0u), v1 = copy_window(c + EX_WIN, 1u);
        }
#pragma unroll
        for (uint32_t q = 0; q < 4u; ++q) {
            const uint32_t word = __ballot_sync(FULL, hit[q] != 0u), j = w0 + q - wb;   // past the last word: no rows
#pragma unroll
            for (int s = 0; s < WPL; ++s)
                if (lane == j / WPL && j % WPL == (uint32_t)s) out.v[s] = word;
        }
        __syncwarp();   // the rows and masks of this batch have been read
    }
    asm volatile("cp.async.wait_all;" ::: "memory");   // none is left for the next use of the rings
    __syncwarp();
    return out;
}

// The test of a D_DATA instruction on a numeric or string role (op word bit 8
// or 9; aux = the op; b = threshold bits, string id or pattern id).
__host__ __device__ __forceinline__ ValueTest value_test(const KBView &kb, uint32_t op_word, uint32_t b) {
    const uint32_t op = (op_word >> 16) & 0xFFu;
    if (op == HEDL_OP_SEQ) return ValueTest{ValueTest::ID_EQ, b, nullptr};
    if (op == HEDL_OP_SCONTAINS) return ValueTest{ValueTest::ID_BIT, 0u, kb.contain + (uint64_t)b * kb.contain_words};
    return ValueTest{op == HEDL_OP_DGE ? ValueTest::GE : op == HEDL_OP_DLE ? ValueTest::LE : ValueTest::EQ, b, nullptr};
}

__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ uint32_t ld_acquire(const uint32_t *p) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

}  // namespace hedl
