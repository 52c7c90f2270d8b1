// Batched evaluation: one persistent interpreter kernel over a work queue of
// (task, tile) items (see plan.cpp for how a batch becomes tasks).
//
// Each CTA pops an item (one task over a tile, or up to SEG_BATCH segments
// over one), waits (bounded) until every task it reads is complete, then its
// warps run it.  A segment task is a
// stack machine whose values are bitset words (one register set per lane,
// deeper stack entries in shared memory), whose leaves load concept rows /
// slots, evaluate data ranges by ballot, or evaluate a lone role restriction
// by the warp's edge-stream CSR walk (role_stream).  A segment's result is
// written to its slot, or, for a hypothesis root, reduced against the example
// sets by popcount (the paper's coverage count, Algorithm 15) with one atomic
// per warp.  A role group (up to 64 restrictions sharing a role and
// direction) runs as two tasks: a transpose of its fillers into one or
// two 32-bit words per individual, and one bit-sliced walk that evaluates all
// of them.
//
// Waits never spin unbounded: each gives up after the plan's timeout, sets an
// abort flag and an error bit, and every CTA then leaves the kernel.
#include <cuda_runtime.h>

#include <cstddef>
#include <cstring>

#include "device_common.cuh"
#include "launch.cuh"

namespace hedl {

namespace {

struct ExecArgs {
    KBView kb;
    uint8_t *ws;
    uint32_t *counts;     // [H][4] or null
    uint32_t *out_bits;   // [H][wp] or null
    uint32_t item_begin, item_end;
    uint32_t ring_words;  // shared-memory words of the concrete-role walk's rings (0: no such role)
    uint32_t use_queue;   // 1: dynamic queue with dependency waits; 0: static striding, no waits
};

template <int NW, int WPL>
struct Smem {
    uint32_t stk[NW][STACK_MAX][WPL][32];
    // the work item's tasks (segments: up to SEG_BATCH): descriptors, the first
    // SEG_CODE instructions, the first leaf rows (bit 0 set: a slot), their number, the tasks' indices
    Seg seg[SEG_BATCH];
    DInsn code[SEG_BATCH][SEG_CODE];
    uint64_t leaf[SEG_BATCH][PF_SLOTS];
    uint32_t n_leaf[SEG_BATCH], task[SEG_BATCH];
    uint32_t item;
    uint32_t ok;
    uint32_t chunk;       // a walk's next chunk of words
    uint32_t pad[1];
    // from here on: for KBs with concrete roles EX_SMEM_WORDS a warp (their walk's
    // rings, ExecArgs::ring_words in all), then a staged plan's filler row (wp words)
    uint32_t tail[1];
};

// The last group with item_begin <= item, from `from` on (a warp; all lanes
// get it).  A CTA's items only grow (the queue hands them out in order; static
// striding steps forward), so the search starts at the CTA's previous group:
// the lanes look at 32 groups with one load each, where a search step by step
// would wait for a load a step.
static_assert(sizeof(Group) == 16, "a group is one 16-byte load");
__device__ __forceinline__ Group find_group(const Group *groups, uint32_t n_groups, uint32_t item, uint32_t &from) {
    const uint32_t lane = threadIdx.x & 31u;
    for (;;) {
        const uint32_t k = from + lane;
        const uint4 x = k < n_groups ? *reinterpret_cast<const uint4 *>(groups + k) : make_uint4(FULL, 0u, 0u, 0u);
        const uint32_t m = __ballot_sync(FULL, x.x <= item);   // a prefix of the lanes: item_begin only grows
        if (m != FULL || from + 31u >= n_groups) {
            const uint32_t l = 31u - __clz(m);   // groups[from].item_begin <= item: lane 0 always holds
            from += l;
            return Group{__shfl_sync(FULL, x.x, l), __shfl_sync(FULL, x.y, l), __shfl_sync(FULL, x.z, l),
                         __shfl_sync(FULL, x.w, l)};
        }
        from += 31u;   // the last of these is the first of the next 32
    }
}

// Bounded wait for one producer task (dep: its index, DEP_FINE if it has fine tiles).
__device__ __forceinline__ bool wait_dep(const PlanHeader &hd, uint32_t dep, uint32_t *done, Counters *ctr,
                                         uint32_t fine_tiles, uint32_t *status) {
    const uint32_t *flag = done + (dep & ~DEP_FINE);
    const uint32_t target = dep & DEP_FINE ? fine_tiles : hd.n_tiles;
    if (ld_acquire(flag) >= target) return true;
    uint64_t t0 = 0, spins = 0;
    const uint64_t max_spins = hd.timeout_ns / 16 + 1000000ull;
    while (ld_acquire(flag) < target) {
        if ((++spins & 15u) == 0u) {   // the clock costs more than a look at the flag
            if (*(volatile uint32_t *)&ctr->abort) return false;
            const uint64_t t = global_ns();
            if (!t0) t0 = t;
            if (t - t0 > hd.timeout_ns || spins > max_spins) {
                atomicOr(status, ST_TIMEOUT);
                atomicExch(&ctr->abort, 1u);
                return false;
            }
        }
        __nanosleep(32);
    }
    return true;
}

// Makes task b of the CTA's work item ready (one warp): its descriptor and
// code go to shared memory, the lanes wait (bounded) for its producers, one
// each, and a segment's leaf table is built: its first PF concept-row and slot
// leaves in code order, which each round of words loads all at once (their
// latencies overlap) before the stack machine takes them in turn.  Returns
// whether every wait succeeded.  The eight warps of a CTA prepare eight
// segments side by side, so that their chains of loads (index, descriptor,
// code, completion counters) and the CTA's barriers are paid once for all of
// them: a batch of 4,096 hypotheses on 10^6 individuals (8,200 segments) 19.8 ms
// against 22.7 with one segment an item.
template <int NW, int WPL>
__device__ bool prepare_task(const ExecArgs &A, const PlanHeader &hd, Smem<NW, WPL> &sm, uint32_t b, uint32_t task,
                             uint32_t *slots, uint32_t *done, Counters *ctr, uint32_t fine_tiles) {
    constexpr uint32_t PF = WPL == 1 ? PF_SLOTS : 2;
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t *src = reinterpret_cast<const uint32_t *>(reinterpret_cast<const Seg *>(A.ws + hd.off_segs) + task);
    const uint32_t x = lane < sizeof(Seg) / 4 ? src[lane] : 0u;
    if (lane < sizeof(Seg) / 4) reinterpret_cast<uint32_t *>(&sm.seg[b])[lane] = x;
    if (lane == 0) sm.task[b] = task;
    static_assert(offsetof(Seg, code_len) == 4 && offsetof(Seg, dep_off) == 16 && offsetof(Seg, dep_cnt) == 20 &&
                      offsetof(Seg, kind) == 28,
                  "the fields are taken from the lanes that loaded them");
    const uint32_t code_off = __shfl_sync(FULL, x, 0), code_len = __shfl_sync(FULL, x, 1);
    const uint32_t dep_off = __shfl_sync(FULL, x, 4), dep_cnt = __shfl_sync(FULL, x, 5);
    const uint32_t kind = __shfl_sync(FULL, x, 7);
    if (kind == TASK_SEGMENT) {
        const DInsn *code = reinterpret_cast<const DInsn *>(A.ws + hd.off_code) + code_off;
        uint32_t n_pf = 0;
        for (uint32_t b0 = 0; b0 < code_len && (b0 == 0 || n_pf < PF); b0 += 32) {
            const uint32_t pc = b0 + lane;
            uint64_t addr = 0;
            bool leaf = false;
            if (pc < code_len) {
                const DInsn d = code[pc];
                if (pc < (uint32_t)SEG_CODE) sm.code[b][pc] = d;
                const uint32_t op = d.op & 0xFFu;
                if (op == D_ATOM) {
                    leaf = true;
                    addr = reinterpret_cast<uint64_t>(A.kb.concepts + (uint64_t)d.a * A.kb.wp);
                } else if (op == D_SLOT) {
                    leaf = true;
                    addr = reinterpret_cast<uint64_t>(slots + (uint64_t)d.ref * A.kb.wp) | 1ull;
                }
            }
            const uint32_t m = __ballot_sync(FULL, leaf);
            const uint32_t rank = n_pf + __popc(m & ((1u << lane) - 1u));
            if (leaf && rank < PF) sm.leaf[b][rank] = addr;
            n_pf = min(PF, n_pf + (uint32_t)__popc(m));
        }
        if (lane == 0) sm.n_leaf[b] = n_pf;
    }
    bool ok = true;
    if (A.use_queue) {
        const uint32_t *deps = reinterpret_cast<const uint32_t *>(A.ws + hd.off_deps) + dep_off;
        for (uint32_t k = lane; k < dep_cnt && ok; k += 32) ok = wait_dep(hd, deps[k], done, ctr, fine_tiles, A.kb.status);
    }
    return __all_sync(FULL, ok);
}

template <int NW, int WPL, bool STAGE, int BLK, bool CONCRETE>
__device__ void run_tile(const ExecArgs &A, const PlanHeader &hd, uint32_t b, uint32_t tile, Smem<NW, WPL> &sm,
                         uint32_t *slots, uint32_t *acc) {
    const KBView &kb = A.kb;
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31u;
    const Seg &seg = sm.seg[b];
    const DInsn *code = seg.code_len <= (uint32_t)SEG_CODE
                            ? sm.code[b]
                            : reinterpret_cast<const DInsn *>(A.ws + hd.off_code) + seg.code_off;
    // a warp covers ww * WPL words a round; with ww < 32, lanes ww..31 hold
    // words of no one: every load, store and walk stops at the warp's limit
    const uint32_t ww = hd.warp_words & 0xFFu;
    const uint32_t rounds = hd.tile_words / (NW * ww * WPL);
    // the leaf rows of prepare_task: the stack machine takes the k-th such leaf from pf[k]
    constexpr int PF = WPL == 1 ? PF_SLOTS : 2;
    const uint32_t n_pf = sm.n_leaf[b];
    const bool score = seg.hyp != NO_HYP && A.counts;
    uint32_t tp = 0, fp = 0;
    // the leaf rows (and example rows) of one round, loaded together
    auto prefetch = [&](uint32_t wb, uint32_t (&pf)[PF][WPL], uint32_t (&pv)[WPL], uint32_t (&nv)[WPL]) {
        const uint32_t lim_p = min(kb.wp, wb + ww * WPL);   // padded row words
#pragma unroll
        for (int k = 0; k < PF; ++k) {
            if ((uint32_t)k < n_pf) {
                const uint64_t a = sm.leaf[b][k];
                if (a & 1ull) load_row_rw<WPL>(reinterpret_cast<const uint32_t *>(a & ~1ull), wb, lane, lim_p, pf[k]);
                else load_row_ro<WPL>(reinterpret_cast<const uint32_t *>(a), wb, lane, lim_p, pf[k]);
            } else {
#pragma unroll
                for (int s = 0; s < WPL; ++s) pf[k][s] = 0u;
            }
        }
        if (score) {
            load_row_ro<WPL>(kb.pos, wb, lane, lim_p, pv);
            load_row_ro<WPL>(kb.neg, wb, lane, lim_p, nv);
        } else {
#pragma unroll
            for (int s = 0; s < WPL; ++s) pv[s] = nv[s] = 0u;
        }
    };
    // the stack machine over one round's words
    auto evaluate = [&](uint32_t wb, const uint32_t (&pf)[PF][WPL], const uint32_t (&pv)[WPL],
                        const uint32_t (&nv)[WPL]) {
        const uint32_t lim_p = min(kb.wp, wb + ww * WPL);   // padded row words
        const uint32_t lim_w = min(kb.w, wb + ww * WPL);    // words holding individuals
        uint32_t n_used = 0;   // concept-row and slot leaves met so far this round
        uint32_t top[WPL];
        uint32_t sp = 0;  // values on the stack, top included
        for (uint32_t pc = 0; pc < seg.code_len; ++pc) {
            const DInsn d = code[pc];
            const uint32_t op = d.op & 0xFFu;
            if (op == D_NOT) {
#pragma unroll
                for (int s = 0; s < WPL; ++s)
                    top[s] = ~top[s] & tail_mask(wb + lane * WPL + s, kb.w, kb.n);
                continue;
            }
            if (op == D_AND || op == D_OR) {
                sp -= 1;
#pragma unroll
                for (int s = 0; s < WPL; ++s) {
                    uint32_t o = sm.stk[warp][sp - 1][s][lane];
                    top[s] = op == D_AND ? (top[s] & o) : (top[s] | o);
                }
                continue;
            }
            // a leaf: spill the current top, compute the new one
            if (sp > 0) {
#pragma unroll
                for (int s = 0; s < WPL; ++s) sm.stk[warp][sp - 1][s][lane] = top[s];
            }
            sp += 1;
            switch (op) {
            case D_ATOM:
            case D_SLOT:
                if (n_used < n_pf) {   // loaded at the start of the round
#pragma unroll
                    for (int s = 0; s < WPL; ++s) {
                        uint32_t x = pf[0][s];
#pragma unroll
                        for (int k = 1; k < PF; ++k)
                            if ((uint32_t)k == n_used) x = pf[k][s];
                        top[s] = x;
                    }
                } else if (op == D_ATOM) {
                    load_row_ro<WPL>(kb.concepts + (uint64_t)d.a * kb.wp, wb, lane, lim_p, top);
                } else {
                    load_row_rw<WPL>(slots + (uint64_t)d.ref * kb.wp, wb, lane, lim_p, top);
                }
                ++n_used;
                break;
            case D_TOP:
#pragma unroll
                for (int s = 0; s < WPL; ++s) top[s] = tail_mask(wb + lane * WPL + s, kb.w, kb.n);
                break;
            case D_BOT:
#pragma unroll
                for (int s = 0; s < WPL; ++s) top[s] = 0u;
                break;
            case D_DATA:
                if ((d.op >> 8) & 3u) {   // a numeric (bit 8) or string (bit 9) concrete role
                    if constexpr (CONCRETE) {
                        const bool str = (d.op >> 9) & 1u;
                        const uint32_t *rp = str ? kb.str[d.a].rp : kb.num[d.a].rp;
                        const uint32_t *vals =
                            str ? kb.str[d.a].ids : reinterpret_cast<const uint32_t *>(kb.num[d.a].vals);
                        const RowWords<WPL> o = exist_run<WPL>(rp, vals, value_test(kb, d.op, d.b), kb.n, lim_w, wb,
                                                               sm.tail + warp * EX_SMEM_WORDS);
#pragma unroll
                        for (int s = 0; s < WPL; ++s) top[s] = o.v[s];
                    }
                } else
                    data_words<WPL>(kb.props + (uint64_t)d.a * kb.prop_stride, (d.op >> 16) & 0xFFu,
                                    __uint_as_float(d.b), kb.n, lim_w, wb, lane, top);
                break;
            default: {  // D_ROLE
                const uint32_t inv = (d.op >> 8) & 1u;
                const DevCSR g = kb.csr[2u * d.a + inv];
                const uint32_t kind = (d.op >> 16) & 0xFFu;
                const uint32_t *filler = STAGE ? sm.tail + A.ring_words
                                         : (d.ref & REF_SLOT) ? slots + (uint64_t)(d.ref & ~REF_SLOT) * kb.wp
                                                              : kb.concepts + (uint64_t)d.ref * kb.wp;
                // with blocks of 4 chunks knowing the filler's memory made the walk 1 % slower (127 to 128.5 us
                // a lone hypothesis on 10^6 individuals), with 8 faster (1,382 to 1,369 us on 10^7)
                const RowWords<WPL> o = role_stream<WPL, BLK, BLK == 8 && !STAGE>(
                    g.rp, g.col, filler, kind, d.b, kb.n, lim_w, wb, STAGE && kind == HEDL_OP_FORALL);
#pragma unroll
                for (int s = 0; s < WPL; ++s) top[s] = o.v[s];
                break;
            }
            }
        }
        if (seg.out_slot != NO_SLOT) store_row<WPL>(slots + (uint64_t)seg.out_slot * kb.wp, wb, lane, lim_p, top);
        if (seg.hyp != NO_HYP) {
            if (A.out_bits) store_row<WPL>(A.out_bits + (uint64_t)seg.hyp * kb.wp, wb, lane, lim_p, top);
            if (score) {
#pragma unroll
                for (int s = 0; s < WPL; ++s) {
                    tp += __popc(top[s] & pv[s]);
                    fp += __popc(top[s] & nv[s]);
                }
            }
        }
    };
    // one round at a time: the round's leaf rows are all requested before the
    // first instruction runs (requesting the next round's as well was slower:
    // twice the prefetch registers, more spills)
    for (uint32_t r = 0; r < rounds; ++r) {
        const uint32_t wb = tile * hd.tile_words + (r * NW + warp) * ww * WPL;
        if (wb >= kb.wp) break;
        uint32_t pf[PF][WPL], pv[WPL], nv[WPL];
        prefetch(wb, pf, pv, nv);
        evaluate(wb, pf, pv, nv);
    }
    if (seg.hyp != NO_HYP && A.counts) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            tp += __shfl_xor_sync(FULL, tp, o);
            fp += __shfl_xor_sync(FULL, fp, o);
        }
        if (lane == 0) {
            if (tp) atomicAdd(acc + 2u * seg.hyp, tp);
            if (fp) atomicAdd(acc + 2u * seg.hyp + 1u, fp);
        }
    }
}

// ------------------------------------------------------------------ bit-sliced role groups
// 32 x 32 bit transpose across a warp: lane r holds row r (bit c = column c)
// on entry and column r on exit.  Five butterfly stages swap the
// off-diagonal blocks of size 16, 8, 4, 2, 1.
__device__ __forceinline__ uint32_t transpose32(uint32_t x, uint32_t lane) {
    const uint32_t masks[5] = {0x0000FFFFu, 0x00FF00FFu, 0x0F0F0F0Fu, 0x33333333u, 0x55555555u};
#pragma unroll
    for (int st = 0; st < 5; ++st) {
        const uint32_t j = 16u >> st, m = masks[st];
        const uint32_t t = __shfl_xor_sync(FULL, x, j);
        x = (lane & j) ? ((x & ~m) | ((t >> j) & m)) : ((x & m) | ((t & m) << j));
    }
    return x;
}

// Transpose task: word p of FT[i], bit s = slice 32p + s's filler at
// individual i (its complement for REF_NEG slices).  The warp takes its words
// four at a time: lane s reads four words of slice 32p + s's row (16 bytes),
// the next four in flight while these are transposed and stored.
template <int NW, int P>
__device__ void run_transpose(const ExecArgs &A, uint32_t ww, const RGroup *gp, uint32_t tile, const uint32_t *slots) {
    const KBView &kb = A.kb;
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31u;
    const uint32_t wb = (tile * NW + warp) * ww, w1 = min(wb + ww, kb.w);
    if (wb >= w1) return;
    const uint32_t n = gp->n;
    const uint32_t *src[P];
    uint32_t x[P];
    bool on[P];
#pragma unroll
    for (int q = 0; q < P; ++q) {
        const uint32_t s = 32u * q + lane;
        on[q] = s < n;
        const uint32_t ref = on[q] ? gp->filler[s] : 0u;
        const uint32_t id = ref & REF_ID;
        src[q] = (ref & REF_SLOT) ? slots + (uint64_t)id * kb.wp : kb.concepts + (uint64_t)id * kb.wp;
        x[q] = (ref & REF_NEG) ? FULL : 0u;
    }
    uint32_t *ft = reinterpret_cast<uint32_t *>(A.ws + gp->ft_off);
    auto load = [&](uint32_t w, uint4 (&v)[P]) {   // w a multiple of 4 below wp: rows are padded to whole quads
#pragma unroll
        for (int q = 0; q < P; ++q)
            v[q] = on[q] ? *reinterpret_cast<const uint4 *>(src[q] + w) : make_uint4(x[q], x[q], x[q], x[q]);
    };
    uint4 nxt[P];
    load(wb, nxt);
#pragma unroll 1
    for (uint32_t w = wb; w < w1; w += 4u) {
        uint32_t v[P][4];
#pragma unroll
        for (int q = 0; q < P; ++q) v[q][0] = nxt[q].x, v[q][1] = nxt[q].y, v[q][2] = nxt[q].z, v[q][3] = nxt[q].w;
        if (w + 4u < w1) load(w + 4u, nxt);
#pragma unroll
        for (uint32_t j = 0; j < 4u; ++j) {
            uint32_t t[P];
#pragma unroll
            for (int q = 0; q < P; ++q) t[q] = transpose32(v[q][j] ^ x[q], lane);
            if (w + j >= w1) break;   // warp-uniform: no individuals there
            if constexpr (P == 1) ft[32ull * (w + j) + lane] = t[0];
            else reinterpret_cast<uint2 *>(ft)[32ull * (w + j) + lane] = make_uint2(t[0], t[1]);
        }
    }
}

// A count per slice: planes c0 < c1 < c2, and over where it has passed 7.
struct Count {
    uint32_t c0, c1, c2, over;
    // adds x, y and z per slice: a full adder compresses them to one sum and one
    // carry, so that three words cost nine operations (one at a time, with
    // saturation at each, seven)
    __device__ __forceinline__ void add3(uint32_t x, uint32_t y, uint32_t z) {
        const uint32_t s = x ^ y ^ z, k = (x & y) | (z & (x | y));
        const uint32_t k0 = c0 & s;
        c0 ^= s;
        const uint32_t k1 = (c1 & k) | (k0 & (c1 | k));
        c1 ^= k ^ k0;
        over |= c2 & k1;
        c2 ^= k1;
    }
    __device__ __forceinline__ void saturate() { c0 |= over, c1 |= over, c2 |= over; }
    __device__ __forceinline__ void clear() { c0 = c1 = c2 = over = 0u; }
};

// a = a + b per slice (3-bit values), saturating at 7.
__device__ __forceinline__ void sat_add3(uint32_t &a0, uint32_t &a1, uint32_t &a2, uint32_t b0, uint32_t b1,
                                         uint32_t b2) {
    const uint32_t s0 = a0 ^ b0, k0 = a0 & b0;
    const uint32_t s1 = a1 ^ b1 ^ k0, k1 = (a1 & b1) | (k0 & (a1 ^ b1));
    const uint32_t s2 = a2 ^ b2 ^ k1, k2 = (a2 & b2) | (k1 & (a2 ^ b2));
    a0 = s0 | k2;
    a1 = s1 | k2;
    a2 = s2 | k2;
}

constexpr uint32_t HEAVY_ROW = 64;   // longer rows are walked by the whole warp
constexpr uint32_t HEAVY_LOADS = 6;  // edges of such a row that a lane has in flight
constexpr uint32_t WALK_BUF = 256;   // 32-bit words of a warp's window buffer

// Walk task: for each individual, the saturating per-slice count of its
// successors' FT words (P words each: 32 P slices), mapped through the
// group's truth tables, transposed back into the output slots (8 bytes a lane
// every two words).  The CTA's warps take the tile's words two at a time (a
// chunk: their individuals' rows form one contiguous edge range) from a shared
// counter, so that a warp whose rows are long takes fewer: with 32 words a warp
// the slowest of eight held 1.84 times the mean's edges on rows of Zipf
// lengths.  A warp streams a chunk's range in windows of WALK_BUF / P edges:
// lane e loads edges e, e + 32, ... of the window (coalesced), gathers their FT
// words and puts them in a per-warp shared-memory buffer; then each lane adds
// the buffer entries of its own rows, three at a time.  The next window's edges
// are loaded while the current window's FT words are gathered, the next chunk's
// row pointers while this one is walked and its first window's edges before
// this one's heavy rows and truth tables; windows that hold no light row's edge
// are skipped.  Rows longer than HEAVY_ROW are walked by the whole warp,
// HEAVY_LOADS edges a lane in flight, and their counts reduced across lanes.
//
// Floor: the gathers, one L1 miss an SM and clock (280 G/s over the chip, for
// 4, 8 or 16 bytes alike).  2,048 refinements at 4 * 10^6 individuals (137
// walks of 40 M edges of Zipf lengths, 5.5 G gathers, 20 ms) take 34.6 ms, 35.4
// without the work items of several segments; 4,096 hypotheses on 10^6 (177
// walks of 6 M edges, 1.1 G gathers, 3.9 ms) 15.9.  What is above it: only the
// edges are loaded a window ahead, so that a warp has no gather in flight while
// it adds, and with short rows most lanes have nothing to add.
//
// The tile's words are wb .. wb + K - 1 (K a multiple of 4) of wp; n_words hold
// the n_indiv individuals; *chunk counts from 0.  A function of its own:
// inlined, its registers raised the spills of the stack machine.
template <int P>
__device__ __noinline__ void run_walk(const DevCSR *csr, const uint32_t *ft, const RGroup *gp, uint32_t n_indiv,
                                      uint32_t n_words, uint32_t wp, uint32_t wb, uint32_t K, uint32_t *slots,
                                      uint32_t *buf, uint32_t *chunk) {
    constexpr uint32_t LOADS = WALK_BUF / (32u * P);   // edges a lane gathers per window
    constexpr uint32_t WIN = 32u * LOADS;
    constexpr uint32_t CW = 2u;                        // words per chunk
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t *__restrict__ rp = csr->rp;
    const uint32_t *__restrict__ col = csr->col;
    const uint32_t n = gp->n;
    // one FT entry (P words) of individual b
    auto ft_at = [&](uint32_t b, uint32_t (&o)[P]) {
        if constexpr (P == 1) {
            o[0] = ft[b];
        } else {
            const uint2 q = reinterpret_cast<const uint2 *>(ft)[b];
            o[0] = q.x;
            o[1] = q.y;
        }
    };
    uint32_t lo[CW], hi[CW];   // this lane's rows of the chunk (none past the last individual)
    auto rows = [&](uint32_t jj, uint32_t (&l)[CW], uint32_t (&h)[CW]) {
#pragma unroll
        for (uint32_t q = 0; q < CW; ++q) {
            const uint32_t w = wb + jj + q, i = w * 32u + lane;
            l[q] = h[q] = 0;
            if (jj < K && w < n_words && i < n_indiv) {
                l[q] = ld_stream(rp + i);
                h[q] = ld_stream(rp + i + 1);
            }
        }
    };
    uint32_t E1 = 0;   // the chunk's edge range ends at its last individual's row end
    auto end_of = [&](const uint32_t (&h)[CW]) {
        uint32_t m = h[0];
#pragma unroll
        for (uint32_t q = 1; q < CW; ++q) m = max(m, h[q]);
        return __reduce_max_sync(FULL, m);
    };
    // first edge at or after `at` that some light row of the chunk holds (E1 if none)
    auto next_light = [&](uint32_t at, const uint32_t (&l)[CW], const uint32_t (&h)[CW], uint32_t e1) {
        uint32_t m = e1;
#pragma unroll
        for (uint32_t q = 0; q < CW; ++q)
            if (h[q] - l[q] <= HEAVY_ROW && h[q] > max(at, l[q])) m = min(m, max(l[q], at));
        return __reduce_min_sync(FULL, m);
    };
    uint32_t cn[LOADS];
    auto fetch = [&](uint32_t at, uint32_t e1) {
#pragma unroll
        for (uint32_t u = 0; u < LOADS; ++u) {
            const uint32_t e = at + 32u * u + lane;
            cn[u] = e < e1 ? ld_stream(col + e) : 0u;
        }
    };
    auto claim = [&]() {   // the first word of the warp's next chunk
        uint32_t k = 0;
        if (lane == 0u) k = atomicAdd(chunk, 1u);
        return __shfl_sync(FULL, k, 0) * CW;
    };
    uint32_t jj = claim(), after;
    rows(jj, lo, hi);
    E1 = end_of(hi);
    uint32_t base = next_light(0, lo, hi, E1);
    if (base < E1) fetch(base, E1);
#pragma unroll 1
    for (; jj < K; jj = after) {
        uint32_t lo2[CW], hi2[CW];   // the next chunk's rows, on their way
        after = claim();
        rows(after, lo2, hi2);
        Count c[CW][P];
#pragma unroll
        for (uint32_t q = 0; q < CW; ++q)
#pragma unroll
            for (int k = 0; k < P; ++k) c[q][k].clear();
        while (base < E1) {   // warp-uniform
            uint32_t b[LOADS];
#pragma unroll
            for (uint32_t u = 0; u < LOADS; ++u) b[u] = cn[u];
            const uint32_t nb = base + WIN, next = next_light(nb, lo, hi, E1);
            if (next < E1) fetch(next, E1);
            uint32_t x[LOADS][P];
#pragma unroll
            for (uint32_t u = 0; u < LOADS; ++u) {
                if (base + 32u * u + lane < E1) {
                    ft_at(b[u], x[u]);
                } else {
#pragma unroll
                    for (int k = 0; k < P; ++k) x[u][k] = 0u;
                }
            }
#pragma unroll
            for (uint32_t u = 0; u < LOADS; ++u) {   // one P-word store per lane: no bank conflicts
                if constexpr (P == 1) buf[32u * u + lane] = x[u][0];
                else reinterpret_cast<uint2 *>(buf)[32u * u + lane] = make_uint2(x[u][0], x[u][1]);
            }
            __syncwarp();
#pragma unroll
            for (uint32_t q = 0; q < CW; ++q) {
                if (hi[q] - lo[q] > HEAVY_ROW) continue;
                const uint32_t k1 = min(hi[q], nb);
#pragma unroll 1
                for (uint32_t e = max(lo[q], base); e < k1; e += 3u) {
                    uint32_t y[3][P];
#pragma unroll
                    for (uint32_t t = 0; t < 3u; ++t) {
                        const bool in = e + t < k1;
                        if constexpr (P == 1) {
                            y[t][0] = in ? buf[e + t - base] : 0u;
                        } else {
                            const uint2 v = in ? reinterpret_cast<const uint2 *>(buf)[e + t - base] : make_uint2(0u, 0u);
                            y[t][0] = v.x, y[t][1] = v.y;
                        }
                    }
#pragma unroll
                    for (int k = 0; k < P; ++k) c[q][k].add3(y[0][k], y[1][k], y[2][k]);
                }
            }
            __syncwarp();
            base = next;
        }
        // the next chunk's first edges, behind which this one's heavy rows and truth tables run
        const uint32_t E2 = end_of(hi2);
        base = next_light(0, lo2, hi2, E2);
        if (base < E2) fetch(base, E2);
        uint32_t outw[P][CW];
#pragma unroll
        for (uint32_t q = 0; q < CW; ++q) {
            uint32_t hm = __ballot_sync(FULL, hi[q] - lo[q] > HEAVY_ROW);
#pragma unroll 1
            while (hm) {
                const uint32_t h = __ffs(hm) - 1;
                hm &= hm - 1;
                const uint32_t hlo = __shfl_sync(FULL, lo[q], h), hhi = __shfl_sync(FULL, hi[q], h);
                Count d[P];
#pragma unroll
                for (int k = 0; k < P; ++k) d[k].clear();
#pragma unroll 1
                for (uint32_t e = hlo + lane; e < hhi; e += 32u * HEAVY_LOADS) {
                    uint32_t to[HEAVY_LOADS], y[HEAVY_LOADS][P];
#pragma unroll
                    for (uint32_t t = 0; t < HEAVY_LOADS; ++t) to[t] = e + 32u * t < hhi ? ld_stream(col + e + 32u * t) : 0u;
#pragma unroll
                    for (uint32_t t = 0; t < HEAVY_LOADS; ++t) {
                        if (e + 32u * t < hhi) {
                            ft_at(to[t], y[t]);
                        } else {
#pragma unroll
                            for (int k = 0; k < P; ++k) y[t][k] = 0u;
                        }
                    }
#pragma unroll
                    for (uint32_t t = 0; t < HEAVY_LOADS; t += 3u)
#pragma unroll
                        for (int k = 0; k < P; ++k) d[k].add3(y[t][k], y[t + 1u][k], y[t + 2u][k]);
                }
                __syncwarp();
#pragma unroll
                for (int k = 0; k < P; ++k) {
                    d[k].saturate();
#pragma unroll
                    for (int s = 16; s > 0; s >>= 1) {
                        const uint32_t e0 = __shfl_xor_sync(FULL, d[k].c0, s), e1 = __shfl_xor_sync(FULL, d[k].c1, s);
                        const uint32_t e2 = __shfl_xor_sync(FULL, d[k].c2, s);
                        sat_add3(d[k].c0, d[k].c1, d[k].c2, e0, e1, e2);
                    }
                    if (lane == h) c[q][k] = d[k];
                }
            }
            const bool valid = (wb + jj + q) * 32u + lane < n_indiv;
#pragma unroll
            for (int k = 0; k < P; ++k) {
                c[q][k].saturate();
                const uint32_t *want = gp->want[k];   // the group's truth table (cached), by the planes of the count
                const uint32_t c0 = c[q][k].c0, c1 = c[q][k].c1, c2 = c[q][k].c2;
                const uint32_t a0 = (c0 & want[1]) | (~c0 & want[0]), a1 = (c0 & want[3]) | (~c0 & want[2]);
                const uint32_t a2 = (c0 & want[5]) | (~c0 & want[4]), a3 = (c0 & want[7]) | (~c0 & want[6]);
                const uint32_t b0 = (c1 & a1) | (~c1 & a0), b1 = (c1 & a3) | (~c1 & a2);
                outw[k][q] = transpose32(valid ? (c2 & b1) | (~c2 & b0) : 0u, lane);   // lane s: slice 32k + s's word
            }
        }
#pragma unroll
        for (int k = 0; k < P; ++k) {
            const uint32_t s = 32u * k + lane;
            if (s < n) {   // aligned: wb + jj is a multiple of CW
                uint32_t *dst = slots + (uint64_t)gp->out[s] * wp + wb + jj;
                *reinterpret_cast<uint2 *>(dst) = make_uint2(outw[k][0], outw[k][1]);
            }
        }
        E1 = E2;
#pragma unroll
        for (uint32_t q = 0; q < CW; ++q) lo[q] = lo2[q], hi[q] = hi2[q];
    }
}

// Copy the segment's filler row into shared memory (all threads of the CTA).
// A FORALL filler is staged complemented (REF_NEG), so the walk counts
// successors outside C without a per-edge complement.
__device__ __forceinline__ void stage_filler(const KBView &kb, const uint32_t *slots, uint32_t ref, uint32_t *dst) {
    const uint32_t id = ref & REF_ID;
    const uint32_t *src = (ref & REF_SLOT) ? slots + (uint64_t)id * kb.wp : kb.concepts + (uint64_t)id * kb.wp;
    const uint32_t x = (ref & REF_NEG) ? 0xFFFFFFFFu : 0u;
    const uint4 *s4 = reinterpret_cast<const uint4 *>(src);
    uint4 *d4 = reinterpret_cast<uint4 *>(dst);
    for (uint32_t q = threadIdx.x; q < kb.wp / 4; q += blockDim.x) {
        uint4 v = s4[q];
        d4[q] = make_uint4(v.x ^ x, v.y ^ x, v.z ^ x, v.w ^ x);
    }
}

// Register budget: every shape is compiled for 768 resident threads per SM
// (80 registers a thread; the prefetching stack machine and the windowed walks
// spill heavily at 64); FULL ones for 2,048 (32 registers, full occupancy, at
// the price of spills).  GROUPS = false leaves the role groups' transposes and
// walks out (for plans without role groups: a lone hypothesis, concrete-role
// restrictions); the rest fits 64 registers, so that build keeps 1,024
// threads per SM for the latency-bound lone walks and value streams.
// CONCRETE = false leaves the concrete-role value walk out, for KBs that have
// no concrete roles: its registers would otherwise raise the spills of the
// whole stack machine.
template <int NW, int WPL, bool STAGE, int BLK, bool FULL = false, bool GROUPS = true, bool CONCRETE = true>
__global__ void __launch_bounds__(NW * 32, (FULL ? 64 : (GROUPS ? 24 : 32)) / NW) exec_kernel(ExecArgs A) {
    // the host sizes the dynamic shared memory (smem_bytes)
    using SmemT = Smem<NW, WPL>;
    static_assert(offsetof(SmemT, tail) ==
                      sizeof(uint32_t) * NW * STACK_MAX * WPL * 32 +
                          SEG_BATCH * (sizeof(Seg) + SEG_CODE * sizeof(DInsn) + PF_SLOTS * sizeof(uint64_t) +
                                       2 * sizeof(uint32_t)) + 16,
                  "the shared-memory layout and its host-side size disagree");
    extern __shared__ __align__(16) uint8_t smem_raw[];
    Smem<NW, WPL> &sm = *reinterpret_cast<Smem<NW, WPL> *>(smem_raw);
    pdl_wait();   // for a plan that upload_kernel puts into the workspace
    const PlanHeader hd = *reinterpret_cast<const PlanHeader *>(A.ws);
    const Group *groups = reinterpret_cast<const Group *>(A.ws + hd.off_groups);
    const uint32_t *gsegs = reinterpret_cast<const uint32_t *>(A.ws + hd.off_gsegs);
    Counters *ctr = reinterpret_cast<Counters *>(A.ws + hd.off_ctr);
    uint32_t *done = reinterpret_cast<uint32_t *>(ctr + 1);
    uint32_t *acc = done + hd.n_segs + 1;
    uint32_t *slots = reinterpret_cast<uint32_t *>(A.ws + hd.off_slots);
    const RGroup *rgroups = reinterpret_cast<const RGroup *>(A.ws + hd.off_rgroups);
    // transposes and walks have tiles of their own: fine_ww words a warp
    const uint32_t fine_ww = hd.warp_words >> 8 & 0xFFu;
    const uint32_t fine_tiles = fine_ww ? (A.kb.wp + NW * fine_ww - 1u) / (NW * fine_ww) : 0u;
    const uint32_t seg_batch = max(hd.warp_words >> 16, 1u);

    // Thread 0 claims the next item as soon as the current one may start (its
    // dependencies are done), so the claim's round trip overlaps the work.
    // Items are claimed in queue order and a CTA holds at most two, the one it
    // runs and the next; every dependency points to an earlier item, so the
    // earliest unfinished item is always running and the queue drains.  (Giving a
    // CTA its index as the first item would save a round trip, but a CTA that
    // another stream's kernel keeps from starting would then hold an item.)
    uint32_t stride_next = A.item_begin + blockIdx.x;
    uint32_t nxt = A.item_end;   // thread 0: the item claimed while the current one runs
    uint32_t g = 0;              // the current item's group
    if (threadIdx.x == 0) {
        sm.item = A.use_queue ? A.item_begin + atomicAdd(&ctr->head, 1u) : stride_next;
        sm.ok = 1u;
    }
    for (;;) {
        __syncthreads();
        const uint32_t item = sm.item;
        if (threadIdx.x == 0) sm.chunk = 0u;
        stride_next += gridDim.x;
        if (item >= A.item_end) break;
        const Group grp = find_group(groups, hd.n_groups, item, g);
        const uint32_t local = item - grp.item_begin;
        // the tasks of an item are of one group and tile
        const uint32_t per = grp.level & GROUP_FINE ? 1u : seg_batch;
        const uint32_t blocks = (grp.n_segs + per - 1u) / per;
        const uint32_t tile = local / blocks, first = local % blocks * per;
        const uint32_t n_tasks = min(per, grp.n_segs - first);
        for (uint32_t b = threadIdx.x >> 5; b < n_tasks; b += NW) {   // a task a warp
            const uint32_t task = gsegs[grp.seg_begin + first + b];
            if (!prepare_task<NW, WPL>(A, hd, sm, b, task, slots, done, ctr, fine_tiles)) sm.ok = 0u;
        }
        __syncthreads();
        if (!sm.ok) break;
        if (A.use_queue && threadIdx.x == 0) nxt = A.item_begin + atomicAdd(&ctr->head, 1u);
        const Seg &seg = sm.seg[0];
        if (seg.kind != TASK_SEGMENT && !GROUPS) {
            // a build without role groups was given a plan with them (the host never does this)
            if (threadIdx.x == 0) {
                atomicOr(A.kb.status, ST_DEVICE_CHECK);
                atomicExch(&ctr->abort, 1u);
            }
        } else if (seg.kind == TASK_TRANSPOSE) {
            if constexpr (GROUPS) {
                const RGroup *gp = rgroups + seg.code_off;
                if (gp->parts == 1) run_transpose<NW, 1>(A, fine_ww, gp, tile, slots);
                else run_transpose<NW, MAX_PARTS>(A, fine_ww, gp, tile, slots);
            }
        } else if (seg.kind == TASK_WALK) {
            if constexpr (GROUPS) {
                // the warp's stack (unused by a walk) holds its window of gathered FT words
                const RGroup *gp = rgroups + seg.code_off;
                const uint32_t wb = tile * NW * fine_ww, K = min(NW * fine_ww, A.kb.wp - wb);
                const uint32_t *ft = reinterpret_cast<const uint32_t *>(A.ws + gp->ft_off);
                uint32_t *buf = &sm.stk[threadIdx.x >> 5][0][0][0];
                if (gp->parts == 1)
                    run_walk<1>(A.kb.csr + gp->role2, ft, gp, A.kb.n, A.kb.w, A.kb.wp, wb, K, slots, buf, &sm.chunk);
                else
                    run_walk<MAX_PARTS>(A.kb.csr + gp->role2, ft, gp, A.kb.n, A.kb.w, A.kb.wp, wb, K, slots, buf, &sm.chunk);
            }
        } else {
            if constexpr (STAGE) {   // one segment an item
                if (seg.filler != NO_FILLER) {
                    stage_filler(A.kb, slots, seg.filler, sm.tail + A.ring_words);
                    __syncthreads();
                }
            }
#pragma unroll 1
            for (uint32_t b = 0; b < n_tasks; ++b)
                run_tile<NW, WPL, STAGE, BLK, CONCRETE>(A, hd, b, tile, sm, slots, acc);
        }
        __syncthreads();
        if (A.use_queue) {
            if (threadIdx.x < n_tasks) {
                __threadfence();
                atomicAdd(done + sm.task[threadIdx.x], 1u);
            }
            if (threadIdx.x == 0) sm.item = *(volatile uint32_t *)&ctr->abort ? A.item_end : nxt;
        } else if (threadIdx.x == 0) {
            sm.item = stride_next;
        }
    }
}

// (TP, FP) accumulators -> (TP, FP, FN, TN).
__global__ void finalize_kernel(KBView kb, const uint8_t *ws, uint32_t *counts) {
    const PlanHeader *hd = reinterpret_cast<const PlanHeader *>(ws);
    const Counters *ctr = reinterpret_cast<const Counters *>(ws + hd->off_ctr);
    const uint32_t *acc = reinterpret_cast<const uint32_t *>(ctr + 1) + hd->n_segs + 1;
    for (uint32_t h = blockIdx.x * blockDim.x + threadIdx.x; h < hd->n_hyps; h += gridDim.x * blockDim.x) {
        const uint32_t tp = acc[2 * h], fp = acc[2 * h + 1];
        uint4 c = make_uint4(tp, fp, kb.n_pos - tp, kb.n_neg - fp);
        *reinterpret_cast<uint4 *>(counts + 4ull * h) = c;
    }
}

// Puts a small plan's image, which comes as the kernel's argument, into the
// workspace.  A host-to-device copy of 2 KB waits for the copy engine and the
// interpreter for it; this is one more short kernel, which the interpreter's
// blocks start behind (pdl_wait).
struct SmallImage {
    uint4 data[SMALL_IMAGE / 16];
};
__global__ void upload_kernel(const __grid_constant__ SmallImage img, uint4 *ws, uint32_t n) {
    pdl_trigger();
    pdl_wait();   // an earlier launch may still use the workspace
    for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) ws[i] = img.data[i];
}

using KernelFn = void (*)(ExecArgs);

// Instantiated launch shapes: warps x words per lane x staging x chunks per
// block of the lone walk (1- and 2-warp CTAs only with one word per lane and no
// staging).
template <bool STAGE, int BLK>
KernelFn pick_t(uint32_t warps, uint32_t wpl) {
    if (wpl == 4) {
        if (warps == 4) return exec_kernel<4, 4, STAGE, BLK>;
        if (warps == 16) return exec_kernel<16, 4, STAGE, BLK>;
        return exec_kernel<8, 4, STAGE, BLK>;
    }
    if constexpr (!STAGE) {
        if (warps == 1) return exec_kernel<1, 1, false, BLK>;
        if (warps == 2) return exec_kernel<2, 1, false, BLK>;
    }
    if (warps == 4) return exec_kernel<4, 1, STAGE, BLK>;
    if (warps == 16) return exec_kernel<16, 1, STAGE, BLK>;
    if (warps == 32) return exec_kernel<32, 1, STAGE, BLK>;
    return exec_kernel<8, 1, STAGE, BLK>;
}

template <int BLK>
KernelFn pick_b(const Tuning &t, bool stage, bool groups, bool concrete) {
    if (t.warps == 8 && t.wpl == 1 && !stage) {   // the common shapes
        if (t.full_occupancy) return exec_kernel<8, 1, false, BLK, true>;
        if (!groups)
            return concrete ? exec_kernel<8, 1, false, BLK, false, false> : exec_kernel<8, 1, false, BLK, false, false, false>;
        if (!concrete) return exec_kernel<8, 1, false, BLK, false, true, false>;
    }
    return stage ? pick_t<true, BLK>(t.warps, t.wpl) : pick_t<false, BLK>(t.warps, t.wpl);
}

KernelFn pick(const Tuning &t, bool stage, bool groups, bool concrete) {
    return t.role_block == 8 ? pick_b<8>(t, stage, groups, concrete) : pick_b<4>(t, stage, groups, concrete);
}

uint32_t ring_words(const hedl_kb *kb, const Tuning &t) { return kb->has_concrete() ? t.warps * EX_SMEM_WORDS : 0u; }

size_t smem_bytes(const hedl_kb *kb, const Tuning &t, bool stage) {
    size_t b = stack_smem_bytes(t) + 16 + 4ull * ring_words(kb, t);   // ... item / ok / pad, rings
    if (stage) b += 4ull * kb->wp;
    return b;
}

}  // namespace

bool use_staging(const hedl_kb *kb, const Tuning &t) {
    return t.stage && t.warps >= 4 && smem_bytes(kb, t, true) <= kb->smem_optin;
}

int exec_occupancy(const hedl_kb *kb, const Tuning &t, bool groups, int *blocks_per_sm) {
    const bool stage = use_staging(kb, t);
    KernelFn fn = pick(t, stage, groups, kb->has_concrete());
    size_t smem = smem_bytes(kb, t, stage);
    // the limit, not this plan's size: plans of other sizes share the kernel
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kb->smem_optin);
    if (e != cudaSuccess) return e;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, fn, (int)(t.warps * 32), smem);
    return e;
}

int upload_small_plan(const PlanImpl *p, void *ws, void *stream) {
    SmallImage img;
    memcpy(img.data, p->image.data(), p->image_bytes);
    return launch_pdl(upload_kernel, 1u, 128u, 0, (cudaStream_t)stream, img, (uint4 *)ws, (uint32_t)(p->image_bytes / 16));
}

int launch_exec(const hedl_kb *kb, const PlanImpl *p, uint32_t *counts, uint32_t *out_bits, void *ws,
                void *stream) {
    cudaStream_t s = (cudaStream_t)stream;
    const Tuning &t = p->tuning;
    KernelFn fn = pick(t, p->staged, p->n_rgroups > 0, kb->has_concrete());
    size_t smem = smem_bytes(kb, t, p->staged);
    int bps = p->bps;
    if (bps < 1) return cudaErrorInvalidConfiguration;
    if (t.ctas_per_sm && (int)t.ctas_per_sm < bps) bps = (int)t.ctas_per_sm;
    ExecArgs A{};
    A.kb = kb->view();
    A.ring_words = ring_words(kb, t);
    A.ws = (uint8_t *)ws;
    A.counts = counts;
    A.out_bits = out_bits;
    const uint32_t n_items = p->n_items;
    if (p->flags & HEDL_LEVELS) {
        // one launch per level; items of a level are independent
        A.use_queue = 0;
        for (uint32_t l = 0; l < p->info.n_levels; ++l) {
            A.item_begin = p->level_items[l];
            A.item_end = p->level_items[l + 1];
            uint32_t n = A.item_end - A.item_begin;
            if (!n) continue;
            uint32_t grid = std::min<uint32_t>(n, (uint32_t)(bps * kb->n_sms));
            fn<<<grid, t.warps * 32, smem, s>>>(A);
            cudaError_t le = cudaGetLastError();
            if (le != cudaSuccess) return le;
        }
    } else {
        A.use_queue = 1;
        A.item_begin = 0;
        A.item_end = n_items;
        uint32_t grid = std::min<uint32_t>(std::max<uint32_t>(n_items, 1), (uint32_t)(bps * kb->n_sms));
        const cudaError_t le = launch_pdl(fn, grid, t.warps * 32, smem, s, A);
        if (le != cudaSuccess) return le;
    }
    if (!counts) return cudaSuccess;
    finalize_kernel<<<std::max<uint32_t>(1, std::min<uint32_t>((p->n_hyps + 255) / 256, 1024)), 256, 0, s>>>(
        kb->view(), (const uint8_t *)ws, counts);
    return cudaGetLastError();
}

}  // namespace hedl
