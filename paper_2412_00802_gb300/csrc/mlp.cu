// The learned surrogate: structural encoder, a 512-512-512-2 MLP with BF16
// weights/activations and FP32 accumulation (forward, backward, Adam), exact
// scores from coverage counts, and a deterministic top-k selection.  The
// paper has no counterpart; the surrogate only orders and prunes the queue of
// exact evaluations.
//
// The dense layers run on tcgen05 (umma.cu).  The comparison engine is a
// warp-level BF16 GEMM (mma.sync m16n8k16, operands staged in shared memory
// and read with ldmatrix, FP32 accumulators in registers) with the same
// epilogues; its split-K mode accumulates weight gradients with atomics.
//
// A training step is six launches: two layers forward (the second also dots
// its rows with the output layer), head_bwd_kernel (output layer, loss and
// its gradients), dH1, both weight gradients, and update_kernel (partial sums
// to gradients, Adam).  Every sum over the batch is first a partial sum of a
// chunk of rows and then a sum over chunks in a fixed order, so a step's
// gradients do not depend on timing.  At batches of 4,096 this took a step
// from 785 us to 57 us: the weight gradient of the output layer
// (584 us) and the bias gradients (2 x 238 us) had been two blocks' loops over
// the whole batch, and the weight gradients had needed four transposes.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <string>
#include <vector>

#include "hedl_internal.h"
#include "launch.cuh"

namespace hedl {
namespace {

constexpr int DI = 512, DH = 512, DO = 2;

// ------------------------------------------------------------------ encoder
__device__ __forceinline__ int arity_of(uint32_t op) {
    if (op == HEDL_OP_NOT || (op >= HEDL_OP_EXISTS && op <= HEDL_OP_EXACTLY)) return 1;
    if (op == HEDL_OP_AND || op == HEDL_OP_OR) return 2;
    return 0;
}

constexpr int ENC_MAXLEN = 256;

// Structural encoding, one warp per program.  Lane l holds instructions l,
// l + 32, ... (one register each up to 32 instructions).  Depths and
// polarities come from the postfix heights: with s_k the operands on the stack
// after instruction k, the parent of k is the first j > k with s_j <= s_k, and
// every such running minimum to the right of k is an ancestor (NOT and ATMOST
// ancestors flip the polarity).  Up to 32 instructions, a ballot per height
// gives every node its parent and pointer jumping its depth; longer programs
// count the minima.  The lanes then count features into shared memory (totals
// by ballots) and write the row as bf16 (counts x 1/4, exact), the two prior
// inputs as bf16 of the caller's values.  The next program's instructions are
// loaded while the current one is counted.
// Signed counts add +1 at polarity 0 and -1 at polarity 1.
//   [  0, 84) op x min(depth, 5)          [ 84,180) concept mod 96, signed
//   [180,244) role mod 32 x inverse       [244,284) restriction kind x depth
//   [284,308) cardinality                 [308,436) property mod 16 x (>=, <=) x bucket / 4, signed
//   [436,493) role-over-atom hash mod 57, signed
//   [493,497) length / 10                 [497,504) statistics sums, signed
//   [504,510) totals, height, constant    [510,512) prior
// stats (or null): n_sc atom scores, then n_grid x 2 x 16 threshold scores.
//
// Bound: 1 KB written a program (67 MB at 65,536: 10 us) against the latency
// of one program's chain (offsets -> instructions -> counts -> row).  One lane
// walking the program with a stack in shared memory, and 2-byte stores, took
// 75 us at 65,536 programs of 13 instructions; this takes 46 us.
constexpr int ENC_WARPS = 8;

// The lane's nodes of a program of at most 32 * N instructions: heights, then
// depth, polarity and the program's height.  Nodes that no root reaches (the
// program is not well formed: a height below the last one's, and all before
// it) get depth 0 and polarity 0.
template <int N>
__device__ __forceinline__ void encode_nodes(const uint64_t (&w)[N], uint32_t L, uint32_t lane, uint32_t (&depth)[N],
                                             uint32_t (&pol)[N], uint32_t &height) {
    int s[N];
    uint32_t flip[N];   // ballot: NOT / ATMOST among the register's 32 instructions
    int base = 0;
#pragma unroll
    for (int r = 0; r < N; ++r) {
        const uint32_t op = (uint32_t)(w[r] & 0xFF), k = 32u * r + lane;
        int v = k < L ? 1 - arity_of(op) : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xFFFFFFFFu, v, o);
            if (lane >= (uint32_t)o) v += t;
        }
        s[r] = base + v;
        base = __shfl_sync(0xFFFFFFFFu, s[r], 31);
        flip[r] = __ballot_sync(0xFFFFFFFFu, k < L && (op == HEDL_OP_NOT || op == HEDL_OP_ATMOST));
    }
    // base is now the height after the last instruction; the last node below it cuts the program
    int cut = -1;
#pragma unroll
    for (int r = 0; r < N; ++r) {
        const uint32_t below = __ballot_sync(0xFFFFFFFFu, 32u * r + lane < L && s[r] < base);
        if (below) cut = 32 * r + 31 - __clz((int)below);
    }
    if constexpr (N == 1) {
        // parent: the first j > k with s_j <= s_k (its own lane if there is none); the heights of the
        // nodes after the cut lie between base and the largest one
        const bool node = lane < L && (int)lane > cut;
        const uint32_t later = ~((2u << lane) - 1u);
        const int top = __reduce_max_sync(0xFFFFFFFFu, node ? s[0] : base);
        uint32_t parent = lane;
        for (int h = base; h <= top; ++h) {   // warp-uniform
            const uint32_t at = __ballot_sync(0xFFFFFFFFu, node && s[0] <= h) & later;
            if (node && s[0] == h && at) parent = (uint32_t)__ffs((int)at) - 1u;
        }
        // ancestors counted by pointer jumping: low half the depth, high half the flips
        uint32_t acc = parent != lane ? 1u + ((flip[0] >> parent & 1u) << 16) : 0u;
        while (__any_sync(0xFFFFFFFFu, parent != lane)) {
            const uint32_t more = __shfl_sync(0xFFFFFFFFu, acc, (int)parent);
            const uint32_t next = __shfl_sync(0xFFFFFFFFu, parent, (int)parent);
            if (parent != lane) acc += more;   // a root's own count is zero
            parent = next == parent ? lane : next;
        }
        depth[0] = acc & 0xFFFFu, pol[0] = acc >> 16 & 1u;
        height = __reduce_max_sync(0xFFFFFFFFu, node ? depth[0] + 1u : 0u);
    } else {
        int low[N];
#pragma unroll
        for (int r = 0; r < N; ++r) depth[r] = pol[r] = 0u, low[r] = s[r];
#pragma unroll
        for (int q = 0; q < N; ++q) {   // ancestors in register q's instructions
            for (uint32_t l = 0; l < 32u && 32u * q + l < L; ++l) {
                const int sj = __shfl_sync(0xFFFFFFFFu, s[q], (int)l);
                const uint32_t f = flip[q] >> l & 1u;
#pragma unroll
                for (int r = 0; r <= q; ++r)
                    if ((r < q || lane < l) && sj <= low[r]) low[r] = sj, depth[r] += 1u, pol[r] ^= f;
            }
        }
        uint32_t ht = 0;
#pragma unroll
        for (int r = 0; r < N; ++r) {
            const int k = (int)(32u * r + lane);
            if (k <= cut) depth[r] = pol[r] = 0u;
            else if ((uint32_t)k < L) ht = max(ht, depth[r] + 1u);
        }
        height = __reduce_max_sync(0xFFFFFFFFu, ht);
    }
}

struct EncTables {
    const float *grid;      // or null
    const int32_t *stats;   // or null
    uint32_t n_grid, n_sc;
};

// Counts a program's features; w: its instructions as in encode_nodes (0 past the end).
template <int N>
__device__ __forceinline__ void encode_program(const uint64_t (&w)[N], uint32_t L, uint32_t lane, int *feat,
                                               const EncTables &t) {
    const float *__restrict__ grid = t.grid;
    const int32_t *__restrict__ stats = t.stats;
    const uint32_t n_grid = t.n_grid, n_sc = t.n_sc;
    uint32_t depth[N], pol[N], height;
    encode_nodes<N>(w, L, lane, depth, pol, height);
    uint64_t left_of_0 = 0ull;   // the instruction before the register's first
    int leaves = 0, roles = 0, datas = 0, nots = 0;
#pragma unroll
    for (int r = 0; r < N; ++r) {
        const uint32_t k = 32u * r + lane;
        uint64_t c = __shfl_up_sync(0xFFFFFFFFu, w[r], 1);   // the instruction before this one
        if (lane == 0) c = left_of_0;
        left_of_0 = __shfl_sync(0xFFFFFFFFu, w[r], 31);
        const uint32_t op = (uint32_t)(w[r] & 0xFF), inv = (uint32_t)((w[r] >> 8) & 1);
        const uint32_t a = (uint32_t)((w[r] >> 16) & 0xFFFF), b = (uint32_t)(w[r] >> 32);
        const bool counted = k < L && op >= HEDL_OP_ATOM && op <= HEDL_OP_DEQ;   // else not an op, or a string restriction
        leaves += __popc(__ballot_sync(0xFFFFFFFFu, counted && arity_of(op) == 0));
        roles += __popc(__ballot_sync(0xFFFFFFFFu, counted && op >= HEDL_OP_EXISTS && op <= HEDL_OP_EXACTLY));
        datas += __popc(__ballot_sync(0xFFFFFFFFu, counted && op >= HEDL_OP_DGE));
        nots += __popc(__ballot_sync(0xFFFFFFFFu, counted && op == HEDL_OP_NOT));
        if (!counted) continue;
        const uint32_t dk = depth[r];
        const int sign = pol[r] ? -1 : 1;
        atomicAdd(&feat[min(dk, 5u) * 14 + op - 1], 1);
        if (op == HEDL_OP_ATOM) {
            atomicAdd(&feat[84 + a % 96], sign);
            if (stats && a < n_sc) atomicAdd(&feat[497 + min(dk / 2, 2u)], sign * stats[a]);
        } else if (op >= HEDL_OP_EXISTS && op <= HEDL_OP_EXACTLY) {
            atomicAdd(&feat[180 + (a % 32) * 2 + inv], 1);
            atomicAdd(&feat[244 + min(dk, 7u) * 5 + (op - HEDL_OP_EXISTS)], 1);
            if (op >= HEDL_OP_ATLEAST) atomicAdd(&feat[284 + (op - HEDL_OP_ATLEAST) * 8 + min(b, 7u)], 1);
            if (k > 0 && (c & 0xFF) == HEDL_OP_ATOM) {   // the filler ends right before its restriction
                const uint32_t cc = (uint32_t)((c >> 16) & 0xFFFF);
                atomicAdd(&feat[436 + ((a * 2 + inv) * 131 + cc) % 57], sign);
                if (stats && cc < n_sc) atomicAdd(&feat[503], sign * stats[cc]);
            }
        } else if (op >= HEDL_OP_DGE) {
            if (op != HEDL_OP_DEQ) {
                const float t = __uint_as_float(b);
                uint32_t q = 0;
                if (grid && a < n_grid && !(t != t))
                    for (int g = 0; g < 15; ++g) q += grid[a * 15 + g] < t ? 1u : 0u;
                atomicAdd(&feat[308 + ((a % 16) * 2 + (op - HEDL_OP_DGE)) * 4 + q / 4], sign);
                if (stats && a < n_grid)
                    atomicAdd(&feat[500 + min(dk / 2, 2u)], sign * stats[n_sc + (a * 2 + (op - HEDL_OP_DGE)) * 16 + q]);
            }
        }
    }
    if (lane == 0) {   // no other lane adds to these
        feat[493 + min(L, 39u) / 10] = 1;
        feat[504] = leaves, feat[505] = roles, feat[506] = datas, feat[507] = nots;
        feat[508] = (int)min(height, 8u) - 1;
        feat[509] = 4;
    }
}

// Programs of more than 32 instructions: a call, so that their registers do not limit the others' occupancy.
template <int N>
__device__ __noinline__ void encode_long(const uint64_t *__restrict__ prog, uint32_t L, int *feat, const EncTables &t) {
    const uint32_t lane = threadIdx.x & 31u;
    uint64_t w[N];
#pragma unroll
    for (int r = 0; r < N; ++r) w[r] = 32u * r + lane < L ? prog[32u * r + lane] : 0ull;
    encode_program<N>(w, L, lane, feat, t);
}

__global__ void __launch_bounds__(32 * ENC_WARPS, 4)
    encode_kernel(const uint64_t *__restrict__ progs, const uint32_t *__restrict__ offs, uint32_t H, EncTables t,
                  const float *__restrict__ prior, __nv_bfloat16 *__restrict__ X) {
    __shared__ __align__(16) int feats[ENC_WARPS][DI];
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int *feat = feats[warp];
    int4 *f4 = reinterpret_cast<int4 *>(feat);
    const bool wide = (reinterpret_cast<uintptr_t>(X) & 15) == 0;   // 16-byte stores
    const uint32_t step = gridDim.x * ENC_WARPS;
    // programs longer than ENC_MAXLEN are encoded by their last ENC_MAXLEN
    // instructions (the root and the nodes nearest to it)
    struct Prog {
        uint64_t w;        // the lane's instruction of a program of at most 32
        uint32_t end, L;
    };
    auto range = [&](uint32_t h, Prog &p) {
        p.end = h < H ? offs[h + 1] : 0u;
        p.L = h < H ? min(p.end - offs[h], (uint32_t)ENC_MAXLEN) : 0u;
    };
    auto load = [&](Prog &p) { p.w = lane < p.L && p.L <= 32u ? progs[p.end - p.L + lane] : 0ull; };
    uint32_t h = blockIdx.x * ENC_WARPS + warp;
    Prog cur, nxt;
    range(h, cur);
    load(cur);
    range(h + step, nxt);
    for (; h < H; h += step) {
        load(nxt);                         // one program ahead
        Prog far;
        range(h + 2u * step, far);         // its range another one
        const float pr = prior && lane >= 30 ? prior[2ull * h + (lane - 30)] : 0.0f;
#pragma unroll
        for (int q = 0; q < DI / 128; ++q) f4[32 * q + lane] = make_int4(0, 0, 0, 0);
        __syncwarp();
        if (cur.L <= 32u) {
            const uint64_t w[1] = {cur.w};
            encode_program<1>(w, cur.L, lane, feat, t);
        } else if (cur.L <= 64u) {
            encode_long<2>(progs + (cur.end - cur.L), cur.L, feat, t);
        } else {
            encode_long<ENC_MAXLEN / 32>(progs + (cur.end - cur.L), cur.L, feat, t);
        }
        cur = nxt;
        nxt = far;
        __syncwarp();
        // the priors take the last two places (never counted); they are not scaled
        const float p0 = __shfl_sync(0xFFFFFFFFu, pr, 30), p1 = __shfl_sync(0xFFFFFFFFu, pr, 31);
        __nv_bfloat16 *row = X + (uint64_t)h * DI;
#pragma unroll
        for (int q = 0; q < DI / 256; ++q) {   // eight features a lane
            const uint32_t at = 32 * q + lane;
            const int4 x = f4[2 * at], y = f4[2 * at + 1];
            float v[8] = {0.25f * (float)x.x, 0.25f * (float)x.y, 0.25f * (float)x.z, 0.25f * (float)x.w,
                          0.25f * (float)y.x, 0.25f * (float)y.y, 0.25f * (float)y.z, 0.25f * (float)y.w};
            if (at == DI / 8 - 1) v[6] = p0, v[7] = p1;
            uint32_t o[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const __nv_bfloat162 z = __floats2bfloat162_rn(v[2 * e], v[2 * e + 1]);
                o[e] = *reinterpret_cast<const uint32_t *>(&z);
            }
            if (wide) {
                reinterpret_cast<uint4 *>(row)[at] = make_uint4(o[0], o[1], o[2], o[3]);
            } else {
#pragma unroll
                for (int e = 0; e < 8; ++e) row[8 * at + e] = __ushort_as_bfloat16((unsigned short)(o[e / 2] >> 16 * (e & 1)));
            }
        }
        __syncwarp();
    }
}

// ------------------------------------------------------------------ tensor-core GEMM
// C[M,N] = sum_k A(m,k) B(k,n), A and B bf16, FP32 accumulation.
//   A_KM: A stored [K][M] (else [M][K]);  B_KN: B stored [K][N] (else [N][K]).
// Tiles: 128 x 128 x 32, 8 warps of 64 x 32, mma.sync.m16n8k16.
constexpr int BM = 128, BN = 128, BK = 32, PAD = 8;

struct GemmArgs {
    const __nv_bfloat16 *A;
    const __nv_bfloat16 *B;
    void *C;
    const float *bias;              // [N] or null
    const __nv_bfloat16 *mask;      // [M][N] (ld = ldc): keep where mask > 0, or null
    int M, N, K, lda, ldb, ldc;
    int relu, out_bf16, atomic;     // atomic: FP32 atomicAdd into C (split-K)
    int k_chunk;                    // K range per blockIdx.z
};

__device__ __forceinline__ void ldsm_x4(uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3, const void *p) {
    uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(a));
}

__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                 "{%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Load a 128 x 32 operand tile into smem as [row][k] (k contiguous); rows are
// M (or N) indices.  KMAJ: the operand is stored [rows][K]; else [K][rows].
template <bool KMAJ>
__device__ __forceinline__ void load_tile(__nv_bfloat16 (*dst)[BK + PAD], const __nv_bfloat16 *src, int rows,
                                          int K, int ld, int r0, int k0) {
    const __nv_bfloat16 zero = __float2bfloat16_rn(0.f);
    if constexpr (KMAJ) {
        for (int idx = threadIdx.x; idx < BM * (BK / 8); idx += blockDim.x) {
            const int r = idx / (BK / 8), kc = (idx % (BK / 8)) * 8;
            const int gr = r0 + r, gk = k0 + kc;
            __nv_bfloat16 *d = &dst[r][kc];
            const __nv_bfloat16 *s = src + (size_t)gr * ld + gk;
            if (gr < rows && gk + 8 <= K && ((reinterpret_cast<uintptr_t>(s) & 15) == 0)) {
                *reinterpret_cast<uint4 *>(d) = *reinterpret_cast<const uint4 *>(s);
            } else {
#pragma unroll
                for (int j = 0; j < 8; ++j) d[j] = (gr < rows && gk + j < K) ? s[j] : zero;
            }
        }
    } else {
        for (int idx = threadIdx.x; idx < BK * (BM / 8); idx += blockDim.x) {
            const int k = idx / (BM / 8), rc = (idx % (BM / 8)) * 8;
            const int gk = k0 + k, gr = r0 + rc;
            const __nv_bfloat16 *s = src + (size_t)gk * ld + gr;
            __nv_bfloat16 v[8];
            if (gk < K && gr + 8 <= rows && ((reinterpret_cast<uintptr_t>(s) & 15) == 0)) {
                *reinterpret_cast<uint4 *>(v) = *reinterpret_cast<const uint4 *>(s);
            } else {
#pragma unroll
                for (int j = 0; j < 8; ++j) v[j] = (gk < K && gr + j < rows) ? s[j] : zero;
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) dst[rc + j][k] = v[j];
        }
    }
}

template <bool A_KM, bool B_KN>
__global__ void __launch_bounds__(256) gemm_kernel(GemmArgs g) {
    __shared__ __align__(16) __nv_bfloat16 As[BM][BK + PAD];
    __shared__ __align__(16) __nv_bfloat16 Bs[BN][BK + PAD];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wm = warp >> 2, wn = warp & 3;          // 2 x 4 warps
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    const int kb = blockIdx.z * g.k_chunk, ke = min(g.K, kb + g.k_chunk);
    float acc[4][4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[i][j][q] = 0.f;
    for (int k0 = kb; k0 < ke; k0 += BK) {
        // operands restricted to this split's K range
        load_tile<!A_KM>(As, g.A, g.M, ke, g.lda, m0, k0);
        load_tile<!B_KN>(Bs, g.B, g.N, ke, g.ldb, n0, k0);
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < BK; kk += 16) {
            uint32_t af[4][4];
#pragma unroll
            for (int mt = 0; mt < 4; ++mt) {
                const int r = wm * 64 + mt * 16 + (lane & 15), c = kk + (lane >> 4) * 8;
                ldsm_x4(af[mt][0], af[mt][1], af[mt][2], af[mt][3], &As[r][c]);
            }
#pragma unroll
            for (int np = 0; np < 2; ++np) {
                uint32_t b0, b1, b2, b3;
                const int r = wn * 32 + np * 16 + (lane & 7) + ((lane >> 4) << 3);
                const int c = kk + ((lane >> 3) & 1) * 8;
                ldsm_x4(b0, b1, b2, b3, &Bs[r][c]);
#pragma unroll
                for (int mt = 0; mt < 4; ++mt) {
                    mma16816(acc[mt][np * 2 + 0], af[mt], b0, b1);
                    mma16816(acc[mt][np * 2 + 1], af[mt], b2, b3);
                }
            }
        }
        __syncthreads();
    }
    // epilogue
#pragma unroll
    for (int mt = 0; mt < 4; ++mt)
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                const int row = m0 + wm * 64 + mt * 16 + (lane >> 2) + half * 8;
                const int col = n0 + wn * 32 + nt * 8 + (lane & 3) * 2;
                if (row >= g.M) continue;
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int cc = col + e;
                    if (cc >= g.N) continue;
                    float v = acc[mt][nt][half * 2 + e];
                    if (g.bias) v += g.bias[cc];
                    if (g.relu) v = fmaxf(v, 0.f);
                    if (g.mask && !(__bfloat162float(g.mask[(size_t)row * g.ldc + cc]) > 0.f)) v = 0.f;
                    if (g.atomic) atomicAdd(reinterpret_cast<float *>(g.C) + (size_t)row * g.ldc + cc, v);
                    else if (g.out_bf16)
                        reinterpret_cast<__nv_bfloat16 *>(g.C)[(size_t)row * g.ldc + cc] = __float2bfloat16_rn(v);
                    else reinterpret_cast<float *>(g.C)[(size_t)row * g.ldc + cc] = v;
                }
            }
}

int gemm(const GemmArgs &a0, bool a_km, bool b_kn, int splits, cudaStream_t s) {
    GemmArgs a = a0;
    splits = std::max(1, splits);
    a.k_chunk = ((a.K + splits - 1) / splits + BK - 1) / BK * BK;
    dim3 grid((a.N + BN - 1) / BN, (a.M + BM - 1) / BM, (a.K + a.k_chunk - 1) / a.k_chunk);
    if (a_km && b_kn) gemm_kernel<true, true><<<grid, 256, 0, s>>>(a);
    else if (a_km) gemm_kernel<true, false><<<grid, 256, 0, s>>>(a);
    else if (b_kn) gemm_kernel<false, true><<<grid, 256, 0, s>>>(a);
    else gemm_kernel<false, false><<<grid, 256, 0, s>>>(a);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ output layer (N = 2)
// Y = u + b3 from the fused output layer's sums u [parts][B][2], a thread a row.
// With map (DEVICE float[5]: mean0, mean1, scale0, scale1, tail weight), the
// output is mapped back to the target scale: Y = (u + b3) * scale + mean.
__global__ void out_map_kernel(const float *u, int parts, const float *b3, float *Y, int B, const float *map) {
    pdl_trigger();
    pdl_wait();
    for (int row = blockIdx.x * blockDim.x + threadIdx.x; row < B; row += gridDim.x * blockDim.x) {
        float u0 = 0.f, u1 = 0.f;
        for (int p = 0; p < parts; ++p) {
            const float2 q = reinterpret_cast<const float2 *>(u)[(size_t)p * B + row];
            u0 += q.x, u1 += q.y;
        }
        u0 += b3[0], u1 += b3[1];
        if (map) {
            u0 = u0 * map[2] + map[0];
            u1 = u1 * map[3] + map[1];
        }
        Y[2 * (size_t)row] = u0;
        Y[2 * (size_t)row + 1] = u1;
    }
}

// The output layer of the mma.sync engine: Y[b][j] = sum_i H2[b][i] W3[j][i] + b3[j],
// mapped as above; one warp per row.
__global__ void out_fwd_kernel(const __nv_bfloat16 *H2, const __nv_bfloat16 *W3, const float *b3, float *Y, int B,
                               const float *map) {
    // warp per row (grid-stride); lane l holds columns 16l .. 16l+15 of both W3 rows
    const int lane = threadIdx.x & 31;
    float w0[16], w1[16];
    {
        const uint4 *p0 = reinterpret_cast<const uint4 *>(W3 + 16 * lane);
        const uint4 *p1 = reinterpret_cast<const uint4 *>(W3 + DH + 16 * lane);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const uint4 a = p0[q], c = p1[q];
            const uint32_t av[4] = {a.x, a.y, a.z, a.w}, cv[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const __nv_bfloat162 x = *reinterpret_cast<const __nv_bfloat162 *>(&av[e]);
                const __nv_bfloat162 y = *reinterpret_cast<const __nv_bfloat162 *>(&cv[e]);
                w0[q * 8 + 2 * e] = __low2float(x), w0[q * 8 + 2 * e + 1] = __high2float(x);
                w1[q * 8 + 2 * e] = __low2float(y), w1[q * 8 + 2 * e + 1] = __high2float(y);
            }
        }
    }
    const int warps = (gridDim.x * blockDim.x) >> 5;
    for (int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; row < B; row += warps) {
        const uint4 *h = reinterpret_cast<const uint4 *>(H2 + (size_t)row * DH + 16 * lane);
        float s0 = 0.f, s1 = 0.f;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const uint4 a = h[q];
            const uint32_t av[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const __nv_bfloat162 x = *reinterpret_cast<const __nv_bfloat162 *>(&av[e]);
                const float lo = __low2float(x), hi = __high2float(x);
                s0 += lo * w0[q * 8 + 2 * e] + hi * w0[q * 8 + 2 * e + 1];
                s1 += lo * w1[q * 8 + 2 * e] + hi * w1[q * 8 + 2 * e + 1];
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            s0 += __shfl_xor_sync(0xFFFFFFFFu, s0, o);
            s1 += __shfl_xor_sync(0xFFFFFFFFu, s1, o);
        }
        if (lane == 0) {
            float u0 = s0 + b3[0], u1 = s1 + b3[1];
            if (map) {
                u0 = u0 * map[2] + map[0];
                u1 = u1 * map[3] + map[1];
            }
            Y[2 * row] = u0;
            Y[2 * row + 1] = u1;
        }
    }
}

// Output layer's backward pass over a chunk of HB_ROWS rows a block.
//   Raw outputs u = sum of y's parts + b3 (b3 null: y is already u), mapped
//   targets t' = (T - mean) / scale, row weight w = 1 + tail * max(0, t'_0)
//   (the upper tail of the first target counts more): dU = 2 w (u - t') / B;
//   loss += w (u - t')^2 / B.
//   dH2[b][i] = (dU[b] . W3[:, i]) * [H2[b][i] > 0], stored as bf16.
// The block's partial sums of dW3[j][i] = dU[b][j] H2[b][i], of db2[i] =
// dH2[b][i] (as stored), of db3 = dU and of the loss go to part[block].  A
// thread owns two columns and walks the rows eight at a time (their loads
// in flight together); HB_ROWS = 32 gives a batch of 4,096 128 blocks.  It is
// bound by reading H2 and writing dH2 (8 MB at 4,096 rows).
constexpr int HB_ROWS = 32, HB_PART = 3 * DH + 4;   // dW3 [2][512], db2 [512], db3 [2], loss
__global__ void __launch_bounds__(256) head_bwd_kernel(const float *y, int parts, const float *b3,
                                                       const __nv_bfloat16 *W3, const float *T, const float *map,
                                                       const __nv_bfloat16 *H2, __nv_bfloat16 *dH2, float *part, int B) {
    __shared__ float2 du[HB_ROWS];
    const int r0 = blockIdx.x * HB_ROWS, rows = min(HB_ROWS, B - r0);
    part += (size_t)blockIdx.x * HB_PART;
    pdl_trigger();
    pdl_wait();
    const int c = 2 * (int)threadIdx.x;
    __nv_bfloat162 h[8];   // the first rows, in flight while dU is computed
    auto fetch = [&](int r) {
#pragma unroll
        for (int k = 0; k < 8; ++k)
            h[k] = r + k < rows ? *reinterpret_cast<const __nv_bfloat162 *>(H2 + (size_t)(r0 + r + k) * DH + c)
                                : __floats2bfloat162_rn(0.f, 0.f);
    };
    fetch(0);
    if (threadIdx.x < HB_ROWS) {   // one warp: a row a lane
        const int b = r0 + (int)threadIdx.x;
        float g0 = 0.f, g1 = 0.f, l = 0.f;
        if ((int)threadIdx.x < rows) {
            float u0 = 0.f, u1 = 0.f;
            for (int p = 0; p < parts; ++p) {
                const float2 q = reinterpret_cast<const float2 *>(y)[(size_t)p * B + b];
                u0 += q.x, u1 += q.y;
            }
            if (b3) u0 += b3[0], u1 += b3[1];
            const float t0 = (T[2 * (size_t)b] - map[0]) / map[2], t1 = (T[2 * (size_t)b + 1] - map[1]) / map[3];
            const float w = 1.f + map[4] * fmaxf(t0, 0.f);
            const float d0 = u0 - t0, d1 = u1 - t1;
            g0 = 2.f * w * d0 / (float)B;
            g1 = 2.f * w * d1 / (float)B;
            l = w * (d0 * d0 + d1 * d1) / (float)B;
        }
        du[threadIdx.x] = make_float2(g0, g1);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            g0 += __shfl_xor_sync(0xFFFFFFFFu, g0, o);
            g1 += __shfl_xor_sync(0xFFFFFFFFu, g1, o);
            l += __shfl_xor_sync(0xFFFFFFFFu, l, o);
        }
        if (threadIdx.x == 0) part[3 * DH] = g0, part[3 * DH + 1] = g1, part[3 * DH + 2] = l;
    }
    __syncthreads();
    const __nv_bfloat162 wa = *reinterpret_cast<const __nv_bfloat162 *>(W3 + c);
    const __nv_bfloat162 wb = *reinterpret_cast<const __nv_bfloat162 *>(W3 + DH + c);
    const float wa0 = __low2float(wa), wa1 = __high2float(wa), wb0 = __low2float(wb), wb1 = __high2float(wb);
    float s00 = 0.f, s01 = 0.f, s10 = 0.f, s11 = 0.f, e0 = 0.f, e1 = 0.f;
#pragma unroll 1
    for (int r = 0; r < rows; r += 8) {
        __nv_bfloat162 now[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) now[k] = h[k];
        if (r + 8 < rows) fetch(r + 8);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if (r + k >= rows) break;
            const float2 d = du[r + k];
            const float h0 = __low2float(now[k]), h1 = __high2float(now[k]);
            s00 += d.x * h0, s01 += d.x * h1;
            s10 += d.y * h0, s11 += d.y * h1;
            const float v0 = h0 > 0.f ? d.x * wa0 + d.y * wb0 : 0.f, v1 = h1 > 0.f ? d.x * wa1 + d.y * wb1 : 0.f;
            const __nv_bfloat162 o = __floats2bfloat162_rn(v0, v1);
            *reinterpret_cast<__nv_bfloat162 *>(dH2 + (size_t)(r0 + r + k) * DH + c) = o;
            e0 += __low2float(o), e1 += __high2float(o);
        }
    }
    *reinterpret_cast<float2 *>(part + c) = make_float2(s00, s01);
    *reinterpret_cast<float2 *>(part + DH + c) = make_float2(s10, s11);
    *reinterpret_cast<float2 *>(part + 2 * DH + c) = make_float2(e0, e1);
}

// Target map from a target set: column means, column standard deviations
// (population; 1 where below 1e-6), the tail weight.  One block, float64 sums.
__global__ void fit_map_kernel(const float *T, int B, float tail, float *map) {
    __shared__ double red[2][1024];
    double s0 = 0, s1 = 0;
    for (int b = threadIdx.x; b < B; b += blockDim.x) s0 += T[2 * b], s1 += T[2 * b + 1];
    red[0][threadIdx.x] = s0, red[1][threadIdx.x] = s1;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) red[0][threadIdx.x] += red[0][threadIdx.x + o], red[1][threadIdx.x] += red[1][threadIdx.x + o];
        __syncthreads();
    }
    const double m0 = red[0][0] / B, m1 = red[1][0] / B;
    __syncthreads();
    double v0 = 0, v1 = 0;
    for (int b = threadIdx.x; b < B; b += blockDim.x) {
        const double d0 = T[2 * b] - m0, d1 = T[2 * b + 1] - m1;
        v0 += d0 * d0, v1 += d1 * d1;
    }
    red[0][threadIdx.x] = v0, red[1][threadIdx.x] = v1;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) red[0][threadIdx.x] += red[0][threadIdx.x + o], red[1][threadIdx.x] += red[1][threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const double sd0 = sqrt(red[0][0] / B), sd1 = sqrt(red[1][0] / B);
        map[0] = (float)m0, map[1] = (float)m1;
        map[2] = sd0 < 1e-6 ? 1.f : (float)sd0;
        map[3] = sd1 < 1e-6 ? 1.f : (float)sd1;
        map[4] = tail;
    }
}

// Column sums of each 128-row tile of dH (the mma.sync engine's db1; tcgen05's epilogue adds its own).
__global__ void __launch_bounds__(256) colsum_kernel(const __nv_bfloat16 *dH, float *out, int B) {
    const int c = 2 * (int)threadIdx.x, r1 = min(((int)blockIdx.x + 1) * 128, B);
    float s0 = 0.f, s1 = 0.f;
#pragma unroll 8
    for (int r = blockIdx.x * 128; r < r1; ++r) {
        const __nv_bfloat162 v = *reinterpret_cast<const __nv_bfloat162 *>(dH + (size_t)r * DH + c);
        s0 += __low2float(v), s1 += __high2float(v);
    }
    *reinterpret_cast<float2 *>(out + (size_t)blockIdx.x * DH + c) = make_float2(s0, s1);
}

// The partial sums of a batch's gradients.
struct GradParts {
    const float *w1, *w2;   // [splits][512][512]
    const float *b1;        // [b1_n][512]: column sums of dH1 by 128-row tile
    const float *head;      // [head_n][HB_PART]
    int splits, b1_n, head_n;
};

struct AdamArgs {
    float *w, *m, *v;
    __nv_bfloat16 *wb;
    float lr, b1, b2, eps, c1, c2;
};

__device__ __forceinline__ float adam_update(const AdamArgs &a, float g, float &m, float &v, float w) {
    m = a.b1 * m + (1.f - a.b1) * g;
    v = a.b2 * v + (1.f - a.b2) * g * g;
    return w - a.lr * (m / a.c1) / (sqrtf(v / a.c2) + a.eps);
}

// Sums the gradients' parts, stores the gradients and the loss and, with ADAM,
// updates the FP32 master weights and their BF16 copies.  The first UP_BIG
// blocks own W1 and W2, four weights a thread; the others own 32 of the
// remaining 2,051 sums each, eight threads a sum (those have up to one part
// per HB_ROWS rows).  Bound by memory: 16 MB of moments, weights and gradients
// plus a megabyte a split and matrix, most of it in L2.
constexpr int UP_BIG = 2 * DH * DH / 4 / 256, UP_SMALL = (4 * DH + 3 + 31) / 32;
template <bool ADAM>
__global__ void __launch_bounds__(256) update_kernel(GradParts p, float *g, float *loss, AdamArgs a) {
    pdl_trigger();
    pdl_wait();
    if (blockIdx.x < UP_BIG) {
        const int e = (int)(blockIdx.x * 256 + threadIdx.x), half = DH * DH / 4;
        const bool second = e >= half;
        const size_t k = second ? e - half : e;   // float4 within the matrix
        const float4 *src = reinterpret_cast<const float4 *>(second ? p.w2 : p.w1) + k;
        const size_t at = (second ? (size_t)(DH * DH + DH) : 0) + 4 * k;   // its place among the parameters
        float4 s = src[0];
        for (int q = 1; q < p.splits; ++q) {
            const float4 x = src[(size_t)q * half];
            s.x += x.x, s.y += x.y, s.z += x.z, s.w += x.w;
        }
        *reinterpret_cast<float4 *>(g + at) = s;
        if constexpr (ADAM) {
            float4 w = *reinterpret_cast<const float4 *>(a.w + at), m = *reinterpret_cast<const float4 *>(a.m + at),
                   v = *reinterpret_cast<const float4 *>(a.v + at);
            w.x = adam_update(a, s.x, m.x, v.x, w.x);
            w.y = adam_update(a, s.y, m.y, v.y, w.y);
            w.z = adam_update(a, s.z, m.z, v.z, w.z);
            w.w = adam_update(a, s.w, m.w, v.w, w.w);
            *reinterpret_cast<float4 *>(a.w + at) = w;
            *reinterpret_cast<float4 *>(a.m + at) = m;
            *reinterpret_cast<float4 *>(a.v + at) = v;
            const __nv_bfloat162 lo = __floats2bfloat162_rn(w.x, w.y), hi = __floats2bfloat162_rn(w.z, w.w);
            *reinterpret_cast<uint2 *>(a.wb + at) =
                make_uint2(*reinterpret_cast<const uint32_t *>(&lo), *reinterpret_cast<const uint32_t *>(&hi));
        }
        return;
    }
    // b1 [512], b2 [512], W3 [1024], b3 [2], the loss
    __shared__ float red[8][33];
    const int lane = threadIdx.x & 31, sub = threadIdx.x >> 5, e = (int)(blockIdx.x - UP_BIG) * 32 + lane;
    const float *src = nullptr;
    size_t stride = HB_PART, at = 0;
    int n = p.head_n;
    if (e < DH) src = p.b1 + e, stride = DH, n = p.b1_n, at = (size_t)DH * DH + e;
    else if (e < 2 * DH) src = p.head + DH + e, at = 2 * (size_t)DH * DH + e;               // db2 at 2 * 512 of a part
    else if (e < 4 * DH) src = p.head + (e - 2 * DH), at = 2 * (size_t)DH * DH + e;         // dW3
    else if (e < 4 * DH + 3) src = p.head + (e - DH), at = 2 * (size_t)DH * DH + e;         // db3, loss
    float s = 0.f;
    if (src)
        for (int q = sub; q < n; q += 8) s += src[(size_t)q * stride];
    red[sub][lane] = s;
    __syncthreads();
    if (sub != 0 || !src) return;
#pragma unroll
    for (int q = 1; q < 8; ++q) s += red[q][lane];
    if (e == 4 * DH + 2) {
        if (loss) *loss = s;
        return;
    }
    g[at] = s;
    if constexpr (ADAM) {
        float m = a.m[at], v = a.v[at];
        const float w = adam_update(a, s, m, v, a.w[at]);
        a.w[at] = w, a.m[at] = m, a.v[at] = v;
        a.wb[at] = __float2bfloat16_rn(w);
    }
}

__global__ void to_bf16_kernel(const float *src, __nv_bfloat16 *dst, size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        dst[i] = __float2bfloat16_rn(src[i]);
}

// accuracy = (TP + TN) / (|P| + |N|), F1 = 2TP / (2TP + FP + FN) (0 if the denominator is 0)
// Statistics table entries from exact scores: round((accuracy - 1/2) * 32), in double.
__global__ void stat_kernel(const float *scores, uint32_t n, int32_t *out) {
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        out[i] = (int32_t)rint(((double)scores[2 * i] - 0.5) * 32.0);
}

// a / b in double, rounded to float.  Below 2^24 both are exact floats, and the
// FP32 quotient is the same value: a quotient of 24-bit integers is either a
// float, or further from every midpoint of two floats than double's rounding
// moves it.  (FP64 divides run at a small fraction of the FP32 rate here.)
__device__ __forceinline__ float ratio(uint64_t a, uint64_t b) {
    if (b < (1u << 24) && a < (1u << 24)) return __fdiv_rn((float)(uint32_t)a, (float)(uint32_t)b);
    return (float)((double)a / (double)b);
}

__global__ void scores_kernel(const uint32_t *counts, uint32_t H, float *T) {
    for (uint32_t h = blockIdx.x * blockDim.x + threadIdx.x; h < H; h += gridDim.x * blockDim.x) {
        const uint4 c = reinterpret_cast<const uint4 *>(counts)[h];
        const uint64_t tot = (uint64_t)c.x + c.y + c.z + c.w, den = 2ull * c.x + c.y + c.z;
        T[2ull * h] = tot > 0 ? ratio((uint64_t)c.x + c.w, tot) : 0.f;
        T[2ull * h + 1] = den > 0 ? ratio(2ull * c.x, den) : 0.f;
    }
}

// ------------------------------------------------------------------ top-k
// Key of a prediction for "larger is better" with ties broken by F1 then by
// smaller index: (accuracy bits, F1 bits) mapped to order-preserving uint32.
__device__ __forceinline__ uint32_t order_key(float x) {
    uint32_t u = __float_as_uint(x);
    if (x != x) return 0u;                      // NaN ranks last
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// The k best of H predictions by a radix select over 64-bit keys (accuracy key
// << 32 | F1 key), in one launch of one cluster of SEL_CTAS blocks; ties go to
// the lowest indices, and the indices come out ascending.
//
// Block r owns a contiguous range of the predictions and walks it in tiles of
// SEL_TILE keys in shared memory; up to SEL_CTAS * SEL_TILE predictions (a
// ranking round's 65,536) a block's range is one tile, read from memory once.
//   1. The bits in which any key differs from the first one: leading bits that
//      all share (sign, most of the exponent) need no pass.
//   2. Up to 10 bits a pass: each block counts its keys that match the bits
//      chosen so far, the cluster adds the counts through distributed shared
//      memory, and every block picks the digit of the k-th largest key by a
//      scan over the 1,024 bins.  A pass ends the search once every key of the
//      chosen bin is wanted.
//   3. Each block's picks are counted, their offsets follow from the blocks
//      before it, and a scan over the tile places them in index order.
// The cluster's barrier replaces a launch: the eight passes of 8 bits had been
// 16 launches whose digit was picked by one thread (11 us each), and the
// compaction one block's walk over all keys (71 us): 171 us at 65,536
// predictions with the scores, 30 us now, most of it two launches and a few
// microseconds a pass.
constexpr uint32_t SEL_CTAS = 8, SEL_THREADS = 1024, SEL_PER = 8, SEL_TILE = SEL_THREADS * SEL_PER;
constexpr uint32_t SEL_BITS = 10, SEL_BINS = 1u << SEL_BITS, SEL_COPIES = 4;
struct SelSmem {
    unsigned long long key[SEL_TILE + SEL_TILE / SEL_PER];   // key i at i + i / SEL_PER: no 8-way bank conflicts
    uint32_t hist[SEL_COPIES][SEL_BINS];                     // the block's counts, a copy per few warps
    uint32_t sum[2][SEL_BINS];                               // ... added up, read by the cluster (two passes apart)
    uint32_t warp_sum[32];
    unsigned long long diff;                                 // bits in which some key differs from the first
    uint32_t n_gt, n_eq;                                     // the block's picks
    uint32_t digit, left, in_bin;
};
static_assert(SEL_BINS == SEL_THREADS, "a thread owns a bin");

__device__ __forceinline__ uint32_t cluster_peer(const void *p, uint32_t rank) {
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return a;
}
__device__ __forceinline__ uint32_t ld_peer(const uint32_t *p, uint32_t rank) {
    uint32_t v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(cluster_peer(p, rank)) : "memory");
    return v;
}
__device__ __forceinline__ unsigned long long ld_peer(const unsigned long long *p, uint32_t rank) {
    unsigned long long v;
    asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(cluster_peer(p, rank)) : "memory");
    return v;
}
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Exclusive prefix sum of v over the block's threads; *total receives the sum.
__device__ __forceinline__ uint32_t block_scan(uint32_t v, uint32_t *warp_sum, uint32_t *total) {
    const uint32_t lane = threadIdx.x & 31u, w = threadIdx.x >> 5;
    uint32_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= (uint32_t)o) incl += t;
    }
    __syncthreads();   // warp_sum may still be read from the scan before
    if (lane == 31) warp_sum[w] = incl;
    __syncthreads();
    uint32_t x = warp_sum[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= (uint32_t)o) x += t;
    }
    *total = __shfl_sync(0xFFFFFFFFu, x, 31);
    const uint32_t before = w ? __shfl_sync(0xFFFFFFFFu, x, (int)(w - 1)) : 0u;
    return before + incl - v;
}

__global__ void __cluster_dims__(SEL_CTAS, 1, 1) __launch_bounds__(SEL_THREADS)
    select_kernel(const float *__restrict__ Y, uint32_t H, uint32_t k, uint32_t *out) {
    extern __shared__ __align__(16) uint8_t sel_raw[];
    SelSmem &sm = *reinterpret_cast<SelSmem *>(sel_raw);
    const uint32_t tid = threadIdx.x, rank = blockIdx.x;   // one cluster: the block's rank in it
    // the block's range, in whole tiles where there are several
    uint64_t per = ((uint64_t)H + SEL_CTAS - 1) / SEL_CTAS;
    if (per > SEL_TILE) per = (per + SEL_TILE - 1) / SEL_TILE * SEL_TILE;
    const uint64_t lo = min((uint64_t)H, rank * per), hi = min((uint64_t)H, lo + per);
    const bool one_tile = per <= SEL_TILE;
    auto make_key = [&](uint64_t i) {
        return ((unsigned long long)order_key(Y[2 * i]) << 32) | order_key(Y[2 * i + 1]);
    };
    auto slot = [](uint32_t i) { return i + i / SEL_PER; };
    // the tile's keys, coalesced; the barrier before it protects the tile read before
    auto load_tile = [&](uint64_t t0) {
        const uint32_t n = (uint32_t)min((uint64_t)SEL_TILE, hi - t0);
        __syncthreads();
        if (n == SEL_TILE) {   // all loads in flight together
            unsigned long long x[SEL_PER];
#pragma unroll
            for (uint32_t q = 0; q < SEL_PER; ++q) x[q] = make_key(t0 + tid + q * SEL_THREADS);
#pragma unroll
            for (uint32_t q = 0; q < SEL_PER; ++q) sm.key[slot(tid + q * SEL_THREADS)] = x[q];
        } else {
            for (uint32_t i = tid; i < n; i += SEL_THREADS) sm.key[slot(i)] = make_key(t0 + i);
        }
        __syncthreads();
        return n;
    };
    const unsigned long long key0 = make_key(0);
    if (tid == 0) sm.diff = 0ull, sm.n_gt = sm.n_eq = 0u;
    for (uint32_t i = tid; i < SEL_COPIES * SEL_BINS; i += SEL_THREADS) (&sm.hist[0][0])[i] = 0u;

    unsigned long long diff = 0ull;
    for (uint64_t t0 = lo; t0 < hi; t0 += SEL_TILE) {
        const uint32_t n = load_tile(t0);
        for (uint32_t i = tid; i < n; i += SEL_THREADS) diff |= sm.key[slot(i)] ^ key0;
    }
    __syncthreads();
    const uint32_t dh = __reduce_or_sync(0xFFFFFFFFu, (uint32_t)(diff >> 32));
    const uint32_t dl = __reduce_or_sync(0xFFFFFFFFu, (uint32_t)diff);
    if ((tid & 31u) == 0) atomicOr(&sm.diff, ((unsigned long long)dh << 32) | dl);
    cluster_barrier();
    diff = 0ull;
    for (uint32_t r = 0; r < SEL_CTAS; ++r) diff |= ld_peer(&sm.diff, r);
    uint32_t rb = diff ? 64u - (uint32_t)__clzll((long long)diff) : 0u;   // low bits still open
    unsigned long long prefix = rb >= 64u ? 0ull : (key0 >> rb) << rb;
    uint32_t left = k;       // wanted among the keys that match the prefix
    bool whole = false;      // all of them are wanted
    for (uint32_t pass = 0; rb > 0u && !whole; ++pass) {
        const uint32_t w = min(SEL_BITS, rb), shift = rb - w, mask = (1u << w) - 1u;
        uint32_t *mine = sm.hist[(tid >> 5) % SEL_COPIES];
        for (uint64_t t0 = lo; t0 < hi; t0 += SEL_TILE) {
            const uint32_t n = one_tile ? (uint32_t)(hi - lo) : load_tile(t0);
            for (uint32_t i = tid; i < n; i += SEL_THREADS) {
                const unsigned long long x = sm.key[slot(i)];
                if (rb >= 64u || (x >> rb) == (prefix >> rb)) atomicAdd(&mine[(uint32_t)(x >> shift) & mask], 1u);
            }
        }
        __syncthreads();
        uint32_t own = 0;
#pragma unroll
        for (uint32_t c = 0; c < SEL_COPIES; ++c) {
            own += sm.hist[c][tid];
            sm.hist[c][tid] = 0u;
        }
        sm.sum[pass & 1u][tid] = own;
        cluster_barrier();
        // thread t owns bin SEL_BINS - 1 - t, so that a prefix sum counts the larger keys
        const uint32_t bin = SEL_BINS - 1u - tid;
        uint32_t cnt = 0;
#pragma unroll
        for (uint32_t r = 0; r < SEL_CTAS; ++r) cnt += ld_peer(&sm.sum[pass & 1u][bin], r);
        uint32_t total;
        const uint32_t larger = block_scan(cnt, sm.warp_sum, &total);
        if (larger < left && left <= larger + cnt) sm.digit = bin, sm.left = left - larger, sm.in_bin = cnt;
        __syncthreads();
        prefix |= (unsigned long long)sm.digit << shift;
        left = sm.left;
        whole = left == sm.in_bin;
        rb = shift;
        __syncthreads();
    }
    // picks: keys above the prefix's range and, of those inside, all (whole) or the first `left`
    const unsigned long long span = rb >= 64u ? ~0ull : (1ull << rb) - 1ull;
    auto above = [&](unsigned long long x) { return whole ? x >= prefix : x > (prefix | span); };
    auto inside = [&](unsigned long long x) { return !whole && x >= prefix && x <= (prefix | span); };
    uint32_t gt = 0, eq = 0;
    for (uint64_t t0 = lo; t0 < hi; t0 += SEL_TILE) {
        const uint32_t n = one_tile ? (uint32_t)(hi - lo) : load_tile(t0);
        for (uint32_t i = tid; i < n; i += SEL_THREADS) {
            const unsigned long long x = sm.key[slot(i)];
            gt += above(x), eq += inside(x);
        }
    }
    gt = __reduce_add_sync(0xFFFFFFFFu, gt), eq = __reduce_add_sync(0xFFFFFFFFu, eq);
    if ((tid & 31u) == 0 && (gt | eq)) atomicAdd(&sm.n_gt, gt), atomicAdd(&sm.n_eq, eq);
    cluster_barrier();
    uint32_t gt_before = 0, eq_before = 0;
    for (uint32_t r = 0; r < rank; ++r) gt_before += ld_peer(&sm.n_gt, r), eq_before += ld_peer(&sm.n_eq, r);
    // a picked key's place: the larger keys before it + the equal ones before it that are taken
    for (uint64_t t0 = lo; t0 < hi; t0 += SEL_TILE) {
        const uint32_t n = one_tile ? (uint32_t)(hi - lo) : load_tile(t0);
        uint32_t g = 0, e = 0;
#pragma unroll
        for (uint32_t q = 0; q < SEL_PER; ++q) {
            const uint32_t i = tid * SEL_PER + q;
            if (i < n) {
                const unsigned long long x = sm.key[slot(i)];
                g += above(x), e += inside(x);
            }
        }
        uint32_t total;
        const uint32_t before = block_scan(g | e << 16, sm.warp_sum, &total);   // at most 8,192 each
        uint32_t pg = gt_before + (before & 0xFFFFu), pe = eq_before + (before >> 16);
#pragma unroll
        for (uint32_t q = 0; q < SEL_PER; ++q) {
            const uint32_t i = tid * SEL_PER + q;
            if (i >= n) break;
            const unsigned long long x = sm.key[slot(i)];
            if (above(x)) out[pg++ + min(pe, left)] = (uint32_t)(t0 + i);
            else if (inside(x)) {
                if (pe < left) out[pg + pe] = (uint32_t)(t0 + i);
                ++pe;
            }
        }
        gt_before += total & 0xFFFFu, eq_before += total >> 16;
    }
    cluster_barrier();   // no block leaves while another may still read its counts
}

}  // namespace
}  // namespace hedl

using namespace hedl;

struct hedl_mlp {
    // FP32 master weights, Adam moments, gradients; BF16 copies for compute;
    // the target map (mean0, mean1, scale0, scale1, tail weight)
    float *w = nullptr, *m = nullptr, *v = nullptr, *g = nullptr, *map = nullptr;
    uint32_t *err = nullptr;                  // device: bit 0 = a tensor-core wait timed out
    hedl::UmmaDevice dev;                     // the device that all of these live on
    unsigned gemm = HEDL_GEMM_TCGEN05;        // engine of the dense layers' forward GEMMs
    __nv_bfloat16 *wb = nullptr;
    size_t n = 0;
    uint32_t step = 0;
};

namespace {

constexpr size_t OFF_W1 = 0, OFF_B1 = OFF_W1 + (size_t)DH * DI, OFF_W2 = OFF_B1 + DH, OFF_B2 = OFF_W2 + (size_t)DH * DH,
                 OFF_W3 = OFF_B2 + DH, OFF_B3 = OFF_W3 + (size_t)DO * DH, N_PARAMS = OFF_B3 + DO;

// K ranges of a weight gradient: 4 give the two 512 x 512 gradients 128 items
// of 128 x 128; a batch below 193 rows has fewer blocks of 64 to split.
int grad_splits(uint32_t B) { return (int)std::min<uint32_t>(4, (B + 63) / 64); }

struct MlpWs {
    __nv_bfloat16 *h1, *h2, *dh1, *dh2;
    float *y;             // [UMMA_MAX_HEAD_TILES][B][2]
    __nv_bfloat16 *x;     // a 16-byte aligned copy of the inputs, if they are not
    float *head, *b1;     // GradParts
    float *w1, *w2;
};

// Lays the workspace out from `ws` (null: only measures it); *end receives its size.
MlpWs carve(void *ws, uint32_t B, size_t *end = nullptr) {
    size_t at = 0;
    uint8_t *base = (uint8_t *)(((uintptr_t)ws + 255) & ~(uintptr_t)255);   // mlp_ws_bytes leaves room for it
    auto take = [&](size_t bytes) {
        uint8_t *r = base + at;
        at += (bytes + 255) & ~size_t(255);
        return r;
    };
    MlpWs w;
    w.h1 = (__nv_bfloat16 *)take((size_t)B * DH * 2);
    w.h2 = (__nv_bfloat16 *)take((size_t)B * DH * 2);
    w.dh1 = (__nv_bfloat16 *)take((size_t)B * DH * 2);
    w.dh2 = (__nv_bfloat16 *)take((size_t)B * DH * 2);
    w.y = (float *)take((size_t)UMMA_MAX_HEAD_TILES * B * DO * 4);
    w.x = (__nv_bfloat16 *)take((size_t)B * DI * 2);
    w.head = (float *)take(((size_t)B + HB_ROWS - 1) / HB_ROWS * HB_PART * 4);
    w.b1 = (float *)take(((size_t)B + 127) / 128 * DH * 4);
    w.w1 = (float *)take((size_t)grad_splits(B) * DH * DI * 4);
    w.w2 = (float *)take((size_t)grad_splits(B) * DH * DH * 4);
    if (end) *end = at;
    return w;
}

size_t mlp_ws_bytes(uint32_t B) {
    size_t n = 0;
    carve(nullptr, B, &n);
    return n + 256;
}

uint32_t grid1(size_t n) { return (uint32_t)std::min<size_t>((n + 255) / 256, 4096); }

// One hidden layer, H = relu(A . W^T + b), on the mma.sync engine.
int dense_relu(const __nv_bfloat16 *A, const __nv_bfloat16 *W, const float *b, __nv_bfloat16 *H, int M, int K,
               cudaStream_t s) {
    GemmArgs a{};
    a.A = A;
    a.B = W;
    a.C = H;
    a.bias = b;
    a.M = M, a.N = DH, a.K = K, a.lda = K, a.ldb = K, a.ldc = DH;
    a.relu = 1, a.out_bf16 = 1;
    return gemm(a, false, false, 1, s);
}

// Both hidden layers and the output layer's sums into w.y, whose parts come
// back in *parts (0: w.y already holds u with b3).  need_h2 = false
// (inference) leaves the second layer's activations unwritten.
int forward_impl(hedl_mlp *mlp, const __nv_bfloat16 *X, uint32_t B, const MlpWs &w, cudaStream_t s, bool need_h2,
                 int *parts) {
    int e;
    if (mlp->gemm == HEDL_GEMM_TCGEN05) {
        UmmaArgs u{X, mlp->wb + OFF_W1, w.h1, mlp->w + OFF_B1, (int)B, DH, DI, DI, DI, DH, 1, 1, mlp->err, nullptr};
        e = umma_gemm(&u, 1, mlp->dev, s);
        if (e) return e;
        UmmaArgs v{w.h1, mlp->wb + OFF_W2, w.h2, mlp->w + OFF_B2, (int)B, DH, DH, DH, DH, DH, 1, 1, mlp->err, nullptr};
        v.w3 = mlp->wb + OFF_W3;
        v.y = w.y;
        v.store = need_h2;
        *parts = DH / umma_tile_n(&v, 1, mlp->dev);
        return umma_gemm(&v, 1, mlp->dev, s);
    }
    e = dense_relu(X, mlp->wb + OFF_W1, mlp->w + OFF_B1, w.h1, (int)B, DI, s);
    if (!e) e = dense_relu(w.h1, mlp->wb + OFF_W2, mlp->w + OFF_B2, w.h2, (int)B, DH, s);
    if (e) return e;
    out_fwd_kernel<<<std::min<uint32_t>((B * 32 + 255) / 256, 148u * 8u), 256, 0, s>>>(
        w.h2, mlp->wb + OFF_W3, mlp->w + OFF_B3, w.y, (int)B, nullptr);
    *parts = 0;
    return cudaGetLastError();
}

// TMA and the 16-byte loads need aligned rows: inputs that are not are copied once.
int aligned_input(const __nv_bfloat16 *&X, uint32_t B, const MlpWs &w, cudaStream_t s) {
    if (((uintptr_t)X & 15) == 0) return 0;
    cudaError_t e = cudaMemcpyAsync(w.x, X, (size_t)B * DI * 2, cudaMemcpyDeviceToDevice, s);
    X = w.x;
    return e;
}

// The batch's gradient parts, up to (not including) update_kernel.
int grads_impl(hedl_mlp *mlp, const __nv_bfloat16 *X, const float *T, uint32_t B, const MlpWs &w, cudaStream_t s,
               GradParts *out) {
    if (B == 0) return cudaErrorInvalidConfiguration;
    int parts = 0, e = aligned_input(X, B, w, s);
    if (!e) e = forward_impl(mlp, X, B, w, s, true, &parts);
    if (e) return e;
    const int M = (int)B, splits = grad_splits(B);
    *out = GradParts{w.w1, w.w2, w.b1, w.head, splits, (M + 127) / 128, (M + HB_ROWS - 1) / HB_ROWS};
    e = launch_pdl(head_bwd_kernel, out->head_n, 256, 0, s, w.y, parts ? parts : 1, parts ? mlp->w + OFF_B3 : nullptr,
                   mlp->wb + OFF_W3, T, mlp->map, w.h2, w.dh2, w.head, M);
    if (e) return e;
    if (mlp->gemm == HEDL_GEMM_TCGEN05) {
        // dH1 = (dH2 . W2) * [H1 > 0]; W2 [out][in] is the MN-major operand
        UmmaArgs d{w.dh2, mlp->wb + OFF_W2, w.dh1, nullptr, M, DH, DH, DH, DH, DH, 0, 1, mlp->err, w.h1};
        d.b_mn = 1;
        d.colsum = w.b1;
        e = umma_gemm(&d, 1, mlp->dev, s);
        if (e) return e;
        // dW1 = dH1^T . X and dW2 = dH2^T . H1: contractions over the batch, both operands MN-major
        UmmaArgs g[2] = {{w.dh1, X, w.w1, nullptr, DH, DI, M, DH, DI, DI, 0, 0, mlp->err, nullptr},
                         {w.dh2, w.h1, w.w2, nullptr, DH, DH, M, DH, DH, DH, 0, 0, mlp->err, nullptr}};
        for (UmmaArgs &a : g) a.a_mn = a.b_mn = 1, a.splits = splits, a.c_split = (size_t)DH * DH;
        return umma_gemm(g, 2, mlp->dev, s);
    }
    out->splits = 1;   // the atomics add every K range into the first part
    e = cudaMemsetAsync(w.w1, 0, (size_t)DH * DI * 4, s);
    if (!e) e = cudaMemsetAsync(w.w2, 0, (size_t)DH * DH * 4, s);
    if (e) return e;
    const int k_splits = std::max(1, std::min((int)(B / 256), 64));
    // dW2 = dH2^T H1   (M = out, N = in, K = batch): A stored [K][M], B stored [K][N]
    GemmArgs a{};
    a.A = w.dh2;
    a.B = w.h1;
    a.C = w.w2;
    a.M = DH, a.N = DH, a.K = M, a.lda = DH, a.ldb = DH, a.ldc = DH;
    a.atomic = 1;
    e = gemm(a, true, true, k_splits, s);
    if (e) return e;
    // dH1 = (dH2 W2) * [H1 > 0]   (M = batch, N = in, K = out): A [M][K], B stored [K][N]
    GemmArgs d{};
    d.A = w.dh2;
    d.B = mlp->wb + OFF_W2;
    d.C = w.dh1;
    d.mask = w.h1;
    d.M = M, d.N = DH, d.K = DH, d.lda = DH, d.ldb = DH, d.ldc = DH;
    d.out_bf16 = 1;
    e = gemm(d, false, true, 1, s);
    if (e) return e;
    colsum_kernel<<<out->b1_n, 256, 0, s>>>(w.dh1, w.b1, M);
    // dW1 = dH1^T X
    a.A = w.dh1;
    a.B = X;
    a.C = w.w1;
    a.N = DI, a.ldb = DI;
    return gemm(a, true, true, k_splits, s);
}

}  // namespace

extern "C" {

int hedl_mlp_create(const float *params, hedl_mlp **out) {
    if (!out || !params) return fail(HEDL_ERR_INVALID_ARG, "NULL argument");
    *out = nullptr;
    auto *m = new hedl_mlp();
    m->n = N_PARAMS;
    cudaError_t e = (cudaError_t)umma_device(&m->dev);
    if (!e) e = cudaMalloc(&m->w, N_PARAMS * 4);
    if (!e) e = cudaMalloc(&m->m, N_PARAMS * 4);
    if (!e) e = cudaMalloc(&m->v, N_PARAMS * 4);
    if (!e) e = cudaMalloc(&m->g, N_PARAMS * 4);
    if (!e) e = cudaMalloc(&m->wb, N_PARAMS * 2);
    if (!e) e = cudaMalloc(&m->map, 7 * 4);
    if (!e) e = cudaMalloc(&m->err, 4);
    if (!e) e = cudaMemset(m->err, 0, 4);
    if (!e) {
        const float ident[7] = {0.f, 0.f, 1.f, 1.f, 0.f, 0.f, 0.f};   // and two zeros behind it
        e = cudaMemcpy(m->map, ident, sizeof(ident), cudaMemcpyHostToDevice);
    }
    if (!e) e = cudaMemcpy(m->w, params, N_PARAMS * 4, cudaMemcpyHostToDevice);
    if (!e) e = cudaMemset(m->m, 0, N_PARAMS * 4);
    if (!e) e = cudaMemset(m->v, 0, N_PARAMS * 4);
    if (!e) {
        to_bf16_kernel<<<grid1(N_PARAMS), 256>>>(m->w, m->wb, N_PARAMS);
        e = cudaDeviceSynchronize();
    }
    if (e) {
        int rc = cuda_fail(e, "hedl_mlp_create");
        hedl_mlp_free(m);
        return rc;
    }
    *out = m;
    return HEDL_OK;
}

void hedl_mlp_free(hedl_mlp *m) {
    if (!m) return;
    cudaDeviceSynchronize();
    cudaFree(m->w);
    cudaFree(m->m);
    cudaFree(m->v);
    cudaFree(m->g);
    cudaFree(m->wb);
    cudaFree(m->map);
    cudaFree(m->err);
    delete m;
}

uint64_t hedl_mlp_param_count(void) { return N_PARAMS; }

int hedl_mlp_get(const hedl_mlp *m, float *params, float *grads, uint32_t *step) {
    if (!m) return fail(HEDL_ERR_INVALID_ARG, "NULL argument");
    cudaError_t e = cudaDeviceSynchronize();
    if (!e && params) e = cudaMemcpy(params, m->w, N_PARAMS * 4, cudaMemcpyDeviceToHost);
    if (!e && grads) e = cudaMemcpy(grads, m->g, N_PARAMS * 4, cudaMemcpyDeviceToHost);
    if (e) return cuda_fail(e, "hedl_mlp_get");
    if (step) *step = m->step;
    return HEDL_OK;
}

int hedl_mlp_get_moments(const hedl_mlp *m, float *first, float *second) {
    if (!m) return fail(HEDL_ERR_INVALID_ARG, "NULL argument");
    cudaError_t e = cudaDeviceSynchronize();
    if (!e && first) e = cudaMemcpy(first, m->m, N_PARAMS * 4, cudaMemcpyDeviceToHost);
    if (!e && second) e = cudaMemcpy(second, m->v, N_PARAMS * 4, cudaMemcpyDeviceToHost);
    return e ? cuda_fail(e, "hedl_mlp_get_moments") : HEDL_OK;
}

int hedl_mlp_workspace_size(uint32_t B, size_t *bytes) {
    if (!bytes) return fail(HEDL_ERR_INVALID_ARG, "NULL argument");
    *bytes = mlp_ws_bytes(B);
    return HEDL_OK;
}

int hedl_encode(const uint64_t *progs, const uint32_t *offs, uint32_t H, const float *grid, uint32_t n_grid,
                const int32_t *stats, uint32_t n_stat_concepts, const float *prior, uint16_t *X, hedl_stream s) {
    if (!progs || !offs || !X) return fail(HEDL_ERR_INVALID_ARG, "NULL argument");
    if (stats && !grid && n_grid) return fail(HEDL_ERR_INVALID_ARG, "threshold statistics need the grid");
    if (H == 0) return HEDL_OK;
    encode_kernel<<<std::min<uint32_t>((H + ENC_WARPS - 1) / ENC_WARPS, 152u * 8u), 32 * ENC_WARPS, 0, (cudaStream_t)s>>>(
        progs, offs, H, EncTables{grid, stats, grid ? n_grid : 0u, stats ? n_stat_concepts : 0u}, prior,
        (__nv_bfloat16 *)X);
    cudaError_t e = cudaGetLastError();
    return e ? cuda_fail(e, "encode launch") : HEDL_OK;
}

int hedl_mlp_forward(hedl_mlp *m, const uint16_t *X, uint32_t B, float *Y, void *ws, size_t ws_bytes,
                     hedl_stream s) {
    if (!m || !X || !Y) return fail(HEDL_ERR_INVALID_ARG, "NULL argument");
    if (!ws || ws_bytes < mlp_ws_bytes(B)) return fail(HEDL_ERR_WORKSPACE_TOO_SMALL, "MLP workspace too small");
    if (B == 0) return cuda_fail(cudaErrorInvalidConfiguration, "mlp forward");
    MlpWs w = carve(ws, B);
    cudaStream_t st = (cudaStream_t)s;
    const __nv_bfloat16 *x = (const __nv_bfloat16 *)X;
    int parts = 0, e = aligned_input(x, B, w, st);
    if (!e) e = forward_impl(m, x, B, w, st, false, &parts);
    if (e) return cuda_fail(e, "mlp forward");
    const float *zero_b3 = m->map + 5;   // two zeros behind the map: b3 when w.y already has it
    e = launch_pdl(out_map_kernel, std::min<uint32_t>((B + 255) / 256, 152u * 8u), 256, 0, st, w.y, parts ? parts : 1,
                   parts ? m->w + OFF_B3 : zero_b3, Y, (int)B, m->map);
    return e ? cuda_fail(e, "mlp forward") : HEDL_OK;
}

int hedl_mlp_gradients(hedl_mlp *m, const uint16_t *X, const float *T, uint32_t B, float *loss, void *ws,
                       size_t ws_bytes, hedl_stream s) {
    if (!m || !X || !T) return fail(HEDL_ERR_INVALID_ARG, "NULL argument");
    if (!ws || ws_bytes < mlp_ws_bytes(B)) return fail(HEDL_ERR_WORKSPACE_TOO_SMALL, "MLP workspace too small");
    MlpWs w = carve(ws, B);
    GradParts p;
    int e = grads_impl(m, (const __nv_bfloat16 *)X, T, B, w, (cudaStream_t)s, &p);
    if (e) return cuda_fail(e, "mlp gradients");
    e = launch_pdl(update_kernel<false>, UP_BIG + UP_SMALL, 256, 0, (cudaStream_t)s, p, m->g, loss, AdamArgs{});
    return e ? cuda_fail(e, "mlp gradients") : HEDL_OK;
}

int hedl_mlp_train_step(hedl_mlp *m, const uint16_t *X, const float *T, uint32_t B, float lr, float *loss,
                        void *ws, size_t ws_bytes, hedl_stream s) {
    if (!m || !X || !T) return fail(HEDL_ERR_INVALID_ARG, "NULL argument");
    if (!ws || ws_bytes < mlp_ws_bytes(B)) return fail(HEDL_ERR_WORKSPACE_TOO_SMALL, "MLP workspace too small");
    MlpWs w = carve(ws, B);
    GradParts p;
    int e = grads_impl(m, (const __nv_bfloat16 *)X, T, B, w, (cudaStream_t)s, &p);
    if (e) return cuda_fail(e, "mlp gradients");
    m->step += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - powf(b1, (float)m->step), c2 = 1.f - powf(b2, (float)m->step);
    e = launch_pdl(update_kernel<true>, UP_BIG + UP_SMALL, 256, 0, (cudaStream_t)s, p, m->g, loss,
                   AdamArgs{m->w, m->m, m->v, m->wb, lr, b1, b2, 1e-8f, c1, c2});
    return e ? cuda_fail(e, "adam launch") : HEDL_OK;
}

int hedl_mlp_fit_target_map(hedl_mlp *m, const float *T, uint32_t B, float tail_weight, hedl_stream s) {
    if (!m || !T) return fail(HEDL_ERR_INVALID_ARG, "NULL argument");
    if (B == 0) return fail(HEDL_ERR_INVALID_ARG, "empty target set");
    if (!(tail_weight >= 0.f)) return fail(HEDL_ERR_INVALID_ARG, "tail_weight must be >= 0");
    fit_map_kernel<<<1, 1024, 0, (cudaStream_t)s>>>(T, (int)B, tail_weight, m->map);
    cudaError_t e = cudaGetLastError();
    return e ? cuda_fail(e, "fit map launch") : HEDL_OK;
}

int hedl_mlp_set_target_map(hedl_mlp *m, const float *map) {
    if (!m || !map) return fail(HEDL_ERR_INVALID_ARG, "NULL argument");
    if (!(map[2] > 0.f) || !(map[3] > 0.f) || !(map[4] >= 0.f))
        return fail(HEDL_ERR_INVALID_ARG, "scales must be > 0 and the tail weight >= 0");
    cudaError_t e = cudaMemcpy(m->map, map, 5 * 4, cudaMemcpyHostToDevice);
    return e ? cuda_fail(e, "set map") : HEDL_OK;
}

int hedl_mlp_set_gemm(hedl_mlp *m, unsigned engine) {
    if (!m) return fail(HEDL_ERR_INVALID_ARG, "NULL argument");
    if (engine != HEDL_GEMM_TCGEN05 && engine != HEDL_GEMM_MMA_SYNC)
        return fail(HEDL_ERR_INVALID_ARG, "engine must be HEDL_GEMM_TCGEN05 or HEDL_GEMM_MMA_SYNC");
    m->gemm = engine;
    return HEDL_OK;
}

int hedl_mlp_status(hedl_mlp *m, hedl_stream s) {
    if (!m) return fail(HEDL_ERR_INVALID_ARG, "NULL argument");
    cudaError_t e = cudaStreamSynchronize((cudaStream_t)s);
    if (e) return cuda_fail(e, "stream synchronize");
    uint32_t st = 0;
    e = cudaMemcpy(&st, m->err, 4, cudaMemcpyDeviceToHost);
    if (e) return cuda_fail(e, "status read");
    if (st) {
        cudaMemset(m->err, 0, 4);
        return fail(HEDL_ERR_TIMEOUT, "a tensor-core completion wait gave up (timeout)");
    }
    return HEDL_OK;
}

int hedl_mlp_get_target_map(const hedl_mlp *m, float *map) {
    if (!m || !map) return fail(HEDL_ERR_INVALID_ARG, "NULL argument");
    cudaError_t e = cudaMemcpy(map, m->map, 5 * 4, cudaMemcpyDeviceToHost);
    return e ? cuda_fail(e, "get map") : HEDL_OK;
}

int hedl_stat_scores(const float *scores, uint32_t n, int32_t *out, hedl_stream s) {
    if (!scores || !out) return fail(HEDL_ERR_INVALID_ARG, "NULL argument");
    if (n == 0) return HEDL_OK;
    stat_kernel<<<grid1(n), 256, 0, (cudaStream_t)s>>>(scores, n, out);
    cudaError_t e = cudaGetLastError();
    return e ? cuda_fail(e, "stat launch") : HEDL_OK;
}

int hedl_scores_from_counts(const uint32_t *counts, uint32_t H, float *scores, hedl_stream s) {
    if (!counts || !scores) return fail(HEDL_ERR_INVALID_ARG, "NULL argument");
    if (H == 0) return HEDL_OK;
    scores_kernel<<<grid1(H), 256, 0, (cudaStream_t)s>>>(counts, H, scores);
    cudaError_t e = cudaGetLastError();
    return e ? cuda_fail(e, "scores launch") : HEDL_OK;
}

int hedl_select_workspace_size(uint32_t H, size_t *bytes) {
    if (!bytes) return fail(HEDL_ERR_INVALID_ARG, "NULL argument");
    *bytes = 8ull * H + 4096 + 256;
    return HEDL_OK;
}

int hedl_select_top(const float *Y, uint32_t H, uint32_t k, uint32_t *idx, void *ws, size_t ws_bytes,
                    hedl_stream s) {
    if (!Y || !idx) return fail(HEDL_ERR_INVALID_ARG, "NULL argument");
    if (k == 0 || k > H) return fail(HEDL_ERR_INVALID_ARG, "k must be in 1..H");
    if (!ws || ws_bytes < 8ull * H + 4096 + 256) return fail(HEDL_ERR_WORKSPACE_TOO_SMALL, "select workspace too small");
    cudaError_t e = allow_smem(select_kernel, sizeof(SelSmem));
    if (e) return cuda_fail(e, "select setup");
    select_kernel<<<SEL_CTAS, SEL_THREADS, sizeof(SelSmem), (cudaStream_t)s>>>(Y, H, k, idx);
    e = cudaGetLastError();
    return e ? cuda_fail(e, "select launch") : HEDL_OK;
}

}  // extern "C"
