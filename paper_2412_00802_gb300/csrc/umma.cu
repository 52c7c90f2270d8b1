// Dense products of the surrogate on the 5th-generation tensor cores:
// C[M][N] = act(A . B^T + bias), bf16 operands, FP32 accumulation in tensor
// memory (TMEM).  An operand is K-major ([rows][K]) or MN-major ([K][rows],
// which lets a weight gradient contract over the batch without transposing).
//
// A persistent kernel: one CTA per SM walks the items (128 x UN output tile,
// K range) blockIdx.x, blockIdx.x + gridDim.x, ... of one or two products.
// Its ten warps have fixed roles:
//   warp 0 (one thread): the TMA producer.  It loads each 64-wide K block of
//     the item's A (128 x 64) and B (UN x 64) (cp.async.bulk.tensor, 128-byte
//     rows in the 128-byte swizzle; a K-major operand is one box, an MN-major
//     one is a box per 64 rows) into a ring of stages, arming the stage's
//     "full" mbarrier with the byte count;
//   warp 1 (one thread): the MMA issuer.  Per K block it waits for a full
//     stage, issues four tcgen05.mma (M 128, N UN, K 16) into one of two
//     UN-column TMEM accumulators and commits them to the stage's "empty"
//     mbarrier; after an item's last block it commits to the accumulator's
//     "tmem full" mbarrier;
//   warps 2-9: the epilogue.  Each reads its 32-lane quarter and one half of
//     the columns of a finished accumulator with tcgen05.ld, adds the bias,
//     applies ReLU or a mask (the backward pass's ReLU derivative), stores
//     bf16 (through shared memory and TMA) or FP32 rows, adds up the tile's
//     columns or the fused output layer's sums where asked, and arrives on the
//     accumulator's "tmem empty" mbarrier.
// With two accumulators, the epilogue of one item overlaps the loads and
// MMAs of the next.
//
// What bounds a layer of many rows: with no epilogue at all the two layers of
// 65,536 rows take 55 us, with no MMAs either 44 (an SM takes in 48 KB a K block
// at 64 B a clock).  Four epilogue warps that stored from registers made it 96
// us (76 without the stores, 64 without the output layer too): one warp a
// scheduler waits out every latency, and its 16-byte stores touch 32 lines
// each.  Eight warps, the next 32 columns loaded ahead, outputs by TMA, bias
// and output weights (as FP32) from shared memory: 68.8 us; a training step of
// 4,096 rows 61 -> 56 us.
//
// Tile width: a layer of a few thousand rows is bound by the latency of one
// item (8 K blocks through one SM), not by the tensor cores, so the tile is
// the widest of 256, 128 and 64 columns that still gives most SMs an item
// (umma_tile_n).
//
// Every wait is bounded: a wait that does not complete within 2 s records an
// error in *err; the CTA then skips the rest of its work and still frees its
// TMEM.
#include <algorithm>

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "hedl_internal.h"
#include "launch.cuh"

namespace hedl {
namespace {

constexpr int UM = 128, UK = 64;
constexpr uint32_t ROW = UK * 2;                     // 128-byte rows of a block
constexpr uint32_t A_BYTES = UM * UK * 2;            // 16 KB
constexpr uint32_t MN_GROUP = 64 * ROW;              // an MN-major box: 64 k rows of 64 elements
constexpr int EPI = 256;                             // threads of the epilogue's eight warps
constexpr int THREADS = 64 + EPI;                    // producer, MMA issuer, epilogue
constexpr int HEAD_N = 512;                          // columns whose bias and output weights fit in shared memory
constexpr uint32_t OUT_BYTES = 32 * 32 * 2;          // a warp's 32 x 32 bf16 outputs
template <int UN>
struct Shape {
    static constexpr uint32_t B_BYTES = UN * UK * 2;
    static constexpr uint32_t STAGE_BYTES = A_BYTES + B_BYTES;
    static constexpr int STAGES = UN == 256 ? 4 : UN == 128 ? 6 : 8;   // 192 KB
    static constexpr uint32_t TMEM_COLS = 2 * UN;                      // two FP32 accumulators
    static constexpr uint32_t OUT_OFF = STAGES * STAGE_BYTES;          // outputs on their way to TMA [8 warps]
    static constexpr uint32_t CS_OFF = OUT_OFF + 8 * OUT_BYTES;        // column sums [4][UN]
    static constexpr uint32_t BIAS_OFF = CS_OFF + 4 * UN * 4;          // [HEAD_N]
    static constexpr uint32_t W3_OFF = BIAS_OFF + HEAD_N * 4;          // [2][HEAD_N], as FP32
    static constexpr uint32_t HS_OFF = W3_OFF + 2 * HEAD_N * 4;        // the other half's output sums [2][128][2]
    static constexpr uint32_t BAR_OFF = HS_OFF + 2 * UM * 2 * 4;
    static constexpr size_t SMEM = BAR_OFF + 256 + 1024;
    // Instruction descriptor, kind::f16: D FP32 (bits 4-5 = 1), A and B BF16
    // (bits 7-9 and 10-12 = 1), operand majors at bits 15 and 16 (0 = K, 1 =
    // MN), N / 8 at bit 17, M / 16 at bit 24.
    static constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(UN >> 3) << 17) |
                                      ((uint32_t)(UM >> 4) << 24);
};

// Shared-memory matrix descriptor of a SWIZZLE_128B operand block as TMA
// wrote it, without its start address / 16: leading byte offset / 16 at bit
// 16, stride byte offset / 16 at bit 32, descriptor version 1, layout type 2.
//   K-major (128-byte rows of 64 k): leading unused (1), stride = 8 rows
//     (1024 B); a K step of 16 advances the start by 32 bytes.
//   MN-major (128-byte rows of 64 m or n, one per k): leading = the next 64
//     m or n (8 KB), stride = 8 k rows (1024 B); a K step of 16 is 2048 bytes.
__device__ __forceinline__ uint64_t smem_desc(bool mn) {
    uint64_t d = (uint64_t)(mn ? MN_GROUP >> 4 : 1u) << 16;
    d |= (uint64_t)((8u * ROW) >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint64_t now_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Waits (one thread) until the barrier's phase of this parity completed, or
// the CTA gave up (*okp cleared elsewhere); false after 2 s or on give-up.
__device__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile uint32_t *okp) {
    const uint64_t t0 = now_ns();
    for (uint32_t i = 0;; ++i) {
        if (mbar_try(bar, parity)) return true;
        if ((i & 255u) == 255u && (!*okp || now_ns() - t0 > 2000000000ull)) return false;
    }
}

__device__ __forceinline__ void tma_2d(uint32_t dst, const CUtensorMap *map, int x, int y, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
        : "memory");
}

// 32 consecutive FP32 accumulator columns of this thread's TMEM lane (no wait).
__device__ __forceinline__ void tmem_ld32(uint32_t ta, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(ta)
        : "memory");
}

// Waits for the loads so far; tied to r, so that nothing reads r earlier.
__device__ __forceinline__ void tmem_wait(uint32_t (&r)[32]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]),
                   "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]),
                   "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]),
                   "+r"(r[30]), "+r"(r[31])::"memory");
}

__device__ __forceinline__ float2 unpack(uint32_t w) {   // two bf16
    return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u));
}
// a += b * c, two FP32 at a time
__device__ __forceinline__ void fma2(float2 &a, float2 b, float2 c) {
    asm("{\n .reg .b64 a, b, c;\n mov.b64 a, {%0, %1};\n mov.b64 b, {%2, %3};\n mov.b64 c, {%4, %5};\n"
        " fma.rn.f32x2 a, b, c, a;\n mov.b64 {%0, %1}, a;\n}"
        : "+f"(a.x), "+f"(a.y)
        : "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
}

// Column sums over the warp's 32 rows of v, one row a lane: a butterfly that
// halves the columns a lane holds at each step; lane l ends with column l's.
__device__ __forceinline__ float colsum32(float (&v)[32], uint32_t lane) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int k = 0; k < o; ++k) {
            const float keep = up ? v[k + o] : v[k], give = up ? v[k] : v[k + o];
            v[k] = keep + __shfl_xor_sync(0xFFFFFFFFu, give, o);
        }
    }
    return v[0];
}

// What the epilogue keeps in shared memory.
struct EpiSmem {
    const float *bias, *w3;   // [N], [2][N]
    uint32_t out;             // this warp's 32 x 32 outputs, rows of 64 bytes in the 64-byte swizzle
};

// Epilogue of 32 columns of one row: bias, ReLU or mask, bf16 or FP32 store,
// the fused output layer's partial sums (of the bf16-rounded outputs, which
// the unfused path stores and reads back; four sums a row of w3, so that the
// FP32 chains are short), the warp's column sums (cs: its 32 entries, or
// null).  All lanes of the warp call together, row < M or not.
//
// A lane holds 64 contiguous bytes of one row: stored from registers, each of
// its 16-byte stores touches 32 lines, and these stores took a fifth of a
// forward pass.  The warp's 32 rows go through shared memory instead (no bank
// conflicts in the 64-byte swizzle), from where TMA writes whole sectors.
__device__ __forceinline__ void emit32(const UmmaArgs &g, const CUtensorMap *tc, void *C, int row, int col,
                                       const uint32_t (&r)[32], const EpiSmem &es, float2 (&a0)[2], float2 (&a1)[2],
                                       float *cs, uint32_t lane) {
    const bool in = row < g.M;
    float v[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
    if (g.bias) {
        const float4 *b4 = reinterpret_cast<const float4 *>(es.bias + col);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const float4 b = b4[q];
            v[4 * q] += b.x;
            v[4 * q + 1] += b.y;
            v[4 * q + 2] += b.z;
            v[4 * q + 3] += b.w;
        }
    }
    if (g.relu) {
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] = fmaxf(v[j], 0.f);
    }
    if (g.mask && in) {   // keep where the mask (e.g. the forward activation) is positive
        const uint4 *mk =
            reinterpret_cast<const uint4 *>(reinterpret_cast<const __nv_bfloat16 *>(g.mask) + (size_t)row * g.ldc + col);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint4 m4 = mk[q];
            const uint32_t mw[4] = {m4.x, m4.y, m4.z, m4.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float2 h = unpack(mw[e]);
                if (!(h.x > 0.f)) v[q * 8 + 2 * e] = 0.f;
                if (!(h.y > 0.f)) v[q * 8 + 2 * e + 1] = 0.f;
            }
        }
    }
    if (g.store && !g.out_bf16 && in) {
        float4 *dst = reinterpret_cast<float4 *>(reinterpret_cast<float *>(C) + (size_t)row * g.ldc + col);
#pragma unroll
        for (int q = 0; q < 8; ++q) dst[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
    }
    uint32_t w[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
        w[j] = *reinterpret_cast<const uint32_t *>(&h);
    }
    if (g.store && g.out_bf16) {
        // the warp's last outputs have been read
        if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
        __syncwarp();
        const uint32_t at = es.out + 64u * lane, x = lane >> 1 & 3u;
#pragma unroll
        for (uint32_t q = 0; q < 4; ++q)
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(at + ((q ^ x) << 4)), "r"(w[4 * q]),
                         "r"(w[4 * q + 1]), "r"(w[4 * q + 2]), "r"(w[4 * q + 3])
                         : "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0 && in) {   // rows past M are cut off
            asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];" ::"l"(
                             reinterpret_cast<uint64_t>(tc)),
                         "r"(col), "r"(row), "r"(es.out)
                         : "memory");
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        }
    }
    if (g.w3) {
        const float4 *x4 = reinterpret_cast<const float4 *>(es.w3 + col);
        const float4 *y4 = reinterpret_cast<const float4 *>(es.w3 + g.N + col);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const float2 h0 = unpack(w[2 * q]), h1 = unpack(w[2 * q + 1]);
            const float4 x = x4[q], y = y4[q];
            fma2(a0[0], h0, make_float2(x.x, x.y));
            fma2(a1[0], h0, make_float2(y.x, y.y));
            fma2(a0[1], h1, make_float2(x.z, x.w));
            fma2(a1[1], h1, make_float2(y.z, y.w));
        }
    }
    if (cs) {
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const float2 h = unpack(w[j]);
            v[2 * j] = in ? h.x : 0.f;
            v[2 * j + 1] = in ? h.y : 0.f;
        }
        cs[lane] = colsum32(v, lane);
    }
}

// One or two products of one launch; product 1's items follow product 0's.
struct Batch {
    CUtensorMap ta[2], tb[2], tc[2];   // tc: bf16 outputs
    UmmaArgs g[2];
    int items0, items;
};

// Item -> (product, tile, K blocks): splits innermost, then column tiles.
// TWO = false (one product) keeps every argument a constant-bank operand.
template <int UN, bool TWO>
struct Item {
    int p, m0, n0, split, kb0, kb1;
    __device__ __forceinline__ Item(const Batch &b, int t) {
        p = TWO && t >= b.items0 ? 1 : 0;
        if (p) t -= b.items0;
        const UmmaArgs &g = b.g[p];
        split = t % g.splits;
        t /= g.splits;
        const int tiles_n = g.N / UN, nk = (g.K + UK - 1) / UK;   // splits <= nk: no range is empty
        m0 = (t / tiles_n) * UM;
        n0 = (t % tiles_n) * UN;
        kb0 = (int)((long)split * nk / g.splits);
        kb1 = (int)((long)(split + 1) * nk / g.splits);
    }
};

template <int UN, bool TWO>
__global__ void __launch_bounds__(THREADS, 1) umma_kernel(const __grid_constant__ Batch b) {
    using S = Shape<UN>;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t *base = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    float *csum = reinterpret_cast<float *>(base + S::CS_OFF);
    uint64_t *full = reinterpret_cast<uint64_t *>(base + S::BAR_OFF);
    uint64_t *empty = full + S::STAGES;
    uint64_t *tfull = empty + S::STAGES;    // [2]: accumulator ready for the epilogue
    uint64_t *tempty = tfull + 2;           // [2]: accumulator drained by the epilogue
    uint32_t *tslot = reinterpret_cast<uint32_t *>(tempty + 2);
    volatile uint32_t *okp = tslot + 1;
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31u;
    pdl_trigger();
    const uint32_t s0 = smem_u32(base);
    const uint32_t full0 = smem_u32(full), empty0 = smem_u32(empty), tfull0 = smem_u32(tfull),
                   tempty0 = smem_u32(tempty);

    if (threadIdx.x == 0) {
        for (int i = 0; i < S::STAGES; ++i) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(full0 + 8u * i) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(empty0 + 8u * i) : "memory");
        }
        for (int i = 0; i < 2; ++i) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tfull0 + 8u * i) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 8;" ::"r"(tempty0 + 8u * i) : "memory");
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        *okp = 1u;
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                     "r"(S::TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t taddr = *tslot;
    pdl_wait();   // everything above overlaps the kernel before

    if (warp == 0 && lane == 0) {
        // producer: the running block count u uses stage u % STAGES
        uint32_t u = 0;
        for (int t = blockIdx.x; t < b.items && *okp; t += gridDim.x) {
            const Item<UN, TWO> it(b, t);
            const UmmaArgs &g = b.g[it.p];
            for (int kb = it.kb0; kb < it.kb1; ++kb, ++u) {
                const uint32_t st = u % S::STAGES;
                if (u >= S::STAGES && !mbar_wait(empty0 + 8u * st, ((u - S::STAGES) / S::STAGES) & 1u, okp)) {
                    *okp = 0u;
                    break;
                }
                const uint32_t fb = full0 + 8u * st, sa = s0 + st * S::STAGE_BYTES;
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(fb), "r"(S::STAGE_BYTES)
                             : "memory");
                if (g.a_mn) {
#pragma unroll
                    for (int q = 0; q < UM / 64; ++q) tma_2d(sa + q * MN_GROUP, &b.ta[it.p], it.m0 + 64 * q, kb * UK, fb);
                } else {
                    tma_2d(sa, &b.ta[it.p], kb * UK, it.m0, fb);
                }
                if (g.b_mn) {
#pragma unroll
                    for (int q = 0; q < UN / 64; ++q)
                        tma_2d(sa + A_BYTES + q * MN_GROUP, &b.tb[it.p], it.n0 + 64 * q, kb * UK, fb);
                } else {
                    tma_2d(sa + A_BYTES, &b.tb[it.p], kb * UK, it.n0, fb);
                }
            }
        }
    } else if (warp == 1 && lane == 0) {
        // MMA issuer: the CTA's j-th item accumulates into buffer j & 1
        uint32_t u = 0, j = 0;
        for (int t = blockIdx.x; t < b.items && *okp; t += gridDim.x, ++j) {
            const Item<UN, TWO> it(b, t);
            const bool amn = b.g[it.p].a_mn, bmn = b.g[it.p].b_mn;
            const uint32_t idesc = S::IDESC | (amn ? 1u << 15 : 0u) | (bmn ? 1u << 16 : 0u);
            const uint64_t adesc = smem_desc(amn), bdesc = smem_desc(bmn);
            const uint32_t astep = amn ? 16u * ROW : 32u, bstep = bmn ? 16u * ROW : 32u;
            const uint32_t bf = j & 1u;
            if (j >= 2 && !mbar_wait(tempty0 + 8u * bf, ((j >> 1) - 1u) & 1u, okp)) {
                *okp = 0u;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t acc_t = taddr + bf * UN;
            bool good = true;
            for (int kb = it.kb0; kb < it.kb1; ++kb, ++u) {
                const uint32_t st = u % S::STAGES;
                if (!mbar_wait(full0 + 8u * st, (u / S::STAGES) & 1u, okp)) {
                    *okp = 0u;
                    good = false;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t sa = s0 + st * S::STAGE_BYTES;
#pragma unroll
                for (int s = 0; s < UK / 16; ++s) {
                    const uint64_t ad = adesc + ((sa + (uint32_t)s * astep) >> 4);   // smem addresses stay below 2^18
                    const uint64_t bd = bdesc + ((sa + A_BYTES + (uint32_t)s * bstep) >> 4);
                    const uint32_t acc = (kb > it.kb0 || s > 0) ? 1u : 0u;
                    asm volatile(
                        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(acc_t),
                        "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
                        : "memory");
                }
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                 empty0 + 8u * st)
                             : "memory");
            }
            if (!good) break;
            // every MMA issued so far completes before this arrives
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                             tfull0 + 8u * bf)
                         : "memory");
        }
    } else if (warp >= 2) {
        // epilogue: warp w reads TMEM lanes 32 (w % 4) .. + 31, the tile rows of that quarter, and one half of the columns
        constexpr int HC = UN / 2;
        const uint32_t q = warp & 3u, half = (warp - 2u) >> 2;
        const int et = (int)threadIdx.x - 64;
        float *bias = reinterpret_cast<float *>(base + S::BIAS_OFF), *w3 = reinterpret_cast<float *>(base + S::W3_OFF);
        const EpiSmem es{bias, w3, s0 + S::OUT_OFF + (warp - 2u) * OUT_BYTES};
        if (b.g[0].bias || b.g[0].w3) {   // one product
            const UmmaArgs &g = b.g[0];
            if (g.bias)
                for (int i = et; i < g.N; i += EPI) bias[i] = g.bias[i];
            if (g.w3)
                for (int i = et; i < 2 * g.N; i += EPI)
                    w3[i] = __bfloat162float(reinterpret_cast<const __nv_bfloat16 *>(g.w3)[i]);
            asm volatile("bar.sync 1, %0;" ::"n"(EPI) : "memory");
        }
        uint32_t j = 0;
        for (int t = blockIdx.x; t < b.items; t += gridDim.x, ++j) {
            const Item<UN, TWO> it(b, t);
            const UmmaArgs &g = b.g[it.p];
            const uint32_t bf = j & 1u;
            uint32_t ok = 1u;
            if (lane == 0) ok = mbar_wait(tfull0 + 8u * bf, (j >> 1) & 1u, okp) ? 1u : 0u;
            ok = __shfl_sync(0xFFFFFFFFu, ok, 0);
            if (g.colsum || g.w3)   // the warps meet at barriers below: they go on, or give up, together
                asm volatile("{\n .reg .pred p, q;\n setp.ne.u32 p, %0, 0;\n bar.red.and.pred q, 1, %1, p;\n"
                             " selp.u32 %0, 1, 0, q;\n}\n"
                             : "+r"(ok)
                             : "n"(EPI)
                             : "memory");
            if (!ok) {
                if (lane == 0) *okp = 0u;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int row = it.m0 + (int)(q * 32 + lane);
            const int n0 = it.n0 + (int)half * HC;
            void *C = reinterpret_cast<float *>(g.C) + (size_t)it.split * g.c_split;   // FP32 outputs
            float2 a0[2] = {}, a1[2] = {};   // the fused output layer
            uint32_t r[2][32];
            const uint32_t ta = taddr + ((q * 32u) << 16) + bf * UN + half * HC;
            tmem_ld32(ta, r[0]);
#pragma unroll
            for (int k = 0; k < HC / 32; ++k) {   // the next 32 columns load while these are worked on
                tmem_wait(r[k & 1]);
                if (k + 1 < HC / 32) {
                    tmem_ld32(ta + 32u * (k + 1), r[(k + 1) & 1]);
                } else {   // the accumulator may be overwritten from here on
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0)
                        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tempty0 + 8u * bf) : "memory");
                }
                emit32(g, &b.tc[it.p], C, row, n0 + 32 * k, r[k & 1], es, a0, a1,
                       g.colsum ? csum + q * UN + half * HC + 32 * k : nullptr, lane);
            }
            if (g.w3) {   // the first half's warp adds the second's sums (two places: one barrier an item is enough)
                float2 *hs = reinterpret_cast<float2 *>(base + S::HS_OFF) + bf * UM + q * 32 + lane;
                const float2 sum = make_float2((a0[0].x + a0[0].y) + (a0[1].x + a0[1].y),
                                               (a1[0].x + a1[0].y) + (a1[1].x + a1[1].y));
                if (half) *hs = sum;
                asm volatile("bar.sync %0, 64;" ::"r"(2u + q) : "memory");
                if (!half && row < g.M)
                    reinterpret_cast<float2 *>(g.y)[(size_t)(it.n0 / UN) * g.M + row] =
                        make_float2(sum.x + hs->x, sum.y + hs->y);
            }
            if (g.colsum) {   // the four quarters' sums, added by the epilogue's threads
                asm volatile("bar.sync 1, %0;" ::"n"(EPI) : "memory");
                for (int c = et; c < UN; c += EPI)
                    g.colsum[(size_t)(it.m0 / UM) * g.N + it.n0 + c] =
                        (csum[c] + csum[UN + c]) + (csum[2 * UN + c] + csum[3 * UN + c]);
                asm volatile("bar.sync 1, %0;" ::"n"(EPI) : "memory");
            }
        }
        if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }
    __syncwarp();
    __syncthreads();
    if (threadIdx.x == 0 && !*okp && b.g[0].err) atomicOr(b.g[0].err, 1u);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(S::TMEM_COLS)
                     : "memory");
}

}  // namespace

bool umma_shape_ok(const UmmaArgs &a) {
    // a K-major operand is contracted in whole 64-wide blocks; an MN-major one
    // has 64-row boxes along M or N and any K (rows past it read as zeros)
    return a.N % 64 == 0 && a.N > 0 && a.K > 0 && (a.a_mn ? a.M % 64 == 0 : a.K % UK == 0) &&
           (a.b_mn || a.K % UK == 0) && a.lda % 8 == 0 && a.ldb % 8 == 0 && a.splits >= 1 &&
           a.splits <= (a.K + UK - 1) / UK &&
           // a K range has a place of its own in FP32 outputs only: bf16 ones leave through one
           // tensor map, and column sums and the output layer's have one place a tile; bias, ReLU
           // and mask would apply to every range
           (a.splits == 1 ||
            (!a.out_bf16 && !a.colsum && !a.w3 && !a.bias && !a.relu && !a.mask && a.c_split % 4 == 0)) &&
           a.ldc % (a.out_bf16 ? 8 : 4) == 0 && ((uintptr_t)a.A & 15) == 0 &&
           ((uintptr_t)a.B & 15) == 0 && ((uintptr_t)a.C & 15) == 0 && ((uintptr_t)a.bias & 15) == 0 &&
           (!a.mask || (a.ldc % 8 == 0 && ((uintptr_t)a.mask & 15) == 0)) &&
           (!(a.bias || a.w3) || a.N <= HEAD_N) &&
           (!a.w3 || (a.y && ((uintptr_t)a.w3 & 15) == 0 && ((uintptr_t)a.y & 7) == 0));
}

namespace {

using EncodeTiled = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                 const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                 CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiled encode_fn() {
    static EncodeTiled fn = nullptr;
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiled>(p);
    }
    return fn;
}

// Tensor map of a row-major bf16 matrix [rows][ld] (cols used): 64-column x box_rows
// boxes in the 128-byte swizzle, rows past the end read as zeros; or 32-column
// boxes in the 64-byte one.
bool make_map(CUtensorMap *m, const void *ptr, int rows, int cols, int ld, int box_rows, int box_cols = UK) {
    EncodeTiled fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    const cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(ptr), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE,
              box_cols == UK ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

long item_count(const UmmaArgs &a, int un) { return (long)((a.M + UM - 1) / UM) * (a.N / un) * a.splits; }

template <int UN, bool TWO>
int launch(const UmmaArgs *a, int count, UmmaDevice &dev, cudaStream_t s) {
    constexpr uint32_t bit = (UN == 256 ? 1u : UN == 128 ? 2u : 4u) << (TWO ? 3 : 0);
    if (!(dev.allowed.load(std::memory_order_relaxed) & bit)) {
        const cudaError_t e = allow_smem(umma_kernel<UN, TWO>, Shape<UN>::SMEM);
        if (e) return (int)e;
        dev.allowed.fetch_or(bit, std::memory_order_relaxed);
    }
    Batch b{};
    for (int p = 0; p < count; ++p) {
        b.g[p] = a[p];
        const bool ok = (a[p].a_mn ? make_map(&b.ta[p], a[p].A, a[p].K, a[p].M, a[p].lda, UK)
                                   : make_map(&b.ta[p], a[p].A, a[p].M, a[p].K, a[p].lda, UM)) &&
                        (a[p].b_mn ? make_map(&b.tb[p], a[p].B, a[p].K, a[p].N, a[p].ldb, UK)
                                   : make_map(&b.tb[p], a[p].B, a[p].N, a[p].K, a[p].ldb, UN)) &&
                        (!a[p].store || !a[p].out_bf16 || make_map(&b.tc[p], a[p].C, a[p].M, a[p].N, a[p].ldc, 32, 32));
        if (!ok) return (int)cudaErrorInvalidValue;
    }
    b.items0 = (int)item_count(a[0], UN);
    b.items = b.items0 + (count > 1 ? (int)item_count(a[1], UN) : 0);
    return (int)launch_pdl(umma_kernel<UN, TWO>, (unsigned)std::min(b.items, dev.sms), THREADS, Shape<UN>::SMEM, s, b);
}

}  // namespace

int umma_device(UmmaDevice *d) {
    int dev = 0;
    const cudaError_t e = cudaGetDevice(&dev);
    return (int)(e ? e : cudaDeviceGetAttribute(&d->sms, cudaDevAttrMultiProcessorCount, dev));
}

int umma_tile_n(const UmmaArgs *a, int count, const UmmaDevice &dev) {
    for (int un : {256, 128}) {
        long items = 0;
        bool fits = true;
        for (int p = 0; p < count; ++p) {
            items += item_count(a[p], un);
            fits = fits && a[p].N % un == 0;
        }
        if (fits && 4 * items >= 3l * dev.sms) return un;
    }
    return 64;
}

int umma_gemm(const UmmaArgs *a, int count, UmmaDevice &dev, void *stream) {
    if (count < 1 || count > 2) return (int)cudaErrorInvalidValue;
    for (int p = 0; p < count; ++p) {
        if (!umma_shape_ok(a[p]) || (count > 1 && (a[p].bias || a[p].w3))) return (int)cudaErrorInvalidValue;
        if (a[p].M <= 0) return 0;
    }
    const int un = umma_tile_n(a, count, dev);
    cudaStream_t s = (cudaStream_t)stream;
    if (count == 1)
        return un == 256   ? launch<256, false>(a, 1, dev, s)
               : un == 128 ? launch<128, false>(a, 1, dev, s)
                           : launch<64, false>(a, 1, dev, s);
    return un == 256   ? launch<256, true>(a, 2, dev, s)
           : un == 128 ? launch<128, true>(a, 2, dev, s)
                       : launch<64, true>(a, 2, dev, s);
}

}  // namespace hedl
