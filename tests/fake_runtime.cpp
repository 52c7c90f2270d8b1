// A stand-in for the CUDA runtime, linked with the library's own objects: it
// launches nothing, keeps "device" memory on the host, and checks or records
// what the library asks of it.  main runs one scenario, named by its argument.
#include <cuda_runtime_api.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <utility>
#include <vector>

#include "hedl_internal.h"

namespace {
struct Launch {
    const void *fn;
    unsigned grid;
    const uint32_t *pos;   // captured launches: the positive examples in the kernel's view of the KB
};
int device = 0;                    // devices 0 and 1, with different numbers of SMs
constexpr int SMS[] = {152, 16};
std::map<std::pair<int, const void *>, size_t> opted;   // (device, kernel) -> shared memory it may use
bool refuse_opt_in = false;        // the next opt-in fails
unsigned last_grid = 0;
const void *last_fn = nullptr;
bool capturing = false;
cudaError_t last = cudaSuccess;
int instantiated = 0;
std::vector<Launch> captured;

cudaError_t launch(const void *fn, dim3 grid, size_t smem, void **args) {
    if (smem > 49152 && smem > opted[{device, fn}]) return cudaErrorInvalidValue;
    last_grid = grid.x, last_fn = fn;
    // the interpreter's and the final kernel's first argument begins with the KBView
    if (capturing) captured.push_back({fn, grid.x, static_cast<const hedl::KBView *>(args[0])->pos});
    return cudaSuccess;
}
struct Config {
    dim3 grid, block;
    size_t smem;
    void *stream;
} config;
}  // namespace

extern "C" {
cudaError_t cudaMalloc(void **p, size_t n) { return (*p = calloc(n ? n : 1, 1)) ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaFree(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemset(void *d, int v, size_t n) { memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { memset(d, v, n); return cudaSuccess; }
cudaError_t cudaGetLastError() { return std::exchange(last, cudaSuccess); }
const char *cudaGetErrorString(cudaError_t) { return "fake error"; }
cudaError_t cudaGetDevice(int *d) { *d = device; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { device = d; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int d) {
    *v = a == cudaDevAttrMultiProcessorCount ? SMS[d] : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448 : 0;
    return cudaSuccess;
}
cudaError_t cudaGetDeviceProperties(cudaDeviceProp *p, int) { memset(p, 0, sizeof *p); return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = reinterpret_cast<cudaStream_t>(&device); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) {
    capturing = true;
    captured.clear();
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) {
    capturing = false;
    *g = reinterpret_cast<cudaGraph_t>(&device);
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *e, cudaGraph_t, unsigned long long) {
    ++instantiated;
    *e = reinterpret_cast<cudaGraphExec_t>(&device);
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *fn, cudaFuncAttribute a, int v) {
    if (std::exchange(refuse_opt_in, false)) return cudaErrorMemoryAllocation;
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) opted[{device, fn}] = (size_t)v;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) { *n = 3; return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void **p, const void *) { *p = nullptr; return cudaErrorInvalidSymbol; }
static int encode_tiled(...) { return 0; }
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **fn, unsigned, unsigned long long, cudaDriverEntryPointQueryResult *r) {
    *fn = reinterpret_cast<void *>(&encode_tiled);
    if (r) *r = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *fn, void **args) { return launch(fn, c->gridDim, c->dynamicSmemBytes, args); }
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, CUstream_st *s) { config = {g, b, smem, s}; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *smem, void *s) {
    *g = config.grid, *b = config.block, *smem = config.smem;
    *static_cast<void **>(s) = config.stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *fn) {
    *k = reinterpret_cast<cudaKernel_t>(const_cast<void *>(fn));
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3, void **args, size_t smem, cudaStream_t) {
    return last = launch(k, grid, smem, args);
}
void **__cudaRegisterFatBinary(void *) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
}

#define REQUIRE(x)                                                                              \
    do {                                                                                        \
        if (!(x)) return printf("line %d: %s (%s)\n", __LINE__, #x, hedl_last_error()), 1;      \
    } while (0)

namespace {
constexpr uint32_t N = 1000, WP = 32;
struct alignas(256) Row { uint32_t w[WP]; };

hedl_kb *load(const Row &concept_row) {
    hedl_kb_desc d{};
    d.n_indiv = N;
    d.n_concepts = 1;
    d.concept_bits = concept_row.w;
    hedl_kb *kb = nullptr;
    hedl_kb_load(&d, HEDL_KB_NO_VALIDATE, nullptr, &kb);
    return kb;
}

// A captured graph holds the examples that it was captured with: after
// hedl_examples_set the next scoring call has to capture anew.
int examples_after_capture(bool one_shot) {
    static Row bits, ex[4];
    hedl_kb *kb = load(bits);
    REQUIRE(kb);
    REQUIRE(hedl_examples_set(kb, ex[0].w, ex[1].w, nullptr) == HEDL_OK);
    const uint64_t prog = HEDL_OP_ATOM;
    const uint32_t offs[2] = {0, 1};
    hedl_plan *plan = nullptr;
    REQUIRE(hedl_plan_batch(kb, &prog, offs, 1, 0, &plan) == HEDL_OK);
    hedl_plan_info info;
    REQUIRE(hedl_plan_info_get(plan, &info) == HEDL_OK);
    void *ws = aligned_alloc(256, (info.workspace_bytes + 255) / 256 * 256);
    alignas(16) static uint32_t counts[4];
    auto score = [&]() {
        return one_shot ? hedl_score_batch(kb, &prog, offs, 1, counts, ws, info.workspace_bytes, 0, nullptr)
                        : hedl_plan_execute(kb, plan, counts, nullptr, ws, info.workspace_bytes, nullptr);
    };
    for (int k = 0; k < 3; ++k) REQUIRE(score() == HEDL_OK);
    REQUIRE(instantiated == 1 && captured.size() == 2 && captured[0].pos == ex[0].w);
    REQUIRE(hedl_examples_set(kb, ex[2].w, ex[3].w, nullptr) == HEDL_OK);
    REQUIRE(score() == HEDL_OK);
    REQUIRE(instantiated == 2 && captured[0].pos == ex[2].w && captured[1].pos == ex[2].w);
    REQUIRE(score() == HEDL_OK && instantiated == 2);   // unchanged: the graph is launched again
    if (!one_shot) REQUIRE(hedl_plan_replay(kb, plan, counts, nullptr, ws, info.workspace_bytes, nullptr) == HEDL_OK && instantiated == 2);
    hedl_plan_free(plan);
    hedl_kb_free(kb);
    free(ws);
    return 0;
}

// The shared memory that a kernel needs is allowed on every device that it
// launches on, and a failure is not kept; grids follow the current device.
int second_device() {
    for (int d : {0, 1, 0}) {
        cudaSetDevice(d);
        alignas(16) static float y[2 * 64];
        static uint32_t idx[4];
        static uint8_t ws[8192];
        refuse_opt_in = true;
        REQUIRE(hedl_select_top(y, 64, 4, idx, ws, sizeof ws, nullptr) == HEDL_ERR_CUDA);
        REQUIRE(hedl_select_top(y, 64, 4, idx, ws, sizeof ws, nullptr) == HEDL_OK);
        std::vector<float> params(hedl_mlp_param_count());
        hedl_mlp *mlp = nullptr;
        REQUIRE(hedl_mlp_create(params.data(), &mlp) == HEDL_OK);
        for (uint32_t rows : {100u, 4096u, 20000u}) {   // tiles of 64, 128 and 256 columns on device 0
            size_t bytes = 0;
            REQUIRE(hedl_mlp_workspace_size(rows, &bytes) == HEDL_OK);
            void *w = malloc(bytes), *x = aligned_alloc(16, 1024ull * rows), *t = malloc(8ull * rows);
            refuse_opt_in = rows == 100u;
            if (refuse_opt_in)
                REQUIRE(hedl_mlp_forward(mlp, (uint16_t *)x, rows, (float *)t, w, bytes, nullptr) == HEDL_ERR_CUDA);
            REQUIRE(hedl_mlp_forward(mlp, (uint16_t *)x, rows, (float *)t, w, bytes, nullptr) == HEDL_OK);
            REQUIRE(hedl_mlp_gradients(mlp, (uint16_t *)x, (float *)t, rows, nullptr, w, bytes, nullptr) == HEDL_OK);
            free(w), free(x), free(t);
        }
        hedl::UmmaDevice dev;
        hedl::UmmaArgs a{};   // a product of many tiles: one block an SM
        alignas(16) static uint8_t operand[16];
        a.A = a.B = a.C = operand;
        a.M = 1 << 16, a.N = a.K = a.lda = a.ldb = a.ldc = 512, a.out_bf16 = 1;
        REQUIRE(hedl::umma_device(&dev) == 0 && hedl::umma_gemm(&a, 1, dev, nullptr) == 0 && last_grid == (unsigned)SMS[d]);
        hedl_mlp_free(mlp);
    }
    return 0;
}

// Products split over K have a place for each range in plain FP32 outputs only.
int split_products() {
    alignas(16) static uint8_t operand[16];
    hedl::UmmaArgs a{};
    a.A = a.B = a.C = operand;
    a.M = a.N = a.K = a.lda = a.ldb = a.ldc = 512, a.splits = 4, a.c_split = 512 * 512;
    REQUIRE(hedl::umma_shape_ok(a));
    auto refused = [&](auto change) {
        hedl::UmmaArgs b = a;
        change(b);
        const bool split = hedl::umma_shape_ok(b);
        b.splits = 1;
        return !split && hedl::umma_shape_ok(b);
    };
    auto *f = reinterpret_cast<float *>(operand);
    REQUIRE(refused([&](hedl::UmmaArgs &b) { b.out_bf16 = 1; }));
    REQUIRE(refused([&](hedl::UmmaArgs &b) { b.colsum = f; }));
    REQUIRE(refused([&](hedl::UmmaArgs &b) { b.w3 = operand, b.y = f; }));
    REQUIRE(refused([&](hedl::UmmaArgs &b) { b.bias = f; }));
    REQUIRE(refused([&](hedl::UmmaArgs &b) { b.relu = 1; }));
    REQUIRE(refused([&](hedl::UmmaArgs &b) { b.mask = operand; }));
    REQUIRE(refused([&](hedl::UmmaArgs &b) { b.c_split = 6; }));
    return 0;
}

// Every launch shape has an interpreter of its own for blocks of 4 and of 8 chunks.
int role_block() {
    static Row bits;
    hedl_kb *kb = load(bits);
    REQUIRE(kb);
    const uint64_t prog = HEDL_OP_ATOM;
    const uint32_t offs[2] = {0, 1};
    static Row out;
    void *ws = aligned_alloc(256, 1 << 20);
    hedl_tuning t;
    REQUIRE(hedl_tuning_get(kb, &t) == HEDL_OK && t.role_block == 4);
    std::map<const void *, int> seen;
    int shapes = 0;
    for (uint32_t full : {0u, 1u})
        for (uint32_t stage : {0u, 1u})
            for (uint32_t wpl : {1u, 4u})
                for (uint32_t warps : {1u, 2u, 4u, 8u, 16u, 32u}) {
                    if ((wpl == 4 && (warps < 4 || warps == 32)) || (full && (warps != 8 || wpl != 1 || stage)) ||
                        (stage && warps < 4))
                        continue;
                    ++shapes;
                    for (uint32_t block : {4u, 8u}) {
                        t.warps_per_cta = warps, t.words_per_lane = wpl, t.stage_fillers = stage;
                        t.full_occupancy = full, t.role_block = block;
                        REQUIRE(hedl_tuning_set(kb, &t) == HEDL_OK);
                        REQUIRE(hedl_eval_concept(kb, &prog, 1, out.w, ws, 1 << 20, HEDL_NO_GRAPH, nullptr) == HEDL_OK);
                        ++seen[last_fn];
                    }
                }
    REQUIRE((int)seen.size() == 2 * shapes);
    hedl_kb_free(kb);
    free(ws);
    return 0;
}

// A workspace of the size that hedl_autotune_workspace_size gives is enough for hedl_autotune.
int autotune_workspace() {
    static Row bits, ex[2];
    hedl_kb *kb = load(bits);
    REQUIRE(kb);
    REQUIRE(hedl_examples_set(kb, ex[0].w, ex[1].w, nullptr) == HEDL_OK);
    for (uint32_t hyps : {1u, 3u, 1000u}) {
        const std::vector<uint64_t> progs(hyps, HEDL_OP_ATOM);
        std::vector<uint32_t> offs(hyps + 1);
        for (uint32_t h = 0; h <= hyps; ++h) offs[h] = h;
        size_t bytes = 0;
        REQUIRE(hedl_autotune_workspace_size(kb, progs.data(), offs.data(), hyps, &bytes) == HEDL_OK);
        void *ws = aligned_alloc(256, (bytes + 255) / 256 * 256);
        REQUIRE(hedl_autotune(kb, progs.data(), offs.data(), hyps, ws, bytes, nullptr, nullptr, nullptr) == HEDL_OK);
        REQUIRE(hedl_autotune(kb, progs.data(), offs.data(), hyps, ws, bytes - 1, nullptr, nullptr, nullptr) ==
                HEDL_ERR_WORKSPACE_TOO_SMALL);
        free(ws);
    }
    hedl_kb_free(kb);
    return 0;
}
}  // namespace

int main(int argc, char **argv) {
    const std::string s = argc > 1 ? argv[1] : "";
    if (s == "examples_plan") return examples_after_capture(false);
    if (s == "examples_one_shot") return examples_after_capture(true);
    if (s == "second_device") return second_device();
    if (s == "split_products") return split_products();
    if (s == "role_block") return role_block();
    if (s == "autotune_workspace") return autotune_workspace();
    return 2;
}
