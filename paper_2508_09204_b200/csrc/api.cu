// C-ABI entry points that tie the kernels together: the routed dequant-GEMM
// call, the device status word, status strings and the launch counter.
#include <atomic>
#include <cstring>

#include "common.cuh"
#include "ptx.cuh"

namespace moqe {

namespace {
std::atomic<unsigned long long> g_launches{0};
// One a device, and zero, when the library's code is loaded there: nothing is allocated or cleared for it, which the first call
// of a process could not do beside a capture (clearing it on the default stream made captures on blocking streams invalid).
__device__ int g_status_word;
std::atomic<int*> g_status_words[64] = {};
std::atomic<int> g_sm_counts[64] = {};
}  // namespace

void count_launch(unsigned n) { g_launches.fetch_add(n, std::memory_order_relaxed); }

int* device_status_word() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    if (int* p = g_status_words[dev].load(std::memory_order_relaxed)) return p;
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_status_word) != cudaSuccess) { cudaGetLastError(); return nullptr; }
    g_status_words[dev].store((int*)p, std::memory_order_relaxed);
    return (int*)p;
}

EncodeTiledFn encode_tiled_fn() {
    static const EncodeTiledFn fn = []() -> EncodeTiledFn {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f, cudaEnableDefault, &q) == cudaSuccess && q == cudaDriverEntryPointSuccess)
            return (EncodeTiledFn)f;
        return nullptr;
    }();
    return fn;
}

int device_sm_count() {
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 148;
    n = g_sm_counts[dev].load(std::memory_order_relaxed);
    if (n == 0) {
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) return 148;
        g_sm_counts[dev].store(n, std::memory_order_relaxed);
    }
    return n;
}

bool ensure_dynamic_smem(const void* kernel, int bytes, std::atomic<unsigned long long>& done) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    const unsigned long long bit = dev >= 0 && dev < 64 ? 1ull << dev : 0ull;
    if (bit && (done.load(std::memory_order_relaxed) & bit)) return true;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess) return false;
    done.fetch_or(bit, std::memory_order_relaxed);
    return true;
}

namespace {

size_t align256(size_t x) { return (x + 255) / 256 * 256; }

// The arrival counters of the split-K kernels have a region of their own (they share it: each leaves it zero) that no kernel
// uses as scratch, so that any of them may follow any other on one workspace.  Above 64 rows its place and size depend on M and
// E alone: one workspace then serves layers of any shape.
struct WsLayout {
    size_t perm, offsets, sort, counters, body, total;
};
size_t counter_bytes(int M, int Np) {
    const size_t a = stream_zero_bytes(M, Np), b = decode_zero_bytes(M), c = tc_zero_bytes();
    return align256(a > b ? (a > c ? a : c) : (b > c ? b : c));
}

WsLayout ws_layout(int M, int Np, int K, int E) {
    WsLayout w;
    size_t off = 0;
    w.perm = off;    off += align256((size_t)M * sizeof(int32_t) + 16);
    w.offsets = off; off += align256((MOQE_MAX_EXPERTS + 2) * sizeof(int32_t));
    w.sort = off;    off += align256(sort_workspace_bytes(M, E));
    w.counters = off; off += counter_bytes(M, Np);
    w.body = off;
    size_t a = stream_workspace_bytes(M, Np, E), b = tc_workspace_bytes(M, K, E, Np), c = decode_workspace_bytes(M);
    const size_t d = dense_workspace_bytes(M, K, E, Np, (K + 127) / 128 * 128);
    a = a > b ? a : b;
    a = a > d ? a : d;
    off += align256(a > c ? a : c);
    w.total = off;
    return w;
}

// Batches beyond the decode kernel's 32 rows: up to this many the streaming kernel, if an expert has groups narrower than
// 128 k (four Qwen experts, layer by layer, streaming / grouped GEMM: 24 rows 25 / 28, 73 / 71, 76 / 107 us; 64 rows
// 32 / 28, 106 / 72, 110 / 108); everything else is the grouped GEMM's (4096 x 4096, three LLaMA experts, 48 rows:
// 30 / 22 us).
constexpr int AUTO_STREAM_MAX_ROWS = 48;
constexpr int LAST_PATH = 6;

bool g_auto_decode = true;   // whether the automatic choice takes a decode kernel where it applies
bool g_auto_dense = true;    // ... and the dense-weights GEMM for large batches on small layers

// 0 = tcgen05 grouped GEMM, 1 = mma.sync streaming kernel, 2 = decode kernel, 3 = dense-weights GEMM (small layers)
int pick_kernel(int path, int M, const moqe_expert* const* ex, int E) {
    if (path == 5) return 2;
    if (path == 6) return 3;
    if (path == 1) return 1;
    if (path == 0) {
        if (g_auto_decode && decode_supported(M, ex, E)) return 2;
        if (M <= AUTO_STREAM_MAX_ROWS && !(g_auto_decode && decode_supported_multi(1, ex, 1, E))) return 1;
        // The dense-weights GEMM has a launch more, streams or re-reads an expert's whole matrix per 128 rows and multiplies grouped
        // experts' weights twice; the grouped GEMM drains every group of 32 k by itself.  Dense / grouped, us, K -> N channels:
        //                   rows    W8-pc W4-pc W4-g32   W4-pc        W8-pc W4-g64   W4-g128
        //   256 ->   64      980    10.3 / 8.2           8.2 / 6.1    9.9 / 7.2      8.9 / 6.5
        //                   3920    10.9 / 10.1          8.2 / 8.5    10.3 / 9.5     9.2 / 8.9
        //                  12544    10.9 / 13.9          8.2 / 10.3   10.3 / 12.3    9.2 / 10.6
        //   256 -> 1024    20000    48.1 / 39.0          33.3 / 27.6  45.7 / 36.9    51.5 / 32.6
        //                  35000    52.4 / 60.5          35.3 / 42.5  49.8 / 56.0    53.3 / 50.7
        //                 100352    120 / 148            90.1 / 109   125 / 138      144 / 128
        //   1024 -> 256    12544    31.8 / 28.5          18.0 / 15.2  31.4 / 20.9    26.7 / 15.8
        //                  50176    59.6 / 51.7          41.0 / 32.5  67.9 / 51.9    67.7 / 38.3
        //                 100352    106 / 112            73.3 / 55.9  111 / 83.5     127 / 71.1
        //   512 ->  512    35000    48.5 / 47.1          31.2 / 26.2  46.5 / 39.0    49.2 / 33.8
        //                 100352    111 / 103            79.0 / 64.0  119 / 96.6     133 / 85.3
        //   512 -> 1024    35000    86.1 / 77.9          53.9 / 45.2  84.0 / 69.6    89.6 / 63.0
        // So rows of 512 k and more are the grouped GEMM's unless a group of 32 k is among the experts (no format, batch, number of
        // experts or scattering of rows was found where it is behind, from 72 to 1024 channels), with one exception: per-channel
        // experts of 512 k whose second pair of channel tiles is mostly padding (512 -> 264, W8-pc W4-pc: 50176 rows 39.2 / 41.0,
        // 100352 71.1 / 73.5; 384 channels 42.6 / 42.1; 576 k 43.2 / 42.8).  The other lines lie where calls with groups of 32 k and
        // layers of 256 k had them when the grouped GEMM drained such groups more slowly; it wins with 512 k and more at many sizes now,
        // not at all (768 -> 384, 50176 rows: 79 / 96).  Small layers below some 3000 rows would do better on it.
        bool fine = false, per_channel = true;
        for (int e = 0; e < E; ++e) { fine |= ex[e]->group == 32; per_channel &= ex[e]->group == 0; }
        const int N = ex[0]->N, K = ex[0]->K;
        const bool padded = per_channel && K < 576 && N > 256 && N <= 320;
        const bool few = (M < (fine && K > N ? 12000 : 30000) || (!fine && K >= 512 && !padded)) && (long long)N * K > 65536;
        return (g_auto_dense && !few && dense_supported(M, N, K, ex, E)) ? 3 : 0;
    }
    return 0;
}

}  // namespace
}  // namespace moqe

using namespace moqe;

extern "C" size_t moqe_routed_qgemm_workspace(int M, int N, int K, int E) {
    if (M < 0 || N <= 0 || K <= 0 || E <= 0) return 0;
    int Np = (N + 127) / 128 * 128;
    return ws_layout(M, Np, K, E).total;
}

namespace {
// Argument checks shared by the single-layer entry points (`ids_or_perm`: row ids, or the sort's perm).  *done: the
// call is complete (an empty batch) when MOQE_OK comes back with it set.
moqe_status single_layer_args(const void* X, const void* ids_or_perm, const void* offsets_or_self, int M,
                              const moqe_expert* const* ex, int E, const void* Y, void* workspace, size_t workspace_bytes,
                              int path, WsLayout& w, int& kernel, bool& done) {
    done = false;
    if (!ex) return MOQE_ERR_NULL;
    if (E <= 0 || M < 0) return MOQE_ERR_SHAPE;
    if (E > MOQE_MAX_EXPERTS) return MOQE_ERR_UNSUPPORTED;
    for (int e = 0; e < E; ++e)
        if (!ex[e]) return MOQE_ERR_NULL;
    const int N = ex[0]->N, K = ex[0]->K;
    for (int e = 1; e < E; ++e)
        if (ex[e]->N != N || ex[e]->K != K) return MOQE_ERR_MISMATCH;
    if (M == 0) { done = true; return MOQE_OK; }
    if (!X || !ids_or_perm || !offsets_or_self || !Y) return MOQE_ERR_NULL;
    if (N % 8 != 0 || K % 8 != 0 || (uintptr_t)X % 16 || (uintptr_t)Y % 16) return MOQE_ERR_UNSUPPORTED;
    if (path < 0 || path > LAST_PATH) return MOQE_ERR_SHAPE;
    w = ws_layout(M, ex[0]->Np, K, E);
    if (!workspace || workspace_bytes < w.total || (uintptr_t)workspace % 256) return MOQE_ERR_WORKSPACE;
    kernel = pick_kernel(path, M, ex, E);
    if (kernel == 2 && !(path == 5 ? decode_supported_multi(M, ex, 1, E) : decode_supported(M, ex, E))) return MOQE_ERR_UNSUPPORTED;
    return MOQE_OK;
}

// the grouped product on sorted rows with the kernel `pick_kernel` chose
moqe_status run_sorted(int kernel, int path, const void* X, int M, const moqe_expert* const* ex, int E, void* Y,
                       const int32_t* perm, const int32_t* offsets, char* base, const WsLayout& w, cudaStream_t st) {
    const int N = ex[0]->N, K = ex[0]->K;
    uint32_t* counters = (uint32_t*)(base + w.counters);
    void* body = base + w.body;
    const size_t body_bytes = w.total - w.body;
    if (kernel == 2) return launch_qgemm_decode_multi(&X, M, 1, ex, E, &Y, perm, offsets, counters, body, body_bytes, st);
    if (kernel == 1) return launch_qgemm_stream(X, M, N, K, ex, E, Y, perm, offsets, counters, body, body_bytes, st);
    if (kernel == 3) return launch_qgemm_dense(X, M, N, K, ex, E, Y, perm, offsets, body, body_bytes, st);
    return launch_qgemm_tc(X, M, N, K, ex, E, Y, perm, offsets, counters, body, body_bytes, path == 3 ? 128 : (path == 4 ? 256 : 0), st);
}
}  // namespace

extern "C" moqe_status moqe_routed_qgemm_path(const void* X_bf16, const int32_t* row_ids, int M,
                                              const moqe_expert* const* h_experts, int E, void* Y_bf16, void* workspace,
                                              size_t workspace_bytes, void* stream, int path) {
    WsLayout w;
    int kernel = 0;
    bool done = false;
    moqe_status s = single_layer_args(X_bf16, row_ids, row_ids, M, h_experts, E, Y_bf16, workspace, workspace_bytes, path, w, kernel, done);
    if (s != MOQE_OK || done) return s;
    cudaStream_t st = (cudaStream_t)stream;
    char* base = (char*)workspace;
    int32_t* perm = (int32_t*)(base + w.perm);
    int32_t* offsets = (int32_t*)(base + w.offsets);
    const size_t zero_bytes = kernel != 3 ? w.body - w.counters : 0;
    s = launch_sort(row_ids, M, E, perm, offsets, base + w.sort, w.counters - w.sort, base + w.counters, zero_bytes, Y_bf16,
                    h_experts[0]->N, st);
    if (s != MOQE_OK) return s;
    return run_sorted(kernel, path, X_bf16, M, h_experts, E, Y_bf16, perm, offsets, base, w, st);
}

extern "C" const char* moqe_routed_qgemm_kernel(int M, const moqe_expert* const* h_experts, int E, int path) {
    if (!h_experts || M <= 0 || E <= 0 || E > MOQE_MAX_EXPERTS || path < 0 || path > LAST_PATH) return nullptr;
    for (int e = 0; e < E; ++e)
        if (!h_experts[e]) return nullptr;
    switch (pick_kernel(path, M, h_experts, E)) {
        case 1: return "qgemm_stream_kernel";
        case 2: return "qgemm_decode_kernel";
        case 3: return "qgemm_dense_kernel";
        default: return "qgemm_tc_kernel";
    }
}

extern "C" moqe_status moqe_routed_qgemm_sorted(const void* X_bf16, const int32_t* perm, const int32_t* offsets, int M,
                                                const moqe_expert* const* h_experts, int E, void* Y_bf16, void* workspace,
                                                size_t workspace_bytes, void* stream, int path) {
    WsLayout w;
    int kernel = 0;
    bool done = false;
    moqe_status s = single_layer_args(X_bf16, perm, offsets, M, h_experts, E, Y_bf16, workspace, workspace_bytes, path, w, kernel, done);
    if (s != MOQE_OK || done) return s;
    return run_sorted(kernel, path, X_bf16, M, h_experts, E, Y_bf16, perm, offsets, (char*)workspace, w, (cudaStream_t)stream);
}

extern "C" moqe_status moqe_routed_qgemm_sorted_multi(const void* const* h_X_bf16, const int32_t* perm, const int32_t* offsets,
                                                      int M, int n_layers, const moqe_expert* const* h_experts, int E,
                                                      void* const* h_Y_bf16, void* workspace, size_t workspace_bytes,
                                                      void* stream) {
    if (!h_experts || !h_X_bf16 || !h_Y_bf16) return MOQE_ERR_NULL;
    if (E <= 0 || M < 0 || n_layers <= 0) return MOQE_ERR_SHAPE;
    if (n_layers * E > MOQE_MAX_EXPERTS) return MOQE_ERR_UNSUPPORTED;
    for (int l = 0; l < n_layers; ++l) {
        for (int e = 0; e < E; ++e)
            if (!h_experts[l * E + e]) return MOQE_ERR_NULL;
        const int N = h_experts[l * E]->N, K = h_experts[l * E]->K;
        for (int e = 1; e < E; ++e)
            if (h_experts[l * E + e]->N != N || h_experts[l * E + e]->K != K) return MOQE_ERR_MISMATCH;
        if (M > 0 && (!h_X_bf16[l] || !h_Y_bf16[l])) return MOQE_ERR_NULL;
        if (N % 8 != 0 || K % 8 != 0 || (uintptr_t)h_X_bf16[l] % 16 || (uintptr_t)h_Y_bf16[l] % 16) return MOQE_ERR_UNSUPPORTED;
    }
    if (M == 0) return MOQE_OK;
    if (!perm || !offsets) return MOQE_ERR_NULL;
    if (!decode_supported_multi(M, h_experts, n_layers, E)) return MOQE_ERR_UNSUPPORTED;
    WsLayout w = ws_layout(M, h_experts[0]->Np, h_experts[0]->K, E);
    if (!workspace || workspace_bytes < w.total || (uintptr_t)workspace % 256) return MOQE_ERR_WORKSPACE;
    char* base = (char*)workspace;
    return launch_qgemm_decode_multi(h_X_bf16, M, n_layers, h_experts, E, h_Y_bf16, perm, offsets, (uint32_t*)(base + w.counters),
                                     base + w.body, w.total - w.body, (cudaStream_t)stream);
}

namespace {
// shared argument checks of the decode-only fused entry points
moqe_status fused_args(const void* X, const int32_t* perm, const int32_t* offsets, int M, const moqe_expert* const* ex, int E,
                       const void* Y, void* workspace, size_t workspace_bytes, WsLayout& w) {
    if (!ex) return MOQE_ERR_NULL;
    if (E <= 0 || M < 0) return MOQE_ERR_SHAPE;
    if (E > MOQE_MAX_EXPERTS) return MOQE_ERR_UNSUPPORTED;
    for (int e = 0; e < E; ++e)
        if (!ex[e]) return MOQE_ERR_NULL;
    const int N = ex[0]->N, K = ex[0]->K;
    for (int e = 1; e < E; ++e)
        if (ex[e]->N != N || ex[e]->K != K) return MOQE_ERR_MISMATCH;
    if (M == 0) return MOQE_OK;
    if (!X || !perm || !offsets || !Y) return MOQE_ERR_NULL;
    if (N % 8 != 0 || K % 8 != 0 || (uintptr_t)X % 16 || (uintptr_t)Y % 16) return MOQE_ERR_UNSUPPORTED;
    if (!decode_supported_multi(M, ex, 1, E)) return MOQE_ERR_UNSUPPORTED;
    w = ws_layout(M, ex[0]->Np, K, E);
    if (!workspace || workspace_bytes < w.total || (uintptr_t)workspace % 256) return MOQE_ERR_WORKSPACE;
    return MOQE_OK;
}
}  // namespace

extern "C" moqe_status moqe_routed_qgemm_sorted_gated(const void* X_bf16, const int32_t* perm, const int32_t* offsets, int M,
                                                      const moqe_expert* const* h_gate, const moqe_expert* const* h_up, int E,
                                                      void* Y_bf16, void* workspace, size_t workspace_bytes, void* stream) {
    if (!h_up) return MOQE_ERR_NULL;
    WsLayout w;
    moqe_status s = fused_args(X_bf16, perm, offsets, M, h_gate, E, Y_bf16, workspace, workspace_bytes, w);
    if (s != MOQE_OK || M == 0) return s;
    for (int e = 0; e < E; ++e)
        if (!h_up[e]) return MOQE_ERR_NULL;
    char* base = (char*)workspace;
    return launch_qgemm_decode_ext(&X_bf16, M, 1, h_gate, h_up, E, &Y_bf16, nullptr, perm, offsets, (uint32_t*)(base + w.counters),
                                   base + w.body, w.total - w.body, (cudaStream_t)stream);
}

extern "C" moqe_status moqe_routed_qgemm_sorted_residual(const void* X_bf16, const int32_t* perm, const int32_t* offsets, int M,
                                                         const moqe_expert* const* h_experts, int E, const void* R_bf16,
                                                         void* Y_bf16, void* workspace, size_t workspace_bytes, void* stream) {
    WsLayout w;
    moqe_status s = fused_args(X_bf16, perm, offsets, M, h_experts, E, Y_bf16, workspace, workspace_bytes, w);
    if (s != MOQE_OK || M == 0) return s;
    if (!R_bf16) return MOQE_ERR_NULL;
    char* base = (char*)workspace;
    return launch_qgemm_decode_ext(&X_bf16, M, 1, h_experts, nullptr, E, &Y_bf16, &R_bf16, perm, offsets,
                                   (uint32_t*)(base + w.counters), base + w.body, w.total - w.body, (cudaStream_t)stream);
}

extern "C" moqe_status moqe_routed_qgemm_workspace_clear(void* workspace, size_t workspace_bytes, int M, int N, int K,
                                                         int E, void* stream) {
    if (M < 0 || N <= 0 || K <= 0 || E <= 0) return MOQE_ERR_SHAPE;
    const int Np = (N + 127) / 128 * 128;
    WsLayout w = ws_layout(M, Np, K, E);
    if (!workspace || workspace_bytes < w.total || (uintptr_t)workspace % 256) return MOQE_ERR_WORKSPACE;
    return cuda_ok(cudaMemsetAsync((char*)workspace + w.counters, 0, w.body - w.counters, (cudaStream_t)stream));
}

extern "C" moqe_status moqe_routed_qgemm(const void* X_bf16, const int32_t* row_ids, int M,
                                         const moqe_expert* const* h_experts, int E, void* Y_bf16, void* workspace,
                                         size_t workspace_bytes, void* stream) {
    return moqe_routed_qgemm_path(X_bf16, row_ids, M, h_experts, E, Y_bf16, workspace, workspace_bytes, stream, 0);
}

extern "C" moqe_status moqe_tune(const char* key, int value) {
    if (!key) return MOQE_ERR_NULL;
    if (!strcmp(key, "stream_tile_cost_w8")) { stream_set_tile_cost(8, value); return MOQE_OK; }
    if (!strcmp(key, "stream_tile_cost_w4")) { stream_set_tile_cost(4, value); return MOQE_OK; }
    if (!strcmp(key, "stream_tile_cost_w3")) { stream_set_tile_cost(3, value); return MOQE_OK; }
    if (!strcmp(key, "auto_decode")) { g_auto_decode = value != 0; return MOQE_OK; }
    if (!strcmp(key, "auto_dense")) { g_auto_dense = value != 0; return MOQE_OK; }
    if (!strcmp(key, "decode_tile_cost_w8")) { decode_set_tile_cost(8, value); return MOQE_OK; }
    if (!strcmp(key, "decode_tile_cost_w4")) { decode_set_tile_cost(4, value); return MOQE_OK; }
    if (!strcmp(key, "decode_tile_cost_w3")) { decode_set_tile_cost(3, value); return MOQE_OK; }
    return MOQE_ERR_UNSUPPORTED;
}

extern "C" moqe_status moqe_async_status(void* stream) {
    if (cudaStreamSynchronize((cudaStream_t)stream) != cudaSuccess) return MOQE_ERR_CUDA;
    int* w = device_status_word();
    if (!w) return MOQE_ERR_ALLOC;
    int v = 0;
    if (cudaMemcpy(&v, w, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return MOQE_ERR_CUDA;
    if (v != 0 && cudaMemset(w, 0, sizeof(int)) != cudaSuccess) return MOQE_ERR_CUDA;
    return (moqe_status)v;
}

namespace moqe {
namespace {
// One thread initialises an mbarrier on which nobody ever arrives and waits for it with the library's bounded wait.
__global__ void selftest_timeout_kernel(int* status, unsigned long long limit_ns, int* returned) {
    __shared__ unsigned long long bar;
    __shared__ int abort_flag;
    if (threadIdx.x == 0) {
        abort_flag = 0;
        mbar_init(smem_u32(&bar), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        const bool ok = mbar_wait_limit(smem_u32(&bar), 0u, &abort_flag, status, limit_ns);
        *returned = ok ? 1 : 2;
    }
}
}  // namespace
}  // namespace moqe

extern "C" moqe_status moqe_selftest_timeout(unsigned limit_us, int* d_returned, void* stream) {
    if (!d_returned) return MOQE_ERR_NULL;
    if (limit_us == 0 || limit_us > 1000000u) return MOQE_ERR_SHAPE;
    int* w = device_status_word();
    if (!w) return MOQE_ERR_ALLOC;
    selftest_timeout_kernel<<<1, 32, 0, (cudaStream_t)stream>>>(w, (unsigned long long)limit_us * 1000ull, d_returned);
    count_launch();
    return cuda_ok(cudaGetLastError());
}

extern "C" const char* moqe_status_str(moqe_status s) {
    switch (s) {
        case MOQE_OK: return "ok";
        case MOQE_ERR_NULL: return "a required pointer is NULL";
        case MOQE_ERR_SHAPE: return "bad or inconsistent size";
        case MOQE_ERR_UNSUPPORTED: return "unsupported format, size or alignment";
        case MOQE_ERR_ALLOC: return "device allocation failed";
        case MOQE_ERR_WORKSPACE: return "workspace missing, misaligned or too small";
        case MOQE_ERR_MISMATCH: return "experts disagree on N or K";
        case MOQE_ERR_CUDA: return "a CUDA call failed";
        case MOQE_ERR_EXPERT_ID: return "an expert id outside [0,E) was seen on the device";
        case MOQE_ERR_TIMEOUT: return "a bounded in-kernel wait ran out";
        case MOQE_ERR_IO: return "file missing, unreadable, unwritable or not a whole expert image";
    }
    return "unknown status";
}

extern "C" unsigned long long moqe_launch_count(void) { return g_launches.load(std::memory_order_relaxed); }
