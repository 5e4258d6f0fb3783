// Host logic of the library on a fake CUDA runtime (no GPU): the library's own objects linked with
// the runtime functions below, which keep "device" memory on the host and launch nothing, but
// record where every allocation, copy, clear and launch went.  Two devices.  A freed block is never
// reused, so a pointer into one is recognised.  Prints "ok" or the first check that failed.
//
// usage: fake_cuda_check <check>
#include <cuda_runtime_api.h>

#include <algorithm>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

#include "arrow.h"

// ---- the fake runtime ----------------------------------------------------------------------
namespace {
struct Block { char* p; size_t bytes; int dev; bool freed; };
struct Launch { std::string name; int dev; cudaStream_t stream; std::vector<char> arg0; };
struct Clear { char* p; size_t bytes; cudaStream_t stream; };
std::vector<Block> g_blocks;
std::vector<Launch> g_launches;
std::vector<Clear> g_clears;
std::map<const void*, std::string> g_names;
thread_local int g_dev = 0;
int g_fail_malloc = -1;        // the number of the cudaMalloc that fails from here on (0: the next)
int g_instantiated = 0;
constexpr size_t kArgBytes = 64;   // of a kernel's first argument that are kept (every argument struct is larger)

Block* find(const void* p) {
    for (Block& b : g_blocks)
        if (p >= b.p && p < b.p + b.bytes) return &b;
    return nullptr;
}
void record(const void* fn, void** args, cudaStream_t s) {
    Launch l{g_names.count(fn) ? g_names[fn] : "?", g_dev, s, {}};
    if (l.name.find("arrow_rows") != std::string::npos || l.name.find("arrow_batch") != std::string::npos ||
        l.name.find("arrow_fused") != std::string::npos || l.name.find("arrow_segments") != std::string::npos)
        l.arg0.assign(static_cast<char*>(args[0]), static_cast<char*>(args[0]) + kArgBytes);
    g_launches.push_back(l);
}
int g_token = 0;
template <class T>
cudaError_t token(T* out) {   // a handle that nobody dereferences
    *out = reinterpret_cast<T>(uintptr_t(++g_token) * 16);
    return cudaSuccess;
}
}  // namespace

extern "C" {
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* fn, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
    g_names[fn] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* fn) {
    *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(fn));
    return cudaSuccess;
}
struct Config { dim3 g, b; size_t smem; void* s; } g_config;
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, void* s) { g_config = {g, b, smem, s}; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* s) {
    *g = g_config.g; *b = g_config.b; *smem = g_config.smem;
    *static_cast<void**>(s) = g_config.s;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void** args, size_t, cudaStream_t s) {
    record(reinterpret_cast<const void*>(k), args, s);
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* fn, void** args) {
    record(fn, args, c->stream);
    return cudaSuccess;
}
cudaError_t cudaLaunchCooperativeKernel(const void* fn, dim3, dim3, void** args, size_t, cudaStream_t s) {
    record(fn, args, s);
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) { *d = g_dev; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { g_dev = d; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 8 : 1;
    return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t bytes) {
    if (g_fail_malloc >= 0 && g_fail_malloc-- == 0) return cudaErrorMemoryAllocation;
    char* q = static_cast<char*>(std::aligned_alloc(256, (bytes + 511) / 256 * 256));
    std::memset(q, 0, bytes);
    g_blocks.push_back({q, bytes, g_dev, false});
    *p = q;
    return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
    if (Block* b = find(p)) b->freed = true;
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t bytes, unsigned) { *p = std::calloc(1, bytes); return cudaSuccess; }
cudaError_t cudaFreeHost(void*) { return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
    std::memmove(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemset(void* p, int v, size_t n) { std::memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t s) {
    g_clears.push_back({static_cast<char*>(p), n, s});
    std::memset(p, v, n);
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void* symbol) { *p = const_cast<void*>(symbol); return cudaSuccess; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
    *f = nullptr;
    *q = cudaDriverEntryPointSymbolNotFound;
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "fake error"; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return token(e); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return token(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return token(s); }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { return token(g); }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) { ++g_instantiated; return token(e); }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
}

// ---- the checks ----------------------------------------------------------------------------
namespace {
#define CHECK(cond)                                                              \
    do {                                                                         \
        if (!(cond)) { std::printf("line %d: %s\n", __LINE__, #cond); return 1; } \
    } while (0)
#define OK(call)                                                                                                    \
    do {                                                                                                            \
        if (int rc_ = (call)) { std::printf("line %d: %s = %d (%s)\n", __LINE__, #call, rc_, arrow_last_error()); return 1; } \
    } while (0)

// A ring of n vertices with self-loops, each vertex also joined to `hubs` hubs (rows that are split).
arrow_handle make(int64_t n, int hubs, int device = -1) {
    std::vector<std::map<int32_t, double>> rows(n);
    for (int64_t v = 0; v < n; ++v)
        for (int64_t u : {v, (v + 1) % n, (v + n - 1) % n}) rows[v][int32_t(u)] = rows[u][int32_t(v)] = 1.0 + double(v % 3);
    for (int h = 0; h < hubs; ++h)
        for (int64_t v = 0; v < n; ++v) rows[v][h] = rows[h][int32_t(v)] = 0.5;
    std::vector<int64_t> rp{0};
    std::vector<int32_t> ci;
    std::vector<double> va;
    for (auto& r : rows) {
        for (auto& e : r) { ci.push_back(e.first); va.push_back(e.second); }
        rp.push_back(int64_t(ci.size()));
    }
    arrow_csr A{};
    A.n = n; A.nnz = int64_t(ci.size()); A.rowptr = rp.data(); A.colidx = ci.data(); A.values = va.data();
    arrow_opts o;
    arrow_opts_default(&o);
    o.device = device;
    o.nthreads = 1;
    arrow_handle h = nullptr;
    return arrow_decompose(&A, 16, &o, &h) == ARROW_OK ? h : nullptr;
}

char* buffer(size_t bytes) {
    void* p = nullptr;
    return cudaMalloc(&p, bytes) == cudaSuccess ? static_cast<char*>(p) : nullptr;
}

// The start of the rows kernel's argument.
struct RowArgsHead {
    const void *long_rowptr, *row_desc, *col, *val, *tile_row, *tile_ent;
    int32_t n_tiles;
};
bool live(const void* p) {
    Block* b = find(p);
    return b && !b->freed;
}

// No launch of a batch kernel since `from` has a descriptor that points into freed memory (the kernels'
// first argument starts with the pointer to the descriptors).
int stale_descriptors(size_t from) {
    int bad = 0;
    for (size_t i = from; i < g_launches.size(); ++i) {
        if (g_launches[i].name.find("arrow_batch") == std::string::npos) continue;
        char* d = nullptr;
        std::memcpy(&d, g_launches[i].arg0.data(), sizeof(d));
        const Block* b = find(d);
        if (!b || b->freed) { ++bad; continue; }
        for (size_t o = 0; o + 8 <= b->bytes; o += 8) {
            void* w = nullptr;
            std::memcpy(&w, b->p + o, 8);
            const Block* t = find(w);
            if (t && t->freed) ++bad;
        }
    }
    return bad;
}

// Calls of the one-launch path on one handle with workspaces of their own may overlap on the GPU, so nothing
// that a call writes apart from Y and the status word lies outside its workspace: the grid barrier's
// arrival count is cleared in the workspace, behind the segment partials and before the FP64 sums.
int own_barrier_count() {
    for (int hubs : {0, 3}) {
        arrow_handle h = make(900, hubs);
        CHECK(h);
        const arrow_tuning t{256, 2048, 4, 70, 0, 1};
        OK(arrow_set_tuning(h, &t));
        arrow_stats st;
        OK(arrow_get_stats(h, &st));
        CHECK((hubs > 0) == (st.segments > 0));
        for (int64_t k : {4, 64, 128})
            for (int flags : {0, ARROW_RESCALE}) {
                size_t bytes = 0;
                OK(arrow_workspace_size(h, k, ARROW_F32, flags, &bytes));
                const char *X = buffer(900 * k * 4), *last = nullptr;
                char* Y = buffer(900 * k * 4);
                for (int call = 0; call < 2; ++call) {
                    char* ws = buffer(bytes);
                    cudaStream_t s = reinterpret_cast<cudaStream_t>(uintptr_t(0x1000 + call));
                    g_clears.clear();
                    g_launches.clear();
                    OK(arrow_spmm_ws(h, X, k, 5, Y, ARROW_F32, flags, ws, bytes, s));
                    CHECK(g_launches.size() == 1 && g_launches[0].name.find("arrow_fused") != std::string::npos);
                    CHECK(g_launches[0].stream == s);
                    CHECK(g_clears.size() == 1 && g_clears[0].stream == s && g_clears[0].bytes == 4);
                    const char* c = g_clears[0].p;
                    CHECK(c != last);
                    last = c;
                    const size_t rows = size_t(900 * k * 4 + 255) / 256 * 256;
                    CHECK(c >= ws + 2 * rows + size_t(st.segments * k * 4) && c + 4 <= ws + bytes);
                    CHECK(uintptr_t(c) % 4 == 0);
                    // the FP64 sums of the rescale start at the next 256-byte boundary at the earliest
                    const size_t part = std::max(size_t(k * 4), size_t(st.segments * k * 4) + 4);
                    CHECK(c + 4 <= ws + 2 * rows + (part + 255) / 256 * 256);
                }
                // a workspace without room for the count still runs the call, kernel by kernel
                const size_t plain = 2 * (size_t(900 * k * 4 + 255) / 256 * 256) +
                                     (size_t(std::max<int64_t>(1, st.segments) * k * 4) + 255) / 256 * 256;
                if (!flags && plain < bytes) {
                    g_launches.clear();
                    OK(arrow_spmm_ws(h, X, k, 5, Y, ARROW_F32, flags, buffer(plain), plain, nullptr));
                    CHECK(g_launches.size() > 5);
                }
                CHECK(flags || arrow_spmm_ws(h, X, k, 5, Y, ARROW_F32, flags, buffer(plain), plain - 256, nullptr) == ARROW_EINVAL);
            }
        arrow_free(h);
    }
    return 0;
}

// A handle on a device that is not current is re-tuned on its own device, and the caller's device stays.
int tuned_on_its_device() {
    arrow_handle h = make(700, 2, 1);
    CHECK(h && g_dev == 0);
    const arrow_tuning shapes[] = {{512, 4096, 4, 70, 0, 0}, {512, 4096, 3, 70, 0, 0}, {64, 1024, 3, 50, 1, 0}};
    for (const arrow_tuning& t : shapes) {
        const size_t blocks = g_blocks.size();
        g_launches.clear();
        OK(arrow_set_tuning(h, &t));
        CHECK(g_dev == 0);
        for (size_t i = blocks; i < g_blocks.size(); ++i) CHECK(g_blocks[i].dev == 1);
        for (const Launch& l : g_launches) CHECK(l.dev == 1);
        arrow_tuning got;
        OK(arrow_get_tuning(h, &got));
        CHECK(std::memcmp(&got, &t, sizeof(t)) == 0);
    }
    // out of range is still refused, with the caller's device current
    const arrow_tuning bad{16, 4096, 3, 70, 0, 0};
    CHECK(arrow_set_tuning(h, &bad) == ARROW_EINVAL && g_dev == 0);
    return 0;
}

// A re-tuning that runs out of device memory leaves the handle as it was: its tuning, and tile tables
// and vertex-id columns that the next call can read.
int failed_retuning() {
    for (int fold : {0, 1})
        for (int fail = 0; fail < 6; ++fail) {
            arrow_handle h = make(700, 2);
            CHECK(h);
            arrow_tuning before, after;
            arrow_stats st, st2;
            OK(arrow_get_tuning(h, &before));
            OK(arrow_get_stats(h, &st));
            const arrow_tuning t{64, 1024, 3, 50, fold, 0};
            g_fail_malloc = fail;
            const int rc = arrow_set_tuning(h, &t);
            const bool failed = g_fail_malloc < 0;
            g_fail_malloc = -1;
            CHECK(rc == (failed ? ARROW_ENOMEM : ARROW_OK));
            OK(arrow_get_tuning(h, &after));
            CHECK(std::memcmp(&after, failed ? &before : &t, sizeof(after)) == 0);
            OK(arrow_get_stats(h, &st2));
            CHECK((st2.tiles == st.tiles) == failed);
            const char* X = buffer(700 * 16 * 4);
            char* Y = buffer(700 * 16 * 4);
            for (int again = 0; again < 2; ++again) {   // then with the tuning applied after all
                g_launches.clear();
                OK(arrow_spmm(h, X, 16, 2, Y, ARROW_F32, 0, nullptr));
                int rows = 0;
                for (const Launch& l : g_launches) {
                    if (l.name.find("arrow_rows") == std::string::npos) continue;
                    RowArgsHead a;
                    std::memcpy(&a, l.arg0.data(), sizeof(a));
                    CHECK(live(a.row_desc) && live(a.col) && live(a.val) && live(a.tile_row) && live(a.tile_ent));
                    const size_t table = size_t(a.n_tiles + 1) * 4;
                    CHECK(find(a.tile_row)->bytes >= table && find(a.tile_ent)->bytes >= table);
                    ++rows;
                }
                CHECK(rows == 2);
                for (const Launch& l : g_launches)
                    if (l.name.find("arrow_segments") != std::string::npos) {
                        const void* lcol = nullptr;   // SegArgs: seg_begin, seg_end, n_seg, lcol
                        std::memcpy(&lcol, l.arg0.data() + 24, sizeof(lcol));
                        CHECK(live(lcol));
                    }
                OK(arrow_set_tuning(h, &t));
                OK(arrow_get_stats(h, &st2));
                CHECK(st2.tiles != st.tiles);
            }
            arrow_free(h);
        }
    return 0;
}

// A batch made before a member is re-tiled walks the new tile tables, whatever part of the tuning
// changed, and captures its graph again.
int retiled_member() {
    arrow_handle h[2] = {make(700, 2), make(300, 0)};
    CHECK(h[0] && h[1]);
    arrow_batch B = nullptr;
    OK(arrow_batch_create(h, 2, &B));
    const int64_t k[2] = {8, 16};
    const void* X[2] = {buffer(700 * 8 * 4), buffer(300 * 16 * 4)};
    void* Y[2] = {buffer(700 * 8 * 4), buffer(300 * 16 * 4)};
    OK(arrow_batch_spmm(B, X, Y, k, 3, ARROW_F32, 0, nullptr));
    OK(arrow_batch_spmm(B, X, Y, k, 3, ARROW_F32, ARROW_GRAPH, nullptr));
    const arrow_tuning shapes[] = {{512, 4096, 4, 70, 0, 0}, {512, 2048, 4, 70, 0, 0}, {64, 2048, 4, 70, 0, 0},
                                   {64, 2048, 3, 70, 0, 0}, {64, 1024, 3, 50, 0, 0}};
    for (const arrow_tuning& t : shapes)
        for (arrow_handle m : h) {
            OK(arrow_set_tuning(m, &t));
            const size_t from = g_launches.size();
            const int graphs = g_instantiated;
            OK(arrow_batch_spmm(B, X, Y, k, 3, ARROW_F32, 0, nullptr));
            OK(arrow_batch_spmm(B, X, Y, k, 3, ARROW_F32, ARROW_GRAPH, nullptr));
            CHECK(g_launches.size() > from);
            CHECK(stale_descriptors(from) == 0);
            CHECK(g_instantiated == graphs + 1);
        }
    // the same tuning again changes nothing: the graph is replayed
    const int graphs = g_instantiated;
    OK(arrow_set_tuning(h[0], &shapes[4]));
    OK(arrow_batch_spmm(B, X, Y, k, 3, ARROW_F32, ARROW_GRAPH, nullptr));
    CHECK(g_instantiated == graphs);
    return 0;
}

}  // namespace

int main(int argc, char** argv) {
    const std::string which = argc > 1 ? argv[1] : "";
    const std::map<std::string, int (*)()> checks{
        {"retiled_member", retiled_member}, {"own_barrier_count", own_barrier_count}, {"tuned_on_its_device", tuned_on_its_device},
        {"failed_retuning", failed_retuning}};
    const auto it = checks.find(which);
    if (it == checks.end()) { std::printf("no check %s\n", which.c_str()); return 2; }
    const int rc = it->second();
    if (rc == 0) std::printf("ok\n");
    return rc;
}
