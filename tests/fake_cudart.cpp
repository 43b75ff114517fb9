// A CUDA runtime for tests of the host code, without a GPU.
//
// Device memory is host memory filled with a pattern.  Copies and memsets wait
// in their stream until it is waited for and are then carried out; a kernel does
// nothing but advance the clock that events record (a unit each, and another
// cost by name through fake_kernel_cost).  The runtime counts misuse (memory
// given back or freed while another stream still has work queued on it), refuses
// the allocations that a test names, and holds memory up to a capacity, to which
// freed memory kept in a pool counts.
#include <cuda_runtime_api.h>

#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <deque>
#include <functional>
#include <map>
#include <set>
#include <string>
#include <utility>
#include <vector>

namespace {

struct Op {
    const char* at[2];  // the ranges it writes and reads
    size_t bytes;
    std::function<void()> run;
};
struct Stream {
    std::deque<Op> ops;
};
struct Event {
    Stream* on = nullptr;
    double at = 0.0;
};
struct Pool {
    uint64_t keep = 0;
    size_t used = 0, held = 0;  // bytes handed out; bytes taken from the device
};
struct Block {
    size_t bytes;
    Pool* pool;
};

Stream g_null;
std::set<Stream*> g_streams{&g_null};
std::map<const char*, Block> g_blocks;
std::set<Pool*> g_pools;
std::map<std::string, double> g_cost;
struct Result {  // what a kernel is to leave behind: a word at an offset of one of its arguments
    std::string kernel;
    int arg;
    size_t offset;
    uint32_t value;
};
std::vector<Result> g_results;
std::map<std::string, unsigned> g_grid;  // blocks of each kernel's last launch
cudaError_t g_last = cudaSuccess;
size_t g_capacity = SIZE_MAX, g_direct = 0;
double g_clock = 0.0;
int g_refuse = 0, g_allocs = 0, g_misuse = 0;

// (filled while the library is loaded, perhaps before this file's own variables exist)
std::map<const void*, std::string>& kernels() {
    static std::map<const void*, std::string> k;
    return k;
}
cudaError_t error(cudaError_t e) {
    if (e != cudaSuccess) g_last = e;
    return e;
}
Stream* stream_of(cudaStream_t s) { return s ? reinterpret_cast<Stream*>(s) : &g_null; }
void drain(Stream* s) {
    while (!s->ops.empty()) {
        Op op = std::move(s->ops.front());
        s->ops.pop_front();
        op.run();
    }
}
void drain_all() {
    for (Stream* s : g_streams) drain(s);
}
void queue(cudaStream_t s, const void* to, const void* from, size_t bytes, std::function<void()> run) {
    stream_of(s)->ops.push_back({{static_cast<const char*>(to), static_cast<const char*>(from)}, bytes, std::move(run)});
}
bool in_use(const char* lo, const char* hi, const Stream* except) {
    for (Stream* s : g_streams)
        if (s != except)
            for (const Op& op : s->ops)
                for (const char* p : op.at)
                    if (p < hi && lo < p + op.bytes) return true;
    return false;
}
size_t taken() {
    size_t n = g_direct;
    for (Pool* p : g_pools) n += p->held;
    return n;
}
void release_pools() {
    for (Pool* p : g_pools)
        if (p->held > p->used) p->held = p->used > p->keep ? p->used : (p->held < p->keep ? p->held : p->keep);
}
cudaError_t take(void** out, size_t bytes, Pool* pool) {
    *out = nullptr;
    if (g_refuse > 0 && --g_refuse == 0) return error(cudaErrorMemoryAllocation);
    const size_t kept = pool ? pool->held - pool->used : 0, more = bytes > kept ? bytes - kept : 0;
    if (more > g_capacity - taken()) return error(cudaErrorMemoryAllocation);
    char* p = static_cast<char*>(std::malloc(bytes ? bytes : 1));
    std::memset(p, 0x5a, bytes);
    g_blocks[p] = {bytes, pool};
    if (pool) {
        pool->used += bytes;
        pool->held += more;
    } else {
        g_direct += bytes;
    }
    ++g_allocs;
    *out = p;
    return cudaSuccess;
}
void give_back(void* at, const Stream* on) {
    auto it = g_blocks.find(static_cast<char*>(at));
    if (it == g_blocks.end()) {
        ++g_misuse;
        return;
    }
    const char* p = it->first;
    if (in_use(p, p + it->second.bytes, on)) ++g_misuse;
    drain_all();  // (the copies still find their memory: a test reads the count)
    if (it->second.pool) it->second.pool->used -= it->second.bytes;
    else g_direct -= it->second.bytes;
    std::free(at);
    g_blocks.erase(it);
}
void launch(const void* f, dim3 grid, void** args, cudaStream_t s) {
    const std::string name = kernels().count(f) ? kernels()[f] : "";
    double cost = 1.0;
    for (const auto& c : g_cost)
        if (name.find(c.first) != std::string::npos) cost = c.second;
    g_grid[name] = grid.x;
    std::vector<std::pair<char*, uint32_t>> writes;
    for (const Result& r : g_results)
        if (name.find(r.kernel) != std::string::npos) writes.emplace_back(*static_cast<char**>(args[r.arg]) + r.offset, r.value);
    queue(s, nullptr, nullptr, 0, [cost, writes] {
        g_clock += cost;
        for (const auto& w : writes) std::memcpy(w.first, &w.second, 4);
    });
}

struct Config {
    dim3 grid, block;
    size_t shared;
    cudaStream_t stream;
};
std::vector<Config> g_config;

}  // namespace

extern "C" {

// ---- for the tests
void fake_refuse_allocation(int which) { g_refuse = which; }  // the which-th from now on; 0: none
void fake_capacity(size_t bytes) { g_capacity = bytes; }
void fake_kernel_cost(const char* part, double units) { g_cost[part] = units; }
void fake_result(const char* part, int arg, size_t offset, uint32_t value) { g_results.push_back({part, arg, offset, value}); }
void fake_no_results() { g_results.clear(); }
unsigned fake_grid(const char* part) {
    for (const auto& g : g_grid)
        if (g.first.find(part) != std::string::npos) return g.second;
    return 0;
}
int fake_allocations() { return g_allocs; }
int fake_misuse() { return g_misuse; }
size_t fake_bytes_live() {
    size_t n = 0;
    for (const auto& b : g_blocks) n += b.second.bytes;
    return n;
}
size_t fake_pool_bytes() {  // handed out from pools
    size_t n = 0;
    for (Pool* p : g_pools) n += p->used;
    return n;
}
int fake_pending() {  // copies, memsets and kernels not yet carried out
    size_t n = 0;
    for (Stream* s : g_streams) n += s->ops.size();
    return (int)n;
}
size_t fake_bytes_taken() { return taken(); }

// ---- registration and launches
void** __cudaRegisterFatBinary(void*) {
    static void* handle;
    return &handle;
}
void __cudaRegisterFatBinaryEnd(void**) {}
char __cudaInitModule(void**) { return 1; }
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
    kernels()[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t shared, void* stream) {
    g_config.push_back({grid, block, shared, static_cast<cudaStream_t>(stream)});
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* shared, void* stream) {
    *grid = g_config.back().grid;
    *block = g_config.back().block;
    *shared = g_config.back().shared;
    *static_cast<cudaStream_t*>(stream) = g_config.back().stream;
    g_config.pop_back();
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
    *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(f));
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3, void** args, size_t, cudaStream_t s) {
    launch(k, grid, args, s);
    return cudaSuccess;
}
cudaError_t cudaLaunchKernel(const void* f, dim3 grid, dim3, void** args, size_t, cudaStream_t s) {
    launch(f, grid, args, s);
    return cudaSuccess;
}
cudaError_t cudaLaunchCooperativeKernel(const void* f, dim3 grid, dim3, void** args, size_t, cudaStream_t s) {
    launch(f, grid, args, s);
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) {
    launch(f, c->gridDim, args, c->stream);
    return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) {
    std::memset(a, 0, sizeof(*a));
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
    *n = 4;
    return cudaSuccess;
}

// ---- device
cudaError_t cudaGetDevice(int* d) {
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : (a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448 : 1);
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() {
    drain_all();
    release_pools();
    return cudaSuccess;
}
cudaError_t cudaGetLastError() { return std::exchange(g_last, cudaSuccess); }

// ---- memory
cudaError_t cudaMalloc(void** p, size_t bytes) { return take(p, bytes, nullptr); }
cudaError_t cudaFree(void* p) {
    if (!p) return cudaSuccess;
    drain_all();
    give_back(p, nullptr);
    return cudaSuccess;
}
cudaError_t cudaMallocHost(void** p, size_t bytes) {
    *p = std::malloc(bytes);
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) {
    drain_all();
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
    *p = nullptr;
    return error(cudaErrorInvalidSymbol);
}
cudaError_t cudaMemPoolCreate(cudaMemPool_t* out, const cudaMemPoolProps*) {
    Pool* p = new Pool();
    g_pools.insert(p);
    *out = reinterpret_cast<cudaMemPool_t>(p);
    return cudaSuccess;
}
cudaError_t cudaMemPoolDestroy(cudaMemPool_t p) {
    g_pools.erase(reinterpret_cast<Pool*>(p));
    delete reinterpret_cast<Pool*>(p);
    return cudaSuccess;
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t p, cudaMemPoolAttr a, void* v) {
    if (a == cudaMemPoolAttrReleaseThreshold) reinterpret_cast<Pool*>(p)->keep = *static_cast<uint64_t*>(v);
    return cudaSuccess;
}
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t p, size_t least) {
    Pool* pool = reinterpret_cast<Pool*>(p);
    if (pool->held > pool->used) pool->held = pool->used > least ? pool->used : (pool->held < least ? pool->held : least);
    return cudaSuccess;
}
cudaError_t cudaMallocFromPoolAsync(void** p, size_t bytes, cudaMemPool_t pool, cudaStream_t) {
    return take(p, bytes, reinterpret_cast<Pool*>(pool));
}
cudaError_t cudaFreeAsync(void* p, cudaStream_t s) {
    give_back(p, stream_of(s));
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* to, const void* from, size_t bytes, cudaMemcpyKind kind, cudaStream_t s) {
    if (kind == cudaMemcpyHostToDevice) {  // pageable: the source has been read when the call returns
        std::vector<char> copy(static_cast<const char*>(from), static_cast<const char*>(from) + bytes);
        queue(s, to, nullptr, bytes, [to, copy] { std::memcpy(to, copy.data(), copy.size()); });
    } else {
        queue(s, to, from, bytes, [to, from, bytes] { std::memmove(to, from, bytes); });
    }
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void* to, const void* from, size_t bytes, cudaMemcpyKind) {
    drain_all();
    std::memmove(to, from, bytes);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* at, int value, size_t bytes, cudaStream_t s) {
    queue(s, at, nullptr, bytes, [at, value, bytes] { std::memset(at, value, bytes); });
    return cudaSuccess;
}

// ---- streams and events
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
    Stream* n = new Stream();
    g_streams.insert(n);
    *s = reinterpret_cast<cudaStream_t>(n);
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) {
    drain(stream_of(s));
    g_streams.erase(stream_of(s));
    delete stream_of(s);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
    drain(stream_of(s));
    release_pools();
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) {
    *e = reinterpret_cast<cudaEvent_t>(new Event());
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t e) {
    drain_all();
    delete reinterpret_cast<Event*>(e);
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
    Event* ev = reinterpret_cast<Event*>(e);
    ev->on = stream_of(s);
    queue(s, nullptr, nullptr, 0, [ev] { ev->at = g_clock; });
    return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t e) {
    if (reinterpret_cast<Event*>(e)->on) drain(reinterpret_cast<Event*>(e)->on);
    return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t e, unsigned) { return cudaEventSynchronize(e); }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t a, cudaEvent_t b) {
    *ms = (float)(reinterpret_cast<Event*>(b)->at - reinterpret_cast<Event*>(a)->at);
    return cudaSuccess;
}

// ---- graphs: none
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return error(cudaErrorNotSupported); }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t*) { return error(cudaErrorNotSupported); }
cudaError_t cudaGraphCreate(cudaGraph_t*, unsigned) { return error(cudaErrorNotSupported); }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t*, cudaGraph_t, unsigned long long) { return error(cudaErrorNotSupported); }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return error(cudaErrorNotSupported); }
cudaError_t cudaGraphConditionalHandleCreate(cudaGraphConditionalHandle*, cudaGraph_t, unsigned, unsigned) {
    return error(cudaErrorNotSupported);
}
cudaError_t cudaGraphAddNode(cudaGraphNode_t*, cudaGraph_t, const cudaGraphNode_t*, const cudaGraphEdgeData*, size_t,
                             cudaGraphNodeParams*) {
    return error(cudaErrorNotSupported);
}

}  // extern "C"
