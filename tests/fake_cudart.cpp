// A CUDA runtime without a GPU, for tests of the library's host code: launches do nothing but are recorded,
// device memory is host memory that is kept track of, uploads from pageable memory are on their way until
// something waits for them, calls can be made to fail or to wait.  Linked with the library's objects by
// tests/test_host_fake_gpu.py.
#include <algorithm>
#include <condition_variable>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <set>
#include <string>
#include <thread>
#include <vector>

#include <cuda_runtime_api.h>

namespace {
std::mutex mu;
std::condition_variable cv;
std::map<const void*, std::string>& kernels() {
    static auto* m = new std::map<const void*, std::string>;
    return *m;
}
struct Launch {
    std::string name;
    uint64_t tables[2];  // the first words of a windowed kernel's second argument: its tables' addresses
    int teams[3];        // of encode_lanes_kernel's: threads a team, teams, input buffers a team
    unsigned grid, block;
    size_t shared;
    bool early;  // may start before the kernel in front has ended
};
std::vector<Launch> launches;
std::map<uintptr_t, size_t> memory;        // live allocations
std::map<uintptr_t, cudaStream_t> pending;  // uploads on their way, by destination
std::set<cudaStream_t> capturing;
std::vector<std::thread::id> freed_by;
cudaError_t fail_launch = cudaSuccess;
thread_local cudaError_t last_error = cudaSuccess;
bool hold_launch = false, hold_malloc = false;
int held = 0;

cudaError_t ret(cudaError_t e) {
    if (e != cudaSuccess) last_error = e;
    return e;
}
void wait_while(bool& flag, std::unique_lock<std::mutex>& lock) {
    if (!flag) return;
    ++held;
    cv.notify_all();
    cv.wait(lock, [&] { return !flag; });
    --held;
}
cudaError_t launch(const void* f, dim3 grid, dim3 block, void** args, size_t shared, bool early) {
    std::unique_lock<std::mutex> lock(mu);
    if (kernels()[f].find("code_window") != std::string::npos) wait_while(hold_launch, lock);
    if (fail_launch != cudaSuccess) return ret(fail_launch);
    Launch l{kernels()[f], {0, 0}, {0, 0, 0}, grid.x, block.x, shared, early};
    if (l.name.find("code_window") != std::string::npos) std::memcpy(l.tables, args[1], sizeof l.tables);
    if (l.name.find("encode_lanes") != std::string::npos) std::memcpy(l.teams, args[1], sizeof l.teams);
    launches.push_back(l);
    return cudaSuccess;
}
}  // namespace

extern "C" {
// ---- what the tests see
int fake_launches() { return static_cast<int>(launches.size()); }
const char* fake_launch_name(int i) { return launches[i].name.c_str(); }
uint64_t fake_launch_table(int i, int which) { return launches[i].tables[which]; }
int fake_launch_teams(int i, int which) { return launches[i].teams[which]; }
unsigned fake_launch_grid(int i) { return launches[i].grid; }
unsigned fake_launch_block(int i) { return launches[i].block; }
unsigned fake_launch_shared(int i) { return static_cast<unsigned>(launches[i].shared); }
int fake_launch_early(int i) { return launches[i].early; }
int fake_live(uint64_t p) {  // does p lie in live memory?
    std::lock_guard<std::mutex> lock(mu);
    auto it = memory.upper_bound(p);
    return it != memory.begin() && (--it, p < it->first + it->second);
}
int fake_allocations() {
    std::lock_guard<std::mutex> lock(mu);
    return static_cast<int>(memory.size());
}
int fake_uploads_pending() {
    std::lock_guard<std::mutex> lock(mu);
    return static_cast<int>(pending.size());
}
void fake_capture(cudaStream_t s, int on) {
    if (on) capturing.insert(s);
    else capturing.erase(s);
}
void fake_fail_launches(int e) { fail_launch = static_cast<cudaError_t>(e); }
void fake_hold(int launch_calls, int malloc_calls) {
    std::lock_guard<std::mutex> lock(mu);
    hold_launch = launch_calls, hold_malloc = malloc_calls;
    cv.notify_all();
}
int fake_wait_until_held(int seconds) {
    std::unique_lock<std::mutex> lock(mu);
    return cv.wait_for(lock, std::chrono::seconds(seconds), [] { return held > 0; });
}
void fake_forget_frees() { freed_by.clear(); }
int fake_frees_by_others() {  // frees by other threads than the caller
    int n = 0;
    for (auto id : freed_by) n += id != std::this_thread::get_id();
    return n;
}
int fake_frees() { return static_cast<int>(freed_by.size()); }
int fake_last_error() { return last_error; }

// ---- the runtime
void** __cudaRegisterFatBinary(void*) {
    static void* handle = nullptr;
    return &handle;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) { kernels()[host] = name; }
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
static thread_local struct {
    dim3 grid, block;
    size_t shared;
    void* stream;
} config;
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t shared, void* stream) {
    config = {grid, block, shared, stream};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* shared, void* stream) {
    *grid = config.grid, *block = config.block, *shared = config.shared;
    *static_cast<void**>(stream) = config.stream;
    return cudaSuccess;
}
cudaError_t cudaLaunchKernel(const void* f, dim3 grid, dim3 block, void** args, size_t shared, cudaStream_t) {
    return launch(f, grid, block, args, shared, false);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) {
    bool early = false;
    for (unsigned i = 0; i < c->numAttrs; ++i)
        early = early || (c->attrs[i].id == cudaLaunchAttributeProgrammaticStreamSerialization && c->attrs[i].val.programmaticStreamSerializationAllowed);
    return launch(f, c->gridDim, c->blockDim, args, c->dynamicSmemBytes, early);
}
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 148 : 232448;
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
// (64 registers a thread)
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int threads, size_t shared) {
    return *n = static_cast<int>(std::min<size_t>(1024 / threads, 233472 / (shared + 1024))), cudaSuccess;
}
cudaError_t cudaGetLastError() {
    const cudaError_t e = last_error;
    last_error = cudaSuccess;
    return e;
}
cudaError_t cudaMalloc(void** p, size_t n) {
    std::unique_lock<std::mutex> lock(mu);
    wait_while(hold_malloc, lock);
    *p = std::aligned_alloc(256, (n + 255) & ~size_t(255));
    memory[reinterpret_cast<uintptr_t>(*p)] = n;
    return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
    std::lock_guard<std::mutex> lock(mu);
    if (!p) return cudaSuccess;
    freed_by.push_back(std::this_thread::get_id());
    memory.erase(reinterpret_cast<uintptr_t>(p));
    pending.erase(reinterpret_cast<uintptr_t>(p));
    std::free(p);
    return cudaSuccess;
}
static cudaError_t upload(void* d, const void* s, size_t n, cudaStream_t stream) {
    std::lock_guard<std::mutex> lock(mu);
    std::memcpy(d, s, n);
    pending[reinterpret_cast<uintptr_t>(d)] = stream;  // staged; on its way
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { return upload(d, s, n, nullptr); }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t st) { return upload(d, s, n, st); }
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
    std::lock_guard<std::mutex> lock(mu);
    for (auto it = pending.begin(); it != pending.end();) it = it->second == s ? pending.erase(it) : std::next(it);
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() {
    std::lock_guard<std::mutex> lock(mu);
    pending.clear();
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
    *s = reinterpret_cast<cudaStream_t>(std::malloc(16));
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) {
    std::free(s);
    return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus* st) {
    *st = capturing.count(s) ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode*) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) {
    *e = reinterpret_cast<cudaEvent_t>(std::malloc(16));
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void* symbol) { return *p = const_cast<void*>(symbol), cudaSuccess; }
}
