// A CUDA runtime without a GPU, for tests of what the assignment engine's host
// code does with device memory: allocations are host address ranges that are
// never handed out twice, copies are memcpy, kernels do not run (their launches
// are recorded).  Any allocation can be made to fail, and the next device-to-host
// copies of one or two words can be given their contents (what a kernel would have
// left there).
#include <cuda_runtime.h>
#include <sys/mman.h>

#include <cstdint>
#include <cstring>
#include <map>
#include <set>
#include <string>
#include <vector>

namespace {
std::map<uintptr_t, size_t> g_live;
std::set<uintptr_t> g_freed;
std::map<const void *, std::string> g_names;
long g_calls = 0, g_fail_at = 0, g_h2d = 0;
std::vector<std::pair<size_t, uint64_t>> g_reads;  // {bytes, value} of the next device-to-host copies
struct {
    dim3 grid, block;
    size_t smem;
    void *stream;
} g_cfg;
struct Launch {
    std::string name;
    int threads, blocks, live, freed;
    size_t smem;
};
std::vector<Launch> g_launches;
thread_local std::string g_error;

// pointer arguments of the kernels, as words to look through: td_trees* take one
// structure by value (its first 32 words), the others scalars and pointers
void count_pointers(const std::string &name, void **args, Launch &l) {
    const bool tree = name.find("td_trees") != std::string::npos;
    const int n_args = name.find("load_routes") != std::string::npos ? 10 : name.find("link_table") != std::string::npos ? 6 : 0;
    for (int i = 0; i < (tree ? 32 : n_args); i++) {
        uintptr_t p;
        std::memcpy(&p, tree ? static_cast<uint64_t *>(args[0]) + i : args[i], 8);
        l.live += (int)g_live.count(p);
        l.freed += (int)g_freed.count(p);
    }
}

// registers a thread, as the compiler reports them
int regs_of(const std::string &name) { return name.find("Li256ELi8E") != std::string::npos ? 32 : 56; }
constexpr size_t kStatic = 160, kReserved = 1024, kSmemSm = 233472, kSmemBlock = 232448;
}  // namespace

int lpsim_fail(int code, const std::string &msg) {
    g_error = msg;
    return code;
}

extern "C" {
const char *lpsim_last_error() { return g_error.c_str(); }
void fake_reset(long fail_at) {
    g_calls = 0;
    g_fail_at = fail_at;
    g_h2d = 0;
    g_reads.clear();
    g_launches.clear();
}
long fake_calls() { return g_calls; }
long fake_uploaded() { return g_h2d; }
long fake_live_bytes() {
    size_t t = 0;
    for (auto &a : g_live) t += a.second;
    return (long)t;
}
void fake_next_read(size_t bytes, uint64_t value) { g_reads.push_back({bytes, value}); }
int fake_launches() { return (int)g_launches.size(); }
const char *fake_launch(int i, int *out) {  // out: threads, blocks, live pointers, freed pointers, shared bytes
    const Launch &l = g_launches[i];
    const int v[5] = {l.threads, l.blocks, l.live, l.freed, (int)l.smem};
    std::memcpy(out, v, sizeof v);
    return l.name.c_str();
}
int fake_occupancy(int threads, int regs, size_t smem) {
    const size_t by_smem = kSmemSm / (smem + kStatic + kReserved), by_regs = 65536 / (regs * threads), by_thr = 2048 / threads;
    if (smem + kStatic > kSmemBlock) return 0;
    return (int)(by_smem < by_regs ? by_smem < by_thr ? by_smem : by_thr : by_regs < by_thr ? by_regs : by_thr);
}

cudaError_t cudaMalloc(void **p, size_t bytes) {
    *p = nullptr;
    if (++g_calls == g_fail_at) return cudaErrorMemoryAllocation;
    void *q = mmap(nullptr, bytes, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
    if (q == MAP_FAILED) return cudaErrorMemoryAllocation;
    *p = q;
    g_live[(uintptr_t)q] = bytes;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
    if (!p) return cudaSuccess;
    auto it = g_live.find((uintptr_t)p);
    if (it == g_live.end()) return cudaErrorInvalidValue;
    madvise(p, it->second, MADV_DONTNEED);  // the address stays taken
    g_freed.insert(it->first);
    g_live.erase(it);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind kind, cudaStream_t) {
    if (kind == cudaMemcpyHostToDevice) g_h2d += (long)n;
    if (kind == cudaMemcpyDeviceToHost && !g_reads.empty() && g_reads.front().first == n) {
        std::memcpy(d, &g_reads.front().second, n);
        g_reads.erase(g_reads.begin());
        return cudaSuccess;
    }
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) {
    std::memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d) { return *d = 0, cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { return *s = nullptr, cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? (int)kSmemBlock : 0;
    return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *a, const void *f) {
    std::memset(a, 0, sizeof *a);
    a->sharedSizeBytes = kStatic;
    a->numRegs = regs_of(g_names[f]);
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *f, int block, size_t smem, unsigned) {
    *n = fake_occupancy(block, regs_of(g_names[f]), smem);
    return cudaSuccess;
}

// what the compiler's host stubs call
void **__cudaRegisterFatBinary(void *) {
    static void *h;
    return &h;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) {
    g_names[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, struct CUstream_st *stream) {
    g_cfg = {grid, block, smem, stream};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *stream) {
    *grid = g_cfg.grid;
    *block = g_cfg.block;
    *smem = g_cfg.smem;
    *static_cast<void **>(stream) = g_cfg.stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) {
    *k = reinterpret_cast<cudaKernel_t>(const_cast<void *>(f));
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3 block, void **args, size_t smem, cudaStream_t) {
    Launch l{g_names[reinterpret_cast<const void *>(k)], (int)block.x, (int)grid.x, 0, 0, smem};
    count_pointers(l.name, args, l);
    g_launches.push_back(l);
    return cudaSuccess;
}
}
