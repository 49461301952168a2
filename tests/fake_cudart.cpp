// A stand-in for the CUDA runtime, linked with the library's own objects in place of it: the library's
// host code runs on a machine without a GPU.  Device memory is host memory, kernels are recorded and not
// run, and a test can make a call fail: an allocation past a budget, a device-side wait that gave up.
#include <cuda_runtime.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

#include "flow_internal.cuh"

namespace {
struct Block {
    size_t bytes;
    cudaMemoryType type;
};
struct Launch {
    std::string name;
    unsigned grid;
    ldpc::flow::Args flow;    // of a flow decoder's kernel
    ldpc::flow::Start start;  // and of the launch before it
};
std::map<char *, Block> g_mem;
std::map<const void *, std::string> g_names;
std::map<const void *, size_t> g_vars;
std::map<const void *, void *> g_var_mem;
std::vector<Launch> g_launches;
std::map<std::string, int> g_calls;
std::map<std::pair<int, const void *>, int> g_smem;  // (device, kernel) -> shared memory it may have
ldpc::flow::Start g_start;
long long g_budget = -1;  // bytes of device memory still to be had (-1: any)
int g_device = 0, g_capturing = 0, g_give_up = 0, g_refused = 0;
cudaError_t g_last = cudaSuccess;
struct {
    dim3 grid, block;
    size_t smem;
    cudaStream_t stream;
} g_config;

cudaError_t fail(cudaError_t e) { return g_last = e; }

cudaError_t launch(const void *fn, dim3 grid, size_t smem, void **args) {
    Launch l;
    l.name = g_names[fn];
    l.grid = grid.x;
    // more than 48 KB of shared memory has to be asked for, on each device
    if (smem > 48 * 1024 && (size_t)g_smem[{g_device, fn}] < smem) {
        ++g_refused;
        return fail(cudaErrorInvalidValue);
    }
    if (l.name.find("start_kernel") != std::string::npos) g_start = *(const ldpc::flow::Start *)args[0];
    if (l.name.find("tile_kernel") != std::string::npos && l.name.find("flow") != std::string::npos) {
        l.flow = *(const ldpc::flow::Args *)args[0];
        l.start = g_start;
        if (g_give_up) *l.flow.err = l.flow.err_tag | g_give_up, g_give_up = 0;
    }
    g_launches.push_back(l);
    return cudaSuccess;
}
}  // namespace

extern "C" {

// --- what a test sets and reads ------------------------------------------------------------------
void fake_reset() {
    g_launches.clear();
    g_calls.clear();
    g_budget = -1;
    g_device = g_capturing = g_give_up = g_refused = 0;
    g_last = cudaSuccess;
}
void *fake_alloc(long long n) {  // device memory of the test's own
    void *p = calloc(n ? n : 1, 1);
    g_mem[(char *)p] = {(size_t)n, cudaMemoryTypeDevice};
    return p;
}
void fake_free(void *p) {
    g_mem.erase((char *)p);
    free(p);
}
void fake_budget(long long bytes) { g_budget = bytes; }
void fake_device(int dev) { g_device = dev; }
void fake_capturing(int on) { g_capturing = on; }
void fake_give_up(int code) { g_give_up = code; }  // the next flow launch gives up a wait
int fake_refused() { return g_refused; }
int fake_calls(const char *name) { return g_calls[name]; }
int fake_launches() { return (int)g_launches.size(); }
const char *fake_launch_name(int i) { return g_launches[i].name.c_str(); }
long long fake_pinned_bytes() {
    long long n = 0;
    for (auto &m : g_mem) n += m.second.type == cudaMemoryTypeHost ? (long long)m.second.bytes : 0;
    return n;
}
// launch i, a flow decoder's: slots, packages, blocks, entries of the phase log, frames, check rows' and
// variables' tiles, syndrome tiles, whether it is a simulation or a streaming decode
void fake_flow(int i, long long *x) {
    const auto &a = g_launches[i].flow;
    const auto &st = g_launches[i].start;
    x[0] = a.W, x[1] = a.P, x[2] = a.blocks, x[3] = a.log_len;
    x[4] = a.sim ? (long long)st.sim.limit : st.code.gamma;
    x[5] = st.code.J * (long long)st.code.rch.d, x[6] = st.code.L * (long long)st.code.vch.d, x[7] = st.code.nsyn;
    x[8] = st.code.N, x[9] = a.sim != nullptr, x[10] = st.code.J;
}

// what a block makes of a log entry's place where it finds the words written for entries n0 and n1 and looks
// for entry n, with a tile of its own (entry_is, entry_whole); kind, package and slot of the entries: their numbers
int fake_entry_is(unsigned n0, unsigned n1, unsigned n) {
    const int is = ldpc::flow::entry_is(ldpc::flow::entry_w1(n1, (int)(n1 & 255), n1 % 152, n1 & 0xffffff), n);
    const auto w0 = ldpc::flow::entry_w0(n0, (int)(n0 % 7), 1, 99999, (int)(n0 & 0x3ffffff));
    return is == ldpc::flow::kEntryHere && !ldpc::flow::entry_whole(w0, n) ? (int)ldpc::flow::kEntryAhead : is;
}

// --- the runtime ---------------------------------------------------------------------------------
void **__cudaRegisterFatBinary(void *) {
    static void *h;
    return &h;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
char __cudaInitModule(void **) { return 1; }
void __cudaRegisterFunction(void **, const char *fn, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *,
                            int *) {
    g_names[fn] = name;
}
void __cudaRegisterVar(void **, char *var, char *, const char *, int, size_t size, int, int) { g_vars[var] = size; }
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, cudaStream_t s) {
    g_config = {grid, block, smem, s};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *s) {
    *grid = g_config.grid, *block = g_config.block, *smem = g_config.smem;
    *(cudaStream_t *)s = g_config.stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *fn) {
    *k = (cudaKernel_t)fn;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3, void **args, size_t smem, cudaStream_t) {
    return launch((const void *)k, grid, smem, args);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *fn, void **args) {
    return launch(fn, c->gridDim, c->dynamicSmemBytes, args);
}
cudaError_t cudaLaunchCooperativeKernel(const void *fn, dim3 grid, dim3, void **args, size_t smem, cudaStream_t) {
    return launch(fn, grid, smem, args);
}
cudaError_t cudaMalloc(void **p, size_t n) {
    ++g_calls["cudaMalloc"];
    *p = nullptr;
    if (g_capturing) return fail(cudaErrorStreamCaptureUnsupported);
    if (g_budget >= 0 && (long long)n > g_budget) return fail(cudaErrorMemoryAllocation);
    if (g_budget >= 0) g_budget -= (long long)n;
    *p = calloc(n ? n : 1, 1);
    g_mem[(char *)*p] = {n, cudaMemoryTypeDevice};
    return cudaSuccess;
}
static cudaError_t release(void *p) {
    if (!p) return cudaSuccess;
    g_mem.erase((char *)p);
    free(p);
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
    if (p) ++g_calls["cudaFree"];
    return release(p);
}
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) {
    ++g_calls["cudaHostAlloc"];
    if (g_capturing) return fail(cudaErrorStreamCaptureUnsupported);
    *p = calloc(n, 1);
    g_mem[(char *)*p] = {n, cudaMemoryTypeHost};
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void *p) { return release(p); }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *q) {
    std::memset(a, 0, sizeof(*a));
    char *p = (char *)q;
    auto f = g_mem.upper_bound(p);
    if (f != g_mem.begin() && p < (--f)->first + (f->second.bytes ? f->second.bytes : 1)) {
        a->type = f->second.type;
        a->devicePointer = a->hostPointer = p;
    }
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void **p, const void *var) {
    void *&m = g_var_mem[var];
    if (!m) m = calloc(g_vars[var], 1);
    *p = m;
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) {
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) {
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) {
    std::memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() {
    ++g_calls["cudaDeviceSynchronize"];
    return g_capturing ? fail(cudaErrorStreamCaptureUnsupported) : cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s) {
    *s = g_capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d) {
    *d = g_device;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : 1;
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *fn, cudaFuncAttribute a, int v) {
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) g_smem[{g_device, fn}] = v;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *, int, size_t) {
    *n = 1;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) {
    *n = 1;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *, const cudaLaunchConfig_t *c) {
    *n = 152 / (int)c->gridDim.x;  // one cluster asked about: a block an SM
    return cudaSuccess;
}
cudaError_t cudaGetLastError() {
    const cudaError_t e = g_last;
    g_last = cudaSuccess;
    return e;
}
const char *cudaGetErrorString(cudaError_t) { return "an error of the stand-in runtime"; }
cudaError_t cudaEventCreate(cudaEvent_t *e) {
    *e = (cudaEvent_t)1;
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) {
    *ms = 0.0f;
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
    *s = nullptr;
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaErrorNotSupported; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *) { return cudaErrorNotSupported; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *, cudaGraph_t, unsigned long long) { return cudaErrorNotSupported; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }

}  // extern "C"
