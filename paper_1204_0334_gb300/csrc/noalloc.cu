// ldpc_decode_noalloc: the block-code decoder for callers that cannot allocate
// device memory.
//
// Some callers cannot call cudaMalloc at decode time: code running inside a
// stream capture that must not add allocation nodes, real-time loops where a
// synchronous allocation would stall the pipeline, or hosts whose memory is
// fully reserved up front by another allocator.  For them the decoder's
// workspace lives in a fixed array compiled into this library (kNoallocBytes,
// 16 MiB, resident on every GPU that loads the library until the process
// exits).  The caller still passes its device input and output buffers.  A
// second array of 1.1 MB holds what the flow decoder schedules by.
//
// The arrays are static __device__ objects of this file.  In host code their
// names are only host-side stand-ins, so their device addresses are looked up
// once per device with cudaGetSymbolAddress (on the first call made with that
// device current) and handed to the kernels as plain pointers.  That call also
// allocates the pinned host words in which the flow decoder reports a wait that
// gave up.
//
// Every call uses the same array, which keeps whatever the previous call left:
// the decode steps initialize everything they read (the flag words and the
// hard-decision words are cleared at the start of every decode, channel LLRs
// and messages are written before they are read).  Two calls whose GPU work
// overlaps -- on two streams, or from two threads -- use the same memory and
// race; serialize them.
#include "flow_internal.cuh"

#include <algorithm>
#include <cstring>
#include <mutex>

namespace ldpc {

constexpr size_t kNoallocBytes = (size_t)16 << 20;

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoallocBytes];

// the flow decoder's slots, phase log and code (not part of the 16 MiB that bound a request)
static __device__ __align__(256) unsigned char g_noalloc_ctl[flow::kMaxSlots * sizeof(flow::Slot) + 256 +
                                                             flow::kMaxLog * sizeof(flow::Entry) + sizeof(flow::Code)];

namespace {
constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mu;
void *g_noalloc_ptr[kMaxDevices] = {}, *g_noalloc_ctl_ptr[kMaxDevices] = {};
constexpr int kErrWords = 1024;
int *g_noalloc_err[kMaxDevices] = {};  // pinned host words the flow decoder reports to, by the code's number

// device addresses of the scratch arrays on the current device (looked up once per device)
ldpc_status noalloc_base(void **out, void **ctl, int **err) {
    int dev = 0;
    LDPC_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) {
        set_error("device index %d out of range", dev);
        return LDPC_EUNSUPPORTED;
    }
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
        void *p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(g_noalloc_scratch)");
        e = cudaGetSymbolAddress(&g_noalloc_ctl_ptr[dev], g_noalloc_ctl);
        if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(g_noalloc_ctl)");
        e = cudaHostAlloc((void **)&g_noalloc_err[dev], kErrWords * sizeof(int), cudaHostAllocMapped);
        if (e != cudaSuccess) return cuda_fail(e, "cudaHostAlloc");
        std::memset(g_noalloc_err[dev], 0, kErrWords * sizeof(int));
        g_noalloc_ptr[dev] = p;
    }
    *out = g_noalloc_ptr[dev];
    *ctl = g_noalloc_ctl_ptr[dev];
    *err = g_noalloc_err[dev];
    return LDPC_OK;
}

size_t align256(size_t x) { return (x + 255) / 256 * 256; }
}  // namespace

// bytes of scratch a decode of gamma frames of code d needs (same buffers as the
// allocating path, rounded to 256-byte boundaries)
static size_t noalloc_need(const QcDesc &d, size_t cap, size_t *off) {
    const size_t P32 = cap / 32;
    size_t o = 0;
    off[0] = o; o += align256((size_t)d.E * cap * 4);   // msg
    off[1] = o; o += align256((size_t)d.N * cap * 4);   // mu
    off[2] = o; o += align256((size_t)d.N * cap * 4);   // post
    off[3] = o; o += align256((size_t)d.N * P32 * 4);   // hw
    off[4] = o; o += align256(P32 * 5 * 4);             // flags
    off[5] = o; o += align256(cap * 2 * 4);             // iters, ok
    off[6] = o; o += align256(8 * sizeof(unsigned long long));  // counters
    off[7] = o; o += align256((P32 + 1) * sizeof(int)); // active-package list
    return o;
}

}  // namespace ldpc

using namespace ldpc;

extern "C" {

ldpc_status ldpc_decode_noalloc(ldpc_code c, const float *llr, int32_t gamma, const ldpc_decode_opts *opts,
                                float *post, uint8_t *hard, int32_t *iters, int32_t *ok, void *stream) {
    if (!c || !llr || gamma < 1 || !opts) {
        set_error("need code, llr, opts and gamma >= 1");
        return LDPC_EINVAL;
    }
    if (pointer_kind(llr) != 0 || (post && pointer_kind(post) != 0) || (hard && pointer_kind(hard) != 0) ||
        (iters && pointer_kind(iters) != 0) || (ok && pointer_kind(ok) != 0)) {
        set_error("ldpc_decode_noalloc takes device buffers only (host buffers would need staging memory)");
        return LDPC_EINVAL;
    }
    ldpc_status st = check_opts(c, opts);
    if (st != LDPC_OK) return st;
    if (opts->algo == LDPC_ALGO_NOMS) {
        set_error("ldpc_decode_noalloc supports sum-product and min-sum");
        return LDPC_EUNSUPPORTED;
    }
    const ldpc_decode_opts o = *opts;
    const size_t cap = ((size_t)gamma + 127) / 128 * 128;
    size_t off[8];
    const size_t need = noalloc_need(c->d, cap, off);
    if (need > kNoallocBytes) {
        set_error("ldpc_decode_noalloc: %d frames of this code need %zu bytes of scratch; the fixed scratch holds "
                  "%zu bytes (about %zu frames of this code)", gamma, need, kNoallocBytes,
                  (size_t)(128.0 * (double)kNoallocBytes / (double)noalloc_need(c->d, 128, off)));
        return LDPC_EINVAL;
    }
    void *base_v = nullptr, *ctl = nullptr;
    int *err = nullptr;
    st = noalloc_base(&base_v, &ctl, &err);
    if (st != LDPC_OK) return st;
    // this code's word, and its number in it: another code may share the word, and is told for itself
    const int tag = (int)(c->number % (INT32_MAX / 8)) * 8;
    err += c->number % kErrWords;
    st = flow_gave_up(err, tag, "an earlier decode of this object in the fixed scratch");
    if (st != LDPC_OK) return st;
    noalloc_need(c->d, cap, off);
    unsigned char *base = (unsigned char *)base_v;
    cudaStream_t s = (cudaStream_t)stream;
    if (!c->sparse) {
        bool on_chip = false;
        st = chip_decode(c->d, llr, gamma, o, post, hard, iters, ok, s, &on_chip);
        if (st != LDPC_OK || on_chip) return st;
    }
    if (!c->sparse && flow_pays(c->d, gamma, o)) {
        // the slots' buffers one after another: a slot takes no more than its package's share of the
        // bytes counted above (the decision words' rounding fits in the iteration counts', not kept here)
        const int V = lanes_per_word(o.msg);
        size_t b[4], at[4], x = 0;
        flow_slot_bytes(c->d, o.msg, o.algo, post != nullptr, b);
        const int W = std::min((gamma + 32 * V - 1) / (32 * V), flow::kMaxSlots);
        for (int i = 0; i < 4; ++i) at[i] = x, x += b[i] * W;
        const FlowMem m{base + at[0], base + at[1], base + at[2], base + at[3], ctl, W, flow::kMaxLog, err, tag};
        return flow_decode(c->d, m, llr, gamma, o, post, hard, iters, ok, s);
    }
    // A private view of the code object whose workspace points into the scratch.  It
    // carries everything the decode steps read from a code: the QC description, and for
    // a general code the flag and the device index tables (which stay owned by c).  The
    // view is never passed to ldpc_code_destroy, the only place a workspace is freed.
    ldpc_code_s view;
    view.d = c->d;
    view.sparse = c->sparse;
    view.sp = c->sp;
    view.device = c->device;
    view.rate = c->rate;
    view.noms = nullptr;
    view.ws.gamma_cap = cap;
    view.ws.msg_bytes = (size_t)c->d.E * cap * 4;
    view.ws.msg = base + off[0];
    view.ws.mu = base + off[1];
    view.ws.post = (float *)(base + off[2]);
    view.ws.hw = (uint32_t *)(base + off[3]);
    view.ws.flags = (uint32_t *)(base + off[4]);
    view.ws.iters = (int32_t *)(base + off[5]);
    view.ws.counters = (unsigned long long *)(base + off[6]);
    view.ws.act = (int *)(base + off[7]);
    st = qc_pack_llr(&view, llr, gamma, o, s);
    if (st != LDPC_OK) return st;
    st = qc_decode_device(&view, gamma, o, post != nullptr, s);
    if (st != LDPC_OK) return st;
    return qc_unpack_outputs(&view, gamma, o, post, hard, iters, ok, s);
}

}  // extern "C"
