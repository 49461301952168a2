// The flow decoder: Algorithm 1 on a batch of frames in one persistent launch.
//
// A decode as a sequence of launches (check pass, variable pass, syndrome, list of running
// packages, thirty times) streams the whole message store through HBM in every pass, leaves the
// chip idle between passes, and launches all iterations whether or not a frame still runs.  Here
// blocks work through tiles: a tile is a few check rows of one package, a few variables, some rows
// of its syndrome, or a piece of the transposes in and out.
//
//  * W packages are in work at a time, each in a slot with its own message, channel-LLR and decision
//    buffers; W is chosen so that the slots' buffers stay in L2, where an in-place copy runs at
//    6.2 TB/s each way against 3.3 through HBM.  A slot whose package is finished takes the next one.
//  * A slot is in one phase: pack the LLRs, check step, variable step, syndrome, output.  Whoever
//    finishes the last tile of a phase opens the slot's next phase: it appends an entry to a log that
//    every block reads.  An entry says how many tiles were opened before it, and tile i of it goes to
//    block (that + i) mod blocks, so the blocks share the tiles evenly without an atomic per tile
//    (handing tiles out by atomics: 3200 cycles a tile in the block's serial part).  With several
//    packages in work the chip stays full through phase ends, and a package stops the moment its
//    frames have.
//  * No tile waits for another, but a phase ends with the last of its tiles, whichever block it fell
//    to: the launch is cooperative, so its blocks (one an SM) are all resident even where another
//    stream's kernel holds SMs.  Every wait has a limit, after which the launch ends and the object
//    reports a timeout.
//  * Within a block, one warp reads the log and starts the bulk copies of its tiles' lines (the rows
//    of a tile meet each circulant in one run of consecutive edges, or two at its wrap: a copy and an
//    address per slot of all the tile's rows, not per edge); 24 warps compute out of shared memory and
//    in place (a row, or a variable, per warp, a frame, or two, or four, per lane); a warp per stage
//    stores the results by bulk copies and counts the tile done once they have landed.
//
// Three stages of 72 KB: a tile arrives while another is computed and a third leaves.  What bounds it
// (n = 18360, FP32, 2048 frames, 30 iterations): the compute warps, 5500 cycles a check tile and 3600
// a variable tile of the 5400 a tile takes on average (66 warp instructions per edge and iteration in all,
// the waiting warps' among them, at 65 % of the issue slots; 1.4 TB/s of the lines are written back to HBM
// although they are read from L2).  15.2 ms before, 11.6 now; the n = 15168 integer min-sum with early
// stop, 4096 frames: 3.18 -> 1.90 ms; 40 frames of the n = 18360 code with early stop: 749 -> 250 us
// (the launches of all 30 iterations are gone); an irregular n = 2532 code, 1000 frames: 886 -> 375 us.
//
// A launch holds every SM until it ends, so long calls are several launches (launch_frames).
//
// Refill mode (the simulation with a frame-error target that cannot be met, and the streaming decode):
// every lane of a slot is a frame slot.  A step of a package is three phases: the syndrome, after which
// frames leave and the next ones enter; the check step with tiles that count wrong bits (or write
// decision rows) and tiles that draw (or read) the new frames' channel LLRs into the slot's lines; the
// variable step.  As many slots as L2 holds give the same counts as the caller's number of slots, since
// a frame's result does not depend on the others.  n = 18360, 32768 frames at 3.5 dB: FP32 68.4 -> 58.9
// ms, FP16 59.8 -> 47.5 ms; the compute warps have a tile 78 % of the time (FP32), the rest is the phases'
// latency at the eight packages that fit.
//
// The arithmetic is that of the pass kernels (qc_pipe.cu), operation by operation.
#include "flow_internal.cuh"

#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <mutex>
#include <new>
#include <utility>

namespace ldpc {
namespace flow {

int resident_blocks(const void *kernel, size_t smem) {
    static std::mutex mu;
    static std::map<std::pair<int, const void *>, int> blocks;  // by device (each has to be asked for the memory)
    int dev = 0, sms = 0, bps = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lk(mu);
    const auto key = std::make_pair(dev, kernel);
    auto f = blocks.find(key);  // each kernel has one shared-memory size
    if (f != blocks.end()) return f->second;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, kernel, kThreads, smem);
    cudaGetLastError();
    try {
        blocks.emplace(key, bps * sms);
    } catch (const std::bad_alloc &) {
    }
    return bps * sms;
}

// rows and variables of a tile by the code's degrees and the storage (as Cfg in flow.cuh)
static void tile_sizes(const QcDesc &d, int FV, int *rows, int *rows1, int *kc) {
    *rows = tile_rows(d.J, d.L);
    *rows1 = *rows / FV;
    *kc = d.J <= 4 ? 4 * kComputeWarps : 2 * kComputeWarps;
}

static uint32_t fill_code(const QcDesc &d, int FV, Code &c) {
    std::memset(&c, 0, sizeof(c));
    int rows, rows1, kc;
    tile_sizes(d, FV, &rows, &rows1, &kc);
    c.J = d.J, c.L = d.L, c.p = d.p, c.N = d.N, c.M = d.M;
    // tiles of equal size within a column, in multiples of four variables
    const int vch = (d.p + kc - 1) / kc;
    c.kc = std::min(kc, ((d.p + vch - 1) / vch + 3) / 4 * 4);
    c.nsyn = (d.M + kSynRows - 1) / kSynRows;
    c.divp = fast_div((uint32_t)d.p);
    c.rch = fast_div((uint32_t)((d.p + rows - 1) / rows));
    c.rch1 = fast_div((uint32_t)((d.p + rows1 - 1) / rows1));
    c.vch = fast_div((uint32_t)((d.p + c.kc - 1) / c.kc));
    std::memcpy(c.sh, d.shift, sizeof(int) * d.J * d.L);
    std::memcpy(c.eo, d.eoff, sizeof(int) * d.J * d.L);
    return std::max(c.J * c.rch1.d + (uint32_t)c.nsyn, c.L * c.vch.d);  // tiles of the largest phase
}

// the code's entry, an empty log, every slot with its first package and its pack phase open; the
// log by all blocks, the rest by the first
constexpr int kStartEntries = 4096;  // entries a block
__global__ void __launch_bounds__(1024) start_kernel(const Start st, const Args a) {
    const int kind = a.sim ? F_SYN : F_PACK;
    for (int n = blockIdx.x * blockDim.x + threadIdx.x; n < a.log_len; n += gridDim.x * blockDim.x) {
        Entry e;
        if (n < a.W) {
            e.w0 = entry_w0((uint32_t)n, kind, 0, a.sim ? 0 : 1, a.sim ? 0 : n);
            e.w1 = entry_w1((uint32_t)n, n, (uint32_t)(((long long)n * st.tiles) % a.blocks), (uint32_t)st.tiles);
        } else {
            const uint32_t before = (uint32_t)(n - a.log_len);  // the sequence number of the lap before
            e.w0 = entry_w0(before, 0, 0, 0, 0);
            e.w1 = entry_w1(before, 0, 0u, 0u);
        }
        a.log[n] = e;
    }
    if (blockIdx.x) return;
    const int *src = reinterpret_cast<const int *>(&st.code);
    int *dst = reinterpret_cast<int *>(a.code);
    const int V = st.V;
    if (a.sim) {
        if (threadIdx.x == 0) *a.sim = st.sim;
        for (int i = threadIdx.x; i < a.W * 128; i += blockDim.x) {
            a.simslots[i / 128].age[i % 128] = 0;
            a.simslots[i / 128].errs[i % 128] = 0;
            if (i % 128 == 0) a.simslots[i / 128].from = a.simslots[i / 128].to = 0ull;
        }
    }
    for (int i = threadIdx.x; i < (int)(sizeof(Code) / 4); i += blockDim.x) dst[i] = src[i];
    if (threadIdx.x == 0) {
        a.ctl->tail = ((unsigned long long)a.W << 40) | ((unsigned long long)a.W * st.tiles);
        a.ctl->next = a.W;
        a.ctl->live = a.W;
        a.ctl->abort = 0;
    }
    const int s = threadIdx.x;
    if (s >= a.W) return;
    Slot &sl = a.slots[s];
    sl.all = 0;
    sl.done = sl.syn_done = 0u;
    for (int v = 0; v < V; ++v) {
        uint32_t valid = 0u;
        for (int ln = 0; ln < 32; ++ln)
            if ((s * 32 + ln) * V + v < st.code.gamma) valid |= 1u << ln;
        sl.dn[v] = a.sim ? 0xffffffffu : ~valid;  // refill mode: no lane has a frame yet
        sl.un[v] = 0u;
    }
}

ldpc_status start(const Args &a, const Start &st, cudaStream_t s) {
    start_kernel<<<(a.log_len + kStartEntries - 1) / kStartEntries, 1024, 0, s>>>(st, a);
    count_launch();
    LDPC_CUDA_TRY(cudaGetLastError());
    return LDPC_OK;
}

}  // namespace flow

using namespace flow;

size_t flow_ctl_bytes(int W, int log_cap) {
    return (size_t)W * sizeof(Slot) + 256 + (size_t)log_cap * sizeof(Entry) + sizeof(Code);
}

// blocks a launch may have on this device (one an SM)
static int flow_blocks() {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return std::max(1, std::min(sms, 1 << kLogBase));
}

void flow_slot_bytes(const QcDesc &d, int msg, int algo, bool post, size_t *b4) {
    const int V = lanes_per_word(msg), FV = algo == LDPC_ALGO_MS ? 1 : V;
    b4[0] = (size_t)d.E * 128;
    b4[1] = (size_t)d.N * 128 * FV;
    b4[2] = post ? (size_t)d.N * 128 * V : 0;
    b4[3] = ((size_t)d.N * V * 4 + 127) / 128 * 128;
}

// L2 the slots' buffers may take: reads of a resident buffer keep their full rate up to about
// 110 MB on this chip (20 TB/s, 13 at 120 MB, 8 past L2)
constexpr size_t kL2Budget = (size_t)96 << 20;

int flow_slots(const QcDesc &d, int msg, int algo, bool post, int P) {
    size_t b[4];
    flow_slot_bytes(d, msg, algo, post, b);
    const size_t one = b[0] + b[1] + b[2] + b[3];
    const size_t fit = kL2Budget / one;
    return (int)std::min<size_t>({(size_t)P, (size_t)kMaxSlots, std::max<size_t>(fit, 4)});
}

// Codes of fewer edges fill a tile badly: a phase has few tiles, each with its fixed cost (2500 cycles).
constexpr int kShortCode = 8000;

// The simulation's frames through flow slots or through launches on all slots (the counts are the
// same): measured on 4 frames a slot, launches / flow, FP32: 3 x 6, p = 64, 1024 slots 1811 / 1208 us,
// 4096 slots 2528 / 3571; 4 x 8, p = 118, 4096 slots 5002 / 5779; 4 x 12, p = 211, 4096 slots 7069 /
// 6013; 4 x 24, p = 765: 68.4 / 59 ms.  FP16 and int8 packages hold two and four times the frames and
// gain throughout.
bool flow_sim_pays(const QcDesc &d, int slots, const ldpc_decode_opts &o) {
    return d.E >= kShortCode || o.msg != LDPC_MSG_F32 || slots <= 2048;
}

// A phase of the flow takes 6 us however few its tiles (8 with FP16 or int8 messages), a pass of its
// own launch 4.5 us: with a fixed iteration count the launches are faster below about 80000 message
// lines (edges times packages).  20 iterations, launches / flow: n = 384, 32 frames (1152 lines) 205 /
// 259 us; 4 x 12, p = 211, 256 frames (81024) 419 / 336; 4 x 24, p = 300, 32 frames (28800) 294 / 355,
// 128 frames (115200) 465 / 394.  Short codes fill a tile badly: 3 x 6, p = 64, 2048 frames (73728)
// 419 / 572, 4 x 8, p = 100, 2048 frames (204800) 720 / 801.  With early stop the flow ends with the
// last frame and its syndrome takes no launches, so it is taken unless the code is short and the
// batch large.  FP32 packages hold the fewest frames, so a large batch has the most phases, and a code
// counts as short there up to 10000 edges (4 x 24, p = 100: 512 frames 557 / 490, 2048 frames 1592 /
// 1735, with early stop 1591 / 1867; 4 x 12, p = 211: 1994 / 1695).
bool flow_pays(const QcDesc &d, int gamma, const ldpc_decode_opts &o) {
    const int W = 32 * lanes_per_word(o.msg);
    const long long lines = (long long)d.E * ((gamma + W - 1) / W);
    const bool shortcode = d.E < kShortCode || (o.msg == LDPC_MSG_F32 && d.E < 10000 && lines > 400000);
    return o.early_stop ? !shortcode || lines < 60000 : !shortcode && lines > 80000;
}

// Frames of one launch: it holds every SM until it ends, so its edges times frames times iterations are
// bounded (2^39: 1.4 s at the 3.9e11 a second of n = 18360, FP32, 30 iterations; 249525 frames of that, so
// what is lost where one launch ends and the next begins, under a millisecond, does not show), but every lane
// in flight gets a frame.
static int64_t launch_frames(const QcDesc &d, int max_iter, int64_t lanes) {
    const int64_t work = std::max<int64_t>(1, (int64_t)d.E * max_iter);
    return std::min<int64_t>((int64_t)1 << 20, std::max(((int64_t)1 << 39) / work, lanes));
}

// a launch on W slots of m: the code's entry, the buffers, the options
static ldpc_status prepare(const QcDesc &d, const FlowMem &m, const ldpc_decode_opts &o, int W, bool post, Start &st, Args &a,
                           uint32_t *tiles) {
    const int V = lanes_per_word(o.msg), FV = o.algo == LDPC_ALGO_MS ? 1 : V;
    std::memset(&st, 0, sizeof(st));
    *tiles = fill_code(d, FV, st.code);
    if (*tiles >= (1u << kLogTiles) || o.max_iter >= (1 << kLogIt)) {
        set_error("code too long: %u tiles a phase", *tiles);
        return LDPC_EINVAL;
    }
    st.code.nparams = o.algo == LDPC_ALGO_NOMS ? o.noms_params : nullptr;
    st.V = V;
    std::memset(&a, 0, sizeof(a));
    size_t b[4];
    flow_slot_bytes(d, o.msg, o.algo, post, b);
    a.slots = (Slot *)m.ctl;
    a.ctl = (Ctl *)((char *)m.ctl + (size_t)m.W * sizeof(Slot));
    a.log = (Entry *)((char *)a.ctl + 256);
    a.code = (Code *)(a.log + m.log_cap);
    a.most_blocks = flow_blocks();
    a.W = std::min(W, log_slots(m.log_cap, a.most_blocks));
    a.msg = (uint32_t *)m.msg, a.mu = (uint32_t *)m.mu, a.post = (float *)m.post, a.hw = (uint32_t *)m.hw;
    a.msg_stride = b[0] / 4, a.mu_stride = b[1] / 4, a.post_stride = b[2] / 4, a.hw_stride = b[3] / 4;
    a.max_iter = o.max_iter, a.early = o.early_stop != 0, a.want_post = post;
    a.clip = o.clip, a.qscale = ldexpf(1.0f, o.frac_bits), a.lsb = ldexpf(1.0f, -o.frac_bits);
    a.err = m.err;
    a.err_tag = m.err_tag;
    return LDPC_OK;
}

static ldpc_status run(const QcDesc &d, const ldpc_decode_opts &o, Args &a, const Start &st, uint32_t tiles, cudaStream_t s) {
    Shape g{d.J, d.L, 1};
    for (int i = 0; i < d.J * d.L; ++i) g.regular &= d.shift[i] >= 0;
    const int grid = (int)std::min<long long>((long long)tiles * a.W, 1 << 20);
    if (o.algo == LDPC_ALGO_MS) return run_ms(a, st, g, grid, s);
    if (o.algo == LDPC_ALGO_NOMS)
        return o.msg == LDPC_MSG_F16 ? run_noms16(a, st, g, grid, s) : run_noms32(a, st, g, grid, s);
    return o.msg == LDPC_MSG_F16 ? run_sp16(a, st, g, grid, s) : run_sp32(a, st, g, grid, s);
}

ldpc_status flow_decode(const QcDesc &d, const FlowMem &m, const float *llr, int gamma, const ldpc_decode_opts &o,
                        float *post, uint8_t *hard, int32_t *iters, int32_t *ok, cudaStream_t s) {
    const int V = lanes_per_word(o.msg), P = (gamma + 32 * V - 1) / (32 * V);
    Start st;
    Args a;
    uint32_t tiles = 0;
    const ldpc_status e = prepare(d, m, o, std::min(m.W, P), post != nullptr, st, a, &tiles);
    if (e != LDPC_OK) return e;
    // with several long packages in work a phase of its own for the syndrome costs no time and saves the
    // check step of a package that has stopped; with few, or short ones, it would add its latency to
    // every iteration (4 x 8, p = 100, 256 frames, FP16: 537 us with, launches 445)
    a.split = a.early && a.W >= 4 && d.E >= kShortCode;
    st.tiles = (d.N + outv(d.J) - 1) / outv(d.J);
    Code &c = st.code;
    const int W = a.W, most = (int)(launch_frames(d, o.max_iter, (int64_t)W * 32 * V) / (32 * V));  // packages a launch
    for (int at = 0; at < P; at += most) {
        const size_t f0 = (size_t)at * 32 * V;
        a.P = std::min(most, P - at);
        a.W = std::min(W, a.P);
        c.gamma = (int)std::min<size_t>(gamma - f0, (size_t)a.P * 32 * V);
        c.llr = llr + f0 * d.N, c.post = post ? post + f0 * d.N : nullptr, c.hard = hard ? hard + f0 * d.N : nullptr;
        c.iters = iters ? iters + f0 : nullptr, c.ok = ok ? ok + f0 : nullptr;
        const ldpc_status r = run(d, o, a, st, tiles, s);
        if (r != LDPC_OK) return r;
    }
    return LDPC_OK;
}

}  // namespace ldpc

// ---------------------------------------------------------------------------
// the workspace a code object keeps
// ---------------------------------------------------------------------------
struct ldpc_flow_ws {
    int frames = 0;                       // that the buffers serve
    size_t cap[5] = {0, 0, 0, 0, 0};
    void *buf[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};  // as FlowMem's
    int log_cap = 0;
    void *sim = nullptr;                  // the simulation's state and its slots' frames
    int *err = nullptr;                   // pinned, device-mapped
    unsigned long long *host = nullptr;   // pinned copy of the simulation's counters
};

namespace ldpc {

void flow_free(ldpc_flow_ws *w) {
    if (!w) return;
    for (void *b : w->buf) cudaFree(b);
    cudaFree(w->sim);
    if (w->host) cudaFreeHost(w->host);
    if (w->err) cudaFreeHost(w->err);
    delete w;
}

// buffers for a decode of `frames` frames, or a simulation on as many frame slots, by every rule and
// message type, with posteriors or without: they are freed for larger ones by a call on more frames only
// (as those of the launches, qc_ensure_workspace), so a captured call stays good while others decode
static ldpc_status flow_ensure(ldpc_code c, int frames, bool sim) {
    auto fail = [&](size_t bytes) {
        cudaGetLastError();
        set_error("device allocation of the decoder's workspace (%zu bytes) failed", bytes);
        return LDPC_ENOMEM;
    };
    if (!c->flow) {
        c->flow = new (std::nothrow) ldpc_flow_ws();
        if (!c->flow) return fail(0);
    }
    ldpc_flow_ws &w = *c->flow;
    if (!w.err) {
        if (cudaHostAlloc((void **)&w.err, 64, cudaHostAllocMapped) != cudaSuccess) {
            w.err = nullptr;
            return fail(64);
        }
        *w.err = 0;
    }
    if (sim && !w.sim) {
        const size_t need = 512 + kMaxSlots * sizeof(SimSlot);
        if (cudaMalloc(&w.sim, need) != cudaSuccess) {
            w.sim = nullptr;
            return fail(need);
        }
    }
    if (sim && !w.host && cudaHostAlloc((void **)&w.host, 64, cudaHostAllocDefault) != cudaSuccess) {
        w.host = nullptr;
        return fail(64);
    }
    if (frames <= w.frames) return LDPC_OK;
    const long long cap = std::min(((long long)frames + 127) / 128 * 128, (long long)INT32_MAX);
    size_t need[5] = {0, 0, 0, 0, 0};
    int most = 1;
    for (int form = 0; form < 6; ++form) {
        static const int msgs[3] = {LDPC_MSG_F32, LDPC_MSG_F16, LDPC_MSG_I8};
        const int msg = msgs[form / 2], algo = msg == LDPC_MSG_I8 ? LDPC_ALGO_MS : LDPC_ALGO_SP;
        const bool post = form % 2 != 0;
        const int wd = 32 * lanes_per_word(msg), W = flow_slots(c->d, msg, algo, post, (int)((cap + wd - 1) / wd));
        size_t b[4];
        flow_slot_bytes(c->d, msg, algo, post, b);
        for (int i = 0; i < 4; ++i) need[i] = std::max(need[i], b[i] * W);
        most = std::max(most, W);
    }
    const int log_cap = std::min(log_entries(most, flow_blocks()), kMaxLog);
    need[4] = flow_ctl_bytes(kMaxSlots, log_cap);
    bool synced = false;
    for (int i = 0; i < 5; ++i) {
        if (need[i] <= w.cap[i]) continue;
        if (!synced) LDPC_CUDA_TRY(cudaDeviceSynchronize());
        synced = true;
        cudaFree(w.buf[i]);
        w.buf[i] = nullptr;
        w.cap[i] = 0;
        if (cudaMalloc(&w.buf[i], need[i]) != cudaSuccess) {
            w.buf[i] = nullptr;
            w.frames = 0;
            return fail(need[i]);
        }
        w.cap[i] = need[i];
    }
    w.log_cap = log_cap;
    w.frames = (int)cap;
    return LDPC_OK;
}

ldpc_status flow_gave_up(int *err, int tag, const char *what) {
    const int e = err ? *(volatile int *)err : 0;
    if (!e || (e & ~7) != tag) return LDPC_OK;
    *err = 0;
    set_error("%s gave up a device-side wait (code %d)", what, e & 7);
    return LDPC_ETIMEOUT;
}

ldpc_status flow_check(const ldpc_code c, const char *what) { return flow_gave_up(c->flow ? c->flow->err : nullptr, 0, what); }

bool flow_ready(const ldpc_code c, int gamma) { return c->flow && gamma <= c->flow->frames; }

ldpc_status flow_decode_code(ldpc_code c, const float *llr, int gamma, const ldpc_decode_opts &o, float *post,
                             uint8_t *hard, int32_t *iters, int32_t *ok, cudaStream_t s) {
    const int V = lanes_per_word(o.msg);
    const int W = flow_slots(c->d, o.msg, o.algo, post != nullptr, (gamma + 32 * V - 1) / (32 * V));
    const ldpc_status e = flow_ensure(c, gamma, false);
    if (e != LDPC_OK) return e;
    const ldpc_flow_ws &w = *c->flow;
    const FlowMem m{w.buf[0], w.buf[1], w.buf[2], w.buf[3], w.buf[4], W, w.log_cap, w.err, 0};
    return flow_decode(c->d, m, llr, gamma, o, post, hard, iters, ok, s);
}

ldpc_status flow_sim_code(ldpc_code c, double sigma, uint64_t seed, uint64_t first_frame, int64_t max_frames, int slots,
                          const ldpc_decode_opts &o, unsigned long long *h, cudaStream_t s, const StreamIO *io) {
    const int V = lanes_per_word(o.msg);
    const int W = flow_slots(c->d, o.msg, o.algo, false, (slots + 32 * V - 1) / (32 * V));
    ldpc_status e = flow_ensure(c, slots, true);
    if (e != LDPC_OK) return e;
    ldpc_flow_ws &w = *c->flow;
    const FlowMem m{w.buf[0], w.buf[1], w.buf[2], w.buf[3], w.buf[4], W, w.log_cap, w.err, 0};
    std::memset(h, 0, 8 * sizeof(*h));
    const int64_t most = launch_frames(c->d, o.max_iter, (int64_t)W * 32 * V);
    for (int64_t at = 0; at < max_frames; at += most) {
        Start st;
        Args a;
        uint32_t tiles = 0;
        e = prepare(c->d, m, o, W, false, st, a, &tiles);
        if (e != LDPC_OK) return e;
        a.sim = (Sim *)w.sim;
        a.simslots = (SimSlot *)((char *)w.sim + 512);
        static_assert(sizeof(Sim) <= 512, "room before the slots");
        st.tiles = st.code.nsyn;
        Sim &si = st.sim;
        si.limit = (unsigned long long)std::min(most, max_frames - at);
        si.first = (io ? 0ull : first_frame) + (unsigned long long)at;
        si.seed = seed;
        si.sigma = (float)sigma;
        si.s2 = (float)(2.0 / (sigma * sigma));
        if (io) {
            si.io = 1;
            si.llr = io->llr, si.hard = io->hard, si.iters = io->iters, si.ok = io->ok;
            si.wide_in = c->d.N % 4 == 0 && ((uintptr_t)io->llr & 15u) == 0;
            si.wide_out = c->d.N % 4 == 0 && ((uintptr_t)io->hard & 3u) == 0;
        }
        e = run(c->d, o, a, st, tiles, s);
        if (e != LDPC_OK) return e;
        LDPC_CUDA_TRY(cudaMemcpyAsync(w.host, a.sim->counters, 64, cudaMemcpyDeviceToHost, s));
        LDPC_CUDA_TRY(cudaStreamSynchronize(s));
        e = flow_check(c, "the simulation");
        if (e != LDPC_OK) return e;
        for (int i = 0; i < 8; ++i) h[i] += w.host[i];
    }
    return LDPC_OK;
}

}  // namespace ldpc
