// Shared declarations of the flow decoder (flow.cu describes it).
#pragma once

#include "ldpc_internal.cuh"

namespace ldpc {
namespace flow {

// One block per SM.  24 compute warps leave 72 registers a thread; with 16 (96 registers) the
// 2048-frame decode of the n = 18360 code took 19.2 ms where 24 took 14.9 (before the other steps):
// the rows are chains of dependent instructions, and warps hide them better than registers.
constexpr int kComputeWarps = 24;
constexpr int kStages = 3;                          // tiles a block holds: in work, arriving, leaving
constexpr int kThreads = (kComputeWarps + 1 + kStages) * 32;  // and the taking warp, a retiring warp per stage
constexpr int kLookLimit = 1 << 24;                 // looks for a new phase before a block gives up (seconds)
constexpr int kMaxSlots = 256;
constexpr int kMaxLog = 1 << 16;                    // entries of the longest phase log
// check rows of a tile: one a compute warp (two of short rows; fewer of 32-edge rows, so that three
// tiles fit in shared memory)
__host__ __device__ constexpr int tile_rows(int J, int L) {
    return J <= 4 && L <= 8 ? 2 * kComputeWarps : (L <= 24 ? kComputeWarps : kComputeWarps * 2 / 3 / 2 * 2);
}
__host__ __device__ constexpr int outv(int J) { return J <= 4 ? 256 : 128; }  // variables of a pack / output tile
static_assert(kComputeWarps % 2 == 0, "row, frame pairs of the first iteration");

enum { kFlowSP = 0, kFlowMS = 1, kFlowNOMS = 2 };
// phases; F_SYN is also a tile of F_CN and F_FIN, the last three are tiles of F_CN in refill mode
enum { F_PACK = 0, F_CN, F_VN, F_FIN, F_OUT, F_SYN, F_EXIT, F_ERR, F_ROWS, F_CHAN };

// the code of a launch and the caller's buffers of its frames
struct Code {
    int J, L, p, N, M;
    int kc;                  // variables of a variable tile (a multiple of 4)
    int nsyn;                // syndrome tiles
    FastDiv divp, rch, rch1, vch;  // p; check tiles per block row (later / first iteration); variable tiles per column
    int gamma;               // frames
    const float *llr;
    float *post;
    uint8_t *hard;
    int32_t *iters, *ok;
    const float *nparams;
    int sh[kMaxJ * kMaxL], eo[kMaxJ * kMaxL];  // [J][L]: shift (-1: zero block), first edge
};

// A phase that has been opened.  w0: kind (3 bits), frames stopped (1), iteration (17), package (26), sequence
// number without its low five bits (17).  w1: tiles (24), the number of tiles opened before it modulo the
// blocks (10), slot (8), sequence number (22).  The words are loaded and stored as a pair, which the memory
// model takes for two accesses in no order: the entries that follow one another in a place are 64 or more
// apart, so the numbers tell a new word from an old one.
constexpr int kLogIt = 17, kLogPk = 26, kLogTiles = 24, kLogBase = 10, kLogSlot = 8, kLogSeq = 22, kLogLow = 5;
constexpr uint32_t kLogMask = (1u << kLogSeq) - 1u;
struct alignas(16) Entry {
    unsigned long long w0, w1;
};
__host__ __device__ inline unsigned long long entry_w0(uint32_t seq, int kind, int stop, int it, int pk) {
    unsigned long long x = (seq & kLogMask) >> kLogLow;
    x = x << kLogPk | (unsigned)pk;
    x = x << kLogIt | (unsigned)it;
    x = x << 1 | (unsigned)stop;
    return x << 3 | (unsigned)kind;
}
__host__ __device__ inline unsigned long long entry_w1(uint32_t seq, int slot, uint32_t base, uint32_t tiles) {
    unsigned long long x = seq & kLogMask;
    x = x << kLogSlot | (unsigned)slot;
    x = x << kLogBase | base;
    return x << kLogTiles | tiles;
}
// what a second word read in entry n's place is: entry n's, a later one's that has overwritten it, or an earlier
enum { kEntryHere = 0, kEntryPast, kEntryAhead };
__host__ __device__ inline int entry_is(unsigned long long w1, uint32_t n) {
    const uint32_t ahead = ((uint32_t)(w1 >> (kLogTiles + kLogBase + kLogSlot)) - n) & kLogMask;
    return ahead == 0u ? kEntryHere : ahead < (kLogMask >> 1) ? kEntryPast : kEntryAhead;
}
// whether the first word read beside it is entry n's too
__host__ __device__ inline bool entry_whole(unsigned long long w0, uint32_t n) {
    return (uint32_t)(w0 >> (4 + kLogIt + kLogPk)) == (n & kLogMask) >> kLogLow;
}

// Entries of the phase log, a power of two.  Entry n is overwritten by entry n + length, which must not be
// opened while some block b has a tile of entry n that it has not read.  Tiles are numbered as they are
// opened and tile t belongs to block t mod blocks, so every `blocks` consecutive tiles hold one of b's.
// b reads the log in order: a phase opened after n with a tile of b does not end before b has read n, and
// its slot opens no other.  With entry n that is at most one such phase a slot, so at most slots * blocks
// tiles, and as many phases, are opened from entry n on (each has a tile but the last of all, which is
// opened when no slot has a phase left).
inline int log_entries(int slots, int blocks) {
    int n = 64;  // more than the 32 entries that are looked at together
    while (n < (long long)slots * blocks + 1) n *= 2;
    return n;
}
// slots that a log of `entries` serves
inline int log_slots(int entries, int blocks) { return (entries - 1) / blocks; }

// a package in work
struct alignas(64) Slot {
    unsigned int done, syn_done;  // finished tiles of the open phase, finished syndrome tiles
    int all;                      // every frame has stopped
    uint32_t dn[4], un[4];        // stopped frames, unsatisfied frames (bit = lane)
    uint32_t ret[4], fresh[4];    // refill mode: frames leaving and entering in this step
};

// Refill mode (the simulation, and the decode of a large batch by streaming): every package lane is a
// frame slot that takes the next frame as soon as its frame stops.
struct Sim {
    unsigned long long next, limit;  // frames handed out, frames to hand out
    unsigned long long first;        // id of frame 0
    unsigned long long counters[8];  // frames, frame errors, bit errors, iterations, undetected, squared bit errors
    unsigned long long seed;
    float sigma, s2;
    const float *llr;                // streaming: the caller's rows, and outputs written as frames leave
    uint8_t *hard;
    int32_t *iters, *ok;
    int io, wide_in, wide_out;       // streaming; rows on 16- / 4-byte boundaries
};
struct SimSlot {
    unsigned long long fid[128], rfid[128];  // frame in the lane, frame that left it in this step
    int age[128];                            // iterations completed
    int pend[128];                           // of the frame that left: 2 * iterations + ok
    int errs[128];                           // its wrong bits
    unsigned long long from, to;             // frames reserved for the slot
};

struct Ctl {
    unsigned long long tail;  // phases opened (24 bits), tiles opened (40)
    int next;                 // packages handed to slots so far
    int live;                 // slots with a package
    int abort;                // a wait ran out
};

struct Args {
    Code *code;
    Slot *slots;
    Ctl *ctl;
    Entry *log;
    int log_len;               // its entries (a power of two)
    int W, P;                  // slots, packages
    uint32_t *msg, *mu, *hw;   // per slot: [E][32], [N][32 FV], [N][V]
    float *post;               // per slot: [N][32 V]
    size_t msg_stride, mu_stride, hw_stride, post_stride;  // words
    int max_iter, early, want_post;
    int split;                 // the early-stop syndrome is a phase of its own
    int blocks, most_blocks;   // of the launch; as many as the log allows
    float clip, qscale, lsb;
    Sim *sim;                  // refill mode, else NULL
    SimSlot *simslots;
    int *err;                  // host word set when a wait ran out: which (1 to 4), beside err_tag
    int err_tag;               // whose launch it is, where objects share a word (a multiple of 8)
};

struct Shape {
    int J, L, regular;
};

// resident blocks of a kernel with kThreads threads (cached per kernel and size)
int resident_blocks(const void *kernel, size_t smem);

// one translation unit per rule
// (start: the launch that opens the first phases, once the number of blocks is known)
struct Start {
    Code code;
    Sim sim;       // refill mode
    int V, tiles;  // lane words' frames; tiles of the first phase
};
ldpc_status run_sp32(Args &a, const Start &st, const Shape &g, int tiles, cudaStream_t s);
ldpc_status run_sp16(Args &a, const Start &st, const Shape &g, int tiles, cudaStream_t s);
ldpc_status run_ms(Args &a, const Start &st, const Shape &g, int tiles, cudaStream_t s);
ldpc_status run_noms32(Args &a, const Start &st, const Shape &g, int tiles, cudaStream_t s);
ldpc_status run_noms16(Args &a, const Start &st, const Shape &g, int tiles, cudaStream_t s);
ldpc_status start(const Args &a, const Start &st, cudaStream_t s);
constexpr int kSynRows = 256;                    // rows of a syndrome tile
constexpr int kErrVars = 128 * kComputeWarps;  // variables of a tile that counts wrong bits or writes decision rows

}  // namespace flow

// the buffers of a flow decode
struct FlowMem {
    void *msg, *mu, *post, *hw;  // W slots each
    void *ctl;                   // flow_ctl_bytes()
    int W, log_cap;              // slots, entries of the phase log
    int *err, err_tag;
};
size_t flow_ctl_bytes(int W, int log_cap);
// slots a decode of P packages keeps in work, and the bytes of one slot's buffers
int flow_slots(const QcDesc &d, int msg, int algo, bool post, int P);
void flow_slot_bytes(const QcDesc &d, int msg, int algo, bool post, size_t *b4);
// whether a decode goes to the flow decoder rather than to a launch per pass
bool flow_pays(const QcDesc &d, int gamma, const ldpc_decode_opts &o);
bool flow_sim_pays(const QcDesc &d, int slots, const ldpc_decode_opts &o);
// Algorithm 1 on gamma frames of a QC code, device buffers in and out (outputs may be NULL)
ldpc_status flow_decode(const QcDesc &d, const FlowMem &m, const float *llr, int gamma, const ldpc_decode_opts &o,
                        float *post, uint8_t *hard, int32_t *iters, int32_t *ok, cudaStream_t s);
// refill mode: frames 0 .. max_frames - 1 (ids from first_frame), drawn by the channel or read from io's
// rows, through min(slots, what stays in L2) frame slots; h: the eight counters.  Waits for the stream.
ldpc_status flow_sim_code(ldpc_code c, double sigma, uint64_t seed, uint64_t first_frame, int64_t max_frames, int slots,
                          const ldpc_decode_opts &o, unsigned long long *h, cudaStream_t s, const StreamIO *io);
// the same on a code object, in a workspace that it keeps
ldpc_status flow_decode_code(ldpc_code c, const float *llr, int gamma, const ldpc_decode_opts &o, float *post,
                             uint8_t *hard, int32_t *iters, int32_t *ok, cudaStream_t s);

// LDPC_ETIMEOUT, once, if a launch with this tag has set its word (no wait: launches that are done by now)
ldpc_status flow_gave_up(int *err, int tag, const char *what);
ldpc_status flow_check(const ldpc_code c, const char *what);
// whether that workspace serves gamma frames as it is
bool flow_ready(const ldpc_code c, int gamma);

// the on-chip decoder of short codes (flow_chip.cu); any: also where another form is faster
ldpc_status chip_decode(const QcDesc &d, const float *llr, int gamma, const ldpc_decode_opts &o, float *post, uint8_t *hard,
                        int32_t *iters, int32_t *ok, cudaStream_t s, bool *taken, bool any = false);

namespace chip {

constexpr int kChipThreads = 512;
constexpr size_t kChipMost = 225 * 1024;  // with the static arrays, below the 227 KB a block may have
// one block an SM, also where registers and shared memory would let two in
constexpr size_t kChipLeast = 116 * 1024;

struct ChipArgs {
    int C, NC;       // blocks of a cluster, variables of a block
    FastDiv divNC;
    int max_iter, early, want_post;
    int any;         // taken also where another form is faster
    float clip, qscale, lsb;
};
size_t bytes(const flow::Code &c, int V, bool ms, bool post, int NC);
// blocks of a cluster so that all P packages are resident, or 0
int pick(const void *kernel, const flow::Code &c, int V, bool ms, const ChipArgs &a, int P);
ldpc_status run_sp32(const flow::Code &c, ChipArgs &a, int P, cudaStream_t s, bool *taken);
ldpc_status run_sp16(const flow::Code &c, ChipArgs &a, int P, cudaStream_t s, bool *taken);
ldpc_status run_ms(const flow::Code &c, ChipArgs &a, int P, cudaStream_t s, bool *taken);
ldpc_status run_noms32(const flow::Code &c, ChipArgs &a, int P, cudaStream_t s, bool *taken);
ldpc_status run_noms16(const flow::Code &c, ChipArgs &a, int P, cudaStream_t s, bool *taken);

}  // namespace chip
}  // namespace ldpc
