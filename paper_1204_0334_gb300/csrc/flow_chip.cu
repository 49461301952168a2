// The on-chip decoder: Algorithm 1 on a few packages of a short code, one launch, a thread-block
// cluster per package.
//
// A short code's pass takes a launch 4.5 us, and a phase of the flow decoder 6, for a few hundred
// nanoseconds of work.  Here the blocks of a cluster divide a package's variables and keep everything of
// theirs in shared memory: channel LLRs, messages (by variable, as in global memory), decision words,
// posteriors.  The variable step is local; the check step reads and writes its edges in the other
// blocks' shared memory; two hardware cluster barriers an iteration, and no spinning.  Early stop ends
// the launch with the package's last frame: the syndrome goes with the check step, a warp per row, a
// lane per edge.
//
// The blocks of a cluster are as many as leave all packages resident at once (16, 8, 4, 2 or 1): more
// blocks a package, fewer rows a warp.  What bounds it is latency: the chain of a row (its remote loads
// in flight together, then the sums and transforms) and the barriers.  n = 384, 32 frames, 30 iterations:
// 283 us by launches, 82 to 86 here (it differs from process to process; 3500 cycles an iteration in the
// check step and its barrier, 2300 in the variable step and its own).
//
// The arithmetic is that of the pass kernels (qc_pipe.cu), operation by operation.
#include "flow_internal.cuh"

#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <mutex>
#include <new>
#include <tuple>

namespace ldpc {
namespace chip {

using namespace flow;

size_t bytes(const Code &c, int V, bool ms, bool post, int NC) {
    const size_t W = 32 * V;
    return (size_t)NC * 4 * ((size_t)c.J * 32 + (ms ? 33 : W + 1) + V + (post ? W + 1 : 0));
}

// Message lines of a block beyond which the passes over the whole chip are faster: an SM works through
// its lines of an iteration one after another.  20 iterations, the faster of launches and flow / here, us,
// at lines a block (and packages): FP32 633: 290 / 263 (1), 329 / 267 (4); 800: 462 / 284 (32).  FP16 320: 298
// / 256 (1); 390: 334 / 264 (2); 400: 372 / 254 (8); 800: 461 / 491 (16), 648 / 507 (32); rows of more than 16
// slots, which take a frame of a word after the other, 375: 341 / 427 (1), with early stop 462 / 450.  int8
// 400: 336 / 226 (8); 600: 299 / 342 (1), 388 / 350 (4); 640: 426 / 349 (8).
static int most_lines(const Code &c, int V, int P, bool early) {
    if (V == 1) return 800;
    if (V == 2) return P >= 24 ? 800 : c.L > 16 && !early ? 250 : 400;
    return P < 4 ? 500 : 800;
}

int pick(const void *kernel, const Code &c, int V, bool ms, const ChipArgs &a, int P) {
    static std::mutex mu;
    // clusters resident at once, one block an SM, by device, kernel and blocks of a cluster
    static std::map<std::tuple<int, const void *, int>, int> active;
    int dev = 0, E = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lk(mu);
    for (int i = 0; i < c.J * c.L; ++i) E += c.sh[i] >= 0 ? c.p : 0;
    for (int C = 16; C >= 1; C /= 2) {
        const int NC = (c.N + C - 1) / C;
        if (bytes(c, V, ms, a.want_post, NC) > kChipMost || (!a.any && E > C * most_lines(c, V, P, a.early))) return 0;  // fewer blocks hold less
        if ((C - 1) * NC >= c.N) continue;  // a block would have no variable
        const auto key = std::make_tuple(dev, kernel, C);
        const auto f = active.find(key);
        int n = f == active.end() ? 0 : f->second;
        if (f == active.end()) {
            cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kChipMost);
            cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
            cudaLaunchConfig_t cfg{};
            cudaLaunchAttribute at[1];
            cfg.gridDim = dim3((unsigned)C);
            cfg.blockDim = dim3(kChipThreads);
            cfg.dynamicSmemBytes = kChipMost;
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = C;
            at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
            cfg.attrs = at;
            cfg.numAttrs = 1;
            if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
                cudaGetLastError();
                n = 0;
            }
            try {
                active.emplace(key, n);
            } catch (const std::bad_alloc &) {
            }
        }
        if (P <= n) return C;
    }
    return 0;
}

}  // namespace chip

using namespace flow;

// Takes a decode whose packages all fit on the chip at once; *taken says whether it did.
ldpc_status chip_decode(const QcDesc &d, const float *llr, int gamma, const ldpc_decode_opts &o, float *post, uint8_t *hard,
                        int32_t *iters, int32_t *ok, cudaStream_t s, bool *taken, bool any) {
    const int V = lanes_per_word(o.msg), P = (gamma + 32 * V - 1) / (32 * V);
    *taken = false;
    if (P > 152 || d.E > 16 * 800) return LDPC_OK;
    Code c;
    std::memset(&c, 0, sizeof(c));
    c.J = d.J, c.L = d.L, c.p = d.p, c.N = d.N, c.M = d.M;
    c.divp = d.divP;
    std::memcpy(c.sh, d.shift, sizeof(int) * d.J * d.L);
    c.gamma = gamma;
    c.llr = llr, c.post = post, c.hard = hard, c.iters = iters, c.ok = ok;
    c.nparams = o.algo == LDPC_ALGO_NOMS ? o.noms_params : nullptr;
    chip::ChipArgs a;
    std::memset(&a, 0, sizeof(a));
    a.any = any;
    a.max_iter = o.max_iter, a.early = o.early_stop != 0, a.want_post = post != nullptr;
    a.clip = o.clip, a.qscale = ldexpf(1.0f, o.frac_bits), a.lsb = ldexpf(1.0f, -o.frac_bits);
    if (o.algo == LDPC_ALGO_MS) return chip::run_ms(c, a, P, s, taken);
    if (o.algo == LDPC_ALGO_NOMS)
        return o.msg == LDPC_MSG_F16 ? chip::run_noms16(c, a, P, s, taken)
                                     : chip::run_noms32(c, a, P, s, taken);
    return o.msg == LDPC_MSG_F16 ? chip::run_sp16(c, a, P, s, taken)
                                 : chip::run_sp32(c, a, P, s, taken);
}

}  // namespace ldpc
