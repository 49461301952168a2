// Decoding of general (not quasi-cyclic) LDPC codes: Algorithm 1 on the QC decoder's package layout, the
// edges of a row (consecutive, edges numbered row by row as in eq. simpleH) and of a variable (the
// column table) from index tables -- the role of the paper's LUT_c / LUT_v (Sec. IV-A) -- instead of
// circulant address arithmetic.  The first iteration starts from messages beta = mu written by an
// initialization pass; the syndrome for early stopping (tested after each complete iteration i >= 1)
// and the final ok flags gather the hard decisions through the row table.
//
// No slot is computed that a row or a variable does not have.  A check row's lines are consecutive: a warp
// holds them in registers, all loads in flight together.  A variable's are scattered: a warp copies those
// of four variables into a ring in shared memory, an item ahead (in registers instead: 81 us, all the
// address arithmetic twice and too few warps).  Sums, transforms and roundings are those of the QC passes.
#include "flow.cuh"

namespace ldpc {

// beta = mu on every edge of every package, in the form the check pass reads:
// sign(mu) phi(|mu|) for sum-product (scaled for FP16), the int8 word for min-sum.
// One thread per (package, edge, lane word).
template <int V, bool MS>
__global__ void sparse_init_kernel(const uint32_t *__restrict__ mu, uint32_t *__restrict__ msg, const int *__restrict__ col,
                                   int N, int E, int P) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long total = (long long)P * E * 32;
    if (i >= total) return;
    const int lane = (int)(i & 31);
    const long long pe = i >> 5;
    const int pk = (int)(pe / E), e = (int)(pe - (long long)pk * E);
    const int n = __ldg(col + e);
    if constexpr (MS) {
        msg[i] = mu[((size_t)pk * N + n) * 32 + lane];
    } else {
        const float *m = reinterpret_cast<const float *>(mu) + ((size_t)pk * N + n) * (32 * V) + lane * V;
        float b[V];
#pragma unroll
        for (int v = 0; v < V; ++v) b[v] = with_sign_of(phi_f(fabsf(m[v])) * XfScale<V>::store, m[v]);
        msg[i] = Lane<V>::pack(b);
    }
}

// syndrome of the hard decisions (eq. hrddcs) through the row table into flag word
// `word` (+v) of each package; one thread per row, a warp ORs its rows
template <int V>
__global__ void sparse_syndrome_kernel(const int *__restrict__ rp, const int *__restrict__ col,
                                       const uint32_t *__restrict__ hw, uint32_t *__restrict__ flags, int M, int N,
                                       int word) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    const int pk = blockIdx.y;
    uint32_t syn[V];
#pragma unroll
    for (int v = 0; v < V; ++v) syn[v] = 0u;
    if (m < M) {
        for (int e = __ldg(rp + m), e1 = __ldg(rp + m + 1); e < e1; ++e) {
            const uint32_t *h = hw + ((size_t)pk * N + __ldg(col + e)) * V;
#pragma unroll
            for (int v = 0; v < V; ++v) syn[v] ^= h[v];
        }
    }
    uint32_t *out = flags + (size_t)pk * 5 * V + word;
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const uint32_t any = __reduce_or_sync(0xffffffffu, syn[v]);
        if (any && (threadIdx.x & 31) == 0) atomicOr(out + v, any);
    }
}

static ldpc_status sparse_syndrome(ldpc_code c, int P, int V, int word, cudaStream_t s) {
    const dim3 grd((c->d.M + 255) / 256, P);
    if (V == 1) sparse_syndrome_kernel<1><<<grd, 256, 0, s>>>(c->sp.rp, c->sp.col, c->ws.hw, c->ws.flags, c->d.M, c->d.N, word);
    else if (V == 2) sparse_syndrome_kernel<2><<<grd, 256, 0, s>>>(c->sp.rp, c->sp.col, c->ws.hw, c->ws.flags, c->d.M, c->d.N, word);
    else sparse_syndrome_kernel<4><<<grd, 256, 0, s>>>(c->sp.rp, c->sp.col, c->ws.hw, c->ws.flags, c->d.M, c->d.N, word);
    count_launch();
    LDPC_CUDA_TRY(cudaGetLastError());
    return LDPC_OK;
}

// Check pass: a row per warp.  n = 6000, 21000 edges, 1024 frames, FP32: 56 us through a ring at 16 slots a row, 38 here.
template <int DC, int V, bool MS>
__global__ void __launch_bounds__(256, DC <= 16 ? 3 : 2)
sparse_cn_kernel(const SparseTab tab, FastDiv divM, int E, uint32_t *__restrict__ msg, const int *__restrict__ act, float clip) {
    const int lane = threadIdx.x & 31, M = (int)divM.d;
    const int total = act[0] * M, step = gridDim.x * (blockDim.x >> 5);
    int item = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    auto row = [&](int it, int &e0, int &deg, uint32_t *&base) {
        const int a = (int)fdiv((uint32_t)it, divM), m = it - a * M;
        e0 = __ldg(tab.rp + m);
        deg = __ldg(tab.rp + m + 1) - e0;
        base = msg + (size_t)__ldg(act + 1 + a) * E * 32 + lane;
    };
    int e0 = 0, deg = 0;
    uint32_t *base = nullptr;
    if (item < total) row(item, e0, deg, base);
    for (; item < total; item += step) {
        uint32_t *S = base + (size_t)e0 * 32;
        const int dg = deg;
        uint32_t x[DC];
#pragma unroll
        for (int l = 0; l < DC; ++l) x[l] = load_if(S + l * 32, l < dg);
        if (item + step < total) row(item + step, e0, deg, base);  // the next row's place, behind the loads
        const uint32_t pm = dg >= 32 ? ~0u : (1u << dg) - 1u;
        if constexpr (MS) {
            uint32_t min1 = 0x7f7f7f7fu, min2 = 0x7f7f7f7fu, sgn = 0u;
#pragma unroll
            for (int l = 0; l < DC; ++l) {
                if (l >= dg) break;  // warp-uniform
                const uint32_t av = __vabsss4(x[l]);
                sgn ^= x[l] & 0x80808080u;
                min2 = __vminu4(min2, __vmaxu4(min1, av));
                min1 = __vminu4(min1, av);
            }
#pragma unroll
            for (int l = 0; l < DC; ++l) {
                if (l >= dg) break;
                const uint32_t eq = __vcmpeq4(__vabsss4(x[l]), min1);
                const uint32_t mag = (min2 & eq) | (min1 & ~eq);
                const uint32_t neg = ((sgn ^ (x[l] & 0x80808080u)) >> 7) & 0x01010101u;
                S[l * 32] = __vadd4(mag ^ (neg * 0xffu), neg);
            }
        } else if constexpr (V == 1) {
            flow::sp_row<DC, false, 1>(pm, clip, ~0u, [&](int l) { return __uint_as_float(x[l]); },
                                       [&](int l, float r) { if (l < dg) S[l * 32] = __float_as_uint(r); });
        } else {
            uint32_t lo[DC];  // the first frame's results
            flow::sp_row<DC, false, 4096>(
                pm, clip, ~0u, [&](int l) { return __half2float(__ushort_as_half((unsigned short)x[l])); },
                [&](int l, float r) { lo[l] = __half_as_ushort(__float2half_rn(r)); });
            flow::sp_row<DC, false, 4096>(
                pm, clip, ~0u, [&](int l) { return __half2float(__ushort_as_half((unsigned short)(x[l] >> 16))); },
                [&](int l, float r) {
                    if (l < dg) S[l * 32] = lo[l] | (uint32_t)__half_as_ushort(__float2half_rn(r)) << 16;
                });
        }
    }
}

// one variable with up to NJ edges (S: the lane's word of the first, on: which are there): messages out,
// decisions and posterior
template <int NJ, int V, bool MS, typename PUT>
__device__ __forceinline__ void sparse_variable(const uint32_t *S, uint32_t on, const float *m, uint32_t q, float clip, float lsb, float *pst,
                                                uint32_t *outb, PUT put) {
    uint32_t x[NJ];
#pragma unroll
    for (int j = 0; j < NJ; ++j) x[j] = (on >> j) & 1u ? S[j * 32] : 0u;
    if constexpr (MS) {
        int tot[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) tot[v] = sbyte(q, v);
#pragma unroll
        for (int j = 0; j < NJ; ++j)
#pragma unroll
            for (int v = 0; v < 4; ++v) tot[v] += sbyte(x[j], v);
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
            uint32_t o = 0u;
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                int b = tot[v] - sbyte(x[j], v);
                b = b > 127 ? 127 : (b < -127 ? -127 : b);
                o |= ((uint32_t)(uint8_t)(int8_t)b) << (8 * v);
            }
            put(j, o);
        }
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            pst[v] = (float)tot[v] * lsb;
            outb[v] = __ballot_sync(0xffffffffu, tot[v] < 0);
        }
    } else {
        float aj[NJ][V], tot[V], bs[NJ][V], ph[NJ][V];
#pragma unroll
        for (int v = 0; v < V; ++v) tot[v] = m[v];
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
            Lane<V>::unpack(x[j], aj[j]);
#pragma unroll
            for (int v = 0; v < V; ++v) tot[v] += aj[j][v];
        }
#pragma unroll
        for (int j = 0; j < NJ; ++j)
#pragma unroll
            for (int v = 0; v < V; ++v) {
                float s = m[v];
#pragma unroll
                for (int j2 = 0; j2 < NJ; ++j2)
                    if (j2 != j) s += aj[j2][v];
                bs[j][v] = s;
            }
        if constexpr (V == 2) {
#pragma unroll
            for (int j = 0; j < NJ; ++j)
                flow::phi_pair<1, 4096>(fminf(fabsf(bs[j][0]), clip), fminf(fabsf(bs[j][1]), clip), ph[j][0], ph[j][1]);
        } else {
#pragma unroll
            for (int j = 0; j < NJ; j += 2)
                flow::phi_pair<1, 1>(fminf(fabsf(bs[j][0]), clip), fminf(fabsf(bs[j + 1][0]), clip), ph[j][0], ph[j + 1][0]);
        }
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
#pragma unroll
            for (int v = 0; v < V; ++v) bs[j][v] = with_sign_of(ph[j][v], bs[j][v]);
            put(j, Lane<V>::pack(bs[j]));
        }
#pragma unroll
        for (int v = 0; v < V; ++v) {
            pst[v] = clipf(tot[v], clip);
            outb[v] = __ballot_sync(0xffffffffu, pst[v] < 0.0f);
        }
    }
}

template <int V, bool MS>
struct SparseStage {
    static constexpr int MUW = MS ? 32 : 32 * V;     // channel-LLR words per variable
    static constexpr int AL = 4 * MUW;               // [variable][edge][32]
    static constexpr int HW = AL + 32 * 32;          // old decision words [variable][V]
    static constexpr int FL = HW + 4 * V;            // done[V], unsat[V]
    static constexpr int WORDS = (FL + 2 * V + 3) & ~3;
};
constexpr int kSparseStages = 2;  // of 5 KB a warp: 24 warps an SM (three: 16)

// Variable pass: four variables per warp and step, each computed for 2, 4, 6 or 8 edges by its degree (an
// edge that is not there adds 0.0 in the same order).  Same code: 86 us computing eight edges a variable, 50 here (66 % issue).
template <int V, bool MS, bool STOP, bool POST>
__global__ void __launch_bounds__(256, 3)
sparse_vn_kernel(const SparseTab tab, FastDiv divG, int N, int E, uint32_t *__restrict__ msg, const uint32_t *__restrict__ mu,
                 uint32_t *__restrict__ hw, uint32_t *__restrict__ flags, float *__restrict__ post,
                 int32_t *__restrict__ iters, const int *__restrict__ act, float clip, float lsb, int it, int par) {
    using St = SparseStage<V, MS>;
    constexpr int W = 32 * V, MUW = St::MUW;
    extern __shared__ __align__(16) uint32_t smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, G = (int)divG.d;
    const int total = act[0] * G, step = gridDim.x * (blockDim.x >> 5);
    uint32_t *ring = smem + warp * kSparseStages * St::WORDS;
    int item = blockIdx.x * (blockDim.x >> 5) + warp;
    // starts the copies of an item; lane t: edge t % 8 of its variable t / 8, -1 where absent
    auto issue = [&](int itm, uint32_t *dst) -> int {
        int mine = -1;
        if (itm < total) {
            const int a = (int)fdiv((uint32_t)itm, divG);
            const int n0 = 4 * (itm - a * G), pk = __ldg(act + 1 + a);
            const int grp = lane >> 3, sub = lane & 7;
            if (n0 + grp < N) {
                const int c0 = __ldg(tab.cptr + n0 + grp), deg = __ldg(tab.cptr + n0 + grp + 1) - c0;
                if (sub < deg) mine = __ldg(tab.cedge + c0 + sub);
#pragma unroll
                for (int h = 0; h < MUW / 32; ++h)
                    cp_async16(dst + grp * MUW + h * 32 + sub * 4,
                               mu + ((size_t)pk * N + n0 + grp) * MUW + h * 32 + sub * 4);
            }
            const uint32_t *gmsg = msg + (size_t)pk * E * 32 + sub * 4;
#pragma unroll
            for (int j = 0; j < 8; ++j) {  // edge j of the four variables
                const int e = __shfl_sync(0xffffffffu, mine, 8 * grp + j);
                if (e >= 0) cp_async16(dst + St::AL + (8 * grp + j) * 32 + sub * 4, gmsg + (size_t)(uint32_t)e * 32);
            }
            if (lane < 4 * V) {
                if (n0 + lane / V < N) cp_async4(dst + St::HW + lane, hw + ((size_t)pk * N + n0) * V + lane);
            } else if (lane >= 32 - 2 * V) {
                const int q = lane - (32 - 2 * V);
                cp_async4(dst + St::FL + q, flags + (size_t)pk * 5 * V + (q < V ? q : (1 + par) * V + (q - V)));
            }
        }
        cp_async_commit();
        return mine;
    };
    int next = issue(item, ring), slot = 0;
    for (; item < total; item += step) {
        const int mine = next;
        next = issue(item + step, ring + (slot ^ 1) * St::WORDS);
        cp_async_wait<1>();
        __syncwarp();
        const uint32_t *S = ring + slot * St::WORDS;
        const int a = (int)fdiv((uint32_t)item, divG);
        const int n0 = 4 * (item - a * G), pk = __ldg(act + 1 + a);
        uint32_t *gm = msg + (size_t)pk * E * 32 + lane;
        const uint32_t present = __ballot_sync(0xffffffffu, mine >= 0);  // bit 8 i + j
        uint32_t frozen[V];
        bool lane_on = false;
#pragma unroll
        for (int v = 0; v < V; ++v) {
            uint32_t dn = S[St::FL + v];
            if (STOP) {
                // whoever reads the done word, before or after it is written here, arrives at the same frames
                const uint32_t newly = ~dn & ~S[St::FL + V + v];
                if (n0 == 0 && lane == 0) {
                    uint32_t *flag = flags + (size_t)pk * 5 * V;
                    if (newly) {
                        flag[v] = dn | newly;
                        for (uint32_t b = newly; b; b &= b - 1)
                            iters[(size_t)pk * W + (__ffs(b) - 1) * V + v] = it - 1;
                    }
                    flag[(1 + (par ^ 1)) * V + v] = 0u;  // cleared for the next check pass
                }
                dn |= newly;
            }
            frozen[v] = dn;
            lane_on |= ((~dn) >> lane) & 1u;
        }
#pragma unroll 2
        for (int i = 0; i < 4; ++i) {
            const int n = n0 + i;
            if (n >= N) break;  // warp-uniform
            const uint32_t on = (present >> (8 * i)) & 255u;
            float m[V], pst[V];
            uint32_t q = 0u, outb[V];
            if constexpr (MS) {
                q = S[i * MUW + lane];
            } else {
#pragma unroll
                for (int v = 0; v < V; ++v) m[v] = __uint_as_float(S[i * MUW + lane * V + v]);
            }
            const uint32_t *A = S + St::AL + i * 256 + lane;
            auto put = [&](int j, uint32_t w) {
                const int e = __shfl_sync(0xffffffffu, mine, 8 * i + j);
                if (e >= 0 && lane_on) gm[(size_t)(uint32_t)e * 32] = w;
            };
            if (!(on & 4u)) sparse_variable<2, V, MS>(A, on, m, q, clip, lsb, pst, outb, put);
            else if (!(on & 16u)) sparse_variable<4, V, MS>(A, on, m, q, clip, lsb, pst, outb, put);
            else if (!(on & 64u)) sparse_variable<6, V, MS>(A, on, m, q, clip, lsb, pst, outb, put);
            else sparse_variable<8, V, MS>(A, on, m, q, clip, lsb, pst, outb, put);
            if (POST && lane_on) {
                float *dst = post + ((size_t)pk * N + n) * W + lane * V;
#pragma unroll
                for (int v = 0; v < V; ++v)
                    if (!((frozen[v] >> lane) & 1u)) dst[v] = pst[v];
            }
            if (lane == 0) {
#pragma unroll
                for (int v = 0; v < V; ++v)
                    hw[((size_t)pk * N + n) * V + v] = (outb[v] & ~frozen[v]) | (S[St::HW + i * V + v] & frozen[v]);
            }
        }
        __syncwarp();
        slot ^= 1;
    }
    cp_async_wait<0>();
}

template <int DC, int V, bool MS>
static void sparse_cn(ldpc_code c, const ldpc_decode_opts &o, cudaStream_t s) {
    auto k = sparse_cn_kernel<DC, V, MS>;
    k<<<persistent_blocks(k, 0), 256, 0, s>>>(c->sp, c->d.divM, c->d.E, (uint32_t *)c->ws.msg, c->ws.act, o.clip);
}

template <int DC>
static void sparse_cn(ldpc_code c, const ldpc_decode_opts &o, cudaStream_t s) {
    if (o.algo == LDPC_ALGO_MS) sparse_cn<DC, 4, true>(c, o, s);
    else if (o.msg == LDPC_MSG_F16) sparse_cn<DC, 2, false>(c, o, s);
    else sparse_cn<DC, 1, false>(c, o, s);
}

static void sparse_cn(ldpc_code c, const ldpc_decode_opts &o, cudaStream_t s) {
    const int dc = c->sp.dc_max;
    if (dc <= 8) sparse_cn<8>(c, o, s);
    else if (dc <= 16) sparse_cn<16>(c, o, s);
    else if (dc <= 24) sparse_cn<24>(c, o, s);
    else sparse_cn<32>(c, o, s);
}

template <int V, bool MS, bool STOP, bool POST>
static void sparse_vn(ldpc_code c, const ldpc_decode_opts &o, int it, int par, cudaStream_t s) {
    auto k = sparse_vn_kernel<V, MS, STOP, POST>;
    const size_t smem = (size_t)8 * kSparseStages * SparseStage<V, MS>::WORDS * 4;
    k<<<persistent_blocks(k, smem), 256, smem, s>>>(c->sp, c->d.divG, c->d.N, c->d.E,
                                              (uint32_t *)c->ws.msg, (const uint32_t *)c->ws.mu, c->ws.hw, c->ws.flags,
                                              c->ws.post, c->ws.iters, c->ws.act, o.clip, ldexpf(1.0f, -o.frac_bits), it, par);
}

template <int V, bool MS>
static void sparse_vn(ldpc_code c, const ldpc_decode_opts &o, bool stop, bool post, int it, int par, cudaStream_t s) {
    if (stop) post ? sparse_vn<V, MS, true, true>(c, o, it, par, s) : sparse_vn<V, MS, true, false>(c, o, it, par, s);
    else post ? sparse_vn<V, MS, false, true>(c, o, it, par, s) : sparse_vn<V, MS, false, false>(c, o, it, par, s);
}

ldpc_status sparse_decode_device(ldpc_code c, int gamma, const ldpc_decode_opts &o, bool want_post, cudaStream_t s) {
    if (o.algo == LDPC_ALGO_NOMS) {
        set_error("the learned min-sum takes QC codes (parameters per circulant)");
        return LDPC_EUNSUPPORTED;
    }
    const int V = lanes_per_word(o.msg), W = 32 * V;
    const int P = (gamma + W - 1) / W;
    ldpc_status st = qc_init_flags(c, gamma, V, s);
    if (st != LDPC_OK) return st;
    LDPC_CUDA_TRY(cudaMemsetAsync(c->ws.hw, 0, (size_t)P * c->d.N * V * 4, s));
    st = qc_compact(c, P, V, s);  // every package starts active
    if (st != LDPC_OK) return st;
    {
        const long long n = (long long)P * c->d.E * 32;
        const unsigned blocks = (unsigned)((n + 255) / 256);
        const uint32_t *mu = (const uint32_t *)c->ws.mu;
        uint32_t *msg = (uint32_t *)c->ws.msg;
        if (o.algo == LDPC_ALGO_MS) sparse_init_kernel<4, true><<<blocks, 256, 0, s>>>(mu, msg, c->sp.col, c->d.N, c->d.E, P);
        else if (V == 2) sparse_init_kernel<2, false><<<blocks, 256, 0, s>>>(mu, msg, c->sp.col, c->d.N, c->d.E, P);
        else sparse_init_kernel<1, false><<<blocks, 256, 0, s>>>(mu, msg, c->sp.col, c->d.N, c->d.E, P);
        count_launch(2);
        LDPC_CUDA_TRY(cudaGetLastError());
    }
    for (int it = 1; it <= o.max_iter; ++it) {
        const bool syn = o.early_stop && it >= 2;
        const int par = it & 1;
        if (syn) {  // early stop: the syndrome of the decisions after it - 1 complete iterations
            st = sparse_syndrome(c, P, V, (1 + par) * V, s);
            if (st != LDPC_OK) return st;
        }
        const int slot_cn = prof_begin(0, s);
        sparse_cn(c, o, s);
        LDPC_CUDA_TRY(cudaGetLastError());
        prof_end(slot_cn, s);
        const int slot_vn = prof_begin(1, s);
        // without early stop only the last iteration's posteriors are read
        const bool keep_post = want_post && (o.early_stop || it == o.max_iter);
        if (o.algo == LDPC_ALGO_MS) sparse_vn<4, true>(c, o, syn, keep_post, it, par, s);
        else if (V == 2) sparse_vn<2, false>(c, o, syn, keep_post, it, par, s);
        else sparse_vn<1, false>(c, o, syn, keep_post, it, par, s);
        LDPC_CUDA_TRY(cudaGetLastError());
        prof_end(slot_vn, s);
        count_launch(2);
        if (o.early_stop && it < o.max_iter) {
            st = qc_compact(c, P, V, s);
            if (st != LDPC_OK) return st;
            count_launch();
        }
    }
    st = sparse_syndrome(c, P, V, 4 * V, s);  // fin words: the last decisions
    if (st != LDPC_OK) return st;
    return qc_finish_frames(c, gamma, o, s);
}

}  // namespace ldpc
