// Device part of the on-chip decoder (flow_chip.cu describes it): a package per thread-block cluster.
#pragma once

#include "flow.cuh"

namespace ldpc {
namespace chip {

using namespace flow;

__device__ __forceinline__ uint32_t at_rank(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ uint32_t ld_far(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void st_far(uint32_t addr, uint32_t v) {
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void st_far_half(uint32_t addr, float x) {
    asm volatile("st.shared::cluster.u16 [%0], %1;" ::"r"(addr), "h"(__half_as_ushort(__float2half_rn(x))) : "memory");
}
__device__ __forceinline__ void or_far(uint32_t addr, uint32_t v) {
    asm volatile("red.relaxed.cluster.shared::cluster.or.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void cluster_sync() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// One row of binary16 messages, both frames of the lane word at once (phi on the pair): the sums and
// roundings of sp_row, slot by slot.  x: the row's words; put(l, word).
template <int DC, bool REG, bool FIX, typename PUT>
__device__ __forceinline__ bool row2(uint32_t pm, float clip, const uint32_t *x, PUT put) {
    float pre[DC][2], acc[2] = {0.0f, 0.0f};
    uint32_t sgn = 0u;
    auto terms = [&](int l, float *t) {
        Lane<2>::unpack(x[l] & 0x7fff7fffu, t);
        if (FIX) t[0] = fminf(t[0], 1e30f), t[1] = fminf(t[1], 1e30f);
    };
#pragma unroll
    for (int l = 0; l < DC; ++l) {
        pre[l][0] = acc[0], pre[l][1] = acc[1];
        float t[2];
        terms(l, t);  // an absent slot's word is 0
        sgn ^= x[l];
        acc[0] += t[0], acc[1] += t[1];
    }
    if (!FIX && __any_sync(0xffffffffu, !(acc[0] < 1e30f) || !(acc[1] < 1e30f))) return false;
    float suf[2] = {0.0f, 0.0f};
#pragma unroll
    for (int l = DC - 1; l >= 0; --l) {
        if (!REG && !((pm >> l) & 1u)) continue;  // warp-uniform
        float t[2], m[2];
        terms(l, t);
        phi_pair<4096, 1>(pre[l][0] + suf[0], pre[l][1] + suf[1], m[0], m[1]);
        suf[0] += t[0], suf[1] += t[1];
        m[0] = fminf(m[0], clip), m[1] = fminf(m[1], clip);
        put(l, Lane<2>::pack(m) ^ ((sgn ^ x[l]) & 0x80008000u));
    }
    return true;
}

// REG: every row has its DC slots, so nothing is under a condition and a row's loads and transforms overlap
template <int DC, int JX, int V, int RULE, bool REG>
__global__ void __launch_bounds__(kChipThreads, 1) chip_kernel(const Code c, const ChipArgs a) {
    constexpr bool MS = RULE == kFlowMS;
    constexpr int W = 32 * V, NW = kChipThreads / 32;
    constexpr int MUP = MS ? 33 : W + 1;  // words of a variable's channel LLRs (one pad word: rows and columns of banks)
    extern __shared__ __align__(16) uint32_t sm[];
    __shared__ uint32_t s_un[2][V];
    __shared__ int s_sh[kMaxJ * kMaxL];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    const int pk = (int)(blockIdx.x / (unsigned)a.C);
    const int NC = a.NC, n0 = (int)rank * NC, nv = max(0, min(NC, c.N - n0));
    uint32_t *msg = sm;                                   // [J][NC][32]
    uint32_t *mu = msg + (size_t)c.J * NC * 32;           // [NC][MUP]
    uint32_t *hw = mu + (size_t)NC * MUP;                 // [NC][V]
    float *post = reinterpret_cast<float *>(hw + (size_t)NC * V);  // [NC][W + 1]
    const uint32_t msg_s = smem_u32(msg), mu_s = smem_u32(mu), hw_s = smem_u32(hw), un_s = smem_u32(&s_un[0][0]);
    for (int i = threadIdx.x; i < c.J * c.L; i += kChipThreads) s_sh[i] = c.sh[i];
    if (threadIdx.x < 2 * V) s_un[threadIdx.x / V][threadIdx.x % V] = 0u;
    // this block's variables of the package's frames
    const int f0 = pk * W;
    for (int f = warp; f < W; f += NW) {
        const float *row = c.llr + (size_t)min(f0 + f, c.gamma - 1) * c.N + n0;
        for (int i = lane; i < nv; i += 32) {
            float x = __ldcs(row + i);
            if (f0 + f >= c.gamma) x = MS ? 1e30f : a.clip;  // frames past the batch
            if constexpr (MS) {
                const float t = fminf(fmaxf(rintf(x * a.qscale), -127.0f), 127.0f);
                reinterpret_cast<int8_t *>(mu)[i * MUP * 4 + f] = (int8_t)t;
            } else {
                reinterpret_cast<float *>(mu)[i * MUP + f] = clipf(x, a.clip);
            }
        }
    }
    uint32_t dn[V];
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const int n = c.gamma - f0 - v, lanes = n <= 0 ? 0 : min(32, (n + V - 1) / V);
        dn[v] = lanes == 32 ? 0u : ~((1u << lanes) - 1u);
    }
    cluster_sync();

    // the syndrome of row (j, r) of lane l's slot: the hard-decision words of its variables
    auto slot = [&](int j, int r, uint32_t &owner, int &i) -> bool {
        const int sh = lane < c.L ? s_sh[j * c.L + lane] : -1;
        if (sh < 0) return false;
        int k = r + sh;
        if (k >= c.p) k -= c.p;
        const uint32_t n = (uint32_t)(lane * c.p + k);
        owner = fdiv(n, a.divNC);
        i = (int)(n - owner * (uint32_t)NC);
        return true;
    };
    auto syndrome = [&](int m, uint32_t *un) {
        const int j = (int)fdiv((uint32_t)m, c.divp), r = m - j * c.p;
        uint32_t owner = 0u;
        int i = 0;
        const bool on = slot(j, r, owner, i);
        const uint32_t at = at_rank(hw_s, owner) + (uint32_t)i * (4 * V);
#pragma unroll
        for (int v = 0; v < V; ++v) un[v] |= __reduce_xor_sync(0xffffffffu, on ? ld_far(at + 4 * v) : 0u);
    };
    auto publish = [&](const uint32_t *un, int par) {  // a warp's unsatisfied frames, to every block
#pragma unroll
        for (int v = 0; v < V; ++v)
            if (un[v] && lane < a.C) or_far(at_rank(un_s + (uint32_t)(par * V + v) * 4, lane), un[v]);
    };

    int it = 1;
    bool all = false;
    for (;; ++it) {
        // check step, and the syndrome of the decisions after it - 1 iterations
        const bool first = it == 1, syn = a.early && it >= 2;
        uint32_t un[V];
#pragma unroll
        for (int v = 0; v < V; ++v) un[v] = 0u;
        for (int m = (int)rank * NW + warp; m < c.M; m += a.C * NW) {
            if (syn) syndrome(m, un);
            const int j = (int)fdiv((uint32_t)m, c.divp), r = m - j * c.p;
            uint32_t owner = 0u;
            int i = 0;
            const bool on = slot(j, r, owner, i);
            const uint32_t pm = __ballot_sync(0xffffffffu, on);
            // where slot `lane`'s message line is, and what this step reads of it
            const uint32_t line = at_rank(msg_s, owner) + (uint32_t)(j * NC + i) * 128;
            const uint32_t from = first ? at_rank(mu_s, owner) + (uint32_t)i * (MUP * 4) : line;
            const uint32_t mine = (first && !MS ? V : 1) * 4 * (uint32_t)lane;  // this lane's word within it
            uint32_t xw[DC];
            auto fetch = [&](int v) {
#pragma unroll
                for (int l = 0; l < DC; ++l) {
                    const uint32_t s = __shfl_sync(0xffffffffu, from, l);
                    xw[l] = REG || ((pm >> l) & 1u) ? ld_far(s + mine + 4 * v) : 0u;
                }
            };
            fetch(0);
            if constexpr (MS) {
                uint32_t min1 = 0x7f7f7f7fu, min2 = 0x7f7f7f7fu, sgn = 0u;
#pragma unroll
                for (int l = 0; l < DC; ++l) {
                    if (!REG && !((pm >> l) & 1u)) continue;  // warp-uniform
                    const uint32_t av = __vabsss4(xw[l]);
                    sgn ^= xw[l] & 0x80808080u;
                    min2 = __vminu4(min2, __vmaxu4(min1, av));
                    min1 = __vminu4(min1, av);
                }
#pragma unroll
                for (int l = 0; l < DC; ++l) {
                    const uint32_t to = __shfl_sync(0xffffffffu, line, l);
                    if (!REG && !((pm >> l) & 1u)) continue;
                    const uint32_t eq = __vcmpeq4(__vabsss4(xw[l]), min1);
                    const uint32_t mag = (min2 & eq) | (min1 & ~eq);
                    const uint32_t sneg = ((sgn ^ (xw[l] & 0x80808080u)) >> 7) & 0x01010101u;
                    st_far(to + 4 * lane, __vadd4(mag ^ (sneg * 0xffu), sneg));
                }
            } else if (RULE == kFlowSP && V == 2 && DC <= 16 && !first) {
                // n = 384, 64 frames, 20 iterations: 89 us with a frame after the other, 80 so; 4 x 16, p = 80,
                // 128 frames with early stop: 351, 275 (wider rows lack
                // the registers)
                auto put = [&](int l, uint32_t w) {
                    const uint32_t to = __shfl_sync(0xffffffffu, line, l);
                    st_far(to + 4 * lane, w);
                };
                if (!row2<DC, REG, false>(pm, a.clip, xw, put)) row2<DC, REG, true>(pm, a.clip, xw, put);
            } else {
                const float2 *prm = nullptr;
                if constexpr (RULE == kFlowNOMS)
                    prm = reinterpret_cast<const float2 *>(c.nparams) + ((size_t)(it - 1) * c.J + j) * c.L;
#pragma unroll 1
                for (int v = 0; v < V; ++v) {
                    if (v > 0 && first) fetch(v);  // the FP32 channel LLR of the word's second frame
                    auto term = [&](int l) -> float {
                        if (V == 1 || first) return __uint_as_float(xw[l]);
                        return __half2float(__ushort_as_half((unsigned short)(xw[l] >> (16 * v))));
                    };
                    auto put = [&](int l, float x) {
                        const uint32_t to = __shfl_sync(0xffffffffu, line, l) + 4 * lane;
                        if (!REG && !((pm >> l) & 1u)) return;
                        if constexpr (V == 1) st_far(to, __float_as_uint(x));
                        else st_far_half(to + 2 * v, x);
                    };
                    if constexpr (RULE == kFlowNOMS) {
                        noms_row<DC, REG>(pm, a.clip, prm, term, put);
                    } else if (first) {
                        float t[DC];
#pragma unroll
                        for (int l = 0; l < DC; ++l) t[l] = with_sign_of(phi_f(fabsf(term(l))), term(l) + 0.0f);
                        sp_row<DC, REG, 1>(pm, a.clip, ~0u, [&](int l) { return t[l]; }, put);
                    } else {
                        sp_row<DC, REG, V == 2 ? 4096 : 1>(pm, a.clip, ~0u, term, put);
                    }
                }
            }
        }
        if (syn) publish(un, it & 1);
        cluster_sync();
        if (syn) {
            uint32_t left = 0u;
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const uint32_t newly = ~dn[v] & ~s_un[it & 1][v];
                if (rank == 0 && warp == 0 && ((newly >> lane) & 1u)) {
                    const int f = f0 + lane * V + v;
                    if (c.iters) c.iters[f] = it - 1;
                    if (c.ok) c.ok[f] = 1;
                }
                dn[v] |= newly;
                left |= ~dn[v];
            }
            all = left == 0u;
            if (all) break;  // every block of the cluster alike
        }
        if (threadIdx.x < V) s_un[(it & 1) ^ 1][threadIdx.x] = 0u;  // read before the last two barriers
        // variable step on this block's variables
        const bool keep_post = a.want_post && (a.early || it == a.max_iter);
        for (int i = warp; i < nv; i += NW) {
            const int l = (int)fdiv((uint32_t)(n0 + i), c.divp);
            const uint32_t pm = __ballot_sync(0xffffffffu, lane < c.J && s_sh[min(lane, c.J - 1) * c.L + l] >= 0);
            uint32_t *S = msg + (size_t)i * 32 + lane;
            const int PITCH = NC * 32;
            uint32_t outb[V];
            float pst[V];
            if constexpr (!MS) {
                const float *mf = reinterpret_cast<const float *>(mu) + i * MUP + lane * V;
                float m[V], aj[JX][V], tot[V], bs[JX][V];
#pragma unroll
                for (int v = 0; v < V; ++v) m[v] = mf[v], tot[v] = m[v];
#pragma unroll
                for (int j = 0; j < JX; ++j) {
#pragma unroll
                    for (int v = 0; v < V; ++v) aj[j][v] = 0.0f;
                    if ((pm >> j) & 1u) {
                        Lane<V>::unpack(S[j * PITCH], aj[j]);
#pragma unroll
                        for (int v = 0; v < V; ++v) tot[v] += aj[j][v];
                    }
                }
#pragma unroll
                for (int j = 0; j < JX; ++j)
#pragma unroll
                    for (int v = 0; v < V; ++v) {
                        float s = m[v];
#pragma unroll
                        for (int j2 = 0; j2 < JX; ++j2)
                            if (j2 != j) s += aj[j2][v];
                        bs[j][v] = s;
                    }
                if constexpr (RULE == kFlowSP) {
                    constexpr int SC = V == 2 ? 4096 : 1;
                    float ph[JX][V];
                    if constexpr (V == 2) {
#pragma unroll
                        for (int j = 0; j < JX; ++j)
                            phi_pair<1, SC>(fminf(fabsf(bs[j][0]), a.clip), fminf(fabsf(bs[j][1]), a.clip), ph[j][0],
                                            ph[j][1]);
                    } else {
#pragma unroll
                        for (int j = 0; j < JX; j += 2)
                            phi_pair<1, SC>(fminf(fabsf(bs[j][0]), a.clip), fminf(fabsf(bs[j + 1][0]), a.clip),
                                            ph[j][0], ph[j + 1][0]);
                    }
#pragma unroll
                    for (int j = 0; j < JX; ++j)
#pragma unroll
                        for (int v = 0; v < V; ++v) bs[j][v] = with_sign_of(ph[j][v], bs[j][v]);
                } else {
#pragma unroll
                    for (int j = 0; j < JX; ++j)
#pragma unroll
                        for (int v = 0; v < V; ++v) bs[j][v] = clipf(bs[j][v], a.clip);
                }
#pragma unroll
                for (int j = 0; j < JX; ++j)
                    if ((pm >> j) & 1u) S[j * PITCH] = Lane<V>::pack(bs[j]);
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    pst[v] = clipf(tot[v], a.clip);
                    outb[v] = __ballot_sync(0xffffffffu, pst[v] < 0.0f);
                }
            } else {
                const uint32_t qw = mu[i * MUP + lane];
                uint32_t aw[JX];
                int tot[4];
#pragma unroll
                for (int v = 0; v < 4; ++v) tot[v] = sbyte(qw, v);
#pragma unroll
                for (int j = 0; j < JX; ++j) {
                    aw[j] = (pm >> j) & 1u ? S[j * PITCH] : 0u;
#pragma unroll
                    for (int v = 0; v < 4; ++v) tot[v] += sbyte(aw[j], v);
                }
#pragma unroll
                for (int j = 0; j < JX; ++j) {
                    if (!((pm >> j) & 1u)) continue;
                    uint32_t o = 0u;
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        int b = tot[v] - sbyte(aw[j], v);
                        b = b > 127 ? 127 : (b < -127 ? -127 : b);
                        o |= ((uint32_t)(uint8_t)(int8_t)b) << (8 * v);
                    }
                    S[j * PITCH] = o;
                }
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    pst[v] = (float)tot[v] * a.lsb;
                    outb[v] = __ballot_sync(0xffffffffu, tot[v] < 0);
                }
            }
            if (keep_post) {
#pragma unroll
                for (int v = 0; v < V; ++v)
                    if (!((dn[v] >> lane) & 1u)) post[(size_t)i * (W + 1) + lane * V + v] = pst[v];
            }
            if (lane == 0) {
#pragma unroll
                for (int v = 0; v < V; ++v)
                    hw[i * V + v] = first ? outb[v] & ~dn[v] : (outb[v] & ~dn[v]) | (hw[i * V + v] & dn[v]);
            }
        }
        cluster_sync();
        if (it == a.max_iter) break;
    }
    if (!all) {
        // the last decisions' syndrome: ok flags of the frames that ran to the end
        uint32_t un[V];
#pragma unroll
        for (int v = 0; v < V; ++v) un[v] = 0u;
        for (int m = (int)rank * NW + warp; m < c.M; m += a.C * NW) syndrome(m, un);
        publish(un, (it & 1) ^ 1);  // cleared in the last variable step
        cluster_sync();
        if (rank == 0 && warp == 0) {
#pragma unroll
            for (int v = 0; v < V; ++v) {
                if ((dn[v] >> lane) & 1u) continue;
                const int f = f0 + lane * V + v;
                if (c.iters) c.iters[f] = a.max_iter;
                if (c.ok) c.ok[f] = (s_un[(it & 1) ^ 1][v] >> lane) & 1u ? 0 : 1;
            }
        }
    } else {
        cluster_sync();  // no block leaves while another may still read its words
    }
    const int nf = min(W, c.gamma - f0);
    for (int f = warp; f < nf; f += NW) {
        const int ln = f / V, v = f % V;
        if (c.hard) {
            uint8_t *row = c.hard + (size_t)(f0 + f) * c.N + n0;
            for (int i = lane; i < nv; i += 32) row[i] = (uint8_t)((hw[i * V + v] >> ln) & 1u);
        }
        if (c.post) {
            float *row = c.post + (size_t)(f0 + f) * c.N + n0;
            for (int i = lane; i < nv; i += 32) row[i] = post[(size_t)i * (W + 1) + f];
        }
    }
}

template <int DC, int JX, int V, int RULE, bool REG>
static ldpc_status launch(const Code &c, ChipArgs &a, int P, cudaStream_t s, bool *taken) {
    auto k = chip_kernel<DC, JX, V, RULE, REG>;
    const int C = pick((const void *)k, c, V, RULE == kFlowMS, a, P);
    *taken = C > 0;
    if (!C) return LDPC_OK;
    a.C = C;
    a.NC = (c.N + C - 1) / C;
    a.divNC = fast_div((uint32_t)a.NC);
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at[1];
    cfg.gridDim = dim3((unsigned)(P * C));
    cfg.blockDim = dim3(kChipThreads);
    cfg.dynamicSmemBytes = std::max(bytes(c, V, RULE == kFlowMS, a.want_post, a.NC), kChipLeast);
    cfg.stream = s;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = C;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    LDPC_CUDA_TRY(cudaLaunchKernelEx(&cfg, k, c, a));
    count_launch();
    LDPC_CUDA_TRY(cudaGetLastError());
    return LDPC_OK;
}

// kernels by row degree: full rows of 6, 8, 12 and 24 slots (without conditions: n = 384, 92 us with them,
// 86 without), else rows of up to 8, 16, 32 slots, some empty; more than four block rows
template <int V, int RULE>
static ldpc_status dispatch(const Code &c, ChipArgs &a, int P, cudaStream_t s, bool *taken) {
    bool regular = true;
    for (int i = 0; i < c.J * c.L; ++i) regular &= c.sh[i] >= 0;
    if (c.J > 4) return launch<32, 8, V, RULE, false>(c, a, P, s, taken);
    if (regular && c.L == 6) return launch<6, 4, V, RULE, true>(c, a, P, s, taken);
    if (regular && c.L == 8) return launch<8, 4, V, RULE, true>(c, a, P, s, taken);
    if (regular && c.L == 12) return launch<12, 4, V, RULE, true>(c, a, P, s, taken);
    if (regular && c.L == 24) return launch<24, 4, V, RULE, true>(c, a, P, s, taken);
    if (c.L <= 8) return launch<8, 4, V, RULE, false>(c, a, P, s, taken);
    if (c.L <= 16) return launch<16, 4, V, RULE, false>(c, a, P, s, taken);
    return launch<32, 4, V, RULE, false>(c, a, P, s, taken);
}

}  // namespace chip
}  // namespace ldpc
