// Device part of the flow decoder (flow.cu describes the scheme): the tile kernel of one
// message rule, and the launch of it.  Included by one translation unit per rule.
#pragma once

#include "flow_internal.cuh"
#include "qc_device.cuh"

#include <algorithm>

namespace ldpc {
namespace flow {

// ---------------------------------------------------------------------------
// mbarriers, bulk copies, fences
// ---------------------------------------------------------------------------
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0u;
}
constexpr int kWaitLimit = 1 << 23;  // tries of one wait (each suspends up to the hardware's time limit)
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
    for (int i = 0; i < kWaitLimit; ++i)
        if (mbar_try(bar, parity)) return true;
    return false;
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void bulk_store(void *dst, uint32_t src, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(src), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void bulk_wait() {  // all but the last N groups are complete
    asm volatile("cp.async.bulk.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void fence_async() { asm volatile("fence.proxy.async;" ::: "memory"); }
__device__ __forceinline__ void fence_async_global() { asm volatile("fence.proxy.async.global;" ::: "memory"); }
__device__ __forceinline__ void fence_async_shared() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void ld_entry(const Entry *p, unsigned long long &w0, unsigned long long &w1) {
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(w0), "=l"(w1) : "l"(p) : "memory");
}
__device__ __forceinline__ void st_entry(Entry *p, unsigned long long w0, unsigned long long w1) {
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(w0), "l"(w1) : "memory");
}
__device__ __forceinline__ uint32_t add_done(unsigned int *p, uint32_t x) {
    uint32_t v;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(v) : "l"(p), "r"(x) : "memory");
    return v;
}
__device__ __forceinline__ int ld_int(const int *p) {
    int v;
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void warps_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kComputeWarps * 32) : "memory"); }  // the compute warps

// ---------------------------------------------------------------------------
// what a tile kernel is built for
// ---------------------------------------------------------------------------
// RULE: sum-product (FP32: V = 1, FP16: V = 2), integer min-sum (V = 4), learned min-sum (V = 1, 2)
template <int DC, int JX, int V, int RULE, bool REG>
struct Cfg {
    static constexpr bool MS = RULE == kFlowMS;
    static constexpr int W = 32 * V;                  // frames of a package
    static constexpr int ROWS = tile_rows(JX, DC);
    static constexpr int FV = MS ? 1 : V;             // channel-LLR words per lane and variable
    static constexpr int ROWS1 = ROWS / FV;           // rows of a first-iteration tile (it reads the channel LLRs)
    static constexpr int KC = JX <= 4 ? 4 * kComputeWarps : 2 * kComputeWarps;  // variables of a tile
    static constexpr int CNW = DC * ROWS * 32;        // words of a check tile
    static constexpr int VNW = KC * (JX + FV) * 32;   // words of a variable tile
    static constexpr int STAGE = CNW > VNW ? CNW : VNW;
    static constexpr int OUTV = outv(JX);             // variables of a pack / output tile
    static constexpr int CHANV = KC * (JX + FV) / FV / 128 * 128;  // variables of a channel tile (whole stage)
    static constexpr int SYNROWS = kSynRows;
    // pack: OUTV lines of W values with one pad value (bytes for min-sum)
    static_assert((MS ? OUTV * (W + 4) / 4 : OUTV * (W + 1)) <= STAGE, "pack tile");
};

struct Desc {
    int kind, rows, j, first, n0, slot, pk, it, post, stop;
    uint32_t pm, tiles;
    uint32_t dn[4];
};

template <int STAGEW, int V>
struct Smem {
    uint32_t stage[kStages][STAGEW];
    Desc desc[kStages];
    int dst[kStages][32];       // check tile: the message line of slot l's first row; variable tile: of block row j
    int n1[kStages][32];        // check tile: rows before the wrap of slot l's circulant, -1: absent
    uint8_t list[kStages][32 * V];  // channel tile: the package's frames that enter, and their ids
    uint32_t fid[kStages][32 * V];  // (less the launch's first)
    uint32_t hw[kStages][4 * kComputeWarps * V];  // variable tile: the decisions so far (where frames have stopped)
    Code code;
    alignas(8) unsigned long long full[kStages], used[kStages], empty[kStages];
};

// ---------------------------------------------------------------------------
// check rules on one row.  S: the lane's word of slot 0 in the stage; slot l's at S[l * PITCH].
// ---------------------------------------------------------------------------
// phi without the clamp at 100, of arguments scaled by 1/IN, times OUT (powers of two, so every
// rounding is that of the unscaled form): the sums that reach it are finite (sp_row)
template <int INV_IN, int OUT>
__device__ __forceinline__ void phi_pair(float x0, float x1, float &y0, float &y1) {
    constexpr float IN = 1.0f / INV_IN, O = (float)OUT;
    const float L2E = 1.44269502f, L2E_LO = 1.92596299e-8f, LN2 = 0.693147182f;
    const f32x2 x = f2(x0, x1);
    const f32x2 na = f2mul(x, f2c(L2E * IN));
    f32x2 alo = f2fma(x, f2c(-L2E * IN), na);
    alo = f2fma(x, f2c(-L2E_LO * IN), alo);
    float n0, n1;
    f2split(na, n0, n1);
    const f32x2 t0 = f2(ex2_approx(-n0), ex2_approx(-n1));
    const f32x2 t = f2fma(t0, f2mul(alo, f2c(LN2)), t0);
    const f32x2 v = f2mul(t, t);
    const f32x2 w = f2mul(f2c(2.0f * O), t);
    f32x2 P = f2fma(f2c(0.147845685f), v, f2c(0.138392285f));
    P = f2fma(P, v, f2c(0.200207084f));
    P = f2fma(P, v, f2c(0.333330393f));
    const f32x2 h = f2fma(w, f2mul(v, P), w);
    const f32x2 y = f2mul(f2c(0.5f * IN), x);
    const f32x2 u = f2mul(y, y);
    f32x2 G = f2fma(f2c(-0.00555368373f * O), u, f2c(0.0216362253f * O));
    G = f2fma(G, u, f2c(-0.0777590200f * O));
    G = f2fma(G, u, f2c(0.333332866f * O));
    G = f2mul(u, G);
    float q0, q1;
    f2split(y, q0, q1);
    const f32x2 lo = f2fma(f2(lg2_approx(q0), lg2_approx(q1)), f2c(-LN2 * O), G);
    float h0, h1, l0, l1;
    f2split(h, h0, h1);
    f2split(lo, l0, l1);
    y0 = x0 < (float)INV_IN ? l0 : h0;
    y1 = x1 < (float)INV_IN ? l1 : h1;
}

// One row of one frame, sum-product: x(l) gives slot l's signed term sign(beta) phi(|beta|) (scaled
// by SC), out(l, alpha) takes the result.  Prefix sums, then the backward sweep adds the suffix
// sums (it reads the terms again: twice the shared-memory reads, but 36 registers fewer); phi on
// pairs of slots.  keep: all ones, or 0 for a frame that has just entered its slot (alpha = 0, so the
// variable step starts it at beta = mu).  An infinite term (beta = 0) counts as 1e30, whose sums give the same result
// (phi = 0) and stay finite, so the sweep needs no clamp: that is checked once a row on the whole sum.
template <int DC, bool REG, int SC, bool FIX, typename X, typename O>
__device__ __forceinline__ float sp_sweep(uint32_t pm, float clip, uint32_t keep, X x, O out) {
    float pre[DC / 2];  // the prefix sums before even slots; those before odd ones are one addition away
    uint32_t sgn = 0u;
    float acc = 0.0f;
    auto term = [&](int l) {
        float t = REG || ((pm >> l) & 1u) ? x(l) : 0.0f;
        if (FIX) t = with_sign_of(fminf(fabsf(t), 1e30f), t);
        return t;
    };
#pragma unroll
    for (int l = 0; l < DC; ++l) {
        const float t = term(l);
        sgn ^= __float_as_uint(t);
        if (l % 2 == 0) pre[l / 2] = acc;
        acc += fabsf(t);
    }
    if (!FIX && __any_sync(0xffffffffu, !(acc < 1e30f))) return 1.0f;
    sgn &= 0x80000000u;
    float suf = 0.0f;
    static_assert(DC % 2 == 0, "slot pairs");
#pragma unroll
    for (int l = DC - 1; l >= 1; l -= 2) {
        if (!REG && ((pm >> (l - 1)) & 3u) == 0u) continue;  // warp-uniform
        const float t0 = term(l), t1 = term(l - 1);
        const float a0 = (pre[l / 2] + fabsf(t1)) + suf;
        suf += fabsf(t0);
        const float a1 = pre[l / 2] + suf;
        suf += fabsf(t1);
        float m0, m1;
        phi_pair<SC, 1>(a0, a1, m0, m1);
        const uint32_t s0 = sgn ^ (__float_as_uint(t0) & 0x80000000u), s1 = sgn ^ (__float_as_uint(t1) & 0x80000000u);
        out(l, __uint_as_float((__float_as_uint(fminf(m0, clip)) ^ s0) & keep));
        out(l - 1, __uint_as_float((__float_as_uint(fminf(m1, clip)) ^ s1) & keep));
    }
    return 0.0f;
}
template <int DC, bool REG, int SC, typename X, typename O>
__device__ __forceinline__ void sp_row(uint32_t pm, float clip, uint32_t keep, X x, O out) {
    if (sp_sweep<DC, REG, SC, false>(pm, clip, keep, x, out) != 0.0f)
        sp_sweep<DC, REG, SC, true>(pm, clip, keep, x, out);
}

// one row of one frame, normalized/offset min-sum: x(l) gives beta, prm(l) the slot's (w, o)
template <int DC, bool REG, typename X, typename O>
__device__ __forceinline__ void noms_row(uint32_t pm, float clip, const float2 *__restrict__ prm, X x, O out) {
    float ab[DC], mn1 = INFINITY, mn2 = INFINITY;
    uint32_t neg = 0u;
#pragma unroll
    for (int l = 0; l < DC; ++l) {
        ab[l] = INFINITY;
        if (REG || ((pm >> l) & 1u)) {
            const float v = x(l);
            ab[l] = fabsf(v);
            neg |= (v < 0.0f ? 1u : 0u) << l;
            mn2 = fminf(mn2, fmaxf(mn1, ab[l]));
            mn1 = fminf(mn1, ab[l]);
        }
    }
    const uint32_t flip = (__popc(neg) & 1u) ? ~neg : neg;
#pragma unroll
    for (int l = 0; l < DC; ++l) {
        if (!REG && !((pm >> l) & 1u)) continue;  // warp-uniform
        const float2 wo = __ldg(prm + l);
        const float m = ab[l] == mn1 ? mn2 : mn1;
        const float mag = fminf(fmaxf(fmaf(wo.x, m, -wo.y), 0.0f), clip);
        out(l, ((flip >> l) & 1u) ? -mag : mag);
    }
}

// check tile: compute warp `warp` takes rows warp, warp + 24, ... of the tile, in place
template <typename C, int DC, int V, int RULE, bool REG>
__device__ __forceinline__ void cn_tile(uint32_t *stage, const Desc &d, int warp, int lane, float clip,
                                        const float2 *__restrict__ prm) {
    constexpr int PITCH = C::ROWS * 32;  // words from one slot's lines to the next slot's
    const uint32_t pm = d.pm;
    if constexpr (RULE == kFlowMS) {
        uint32_t keep = 0u;  // bytes of the frames that have not just entered
#pragma unroll
        for (int v = 0; v < 4; ++v) keep |= ((d.dn[v] >> lane) & 1u) ? 0u : 0xffu << (8 * v);
        for (int r = warp; r < d.rows; r += kComputeWarps) {
            uint32_t *S = stage + r * 32 + lane;
            uint32_t ab[DC], sg[DC];
            uint32_t min1 = 0x7f7f7f7fu, min2 = 0x7f7f7f7fu, sgn = 0u;
#pragma unroll
            for (int l = 0; l < DC; ++l) {
                ab[l] = sg[l] = 0u;
                if (REG || ((pm >> l) & 1u)) {
                    const uint32_t x = S[l * PITCH];
                    const uint32_t av = __vabsss4(x);
                    sg[l] = x & 0x80808080u;
                    ab[l] = av;
                    sgn ^= sg[l];
                    min2 = __vminu4(min2, __vmaxu4(min1, av));
                    min1 = __vminu4(min1, av);
                }
            }
#pragma unroll
            for (int l = 0; l < DC; ++l) {
                if (!REG && !((pm >> l) & 1u)) continue;  // warp-uniform
                const uint32_t eq = __vcmpeq4(ab[l], min1);
                const uint32_t mag = (min2 & eq) | (min1 & ~eq);
                const uint32_t sneg = ((sgn ^ sg[l]) >> 7) & 0x01010101u;
                S[l * PITCH] = __vadd4(mag ^ (sneg * 0xffu), sneg) & keep;
            }
        }
    } else if (d.first && V == 2) {
        // first iteration from the FP32 channel LLRs, two frames per lane: warps take (row, frame); the
        // results, half the size, go where the inputs were once every warp has read its own
        static_assert(C::ROWS1 * 2 == C::ROWS || V != 2, "row, frame pairs");
        for (int q0 = 0; q0 < 2 * C::ROWS1; q0 += kComputeWarps) {
            const int q = q0 + warp, r = q >> 1, v = q & 1;
            const bool on = r < d.rows;
            const float *S = reinterpret_cast<const float *>(stage) + r * 64 + lane * 2 + v;
            __half *D = reinterpret_cast<__half *>(stage) + r * 64 + lane * 2 + v;
            float x[DC];
#pragma unroll
            for (int l = 0; l < DC; ++l) x[l] = on && (REG || ((pm >> l) & 1u)) ? S[l * PITCH] : 0.0f;
            warps_sync();
            if (!on) continue;
            auto put = [&](int l, float a) {
                if (REG || ((pm >> l) & 1u)) D[l * PITCH * 2] = __float2half_rn(a);
            };
            if constexpr (RULE == kFlowNOMS) {
                noms_row<DC, REG>(pm, clip, prm, [&](int l) { return x[l]; }, put);
            } else {
                // x + 0 turns -0 into +0 (the sign of a channel LLR is that of x < 0)
                sp_row<DC, REG, 1>(pm, clip, ~0u, [&](int l) { return with_sign_of(phi_f(fabsf(x[l])), x[l] + 0.0f); }, put);
            }
        }
    } else {
        for (int r = warp; r < d.rows; r += kComputeWarps) {
            uint32_t *S = stage + r * 32 + lane;
            if constexpr (V == 1) {
                auto put = [&](int l, float a) {
                    if (REG || ((pm >> l) & 1u)) S[l * PITCH] = __float_as_uint(a);
                };
                if constexpr (RULE == kFlowNOMS) {
                    noms_row<DC, REG>(pm, clip, prm, [&](int l) { return __uint_as_float(S[l * PITCH]); }, put);
                } else {
                    if (d.first) {
#pragma unroll 4
                        for (int l = 0; l < DC; ++l) {
                            if (!REG && !((pm >> l) & 1u)) continue;  // warp-uniform
                            const float x = __uint_as_float(S[l * PITCH]);
                            S[l * PITCH] = __float_as_uint(with_sign_of(phi_f(fabsf(x)), x + 0.0f));
                        }
                    }
                    sp_row<DC, REG, 1>(pm, clip, ((d.dn[0] >> lane) & 1u) - 1u,
                                       [&](int l) { return __uint_as_float(S[l * PITCH]); }, put);
                }
            } else {
                // the two frames of a lane word one after the other, each through its half of the words
                __half *H = reinterpret_cast<__half *>(S);
#pragma unroll 1
                for (int v = 0; v < V; ++v) {
                    auto get = [&](int l) { return __half2float(H[l * PITCH * 2 + v]); };
                    auto put = [&](int l, float a) {
                        if (REG || ((pm >> l) & 1u)) H[l * PITCH * 2 + v] = __float2half_rn(a);
                    };
                    if constexpr (RULE == kFlowNOMS) noms_row<DC, REG>(pm, clip, prm, get, put);
                    else sp_row<DC, REG, 4096>(pm, clip, ((d.dn[v] >> lane) & 1u) - 1u, get, put);
                }
            }
        }
    }
}

// variable tile: warp `warp` takes variables warp, warp + 24, ...; beta (or its transform) in place,
// decision words and posteriors to global memory
template <typename C, int JX, int V, int RULE, bool REG>
__device__ __forceinline__ void vn_tile(uint32_t *stage, const uint32_t *hwold, const Desc &d, int warp, int lane,
                                        float clip, float lsb, uint32_t *__restrict__ hw, float *__restrict__ post) {
    constexpr int PITCH = C::KC * 32;
    const uint32_t pm = d.pm;
    uint32_t frozen[V], any = 0u;
#pragma unroll
    for (int v = 0; v < V; ++v) frozen[v] = d.dn[v], any |= d.dn[v];
#pragma unroll (V == 1 ? 4 : 1)
    for (int i = warp; i < d.rows; i += kComputeWarps) {
        uint32_t *S = stage + i * 32 + lane;
        uint32_t outb[V];
        float pst[V];
        if constexpr (RULE != kFlowMS) {
            const float *mf = reinterpret_cast<const float *>(stage + JX * PITCH) + (i * 32 + lane) * V;
            float m[V], aj[JX][V], tot[V], bs[JX][V];
            if constexpr (V == 2) {
                const float2 t = *reinterpret_cast<const float2 *>(mf);
                m[0] = t.x, m[1] = t.y;
            } else {
                m[0] = mf[0];
            }
#pragma unroll
            for (int v = 0; v < V; ++v) tot[v] = m[v];
#pragma unroll
            for (int j = 0; j < JX; ++j) {
#pragma unroll
                for (int v = 0; v < V; ++v) aj[j][v] = 0.0f;
                if (REG || ((pm >> j) & 1u)) {
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
                // the check rule sums phi(|beta|): evaluate it here, from the unrounded beta, keep beta's sign
                constexpr int SC = V == 2 ? 4096 : 1;
                float ph[JX][V];
                if constexpr (V == 2) {
#pragma unroll
                    for (int j = 0; j < JX; ++j) {
                        if (!REG && !((pm >> j) & 1u)) continue;
                        phi_pair<1, SC>(fminf(fabsf(bs[j][0]), clip), fminf(fabsf(bs[j][1]), clip), ph[j][0], ph[j][1]);
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < JX; j += 2) {
                        if (!REG && ((pm >> j) & 3u) == 0u) continue;
                        phi_pair<1, SC>(fminf(fabsf(bs[j][0]), clip), fminf(fabsf(bs[j + 1][0]), clip), ph[j][0],
                                        ph[j + 1][0]);
                    }
                }
#pragma unroll
                for (int j = 0; j < JX; ++j)
#pragma unroll
                    for (int v = 0; v < V; ++v) bs[j][v] = with_sign_of(ph[j][v], bs[j][v]);
            } else {
#pragma unroll
                for (int j = 0; j < JX; ++j)
#pragma unroll
                    for (int v = 0; v < V; ++v) bs[j][v] = clipf(bs[j][v], clip);
            }
#pragma unroll
            for (int j = 0; j < JX; ++j)
                if (REG || ((pm >> j) & 1u)) S[j * PITCH] = Lane<V>::pack(bs[j]);
#pragma unroll
            for (int v = 0; v < V; ++v) {
                pst[v] = clipf(tot[v], clip);
                outb[v] = __ballot_sync(0xffffffffu, pst[v] < 0.0f);
            }
        } else {
            const uint32_t qw = stage[JX * PITCH + i * 32 + lane];
            uint32_t aw[JX];
            int tot[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) tot[v] = sbyte(qw, v);
#pragma unroll
            for (int j = 0; j < JX; ++j) {
                aw[j] = REG || ((pm >> j) & 1u) ? S[j * PITCH] : 0u;
#pragma unroll
                for (int v = 0; v < 4; ++v) tot[v] += sbyte(aw[j], v);
            }
#pragma unroll
            for (int j = 0; j < JX; ++j) {
                if (!REG && !((pm >> j) & 1u)) continue;
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
                pst[v] = (float)tot[v] * lsb;
                outb[v] = __ballot_sync(0xffffffffu, tot[v] < 0);
            }
        }
        if (d.post) {
            float *dst = post + ((size_t)(d.n0 + i) * 32 + lane) * V;
#pragma unroll
            for (int v = 0; v < V; ++v)
                if (!((frozen[v] >> lane) & 1u)) dst[v] = pst[v];
        }
        if (any) {  // the stopped frames keep their decisions
#pragma unroll
            for (int v = 0; v < V; ++v) outb[v] = (outb[v] & ~frozen[v]) | (hwold[i * V + v] & frozen[v]);
        }
        if (lane == 0) {
            uint32_t *h = hw + (size_t)(d.n0 + i) * V;
            if constexpr (V == 1) h[0] = outb[0];
            else if constexpr (V == 2) *reinterpret_cast<uint2 *>(h) = make_uint2(outb[0], outb[1]);
            else *reinterpret_cast<uint4 *>(h) = make_uint4(outb[0], outb[1], outb[2], outb[3]);
        }
    }
}

// pack tile: channel LLRs of OUTV variables, frame-major rows of the caller -> package lines
template <typename C, int V, bool MS>
__device__ __forceinline__ void pack_tile(uint32_t *stage, const Code &c, const Desc &d, int warp, int lane, float clip,
                                          float qscale, void *__restrict__ mu) {
    constexpr int W = C::W;
    const int f0 = d.pk * W;
    const int nv = min(C::OUTV, c.N - d.n0);
    for (int f = warp; f < W; f += kComputeWarps) {
        // unconditional loads (of the last frame and variable where there is none), so that they overlap
        const float *row = c.llr + (size_t)min(f0 + f, c.gamma - 1) * c.N + d.n0;
        float x[C::OUTV / 32];
#pragma unroll
        for (int q = 0; q < C::OUTV / 32; ++q) x[q] = __ldcs(row + min(q * 32 + lane, nv - 1));
        if (f0 + f >= c.gamma)
#pragma unroll
            for (int q = 0; q < C::OUTV / 32; ++q) x[q] = MS ? 1e30f : clip;  // frames past the batch
#pragma unroll
        for (int q = 0; q < C::OUTV / 32; ++q) {
            const int i = q * 32 + lane;
            if constexpr (MS) {
                const float t = fminf(fmaxf(rintf(x[q] * qscale), -127.0f), 127.0f);
                reinterpret_cast<int8_t *>(stage)[i * (W + 4) + f] = (int8_t)t;
            } else {
                reinterpret_cast<float *>(stage)[i * (W + 1) + f] = clipf(x[q], clip);
            }
        }
    }
    warps_sync();
    for (int i = warp; i < nv; i += kComputeWarps) {
        if constexpr (MS) {
            reinterpret_cast<uint32_t *>(mu)[(size_t)(d.n0 + i) * 32 + lane] = stage[i * (W + 4) / 4 + lane];
        } else {
            const float *s = reinterpret_cast<const float *>(stage) + i * (W + 1) + lane * V;
            float *o = reinterpret_cast<float *>(mu) + ((size_t)(d.n0 + i) * 32 + lane) * V;
            if constexpr (V == 2) *reinterpret_cast<float2 *>(o) = make_float2(s[0], s[1]);
            else o[0] = s[0];
        }
    }
    warps_sync();  // the stage is handed on
}

// output tile: decisions and posteriors of OUTV variables -> the caller's frame-major rows
template <typename C, int V>
__device__ __forceinline__ void out_tile(uint32_t *stage, const Code &c, const Desc &d, int warp, int lane,
                                         const uint32_t *__restrict__ hw, const float *__restrict__ post) {
    constexpr int W = C::W, NV = C::OUTV;
    const int f0 = d.pk * W, nf = min(W, c.gamma - f0);
    const int nv = min(NV, c.N - d.n0);
    if (c.hard) {
        for (int x = warp * 32 + lane; x < nv * V; x += kComputeWarps * 32) stage[x] = __ldcg(hw + (size_t)d.n0 * V + x);
        warps_sync();
        for (int f = warp; f < nf; f += kComputeWarps) {
            uint8_t *row = c.hard + (size_t)(f0 + f) * c.N + d.n0;
            const int ln = f / V, v = f % V;
#pragma unroll
            for (int q = 0; q < NV / 32; ++q) {
                const int i = q * 32 + lane;
                if (i < nv) row[i] = (uint8_t)((stage[i * V + v] >> ln) & 1u);
            }
        }
        warps_sync();
    }
    if (c.post) {
        // half of the tile at a time for the wide packages
        constexpr int H = NV * (W + 1) <= C::STAGE ? NV : NV / 4;
        for (int h0 = 0; h0 < nv; h0 += H) {
            const int hn = min(H, nv - h0);
#pragma unroll 4
            for (int i = warp; i < hn; i += kComputeWarps)
#pragma unroll
                for (int v = 0; v < V; ++v)
                    reinterpret_cast<float *>(stage)[i * (W + 1) + v * 32 + lane] =
                        __ldcg(post + (size_t)(d.n0 + h0 + i) * W + v * 32 + lane);
            warps_sync();
            for (int f = warp; f < nf; f += kComputeWarps) {
                float *row = c.post + (size_t)(f0 + f) * c.N + d.n0 + h0;
                for (int i = lane; i < hn; i += 32) row[i] = reinterpret_cast<const float *>(stage)[i * (W + 1) + f];
            }
            warps_sync();
        }
    }
}

// syndrome tile: 256 check rows of the package's decisions, eq. (hrddcs); unsatisfied frames to un
template <int V>
__device__ __forceinline__ void syn_tile(const Code &c, const Desc &d, int warp, int lane,
                                         const uint32_t *__restrict__ hw, uint32_t *__restrict__ un) {
    if (warp >= kSynRows / 32) return;
    const int m = d.n0 + warp * 32 + lane;
    uint32_t syn[V];
#pragma unroll
    for (int v = 0; v < V; ++v) syn[v] = 0u;
    if (m < c.M) {
        const int j = (int)fdiv((uint32_t)m, c.divp), r = m - j * c.p;
        constexpr int B = 24 / V;  // edges whose loads are in flight together
        for (int l0 = 0; l0 < c.L; l0 += B) {
            uint32_t w[B][V];
#pragma unroll
            for (int i = 0; i < B; ++i) {
                // absent edges read word 0 and are masked: loads under a condition are not overlapped
                // (4900 cycles for eight, against 2300)
                const int l = l0 + i;
                const int a = l < c.L ? c.sh[j * c.L + l] : -1;
                int k = r + a;
                if (k >= c.p) k -= c.p;
                const uint32_t on = a >= 0 ? 0xffffffffu : 0u;
                const uint32_t *h = hw + (a >= 0 ? ((size_t)l * c.p + k) * V : (size_t)0);
#pragma unroll
                for (int v = 0; v < V; ++v) w[i][v] = __ldcg(h + v) & on;
            }
#pragma unroll
            for (int i = 0; i < B; ++i)
#pragma unroll
                for (int v = 0; v < V; ++v) syn[v] ^= w[i][v];
        }
    }
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const uint32_t o = __reduce_or_sync(0xffffffffu, syn[v]);
        if (lane == 0 && o) atomicOr(un + v, o);
    }
}

// refill mode: wrong bits (all-zero codeword) of the frames that leave, from their last decisions
template <int V>
__device__ __forceinline__ void err_tile(const Code &c, const Desc &d, int warp, int lane,
                                         const uint32_t *__restrict__ hw, int *__restrict__ errs) {
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const uint32_t ret = d.dn[v];
        if (!ret) continue;
        uint32_t w[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int n = d.n0 + warp * 128 + q * 32 + lane;
            w[q] = n < c.N ? __ldcg(hw + (size_t)n * V + v) & ret : 0u;
        }
        int cnt = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q)
            for (uint32_t m = __ballot_sync(0xffffffffu, w[q] != 0u); m; m &= m - 1)  // mostly none
                cnt += (__shfl_sync(0xffffffffu, w[q], __ffs(m) - 1) >> lane) & 1u;
        if (cnt) atomicAdd(errs + lane * V + v, cnt);
    }
}

// streaming: the decisions of the frames that leave, to their rows of the caller's bytes
template <int V>
__device__ __forceinline__ void rows_tile(const Code &c, const Sim &si, const SimSlot &ss, const Desc &d, int warp, int lane,
                                          const uint32_t *__restrict__ hw) {
    const int n0 = d.n0 + warp * 128;
    if (n0 >= c.N) return;
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const uint32_t ret = d.dn[v];
        if (!ret) continue;
        uint32_t w[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int n = n0 + (si.wide_out ? 4 * lane + e : 32 * e + lane);
            w[e] = n < c.N ? __ldcg(hw + (size_t)n * V + v) : 0u;
        }
        for (uint32_t m = ret; m; m &= m - 1) {
            const int ln = __ffs(m) - 1;
            uint8_t *row = si.hard + __ldcg(&ss.rfid[ln * V + v]) * (unsigned long long)c.N + n0;
            if (si.wide_out) {
                const uint32_t x = ((w[0] >> ln) & 1u) | (((w[1] >> ln) & 1u) << 8) | (((w[2] >> ln) & 1u) << 16) |
                                   (((w[3] >> ln) & 1u) << 24);
                if (n0 + 4 * lane < c.N) reinterpret_cast<uint32_t *>(row)[lane] = x;
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (n0 + 32 * e + lane < c.N) row[32 * e + lane] = (uint8_t)((w[e] >> ln) & 1u);
            }
        }
    }
}

// refill mode: channel LLRs of the frames that enter, into the lines of CHANV variables (in the stage):
// drawn from the channel, or read from the caller's rows
template <typename C, int V, bool MS>
__device__ __forceinline__ void chan_tile(uint32_t *stage, const uint8_t *list, const uint32_t *fid, const Code &c,
                                          const Sim &si, const Desc &d, int warp, int lane, float clip, float qscale) {
    constexpr int Q = C::CHANV / 4;
    const int nf = d.rows, total = nf * Q;
    // a few frames do not fill the warps: start with another warp in each tile
    const int first = (warp + d.n0 / C::CHANV * 13) % kComputeWarps;
    for (int x = first * 32 + lane; x < total; x += kComputeWarps * 32) {
        // neighbouring lanes: other frames (other banks), or the next quarter-words of the row they read
        const int i = si.io ? x / Q : x % nf, q = si.io ? x % Q : x / nf;
        const int f = list[i], n = d.n0 + 4 * q;
        if (n >= c.N) continue;
        const unsigned long long F = si.first + fid[i];
        float y[4];
        if (si.io) {
            const float *row = si.llr + F * (unsigned long long)c.N + n;
            if (si.wide_in) {
                const float4 t = __ldcs(reinterpret_cast<const float4 *>(row));
                y[0] = t.x, y[1] = t.y, y[2] = t.z, y[3] = t.w;
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e) y[e] = n + e < c.N ? __ldcs(row + e) : 0.0f;
            }
        } else {
            channel_quad(si.seed, F, n >> 2, si.sigma, si.s2, y);
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if (n + e >= c.N) break;
            if constexpr (MS) {
                const float t = fminf(fmaxf(rintf(y[e] * qscale), -127.0f), 127.0f);
                reinterpret_cast<int8_t *>(stage)[(4 * q + e) * C::W + f] = (int8_t)t;
            } else {
                reinterpret_cast<float *>(stage)[(4 * q + e) * C::W + f] = clipf(y[e], clip);
            }
        }
    }
}

// ---------------------------------------------------------------------------
// the control warp
// ---------------------------------------------------------------------------
// A block's place in the log of opened phases: tile i of a phase goes to block (base + i) mod blocks,
// so every block finds its own tiles by reading the log and none is handed out by an atomic.
struct Place {
    uint32_t n = 0u;       // entry in hand (once idx is set), else the next to look at
    uint32_t first = 0u;   // the lanes hold entries first .. first + 31
    unsigned long long w0 = 0ull, w1 = 0ull;
    uint32_t idx = ~0u;    // this block's next tile of the entry in hand
    unsigned long long e0 = 0ull, e1 = 0ull;
    bool loaded = false;
};
__device__ __forceinline__ uint32_t bits(unsigned long long x, int at, int n) {
    return (uint32_t)(x >> at) & ((1u << n) - 1u);
}

// This block's next tile (its number in pl.idx - blocks, its phase in pl.e0, pl.e1); false: every
// package is done (or the kernel gives up).
__device__ __forceinline__ bool take(const Args &a, int lane, Place &pl, uint32_t &idx) {
    if (pl.idx != ~0u) {
        if (pl.idx < bits(pl.e1, 0, kLogTiles)) {
            idx = pl.idx;
            pl.idx += gridDim.x;
            return true;
        }
        pl.idx = ~0u;
        ++pl.n;
    }
    for (int tries = 0;;) {
        if (!pl.loaded || pl.n - pl.first >= 32u) {
            pl.first = pl.n;
            ld_entry(a.log + ((pl.n + lane) & (uint32_t)(a.log_len - 1)), pl.w0, pl.w1);
            pl.loaded = true;
        }
        const int at = (int)(pl.n - pl.first);
        pl.e1 = __shfl_sync(0xffffffffu, pl.w1, at);
        int is = entry_is(pl.e1, pl.n);
        if (is == kEntryHere) {
            const uint32_t base = bits(pl.e1, kLogTiles, kLogBase), tiles = bits(pl.e1, 0, kLogTiles);
            const uint32_t i = blockIdx.x >= base ? blockIdx.x - base : blockIdx.x + gridDim.x - base;
            if (i >= tiles && tiles) {
                ++pl.n;  // none of its tiles is this block's
                continue;
            }
            pl.e0 = __shfl_sync(0xffffffffu, pl.w0, at);
            if (entry_whole(pl.e0, pl.n)) {
                if (!tiles) return false;  // F_EXIT
                __threadfence();  // the phase's inputs were written before it was opened
                fence_async_global();  // by other blocks' bulk copies too, and bulk copies read them next
                idx = i;
                pl.idx = i + gridDim.x;
                return true;
            }
            is = kEntryAhead;
        }
        if (is == kEntryPast) {
            ++pl.n;  // overwritten: it had no tile of this block's (log_entries)
            continue;
        }
        // not opened yet
        pl.loaded = false;
        if ((++tries & 15) == 0) {
            if (ld_int(&a.ctl->abort)) return false;
            if (tries > kLookLimit) {
                if (lane == 0) atomicExch(&a.ctl->abort, 1), *(volatile int *)a.err = a.err_tag | 1;
                return false;
            }
        }
    }
}

// opens a slot's next phase (one lane)
template <typename C>
__device__ __forceinline__ void open_phase(const Args &a, Slot &sl, int slot, const Code &c, int pk, int kind, int it,
                                           int stop) {
    uint32_t tiles = 0;
    switch (kind) {
        case F_CN:
            if (a.sim) {  // it: bit 0 frames leave, 1 enter, 2 run
                tiles = (it & 1 ? (c.N + kErrVars - 1) / kErrVars : 0) + (it & 2 ? (c.N + C::CHANV - 1) / C::CHANV : 0) +
                        (it & 4 ? c.J * c.rch.d : 0);
                break;
            }
            tiles = (a.early && !a.split && it >= 2 ? c.nsyn : 0) + c.J * (it == 1 ? c.rch1.d : c.rch.d); break;
        case F_VN: tiles = c.L * c.vch.d; break;
        case F_FIN:
        case F_SYN: tiles = c.nsyn; break;
        case F_PACK:
        case F_OUT: tiles = (c.N + C::OUTV - 1) / C::OUTV; break;
        default: break;
    }
    sl.done = 0u;
    sl.syn_done = 0u;
    const unsigned long long t = atomicAdd(&a.ctl->tail, (1ull << 40) | tiles);
    const uint32_t n = (uint32_t)(t >> 40), base = (uint32_t)((t & ((1ull << 40) - 1ull)) % gridDim.x);
    __threadfence();
    st_entry(a.log + (n & (uint32_t)(a.log_len - 1)), entry_w0(n, kind, stop, it, pk), entry_w1(n, slot, base, tiles));
}

// the slot's next package, or the end (one lane)
template <typename C, int V>
__device__ __forceinline__ void next_package(const Args &a, const Code &c, Slot &sl, int slot) {
    const int g = atomicAdd(&a.ctl->next, 1);
    if (g >= a.P) {
        __threadfence();
        if (atomicSub(&a.ctl->live, 1) == 1) open_phase<C>(a, sl, slot, c, 0, F_EXIT, 0, 0);
        return;
    }
    uint32_t stop = 0u;
    sl.all = 0;
    for (int v = 0; v < V; ++v) {
        const int n = c.gamma - g * C::W - v;  // frames v, V + v, ... of the package
        const int lanes = n <= 0 ? 0 : min(32, (n + V - 1) / V);
        const uint32_t valid = lanes == 32 ? 0xffffffffu : (1u << lanes) - 1u;
        sl.dn[v] = ~valid;
        sl.un[v] = 0u;
        stop |= ~valid;
    }
    open_phase<C>(a, sl, slot, c, g, F_PACK, 1, stop != 0u);
}

// what finish() needs of a tile
struct Fin {
    int kind, slot, pk, it, stop;
    uint32_t tiles;
};

// Refill mode, one step of a package complete up to its syndrome (the whole warp): frames whose
// decisions satisfy every check, or that have run max_iter iterations, leave; the next frames take
// their lanes.  Returns what the next check phase has to do (bit 0: frames leave, 1: enter, 2: run).
template <typename C, int V>
__device__ __forceinline__ int refill(const Args &a, Slot &sl, SimSlot &ss, int lane) {
    Sim &si = *a.sim;
    int what = 0;
    // everything the decision needs in one round of loads
    uint32_t D[V], U[V];
    int age[V];
    unsigned long long id[V];
#pragma unroll
    for (int v = 0; v < V; ++v) {
        D[v] = __ldcg(&sl.dn[v]), U[v] = __ldcg(&sl.un[v]);
        age[v] = __ldcg(&ss.age[lane * V + v]);
        id[v] = __ldcg(&ss.fid[lane * V + v]);
    }
    const unsigned long long handed = __ldcg(&si.next);
    unsigned long long from = __ldcg(&ss.from), to = __ldcg(&ss.to);  // ids the slot has reserved
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const int f = lane * V + v;
        const bool running = !((D[v] >> lane) & 1u), sat = !((U[v] >> lane) & 1u);
        const bool ret = running && ((a.early && age[v] >= 1 && sat) || age[v] >= a.max_iter);
        if (ret) {
            ss.rfid[f] = id[v];
            ss.pend[f] = 2 * age[v] + (sat ? 1 : 0);
            if (si.io) {
                if (si.iters) si.iters[id[v]] = age[v];
                if (si.ok) si.ok[id[v]] = sat ? 1 : 0;
            }
        }
        const uint32_t want = __ballot_sync(0xffffffffu, !running || ret);
        const int need = __popc(want), have = (int)(to - from);
        unsigned long long more = ~0ull >> 1;
        int got = 0;
        if (need > have && handed < si.limit) {
            // while many frames remain, reserve ahead: one atomic every few steps
            got = si.limit - handed > 256ull * gridDim.x ? need - have + C::W : need - have;
            if (lane == 0) more = atomicAdd(&si.next, (unsigned long long)got);
            more = __shfl_sync(0xffffffffu, more, 0);
        }
        const int at = __popc(want & ((1u << lane) - 1u));
        const unsigned long long idx = at < have ? from + at : more + (unsigned)(at - have);
        const bool fill = ((want >> lane) & 1u) && idx < si.limit;
        if (need <= have) from += need;
        else if (got) from = more + (unsigned)(need - have), to = more + (unsigned)got;
        else from = to;
        if (fill) {
            ss.fid[f] = si.first + idx;
            ss.age[f] = 0;
        } else if (running && !ret) {
            ss.age[f] = age[v] + 1;
        }
        const uint32_t retw = __ballot_sync(0xffffffffu, ret), fillw = __ballot_sync(0xffffffffu, fill);
        const uint32_t dn = (D[v] | retw) & ~fillw;
        if (lane == 0) {
            sl.dn[v] = dn;
            sl.un[v] = 0u;
            sl.ret[v] = retw;
            sl.fresh[v] = fillw;
        }
        what |= (retw ? 1 : 0) | (fillw ? 2 : 0) | (dn != 0xffffffffu ? 4 : 0);
    }
    if (lane == 0) ss.from = from, ss.to = to;
    // no rows to write and nothing to count: streaming without decisions
    if (si.io && !si.hard) what &= ~1;
    return what;
}

// the frames that left in this step join the totals (the whole warp)
template <int V>
__device__ __forceinline__ void tally(const Args &a, Slot &sl, SimSlot &ss, int lane) {
    unsigned long long t[6] = {0, 0, 0, 0, 0, 0};
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const int f = lane * V + v;
        if (!((__ldcg(&sl.ret[v]) >> lane) & 1u)) continue;
        const int pr = __ldcg(&ss.pend[f]), e = __ldcg(&ss.errs[f]);
        ss.errs[f] = 0;
        t[0] += 1;
        t[1] += e > 0;
        t[2] += (unsigned long long)e;
        t[3] += (unsigned long long)(pr >> 1);
        t[4] += e > 0 && (pr & 1);
        t[5] += (unsigned long long)e * (unsigned long long)e;
    }
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        for (int o = 16; o > 0; o >>= 1) t[i] += __shfl_xor_sync(0xffffffffu, t[i], o);
        if (lane == 0 && t[i]) atomicAdd(&a.sim->counters[i], t[i]);
    }
}

// a slot has no frame left (one lane)
template <typename C>
__device__ __forceinline__ void end_slot(const Args &a, const Code &c, Slot &sl, int slot) {
    __threadfence();
    if (atomicSub(&a.ctl->live, 1) == 1) open_phase<C>(a, sl, slot, c, 0, F_EXIT, 0, 0);
}

// finish() in refill mode: syndrome, check and variable phases in turn
template <typename C, int V>
__device__ __forceinline__ void finish_refill(const Args &a, const Code &c, const Fin &d, int lane) {
    Slot &sl = a.slots[d.slot];
    SimSlot &ss = a.simslots[d.slot];
    __syncwarp();
    uint32_t o = 0u;
    if (lane == 0) o = add_done(&sl.done, 1u);
    o = __shfl_sync(0xffffffffu, o, 0);
    if (o + 1 != d.tiles) return;
    if (d.kind == F_SYN) {
        const int what = refill<C, V>(a, sl, ss, lane);
        __syncwarp();  // opening the phase publishes what the lanes wrote
        if (lane == 0) {
            if (what) open_phase<C>(a, sl, d.slot, c, 0, F_CN, what, 0);
            else end_slot<C>(a, c, sl, d.slot);
        }
    } else if (d.kind == F_VN) {
        if (lane == 0) open_phase<C>(a, sl, d.slot, c, 0, F_SYN, 0, 0);
    } else {
        if ((d.it & 1) && !a.sim->io) tally<V>(a, sl, ss, lane);
        __syncwarp();
        if (lane == 0) {
            if (d.it & 4) open_phase<C>(a, sl, d.slot, c, 0, F_VN, 0, 0);
            else end_slot<C>(a, c, sl, d.slot);
        }
    }
    __syncwarp();
}

// a tile is done: counts it, and opens the slot's next phase with its last one (the whole warp)
template <typename C, int V>
__device__ __forceinline__ void finish(const Args &a, const Code &c, const Fin &d, int lane) {
    Slot &sl = a.slots[d.slot];
    if (a.sim) return finish_refill<C, V>(a, c, d, lane);
    const bool fin = d.it < 0;  // the final syndrome
    if (d.kind == F_SYN) {
        uint32_t o = 0u;
        if (lane == 0) o = add_done(&sl.syn_done, 1u);
        o = __shfl_sync(0xffffffffu, o, 0);
        if (o + 1 == (uint32_t)c.nsyn) {
            // the syndrome of the decisions after it - 1 iterations is complete: frames stop here
            uint32_t all = 0xffffffffu, dn[V], un[V];
#pragma unroll
            for (int v = 0; v < V; ++v) dn[v] = __ldcg(&sl.dn[v]), un[v] = __ldcg(&sl.un[v]);
            __syncwarp();
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const uint32_t newly = fin ? ~dn[v] : ~dn[v] & ~un[v];  // at the end every frame that still runs
                const int f = d.pk * C::W + lane * V + v;
                if ((newly >> lane) & 1u) {
                    if (c.iters) c.iters[f] = fin ? a.max_iter : d.it - 1;
                    if (c.ok) c.ok[f] = (un[v] >> lane) & 1u ? 0 : 1;
                }
                if (lane == 0) {
                    sl.dn[v] = dn[v] | newly;
                    sl.un[v] = 0u;
                }
                all &= dn[v] | newly;
            }
            if (lane == 0 && !fin && all == 0xffffffffu) sl.all = 1;
        }
    }
    __syncwarp();
    if (lane == 0 && add_done(&sl.done, 1u) + 1 == d.tiles) {
        // the phase is complete: the next one
        const bool outs = c.hard || c.post;
        int it = fin ? 0 : d.it, nk = -1, stop = d.stop, all = 0;
        // the check phase's kind, also for the syndrome tiles that were part of it
        const int kind = d.kind != F_SYN ? d.kind : (fin ? F_FIN : (a.split ? F_SYN : F_CN));
        if (a.early && it >= 2 && (kind == F_SYN || kind == F_CN)) {  // frames may have stopped
            uint32_t dn = 0u;
            all = __ldcg(&sl.all);
#pragma unroll
            for (int v = 0; v < V; ++v) dn |= __ldcg(&sl.dn[v]);
            stop = dn != 0u;
        }
        switch (kind) {
            case F_PACK: nk = F_CN, it = 1; break;
            case F_SYN: nk = all ? F_OUT : F_CN; break;
            case F_CN: nk = all ? F_OUT : F_VN; break;
            case F_VN:
                if (it == a.max_iter) nk = F_FIN;
                else nk = a.split ? F_SYN : F_CN, ++it;
                break;
            case F_FIN: nk = F_OUT; break;
            default: break;
        }
        if (nk == F_OUT && !outs) nk = -1;
        if (nk >= 0) open_phase<C>(a, sl, d.slot, c, d.pk, nk, it, stop);
        else next_package<C, V>(a, c, sl, d.slot);
    }
    __syncwarp();
}

// ---------------------------------------------------------------------------
// the kernel: compute warps, a taking warp, a retiring warp per stage; one persistent block per SM
// ---------------------------------------------------------------------------
template <typename C, int JX, int V, typename SM>
__device__ __forceinline__ void taking_warp(const Args &a, SM &sm, int lane) {
    Place pl;
    uint32_t ph = 1u;
    for (int head = 0;;) {
        uint32_t idx = 0u;  // taken while the stage empties
        bool on = take(a, lane, pl, idx);
        if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&sm.empty[head]), ph))) {
            if (lane == 0) atomicExch(&a.ctl->abort, 1), *(volatile int *)a.err = a.err_tag | 3;
            on = false;
        }
        const uint32_t bar = smem_u32(&sm.full[head]);
        Desc &d = sm.desc[head];
        if (!on) {
            // every stage's retiring warp sees the end, the compute warps at the first
            for (int q = 0; q < kStages; ++q, head = head + 1 == kStages ? 0 : head + 1, ph ^= head == 0) {
                if (q > 0 && !mbar_wait(smem_u32(&sm.empty[head]), ph)) return;
                if (lane == 0) {
                    sm.desc[head].kind = F_EXIT;
                    mbar_arrive(smem_u32(&sm.full[head]));
                }
            }
            return;
        }
        int kind = (int)bits(pl.e0, 0, 3), it = (int)bits(pl.e0, 4, kLogIt);
        const bool stop = bits(pl.e0, 3, 1) != 0u;
        const int pk = (int)bits(pl.e0, 4 + kLogIt, kLogPk);
        const int slot = (int)bits(pl.e1, kLogTiles + kLogBase, kLogSlot);
        const Code &c = sm.code;
        if (kind == F_FIN) {
            kind = F_SYN;
            it = -1;
        } else if (kind == F_CN && a.sim) {
            const uint32_t ne = it & 1 ? (c.N + kErrVars - 1) / kErrVars : 0;
            const uint32_t nc = it & 2 ? (c.N + C::CHANV - 1) / C::CHANV : 0;
            if (idx < ne) kind = a.sim->io ? F_ROWS : F_ERR;
            else if (idx < ne + nc) kind = F_CHAN, idx -= ne;
            else idx -= ne + nc;
        } else if (kind == F_CN && a.early && !a.split && it >= 2) {
            if (idx < (uint32_t)c.nsyn) kind = F_SYN;
            else idx -= c.nsyn;
        }
        if (lane == 0) {
            d.kind = kind;
            d.slot = slot;
            d.pk = pk;
            d.it = it;
            d.stop = stop;
            d.tiles = bits(pl.e1, 0, kLogTiles);
        }
        uint32_t *stage = sm.stage[head];
        const char *msg = reinterpret_cast<const char *>(a.msg + (size_t)slot * a.msg_stride);
        const char *mu = reinterpret_cast<const char *>(a.mu + (size_t)slot * a.mu_stride);
        if (kind == F_CN) {
            const bool first = it == 1 && !a.sim;
            const FastDiv &dv = first ? c.rch1 : c.rch;
            const int R = first ? C::ROWS1 : C::ROWS;
            const int j = (int)fdiv(idx, dv), r0 = (int)(idx - (uint32_t)j * dv.d) * R;
            const int rows = min(R, c.p - r0);
            const int sh = lane < c.L ? c.sh[j * c.L + lane] : -1;
            const uint32_t pm = __ballot_sync(0xffffffffu, sh >= 0);
            const int lb = first ? 128 * C::FV : 128;
            int k0 = 0, n1 = -1, line = 0;
            if (sh >= 0) {
                k0 = r0 + sh;
                if (k0 >= c.p) k0 -= c.p;
                n1 = min(rows, c.p - k0);
                line = c.eo[j * c.L + lane] + k0;
            }
            sm.dst[head][lane] = line;
            sm.n1[head][lane] = n1;
            if (lane == 0) {
                d.rows = rows;
                d.j = j;
                d.first = first;
                d.pm = pm;
#pragma unroll
                for (int v = 0; v < V; ++v) d.dn[v] = a.sim ? __ldcg(&a.slots[slot].fresh[v]) : 0u;
                mbar_arrive_tx(bar, (uint32_t)(__popc(pm) * rows * lb));
            }
            __syncwarp();
            if (sh >= 0) {
                const uint32_t dst = smem_u32(stage + lane * C::ROWS * 32);
                const char *src = first ? mu + ((size_t)lane * c.p + k0) * lb : msg + (size_t)line * 128;
                bulk_load(dst, src, (uint32_t)(n1 * lb), bar);
                if (n1 < rows) bulk_load(dst + n1 * lb, src - (size_t)k0 * lb, (uint32_t)((rows - n1) * lb), bar);
            }
        } else if (kind == F_VN) {
            const int l = (int)fdiv(idx, c.vch), k0 = (int)(idx - (uint32_t)l * c.vch.d) * c.kc;
            const int K = min(c.kc, c.p - k0), n0 = l * c.p + k0;
            const int sh = lane < c.J ? c.sh[lane * c.L + l] : -1;
            const uint32_t pm = __ballot_sync(0xffffffffu, sh >= 0);
            const int line = sh >= 0 ? c.eo[lane * c.L + l] + k0 : 0;
            sm.dst[head][lane] = line;
            uint32_t dn[V];
#pragma unroll
            for (int v = 0; v < V; ++v) dn[v] = stop ? __ldcg(&a.slots[slot].dn[v]) : 0u;  // refill mode: none kept
            if (stop) {  // the decisions of the stopped frames (none yet in the first iteration)
                const uint32_t *h = a.hw + (size_t)slot * a.hw_stride + (size_t)n0 * V;
                for (int q = lane; q < K * V; q += 32) sm.hw[head][q] = it > 1 ? __ldcg(h + q) : 0u;
                __syncwarp();
            }
            if (lane == 0) {
                d.rows = K;
                d.n0 = n0;
                d.pm = pm;
                d.post = a.want_post && (a.early || it == a.max_iter);
#pragma unroll
                for (int v = 0; v < V; ++v) d.dn[v] = dn[v];
                mbar_arrive_tx(bar, (uint32_t)((__popc(pm) + C::FV) * K * 128));
            }
            __syncwarp();
            if (sh >= 0)
                bulk_load(smem_u32(stage + lane * C::KC * 32), msg + (size_t)line * 128, (uint32_t)(K * 128), bar);
            if (lane == 31)
                bulk_load(smem_u32(stage + JX * C::KC * 32), mu + (size_t)n0 * 128 * C::FV,
                          (uint32_t)(K * 128 * C::FV), bar);
        } else if (kind == F_CHAN) {
            const int n0 = (int)idx * C::CHANV, K = min(C::CHANV, c.N - n0);
            int nf = 0;  // the list of the frames that enter
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const uint32_t w = __ldcg(&a.slots[slot].fresh[v]);
                if ((w >> lane) & 1u) {
                    const int at = nf + __popc(w & ((1u << lane) - 1u));
                    sm.list[head][at] = (uint8_t)(lane * V + v);
                    sm.fid[head][at] = (uint32_t)(__ldcg(&a.simslots[slot].fid[lane * V + v]) - a.sim->first);
                }
                nf += __popc(w);
            }
            __syncwarp();
            if (lane == 0) {
                d.n0 = n0;
                d.rows = nf;
                d.j = K;
                mbar_arrive_tx(bar, (uint32_t)(K * 128 * C::FV));
                bulk_load(smem_u32(stage), mu + (size_t)n0 * 128 * C::FV, (uint32_t)(K * 128 * C::FV), bar);
            }
        } else if (lane == 0) {
            d.n0 = (int)idx * (kind == F_SYN ? C::SYNROWS : (kind == F_ERR || kind == F_ROWS ? kErrVars : C::OUTV));
            if (kind == F_ERR || kind == F_ROWS) {
#pragma unroll
                for (int v = 0; v < V; ++v) d.dn[v] = __ldcg(&a.slots[slot].ret[v]);
            }
            mbar_arrive(bar);
        }
        __syncwarp();
        if (++head == kStages) head = 0, ph ^= 1u;
    }
}

// Stores the results of one stage's tiles and counts them done.
template <typename C, int V, typename SM>
__device__ __forceinline__ void retiring_warp(const Args &a, SM &sm, int st, int lane) {
    for (uint32_t ph = 0u;; ph ^= 1u) {
        if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&sm.used[st]), ph))) {
            if (lane == 0) atomicExch(&a.ctl->abort, 1), *(volatile int *)a.err = a.err_tag | 4;
            return;
        }
        const Desc &d = sm.desc[st];
        const int kind = d.kind;
        if (kind == F_EXIT) return;
        const Fin n{kind, d.slot, d.pk, d.it, d.stop, d.tiles};
        const Code &c = sm.code;
        if (kind == F_CN || kind == F_VN) {
            char *msg = reinterpret_cast<char *>(a.msg + (size_t)d.slot * a.msg_stride);
            const uint32_t src = smem_u32(sm.stage[st] + lane * (kind == F_CN ? C::ROWS : C::KC) * 32);
            if ((d.pm >> lane) & 1u) {
                const size_t line = (size_t)sm.dst[st][lane];
                const int rows = d.rows;
                if (kind == F_CN) {
                    const int n1 = sm.n1[st][lane];
                    bulk_store(msg + line * 128, src, (uint32_t)(n1 * 128));
                    if (n1 < rows)  // past the wrap: the circulant's first line
                        bulk_store(msg + (size_t)c.eo[d.j * c.L + lane] * 128, src + n1 * 128,
                                   (uint32_t)((rows - n1) * 128));
                } else {
                    bulk_store(msg + line * 128, src, (uint32_t)(rows * 128));
                }
            }
            bulk_commit();
            bulk_wait_read();
        } else if (kind == F_CHAN) {
            if (lane == 0)
                bulk_store(reinterpret_cast<char *>(a.mu + (size_t)d.slot * a.mu_stride) + (size_t)d.n0 * 128 * C::FV,
                           smem_u32(sm.stage[st]), (uint32_t)(d.j * 128 * C::FV));
            bulk_commit();
            bulk_wait_read();
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&sm.empty[st]));  // the stage is free
        bulk_wait<0>();
        __syncwarp();
        finish<C, V>(a, c, n, lane);
    }
}

template <int DC, int JX, int V, int RULE, bool REG>
__global__ void __launch_bounds__(kThreads, 1) tile_kernel(const Args a) {
    using C = Cfg<DC, JX, V, RULE, REG>;
    using SM = Smem<C::STAGE, V>;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    SM &sm = *reinterpret_cast<SM *>(smem_raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(smem_u32(&sm.full[s]), 1);
            mbar_init(smem_u32(&sm.used[s]), kComputeWarps);
            mbar_init(smem_u32(&sm.empty[s]), 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_async();
    }
    const int *src = reinterpret_cast<const int *>(a.code);
    int *dst = reinterpret_cast<int *>(&sm.code);
    for (int i = threadIdx.x; i < (int)(sizeof(Code) / 4); i += blockDim.x) dst[i] = src[i];
    __syncthreads();
    if (warp == kComputeWarps) return taking_warp<C, JX, V>(a, sm, lane);
    if (warp > kComputeWarps) return retiring_warp<C, V>(a, sm, warp - kComputeWarps - 1, lane);

    int st = 0, left = 0;
    uint32_t ph = 0u;
    for (;;) {
        if (!mbar_wait(smem_u32(&sm.full[st]), ph)) {
            if (lane == 0) atomicExch(&a.ctl->abort, 1), *(volatile int *)a.err = a.err_tag | 2;
            return;
        }
        const Desc &d = sm.desc[st];
        const int kind = d.kind;
        uint32_t *stage = sm.stage[st];
        const size_t slot = (size_t)d.slot;
        const Code &c = sm.code;
        if (kind == F_CN) {
            const float2 *prm = nullptr;
            if constexpr (RULE == kFlowNOMS) {
                prm = reinterpret_cast<const float2 *>(c.nparams) + ((size_t)(d.it - 1) * c.J + d.j) * c.L;
            }
            cn_tile<C, DC, V, RULE, REG>(stage, d, warp, lane, a.clip, prm);
        } else if (kind == F_VN) {
            vn_tile<C, JX, V, RULE, REG>(stage, sm.hw[st], d, warp, lane, a.clip, a.lsb, a.hw + slot * a.hw_stride,
                                         a.post + slot * a.post_stride);
        } else if (kind == F_SYN) {
            syn_tile<V>(c, d, warp, lane, a.hw + slot * a.hw_stride, a.slots[d.slot].un);
        } else if (kind == F_PACK) {
            pack_tile<C, V, C::MS>(stage, c, d, warp, lane, a.clip, a.qscale, a.mu + slot * a.mu_stride);
        } else if (kind == F_CHAN) {
            chan_tile<C, V, C::MS>(stage, sm.list[st], sm.fid[st], c, *a.sim, d, warp, lane, a.clip, a.qscale);
        } else if (kind == F_ERR) {
            err_tile<V>(c, d, warp, lane, a.hw + slot * a.hw_stride, a.simslots[slot].errs);
        } else if (kind == F_ROWS) {
            rows_tile<V>(c, *a.sim, a.simslots[slot], d, warp, lane, a.hw + slot * a.hw_stride);
        } else if (kind == F_OUT) {
            out_tile<C, V>(stage, c, d, warp, lane, a.hw + slot * a.hw_stride,
                           a.post + slot * a.post_stride);
        }
        // results in shared memory (and the channel LLRs in global memory) are moved by bulk copies next
        if (kind == F_PACK) fence_async();
        else fence_async_shared();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&sm.used[st]));
        if (kind == F_EXIT && ++left == kStages) return;
        if (++st == kStages) st = 0, ph ^= 1u;
    }
}

template <int DC, int JX, int V, int RULE, bool REG>
static ldpc_status launch(Args &a, const Start &st, int tiles, cudaStream_t s) {
    using C = Cfg<DC, JX, V, RULE, REG>;
    auto k = tile_kernel<DC, JX, V, RULE, REG>;
    const size_t smem = sizeof(Smem<C::STAGE, V>);
    const int most = resident_blocks((const void *)k, smem);
    if (most < 1) {
        set_error("the flow kernel does not fit an SM (%zu bytes of shared memory)", smem);
        return LDPC_ECUDA;
    }
    a.blocks = std::min({tiles, most, a.most_blocks});
    a.log_len = log_entries(a.W, a.blocks);
    const ldpc_status e = start(a, st, s);
    if (e != LDPC_OK) return e;
    // cooperative: all blocks resident or none, whatever else runs on the device
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at[1];
    cfg.gridDim = dim3((unsigned)a.blocks);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    LDPC_CUDA_TRY(cudaLaunchKernelEx(&cfg, k, a));
    count_launch();
    LDPC_CUDA_TRY(cudaGetLastError());
    return LDPC_OK;
}

// the kernel for a code's degrees: L up to 8, 16, 24 (regular: 24 x 4 without zero blocks) or 32
// slots a row, J up to 4 or 8
template <int V, int RULE>
static ldpc_status dispatch(Args &a, const Start &st, const Shape &g, int tiles, cudaStream_t s) {
    if (g.J <= 4) {
        if (g.L <= 8) return launch<8, 4, V, RULE, false>(a, st, tiles, s);
        if (g.L <= 16) return launch<16, 4, V, RULE, false>(a, st, tiles, s);
        if (g.regular && g.L == 24 && g.J == 4) return launch<24, 4, V, RULE, true>(a, st, tiles, s);
        if (g.L <= 24) return launch<24, 4, V, RULE, false>(a, st, tiles, s);
        return launch<32, 4, V, RULE, false>(a, st, tiles, s);
    }
    if (g.L <= 16) return launch<16, 8, V, RULE, false>(a, st, tiles, s);
    return launch<32, 8, V, RULE, false>(a, st, tiles, s);
}

}  // namespace flow
}  // namespace ldpc
