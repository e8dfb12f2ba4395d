// Training of the neural normalized min-sum decoder on sm_103a: Algorithm 1 (Sec. 2 of
// arXiv 2508.07879) with the scale alpha replaced by a learned weight w[t][e] per iteration and
// edge, unrolled over T iterations, trained on the BCE of the soft outputs sigma(-Q).
//
//   nms_forward_kernel   T iterations of the learned check step and the exact variable step of the decoder
//                        kernels (so FP32 messages are bit-identical to the learned decoder's), the per-shot
//                        loss sum_t lambda_t / N sum_n BCE(sigma(-Q^t_n), y_n) (lambda_t = 1/T unless
//                        given), and, per iteration and check, the
//                        compressed check state: min1, min2, the positions attaining them (lowest on
//                        ties), the sign bits of the inputs and the syndrome-flipped total sign.
//   nms_backward_kernel  the reverse sweep.  It stores no message: every r^(t) is recomputed from
//                        the recorded state (r_{m,n} = sign * (w * (n == idx1 ? min2 : min1))),
//                        Q^(t) from those r, and the gradient flows
//                          dL/dr_{m,n}   = dL/dQ_n + sum_{i != m} dL/dq_{i,n}      (variable step)
//                          dL/dw_{m,n}   = dL/dr_{m,n} * sign * min_{j != n}|q_j|
//                          dL/dq_{m,idx1} = sum_{n != idx1} dL/dr_{m,n} w sign * sign(q_idx1)
//                          dL/dq_{m,idx2} = dL/dr_{m,idx1} w sign * sign(q_idx2)     (all other q: 0)
//                        Weight gradients are added into one L2-resident buffer with global
//                        reductions, so the order of the sum over shots follows the schedule: the
//                        last bits of a gradient can differ between calls.  The next step can make
//                        much more of them: min-sum's gradient jumps where a minimum changes place, so a
//                        weight that is off in its last bit moves one shot's whole share.  LP-1054, 4096
//                        shots, T = 20: two runs of a step differ by 5e-7 of the gradient's norm, 30 of
//                        its 74400 weights then differ in the last bit, and after one more step the two
//                        gradients are more than 2e-5 apart for 3 of 10 inputs (up to 4e-3).
//
// Forward, L = 1 or 2 shots per block: two shots share every weight, edge list and prior, their messages sit in one
// 8-byte slot per edge (as in the two-shots-per-block decoder), their sums and products are packed FP32
// operations.  Weights and their gradient lie in groups of four edges (two where a row's length asks for it), so a
// check moves four of them per instruction and a warp whole sectors; a lane's edge slots come four to a load.
// Backward, one shot per block, a few blocks an SM that take the shots in waves: a shot's gradient is one fixed
// chain of roundings, and the sum over shots, whose rounding is the largest error of a gradient, keeps the order of those
// waves (plan_backward in qldpc_learned.cpp).
// What bounds both kernels is instruction issue and the latency of short chains between barriers, not
// memory: the recorded state (16 bytes per check, iteration and shot, written once and read from L2 after
// a prefetch) and the gradient's reductions are the only traffic.
// LP-1054, 4096 shots, T = 20, syndrome loss: forward 1107 -> 669 us, backward 2711 -> 1572 us
// (error loss 790 -> 605 and 1690 -> 1038).
#pragma once

#include <cstdint>
#include <type_traits>

#include <cuda_runtime.h>

#include "msa_kernel.cuh"
#include "msa_launch.h"

namespace qldpc {
namespace kern {

// ---------------------------------------------------------------------------------------------
// The same number of L shots: a float or a pair, with lane-wise operations rounded to nearest
// ---------------------------------------------------------------------------------------------
template <int L>
struct Lanes {
    using word = float;
    static __device__ __forceinline__ word all(float x) { return x; }
    static __device__ __forceinline__ word add(word a, word b) { return __fadd_rn(a, b); }
    static __device__ __forceinline__ word sub(word a, word b) { return __fsub_rn(a, b); }
    static __device__ __forceinline__ word mul(word a, word b) { return __fmul_rn(a, b); }
    static __device__ __forceinline__ float get(word a, int) { return a; }
    static __device__ __forceinline__ void set(word &a, int, float x) { a = x; }
};
#define QLDPC_PACKED2(name, op)                                                                 \
    static __device__ __forceinline__ word name(word a, word b)                                 \
    {                                                                                           \
        unsigned long long x, y, r;                                                             \
        asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "f"(a.x), "f"(a.y));                            \
        asm("mov.b64 %0, {%1, %2};" : "=l"(y) : "f"(b.x), "f"(b.y));                            \
        asm(op " %0, %1, %2;" : "=l"(r) : "l"(x), "l"(y));                                      \
        word o;                                                                                 \
        asm("mov.b64 {%0, %1}, %2;" : "=f"(o.x), "=f"(o.y) : "l"(r));                           \
        return o;                                                                               \
    }
template <>
struct Lanes<2> {
    using word = float2;
    static __device__ __forceinline__ word all(float x) { return make_float2(x, x); }
    QLDPC_PACKED2(add, "add.rn.f32x2")
    QLDPC_PACKED2(mul, "mul.rn.f32x2")
    static __device__ __forceinline__ word sub(word a, word b) { return add(a, make_float2(-b.x, -b.y)); }
    static __device__ __forceinline__ float get(word a, int l) { return l ? a.y : a.x; }
    static __device__ __forceinline__ void set(word &a, int l, float x) { (l ? a.y : a.x) = x; }
};
#undef QLDPC_PACKED2

__device__ __forceinline__ float with_sign(float mag, uint32_t bit31) { return __uint_as_float(__float_as_uint(mag) ^ bit31); }
__device__ __forceinline__ uint32_t sign_of(float x) { return __float_as_uint(x) & 0x80000000u; }

__device__ __forceinline__ float softplus(float x) { return fmaxf(x, 0.0f) + log1pf(expf(-fabsf(x))); }
__device__ __forceinline__ float sigmoid(float x) { return 1.0f / (1.0f + expf(-x)); }

// Sum over the block (deterministic order); every thread gets the total.
__device__ __forceinline__ float block_sum(float v, float *red)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = (blockDim.x + 31) >> 5;
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    float t = 0.0f;
    for (int i = 0; i < nw; ++i) t += red[i];
    return t;
}

// Weights and their gradient: the edges of a row in groups of G, a group's values of all checks one after
// another, so that a warp's 32 checks move whole sectors with one G-wide load or reduction (edge j of check
// c at edge_at<G>(c, j, M); rows are padded with zeros to whole groups).
template <int DC, bool UNIFORM>
__host__ __device__ constexpr int edge_group()
{
    return train_group(DC, UNIFORM);
}

// The weights of check c: DC values, 0 past the row's end.
template <int DC, bool UNIFORM>
__device__ __forceinline__ void load_row(const float *__restrict__ rows, int M, int c, int deg, float (&w)[DC])
{
    constexpr int G = edge_group<DC, UNIFORM>();
#pragma unroll
    for (int j = 0; j < DC; j += G) {
        float v[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        if (UNIFORM || j < deg) {
            const float *at = rows + train_edge_at(G, c, j, M);
            if constexpr (G == 2) {
                const float2 x = __ldg(reinterpret_cast<const float2 *>(at));
                v[0] = x.x;
                v[1] = x.y;
            } else {
                const float4 x = __ldg(reinterpret_cast<const float4 *>(at));
                v[0] = x.x;
                v[1] = x.y;
                v[2] = x.z;
                v[3] = x.w;
            }
        }
#pragma unroll
        for (int i = 0; i < G; ++i)
            if (j + i < DC) w[j + i] = v[i];
    }
}

// ---------------------------------------------------------------------------------------------
// Syndrome loss.  With t_v = tanh(Q_v / 2), P_c = (1 + (-1)^s prod_{v in c} t_v) / 2 is the
// probability that row c's parity under independent bits sigma(-Q) equals s.  Each variable
// stores, on its edge slots, its log-magnitude code
//   lm_v = sign(Q_v) * (-log |t_v|),  -log |t_v| = log1p(e^-|Q_v|) - log1p(-e^-|Q_v|)  (+inf at Q = 0),
// computed once per variable.  A check then has prod |t| = exp(A), A = -sum |lm|, and a violated,
// confident check gets P = -expm1(A) / 2 without the cancellation of 1 - prod (|t| rounds to 1
// long before 1 - |t| is negligible).  (u = 1 - |t| from one exponential and a division, and 1 - prod (1 - u)
// term by term, would spare the logarithms and an exponential per edge: 516 and 830 us.  It loses bits of |t|
// for Q near 0: with priors of 0.01 and T = 2 a shot's gradient is 7e-6 from 64 bits against 1.8e-6.)
// ---------------------------------------------------------------------------------------------
constexpr float kSynLossFloor = 1e-7f;

// The sign travels in the sign bit (also on a magnitude of 0, where |Q| is so large that |t| = 1).
__device__ __forceinline__ float log_magnitude_code(float Q)
{
    const float x = expf(-fabsf(Q));
    const float mag = log1pf(x) - log1pf(-x);   // -log |tanh(Q/2)| >= 0
    return __uint_as_float(__float_as_uint(mag) | (Q < 0.0f ? 0x80000000u : 0u));
}
// d tanh(Q/2) / dQ = sech^2(Q/2) / 2 (no cancellation for large |Q|)
__device__ __forceinline__ float half_sech2_half(float Q)
{
    const float ch = coshf(0.5f * Q);
    return 0.5f / (ch * ch);
}

// P_c of L shots from the codes in check c's slots; s_bits: bit l = s_c of shot l.  WANT_T: the signed t_j.
template <int L, int DC, bool UNIFORM, bool WANT_T>
__device__ __forceinline__ void parity_match(int c, int M, int deg, uint32_t s_bits,
                                             const typename Lanes<L>::word *__restrict__ ts, float (&P)[L],
                                             typename Lanes<L>::word (&t)[DC])
{
    using V = Lanes<L>;
    using word = typename V::word;
    word A = V::all(0.0f);
    uint32_t neg[L];
#pragma unroll
    for (int l = 0; l < L; ++l) neg[l] = s_bits << (31 - l);
#pragma unroll
    for (int j = 0; j < DC; ++j) {
        if (UNIFORM || j < deg) {
            const word code = ts[j * M + c];
            word minus;                        // -|lm| = log |t|
#pragma unroll
            for (int l = 0; l < L; ++l) {
                neg[l] ^= __float_as_uint(V::get(code, l));
                V::set(minus, l, -fabsf(V::get(code, l)));
            }
            A = V::add(A, minus);
            if constexpr (WANT_T) {
#pragma unroll
                for (int l = 0; l < L; ++l) V::set(t[j], l, with_sign(expf(V::get(minus, l)), sign_of(V::get(code, l))));
            }
        } else if constexpr (WANT_T) {
            t[j] = V::all(1.0f);
        }
    }
#pragma unroll
    for (int l = 0; l < L; ++l)
        P[l] = (neg[l] >> 31) ? -0.5f * expm1f(V::get(A, l)) : 0.5f * (1.0f + expf(V::get(A, l)));
}

template <int L, int DC, bool UNIFORM>
__device__ __forceinline__ void syndrome_term(int c, int M, int deg, uint32_t s_bits,
                                              const typename Lanes<L>::word *__restrict__ ts, float (&term)[L])
{
    float P[L];
    typename Lanes<L>::word none[DC];
    parity_match<L, DC, UNIFORM, false>(c, M, deg, s_bits, ts, P, none);
#pragma unroll
    for (int l = 0; l < L; ++l) term[l] = -logf(fmaxf(P[l], kSynLossFloor));
}

// d(syndrome term)/d t_j = -(1 / P) (-1)^s / 2 prod_{i != j} t_i (0 at the floor), written over the
// codes of check c.
template <int DC, bool UNIFORM>
__device__ __forceinline__ void syndrome_term_grad(int c, int M, int deg, uint32_t s_bit, float *__restrict__ ts)
{
    float P[1], t[DC], pre[DC];
    parity_match<1, DC, UNIFORM, true>(c, M, deg, s_bit, ts, P, t);
    const float coef = P[0] > kSynLossFloor ? (s_bit & 1u ? 0.5f : -0.5f) / P[0] : 0.0f;
    float run = 1.0f;
#pragma unroll
    for (int j = 0; j < DC; ++j) {
        pre[j] = run;                        // t_0 ... t_{j-1}
        run = __fmul_rn(run, t[j]);
    }
    float suf = 1.0f;                        // t_{j+1} ... t_{deg-1}
#pragma unroll
    for (int j = DC - 1; j >= 0; --j) {
        if (UNIFORM || j < deg) {
            ts[j * M + c] = __fmul_rn(coef, __fmul_rn(pre[j], suf));
            suf = __fmul_rn(suf, t[j]);
        }
    }
}

// ---------------------------------------------------------------------------------------------
// Forward
// ---------------------------------------------------------------------------------------------
// Learned check step for check c: r = sign * (w * min over the others), written in place of q, and the
// recorded state of shot l at st[l] (not where st[l] is null).
template <int L, int DC, bool UNIFORM>
__device__ __forceinline__ void train_check(int c, int M, int deg, uint32_t s_bits,
                                            typename Lanes<L>::word *__restrict__ slots, const float *__restrict__ w,
                                            uint4 *const (&st)[L])
{
    using V = Lanes<L>;
    float q[L][DC], wv[DC], m2[L];
    uint32_t sum[L];
    load_row<DC, UNIFORM>(w, M, c, deg, wv);
#pragma unroll
    for (int j = 0; j < DC; ++j) {
        if (UNIFORM || j < deg) {
            const typename V::word v = slots[j * M + c];
#pragma unroll
            for (int l = 0; l < L; ++l) q[l][j] = V::get(v, l);
        }
    }
#pragma unroll
    for (int l = 0; l < L; ++l) {
        float m1;
        uint32_t sx;
        row_minima<F32, DC, UNIFORM>(q[l], deg, m1, m2[l], sx);
        const uint32_t negall = ((s_bits >> l) ^ (sx >> 31)) & 1u;
        sum[l] = other_sum(m1, m2[l], negall << 31);
        uint32_t signs = 0, at1 = 0, at2 = 0;
#pragma unroll
        for (int j = DC - 1; j >= 0; --j) {
            if (UNIFORM || j < deg) {
                signs = __funnelshift_l(__float_as_uint(q[l][j]), signs, 1);
                if (fabsf(q[l][j]) == m1) at1 |= 1u << j;
                if (fabsf(q[l][j]) == m2[l]) at2 |= 1u << j;
            }
        }
        // the lowest position of the minimum, and the lowest other position of the second smallest (0 where
        // a NaN hides them, so that an index always names an edge)
        const int i1 = at1 ? __ffs(int(at1)) - 1 : 0;
        at2 &= ~(1u << i1);
        const int i2 = at2 ? __ffs(int(at2)) - 1 : 0;
        if (st[l])
            st[l][c] = make_uint4(__float_as_uint(m1), __float_as_uint(m2[l]), signs,
                                  uint32_t(i1) | (uint32_t(i2) << 8) | (negall << 16));
    }
#pragma unroll
    for (int j = 0; j < DC; ++j) {
        if (UNIFORM || j < deg) {
            typename V::word o;
#pragma unroll
            for (int l = 0; l < L; ++l) V::set(o, l, other_min(q[l][j], m2[l], sum[l]));
            slots[j * M + c] = V::mul(V::all(wv[j]), o);
        }
    }
}

// Per-lane inputs: the prior of the variable in lane u, and its targets (bit l: shot l; kIdleLane where the
// lane holds no variable: its prior is 0, its edges are scratch slots and it adds nothing to the loss).
constexpr uint8_t kIdleLane = 0x80;
__device__ __forceinline__ float lane_prior(const DeviceGraph &g, const float *prior, int u)
{
    const uint32_t v = __ldg(g.vperm + u);
    return v < uint32_t(g.n) ? prior[v] : 0.0f;
}
template <int L>
__device__ __forceinline__ uint8_t lane_targets(const DeviceGraph &g, const uint8_t *target, const int (&shot)[L], int u)
{
    const uint32_t v = __ldg(g.vperm + u);
    if (v >= uint32_t(g.n)) return kIdleLane;
    uint8_t y = 0;
#pragma unroll
    for (int l = 0; l < L; ++l) y |= uint8_t((target[size_t(shot[l]) * g.n + v] & 1u) << l);
    return y;
}

// The block's shots; one past the batch's end takes the first one's inputs and leaves no output.
template <int L>
__device__ __forceinline__ void block_shots(int batch, int (&shot)[L], bool (&real)[L])
{
#pragma unroll
    for (int l = 0; l < L; ++l) {
        const int64_t b = int64_t(blockIdx.x) * L + l;
        real[l] = b < batch;
        shot[l] = real[l] ? int(b) : int(blockIdx.x) * L;
    }
}

template <int L>
__device__ __forceinline__ uint8_t check_bits(const uint8_t *syn, const int (&shot)[L], int M, int c)
{
    uint8_t s = 0;
#pragma unroll
    for (int l = 0; l < L; ++l) s |= uint8_t((syn[size_t(shot[l]) * M + c] & 1u) << l);
    return s;
}

// SYN: the syndrome loss (compiled separately, so the error-loss kernels carry none of its code).
template <int L, int DC, bool UNIFORM, int DV, bool SYN>
__global__ void __launch_bounds__(kTrainThreads, DC <= 8 ? 3 : 1) nms_forward_kernel(const __grid_constant__ TrainParams p)
{
    using V = Lanes<L>;
    using word = typename V::word;
    const DeviceGraph &G = p.g;
    const int M = G.m, N = G.n, NV = G.nv, T = blockDim.x, tid = threadIdx.x;
    extern __shared__ __align__(16) unsigned char smem[];
    const TrainLayout lay = train_layout(M, NV, G.dc_max, L, false, SYN);
    word *slots = reinterpret_cast<word *>(smem + lay.slot_off);
    word *ts = reinterpret_cast<word *>(smem + lay.r_off);        // syndrome loss: each edge's variable's code
    float *gam = reinterpret_cast<float *>(smem + lay.g_off);
    uint8_t *y = smem + lay.y_off;
    uint8_t *sb = smem + lay.s_off;
    __shared__ float red[32];
    int shot[L];
    bool real[L];
    block_shots<L>(p.batch, shot, real);

    for (int c = tid; c < M; c += T) sb[c] = check_bits<L>(p.syn, shot, M, c);
    for_lanes<DV>(G, tid, T, [&](auto deg, int u) {
        constexpr int D = decltype(deg)::value;
        const float g = F32::quantize(lane_prior(G, p.prior, u));
        gam[u] = g;
        if constexpr (!SYN) y[u] = lane_targets<L>(G, p.target, shot, u);
        uint32_t e[D > 0 ? D : 1];
        lane_slots<D, sizeof(word)>(G.vslot16, NV, u, e);
#pragma unroll
        for (int i = 0; i < D; ++i) *at_bytes(slots, e[i]) = V::all(g);
    });
    __syncthreads();
    float acc[L];
#pragma unroll
    for (int l = 0; l < L; ++l) acc[l] = 0.0f;
    // uniform lambda: sum the terms and scale once by 1/(T K); else weight each iteration's terms
    // (K = N variables for the error loss, M checks for the syndrome loss)
    const float K = float(SYN ? M : N);
    const float inv = p.loss_w ? 1.0f / K : 1.0f / (float(p.T) * K);
    for (int k = 0; k < p.T; ++k) {
        const float *wk = p.w + size_t(k) * M * p.wstride;
        uint4 *st[L];
#pragma unroll
        for (int l = 0; l < L; ++l) st[l] = real[l] ? p.state + (size_t(shot[l]) * p.T + k) * M : nullptr;
        // syndrome loss of iteration k-1 (its code slots are complete) beside the check step of k
        const float lw_prev = (SYN && k > 0) ? (p.loss_w ? __ldg(p.loss_w + k - 1) : 1.0f) : 0.0f;
        for (int c = tid; c < M; c += T) {
            const int deg = UNIFORM ? DC : int(__ldg(G.rdeg + c));
            if (SYN && k > 0) {
                float term[L];
                syndrome_term<L, DC, UNIFORM>(c, M, deg, sb[c], ts, term);
#pragma unroll
                for (int l = 0; l < L; ++l) acc[l] += lw_prev * term[l];
            }
            train_check<L, DC, UNIFORM>(c, M, deg, sb[c], slots, wk, st);
        }
        __syncthreads();
        const bool lastk = k + 1 == p.T;
        const float lw = p.loss_w ? __ldg(p.loss_w + k) : 1.0f;
        for_lanes<DV>(G, tid, T, [&](auto deg, int u) {
            constexpr int D = decltype(deg)::value;
            uint32_t e[D > 0 ? D : 1];
            word r[D > 0 ? D : 1], pre[D + 1];
            lane_slots<D, sizeof(word)>(G.vslot16, NV, u, e);
#pragma unroll
            for (int i = 0; i < D; ++i) r[i] = *at_bytes(slots, e[i]);
            pre[0] = V::all(gam[u]);
#pragma unroll
            for (int i = 0; i < D; ++i) pre[i + 1] = V::add(pre[i], r[i]);
            const word Q = pre[D];
#pragma unroll
            for (int i = 0; i < D; ++i) {
                word q = pre[i];
#pragma unroll
                for (int h = i + 1; h < D; ++h) q = V::add(q, r[h]);
                *at_bytes(slots, e[i]) = q;
            }
            if constexpr (SYN) {
                word code;
#pragma unroll
                for (int l = 0; l < L; ++l) V::set(code, l, log_magnitude_code(V::get(Q, l)));
#pragma unroll
                for (int i = 0; i < D; ++i) *at_bytes(ts, e[i]) = code;
            } else if (y[u] != kIdleLane) {
#pragma unroll
                for (int l = 0; l < L; ++l) {
                    const float q = V::get(Q, l);
                    acc[l] += lw * ((y[u] >> l) & 1u ? softplus(q) : softplus(-q));
                }
            }
            if (lastk && p.post) {
                const uint32_t v = __ldg(G.vperm + u);
#pragma unroll
                for (int l = 0; l < L; ++l)
                    if (v < uint32_t(N) && real[l]) p.post[size_t(shot[l]) * N + v] = V::get(Q, l);
            }
        });
        __syncthreads();
    }
    if (SYN) {   // the last iteration's syndrome loss
        const float lw = p.loss_w ? __ldg(p.loss_w + p.T - 1) : 1.0f;
        for (int c = tid; c < M; c += T) {
            float term[L];
            syndrome_term<L, DC, UNIFORM>(c, M, UNIFORM ? DC : int(__ldg(G.rdeg + c)), sb[c], ts, term);
#pragma unroll
            for (int l = 0; l < L; ++l) acc[l] += lw * term[l];
        }
    }
#pragma unroll
    for (int l = 0; l < L; ++l) {
        const float total = block_sum(acc[l], red);
        if (tid == 0 && real[l]) p.loss[shot[l]] = total * inv;
    }
}

// ---------------------------------------------------------------------------------------------
// Backward
// ---------------------------------------------------------------------------------------------
// Bring one iteration's recorded state (16 bytes per check) of a shot into L2.
__device__ __forceinline__ void prefetch_state(const uint4 *st, int M, int tid, int T)
{
    for (int i = 8 * tid; i < M; i += 8 * T) asm volatile("prefetch.global.L2 [%0];" ::"l"(st + i));
}

// r of check c recomputed from its recorded state and its edges' weights (bit-identical to the
// forward's r).
template <int DC, bool UNIFORM>
__device__ __forceinline__ void recompute_r(int c, int M, int deg, const uint4 &st, const float (&w)[DC], float *__restrict__ rs)
{
    const uint32_t flip = st.z ^ (0u - ((st.w >> 16) & 1u));   // bit j: the sign of r_j
#pragma unroll
    for (int j = 0; j < DC; ++j)
        if (UNIFORM || j < deg)
            rs[j * M + c] = __fmul_rn(w[j], with_sign(__uint_as_float(j == int(st.w & 0xffu) ? st.y : st.x),
                                                      (flip << (31 - j)) & 0x80000000u));
}

// One shot per block, shots blockIdx.x, blockIdx.x + gridDim.x, ... (plan_backward in qldpc_learned.cpp).
template <int DC, bool UNIFORM, int DV, bool SYN>
__global__ void __launch_bounds__(kTrainThreads, DC <= 8 ? 2 : 1) nms_backward_kernel(const __grid_constant__ TrainParams p)
{
    const DeviceGraph &G = p.g;
    const int M = G.m, N = G.n, NV = G.nv, T = blockDim.x, tid = threadIdx.x;
    const size_t S = size_t(M) * p.wstride;
    extern __shared__ __align__(16) unsigned char smem[];
    const TrainLayout lay = train_layout(M, NV, G.dc_max, 1, true, SYN);
    float *gs = reinterpret_cast<float *>(smem + lay.slot_off);   // dL/dq (next iteration), then dL/dr
    float *rs = reinterpret_cast<float *>(smem + lay.r_off);      // recomputed r of the current iteration
    // Syndrome loss: once Q^(k) is formed, each variable overwrites its own r slots with its code
    // (no other thread reads them), and each check then replaces the codes with d(term)/d t.
    float *ts = rs;
    float *qlane = reinterpret_cast<float *>(smem + lay.q_off);   // syndrome loss: Q^(k) per lane
    float *gam = reinterpret_cast<float *>(smem + lay.g_off);
    uint8_t *y = smem + lay.y_off;
    uint8_t *sb = smem + lay.s_off;
    for (int u = tid; u < NV; u += T) gam[u] = F32::quantize(lane_prior(G, p.prior, u));
    for (int b = blockIdx.x; b < p.batch; b += gridDim.x) {   // (the last iteration's barrier closes a shot)
        const int shot[1] = {b};
        const uint4 *st = p.state + size_t(b) * p.T * M;
        const float gscale = p.grad_loss[b] * (1.0f / float(SYN ? M : N));
        if (p.T > 1) prefetch_state(st + size_t(p.T - 2) * M, M, tid, T);

        // iteration T: recompute r; dL/dq of iteration T+1 is zero
        for (int c = tid; c < M; c += T) {
            const int deg = UNIFORM ? DC : int(__ldg(G.rdeg + c));
            if (SYN) sb[c] = check_bits<1>(p.syn, shot, M, c);
            float w[DC];
            const uint4 s = __ldg(st + size_t(p.T - 1) * M + c);
            load_row<DC, UNIFORM>(p.w + size_t(p.T - 1) * S, M, c, deg, w);
            recompute_r<DC, UNIFORM>(c, M, deg, s, w, rs);
#pragma unroll
            for (int j = 0; j < DC; ++j)
                if (UNIFORM || j < deg) gs[j * M + c] = 0.0f;
        }
        if constexpr (!SYN)
            for (int u = tid; u < NV; u += T) y[u] = lane_targets<1>(G, p.target, shot, u);
        __syncthreads();
        for (int k = p.T - 1; k >= 0; --k) {
            if (k > 1) prefetch_state(st + size_t(k - 2) * M, M, tid, T);
            const float gk = __fmul_rn(gscale, p.loss_w ? __ldg(p.loss_w + k) : 1.0f / float(p.T));
            if constexpr (SYN) {
                // the code of Q^(k) on every edge slot, then each check's d(loss term)/d t in its place
                for_lanes<DV>(G, tid, T, [&](auto deg, int u) {
                    constexpr int D = decltype(deg)::value;
                    uint32_t e[D > 0 ? D : 1];
                    lane_slots<D, sizeof(float)>(G.vslot16, NV, u, e);
                    float Q = gam[u];
#pragma unroll
                    for (int i = 0; i < D; ++i) Q = __fadd_rn(Q, *at_bytes(rs, e[i]));
                    const float code = log_magnitude_code(Q);
                    qlane[u] = Q;
#pragma unroll
                    for (int i = 0; i < D; ++i) *at_bytes(ts, e[i]) = code;
                });
                __syncthreads();
                for (int c = tid; c < M; c += T)
                    syndrome_term_grad<DC, UNIFORM>(c, M, UNIFORM ? DC : int(__ldg(G.rdeg + c)), sb[c], ts);
                __syncthreads();
            }
            // variable side: dL/dQ^(k) (error loss: Q^(k) from the recomputed r), and dL/dr for every edge
            for_lanes<DV>(G, tid, T, [&](auto deg, int u) {
                constexpr int D = decltype(deg)::value;
                uint32_t e[D > 0 ? D : 1];
                float g[D > 0 ? D : 1], sum = 0.0f, gQ;
                lane_slots<D, sizeof(float)>(G.vslot16, NV, u, e);
#pragma unroll
                for (int i = 0; i < D; ++i) {
                    g[i] = *at_bytes(gs, e[i]);
                    sum = __fadd_rn(sum, g[i]);
                }
                if constexpr (SYN) {
                    float H = 0.0f;
#pragma unroll
                    for (int i = 0; i < D; ++i) H = __fadd_rn(H, *at_bytes(ts, e[i]));
                    gQ = __fmul_rn(__fmul_rn(gk, half_sech2_half(qlane[u])), H);
                } else {
                    float Q = gam[u];
#pragma unroll
                    for (int i = 0; i < D; ++i) Q = __fadd_rn(Q, *at_bytes(rs, e[i]));
                    gQ = __fmul_rn(gk, float(y[u] & 1u) - sigmoid(-Q));
                }
#pragma unroll
                for (int i = 0; i < D; ++i) *at_bytes(gs, e[i]) = __fadd_rn(gQ, __fsub_rn(sum, g[i]));
            });
            __syncthreads();
            // check side: weight gradient, dL/dq of iteration k, and r of iteration k-1
            for (int c = tid; c < M; c += T) {
                const int deg = UNIFORM ? DC : int(__ldg(G.rdeg + c));
                constexpr int GW = edge_group<DC, UNIFORM>(), PAD = (DC + GW - 1) / GW * GW;
                float w[DC], dw[PAD];
                const uint4 s = __ldg(st + size_t(k) * M + c);
                load_row<DC, UNIFORM>(p.w + size_t(k) * S, M, c, deg, w);
                uint4 sp{};
                if (k > 0) sp = __ldg(st + size_t(k - 1) * M + c);
                const uint32_t flip = s.z ^ (0u - ((s.w >> 16) & 1u));
                const int i1 = int(s.w & 0xffu), i2 = int((s.w >> 8) & 0xffu);
                float rest = 0.0f, own = 0.0f;     // sum of gr w sign over the edges but idx1, and idx1's
#pragma unroll
                for (int j = 0; j < PAD; ++j) {
                    dw[j] = 0.0f;
                    if (j < DC && (UNIFORM || j < deg)) {
                        const float sg = with_sign(gs[j * M + c], (flip << (31 - j)) & 0x80000000u);   // gr * sign
                        const float t = __fmul_rn(sg, w[j]);
                        dw[j] = __fmul_rn(sg, __uint_as_float(j == i1 ? s.y : s.x));
                        if (j == i1)
                            own = t;
                        else
                            rest = __fadd_rn(rest, t);
                        gs[j * M + c] = 0.0f;
                    }
                }
                float *out = p.partial + size_t(k) * S;
#pragma unroll
                for (int j = 0; j < PAD; j += GW)     // (results unused: reductions; 0 past the row's end)
                    if (UNIFORM || j < deg) {
                        float *at = out + train_edge_at(GW, c, j, M);
                        if constexpr (GW == 2)
                            atomicAdd(reinterpret_cast<float2 *>(at), make_float2(dw[j], dw[j + 1]));
                        else
                            atomicAdd(reinterpret_cast<float4 *>(at), make_float4(dw[j], dw[j + 1], dw[j + 2], dw[j + 3]));
                    }
                // dL/dq is 0 but at the positions of the two minima
                gs[i1 * M + c] = (s.z >> i1) & 1u ? -rest : rest;
                gs[i2 * M + c] = (s.z >> i2) & 1u ? -own : own;
                if (k > 0) {
                    load_row<DC, UNIFORM>(p.w + size_t(k - 1) * S, M, c, deg, w);
                    recompute_r<DC, UNIFORM>(c, M, deg, sp, w, rs);
                }
            }
            __syncthreads();
        }
    }
}

}  // namespace kern

// Compiled training variants: uniform row degree 6..8 with column-degree bucket 4 or 8, or a row-degree
// bucket 8 with column-degree bucket 8 or 16 (forward: for one and two shots per block); longer rows take one
// shot per block.
#define QLDPC_TRAIN_SHORT(X)                                                                    \
    X(6, true, 4) X(6, true, 8) X(7, true, 4) X(7, true, 8) X(8, true, 4) X(8, true, 8)        \
    X(8, false, 8) X(8, false, 16)
#define QLDPC_TRAIN_LONG(X) X(16, false, 8) X(16, false, 16) X(32, false, 8) X(32, false, 16)

template <int L>
const void *forward_kernel(const TrainChoice &tc, int loss_kind)
{
    const bool syn = loss_kind == kLossSyndrome;
#define QLDPC_K(DCV, UNI, DVV)                                                                  \
    if (tc.dc == DCV && tc.uniform == UNI && tc.dvb == DVV)                                     \
        return syn ? reinterpret_cast<const void *>(&kern::nms_forward_kernel<L, DCV, UNI, DVV, true>) \
                   : reinterpret_cast<const void *>(&kern::nms_forward_kernel<L, DCV, UNI, DVV, false>);
    QLDPC_TRAIN_SHORT(QLDPC_K)
    if constexpr (L == 1) {
        QLDPC_TRAIN_LONG(QLDPC_K)
    }
#undef QLDPC_K
    return nullptr;
}

}  // namespace qldpc
