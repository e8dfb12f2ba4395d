// Flooding normalized min-sum decoder driven by a syndrome -- Algorithm 1 ("MSA for
// syndrome-based LDPC decoding"), Sec. 2 of arXiv 2508.07879 -- for sm_103a.
//
// Two kernels share the arithmetic below and one shared-memory layout:
//
//   msa_batch_kernel    throughput: one block per shot, persistent over the batch, one thread per
//                       check in the check step and one thread per variable in the variable step;
//                       16-bit edge lists are read through the read-only path (L1-resident).
//   msa_latency_kernel  single shots and moderate batches: the same steps, but every thread keeps its edge
//                       lists, degrees, priors and a-posteriori LLRs in registers for the whole
//                       launch, so an iteration touches only shared memory.
//
// Layout (a GB300 design, not the paper's per-iteration launches over global memory):
//   * every edge message of a shot lives in shared memory, in place: the check step overwrites
//     q_{m,n} with r_{m,n}, the variable step overwrites r with the next q.  Slots are check-major
//     (slot j*M + m, 4 bytes FP32 / 2 bytes INT16), so 32 consecutive checks touch 32 consecutive
//     slots;
//   * the stop test H e^T = s is kept incrementally: check m owns a parity word
//     (bit 1 = s_m, bit 0 = s_m XOR the decisions of its variables); a variable whose decision
//     flips XORs bit 0 of its checks' words (shared-memory atomics, exact).  The next check step
//     reads one word per check and the block settles the test with one __syncthreads_and, so an
//     iteration costs two block barriers (the paper's kernel: four);
//   * the check step keeps no argmin: min over S_v(m)\n is min2 where |q_n| equals min1 and min1
//     elsewhere (min2 = min1 when the minimum is shared), which is exact (FP32: other_min below).
//
// Arithmetic is operation-for-operation that of the CPU oracle:
//   r = sign * (alpha * min_{j != n} |q_j|)
//   q_{m,n} = gamma_n + sum_{i != m} r_{i,n}        ascending check order, prefixes reused
//   Q_n = gamma_n + sum_i r_{i,n}                   ascending check order
// so FP32 results are bit-identical (every add/multiply is an explicit round-to-nearest intrinsic,
// nothing is fused or reassociated) and INT16 results are exact integer arithmetic.
// (A lane-per-edge check step with warp-shuffle reductions, a two-lanes-per-check step and a
// thread-block-cluster split of one shot over several SMs were all measured slower on GB300.)
#pragma once

#include <cstdint>
#include <type_traits>

#include <cuda_runtime.h>

#include "msa_launch.h"

namespace qldpc {
namespace kern {

// ---------------------------------------------------------------------------------------------
// Precision policies: arithmetic and the slot format
// ---------------------------------------------------------------------------------------------
struct F32 {
    using acc_t = float;    // variable-node sums, Q_n
    using mag_t = float;    // |q| and scaled minima
    using msg_t = float;    // a slot
    // g + 0 is g except that -0 becomes +0; with no -0 prior no message is ever -0 (a rounded sum
    // is -0 only when every term is), so the sign bit of a message equals [message < 0].
    static __device__ __forceinline__ acc_t quantize(float g) { return __fadd_rn(g, 0.0f); }
    static __device__ __forceinline__ acc_t add(acc_t a, acc_t b) { return __fadd_rn(a, b); }
    // layered schedule: Q - r_old, and the check's input clamped to the message range (none here)
    static __device__ __forceinline__ acc_t sub(acc_t Q, acc_t r) { return __fsub_rn(Q, r); }
    static __device__ __forceinline__ acc_t clampq(acc_t x) { return x; }
    static __device__ __forceinline__ bool neg(float x) { return x < 0.0f; }
    static __device__ __forceinline__ mag_t mag(acc_t x) { return fabsf(x); }
    static __device__ __forceinline__ mag_t mag_init() { return __int_as_float(0x7f800000); }
    static __device__ __forceinline__ mag_t mn(mag_t a, mag_t b) { return fminf(a, b); }
    static __device__ __forceinline__ mag_t mx(mag_t a, mag_t b) { return fmaxf(a, b); }
    // three-input minimum (sm_100 and later)
    static __device__ __forceinline__ mag_t mn3(mag_t a, mag_t b, mag_t c)
    {
        float r;
        asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
        return r;
    }
    // bit 31 = [x < 0] (valid because no message is -0)
    static __device__ __forceinline__ uint32_t sign_word(acc_t x) { return __float_as_uint(x); }
    static __device__ __forceinline__ float post(acc_t a) { return a; }
    static __device__ __forceinline__ msg_t to_msg(acc_t q) { return q; }
};

// Fixed point with 32-bit accumulation: LLR * 2^FRAC, messages clamped to +-LIM.
//   I16: 8 fractional bits, +-32767;  I8: 2 fractional bits, +-127.
template <class MSG, int FRAC, int LIM>
struct IFix {
    static constexpr int kFrac = FRAC, kLim = LIM;
    using acc_t = int32_t;
    using mag_t = int32_t;
    using msg_t = MSG;
    // gamma_q = clamp(round_half_away(gamma * 2^FRAC), -LIM, LIM); the scaling is exact in binary32
    static __device__ __forceinline__ acc_t quantize(float g)
    {
        float t = roundf(g * float(1 << FRAC));
        t = fminf(fmaxf(t, -float(LIM)), float(LIM));
        return static_cast<int32_t>(t);
    }
    static __device__ __forceinline__ acc_t add(acc_t a, acc_t b) { return a + b; }
    // layered schedule: Q - r_old exactly in 32 bits, and the check's input q = clamp(Q - r_old)
    static __device__ __forceinline__ acc_t sub(acc_t Q, acc_t r) { return Q - r; }
    static __device__ __forceinline__ acc_t clampq(acc_t x) { return max(-LIM, min(LIM, x)); }
    static __device__ __forceinline__ bool neg(int32_t x) { return x < 0; }
    static __device__ __forceinline__ mag_t mag(acc_t x) { return abs(x); }
    static __device__ __forceinline__ mag_t mag_init() { return 0x7fffffff; }
    static __device__ __forceinline__ mag_t mn(mag_t a, mag_t b) { return min(a, b); }
    static __device__ __forceinline__ mag_t mx(mag_t a, mag_t b) { return max(a, b); }
    static __device__ __forceinline__ mag_t mn3(mag_t a, mag_t b, mag_t c) { return __vimin3_s32(a, b, c); }
    // |r| = floor(min * alpha_q / 2^15); min <= 32767 and alpha_q <= 2^15 keep it in 31 bits
    static __device__ __forceinline__ mag_t scale(mag_t m, const LaunchParams &p)
    {
        return (m * p.alpha_q) >> 15;
    }
    static __device__ __forceinline__ uint32_t sign_word(acc_t x) { return uint32_t(x); }
    // sign * m with sign = (-1)^{negall} * sign(x), in two steps: the check's factor on a magnitude once, then each edge's
    // own sign
    static __device__ __forceinline__ mag_t presign(mag_t m, uint32_t negall) { return negall ? -m : m; }
    static __device__ __forceinline__ acc_t apply_sign(mag_t pm, acc_t x) { return x < 0 ? -pm : pm; }
    static __device__ __forceinline__ float post(acc_t a) { return float(a) * (1.0f / float(1 << FRAC)); }
    static __device__ __forceinline__ msg_t to_msg(acc_t q) { return msg_t(max(-LIM, min(LIM, q))); }
};
using I16 = IFix<int16_t, 8, 32767>;
using I8 = IFix<int8_t, 2, 127>;

// The same arithmetic with 4-byte slots.  The variable lanes are packed so that a warp's slots fall in distinct
// 4-byte banks; 2- and 1-byte slots share banks (1.5 wavefronts an access on LP-1054) and need conversions.  The
// single-shot kernel, whose shared memory is never short, keeps its messages so.  Not INT8 rows of more than 16 edges:
// a check's loads then leave no time to its barriers, and bytes take a quarter of the wavefronts (120 rows of 24 at error
// rate 0.05, one shot 150 us with 4-byte slots, 131 with bytes; INT16 152 and 154).
template <class P, int DC>
struct WideSlots {
    using type = P;
};
template <class MSG, int FRAC, int LIM, int DC>
struct WideSlots<IFix<MSG, FRAC, LIM>, DC> {
    using type = IFix<typename std::conditional<sizeof(MSG) == 1 && (DC > 16), MSG, int32_t>::type, FRAC, LIM>;
};

template <class T>
__device__ __forceinline__ T *at_bytes(T *base, uint32_t offset)
{
    return reinterpret_cast<T *>(reinterpret_cast<unsigned char *>(base) + offset);
}

template <class P>
__device__ __forceinline__ typename P::acc_t load_msg(const typename P::msg_t *s, uint32_t i)
{
    return typename P::acc_t(s[i]);
}

// Flip the decision bit of one check's parity word (exact: integer XOR in shared memory).
__device__ __forceinline__ void flip_check(uint32_t *parity, uint32_t m) { atomicXor(parity + m, 1u); }

// Edge-list entries are slot indices j*M + m; the check of a slot is needed only when a decision
// flips: m = slot - M * floor(slot / M), the quotient by a multiply-high with a magic number the
// host verified for every slot (Granlund and Montgomery, PLDI 1994).
struct CheckOf {
    uint32_t M, magic, shift;
    __device__ __forceinline__ CheckOf() : M(1u), magic(0u), shift(0u) {}
    __device__ __forceinline__ explicit CheckOf(const DeviceGraph &g)
        : M(uint32_t(g.m)), magic(g.m_magic), shift(uint32_t(g.m_shift)) {}
    __device__ __forceinline__ uint32_t operator()(uint32_t slot) const
    {
        return M == 1u ? 0u : slot - M * (__umulhi(slot, magic) >> shift);
    }
};

// The two smallest of a[LO .. LO+N), with multiplicity, as a balanced tree: the two smallest of
// {x1 <= x2} and {y1 <= y2} together are min(x1, y1) and min(max(x1, y1), x2, y2).  Every step is
// an exact minimum or maximum, so any grouping gives the same pair; the tree only shortens the
// chain of dependent operations (depth 5 for eight magnitudes against 7 for a running pair).
// Ops supplies mn, mx and mn3 (three-input minimum) on magnitudes of type M.
template <class Ops, int LO, int N, class M>
__device__ __forceinline__ void min2_tree(const M *a, M &m1, M &m2)
{
    static_assert(N >= 2, "two magnitudes at least");
    if constexpr (N == 2) {
        m1 = Ops::mn(a[LO], a[LO + 1]);
        m2 = Ops::mx(a[LO], a[LO + 1]);
    } else if constexpr (N == 3) {
        const M lo = Ops::mn(a[LO + 1], a[LO + 2]), hi = Ops::mx(a[LO + 1], a[LO + 2]);
        m1 = Ops::mn(a[LO], lo);
        m2 = Ops::mn(Ops::mx(a[LO], lo), hi);
    } else {
        constexpr int H = (N / 2) % 2 == 0 || N == 5 ? N / 2 : N / 2 + 1;   // halves of >= 2
        M x1, x2, y1, y2;
        min2_tree<Ops, LO, H>(a, x1, x2);
        min2_tree<Ops, LO + H, N - H>(a, y1, y2);
        m1 = Ops::mn(x1, y1);
        m2 = Ops::mn3(Ops::mx(x1, y1), x2, y2);
    }
}

// The two smallest magnitudes of a row, with multiplicity (m2 = m1 when the minimum is shared).
// Rows of exact degree take the magnitudes in pairs (lo, hi): the second smallest of {m1 <= m2}
// and {lo <= hi} is min(max(m1, lo), m2, hi), one three-input minimum (an odd degree starts from
// m1 = the first magnitude, m2 = +inf); rows of varying degree stream them one at a time.  Either
// way the result is the exact pair of minima.  (A balanced tree, min2_tree, shortens the chain but
// keeps every magnitude live at once: in the FP32 kernels that cost a resident block per SM.)
template <class P, int DC, bool UNIFORM>
__device__ __forceinline__ void two_smallest(const typename P::acc_t *q, int deg, typename P::mag_t &m1,
                                             typename P::mag_t &m2)
{
    using mag_t = typename P::mag_t;
    if constexpr (UNIFORM && DC >= 2) {
        constexpr int j0 = DC % 2 == 0 ? 2 : 1;
        if constexpr (DC % 2 == 0) {
            m1 = P::mn(P::mag(q[0]), P::mag(q[1]));
            m2 = P::mx(P::mag(q[0]), P::mag(q[1]));
        } else {
            m1 = P::mag(q[0]);
            m2 = P::mag_init();
        }
#pragma unroll
        for (int j = j0; j < DC; j += 2) {
            const mag_t a = P::mag(q[j]), b = P::mag(q[j + 1]);
            const mag_t lo = P::mn(a, b), hi = P::mx(a, b);
            m2 = P::mn3(P::mx(m1, lo), m2, hi);
            m1 = P::mn(m1, lo);
        }
    } else {
        m1 = P::mag_init();
        m2 = P::mag_init();
#pragma unroll
        for (int j = 0; j < DC; ++j) {
            if (UNIFORM || j < deg) {
                const mag_t a = P::mag(q[j]);
                m2 = P::mn(m2, P::mx(m1, a));
                m1 = P::mn(m1, a);
            }
        }
    }
}

// min(|a|, |b|) carrying the sign sign(a) xor sign(b) (sm_86 and later)
__device__ __forceinline__ float min_xorsign_abs(float a, float b)
{
    float d;
    asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
    return d;
}

// The two smallest FP32 magnitudes of a row of exactly DC messages, two at a time, with the parity of
// the signs riding on the smallest: |m1s| = min |q|, the sign bit of m1s = xor of every sign bit; m2
// the second smallest magnitude (with multiplicity).  The same pairs of minima and maxima as
// two_smallest, so the same values.
template <int DC>
__device__ __forceinline__ void two_smallest_signed(const float *q, float &m1s, float &m2)
{
    constexpr int j0 = DC % 2 == 0 ? 2 : 1;
    if constexpr (DC % 2 == 0) {
        m1s = min_xorsign_abs(q[0], q[1]);
        m2 = fmaxf(fabsf(q[0]), fabsf(q[1]));
    } else {
        m1s = q[0];
        m2 = F32::mag_init();
    }
#pragma unroll
    for (int j = j0; j < DC; j += 2) {
        const float lo = min_xorsign_abs(q[j], q[j + 1]);
        const float hi = fmaxf(fabsf(q[j]), fabsf(q[j + 1]));
        m2 = F32::mn3(fmaxf(fabsf(m1s), fabsf(lo)), m2, hi);
        m1s = min_xorsign_abs(m1s, lo);
    }
}

// sign * min over the other messages, for one FP32 message q of a row with smallest magnitudes m1 <= m2:
// min(|q|, m2) is m1 where q holds the minimum and m2 elsewhere, so the minimum over the others is the
// one of the two that it is not, and since the bits of non-negative floats are whole numbers it is
// bits(m1) + bits(m2) - bits(min(|q|, m2)), exactly.  The sign of q rides along (min.xorsign with m2 >= 0: its
// bit survives the subtraction modulo 2^32) and the check's factor sits in the sum's bit 31.  Two
// instructions where a comparison, a selection and a sign XOR took three, and one on the ALU pipe
// (which bounds the kernels) instead of three.  A NaN q counts as not holding the minimum, as in the comparison.
// LP-1054, 65536 shots at p = 0.05 in pairs: 3958 -> 3627 us; rows of 9 on [H | I], 8191 shots: 926 -> 849 us;
// learned, 16384 shots: 752 -> 727 us.  (An XOR of the three bit patterns serves as well but stays on the ALU
// pipe: 3693 us.)
__device__ __forceinline__ uint32_t other_sum(float m1, float m2, uint32_t factor_bit31)
{
    return __float_as_uint(m1) + __float_as_uint(m2) + factor_bit31;
}
__device__ __forceinline__ float other_min(float q, float m2, uint32_t sum)
{
    return __uint_as_float(sum - __float_as_uint(min_xorsign_abs(q, m2)));
}

// The check update's reductions of one row: its two smallest magnitudes m1 <= m2 (with multiplicity)
// and the parity of its messages' sign bits (bit 31 of sx).  FP32 rows of exact degree take the parity
// with the smallest magnitude (one instruction per pair of messages fewer); the others xor the signs.
template <class P, int DC, bool UNIFORM>
__device__ __forceinline__ void row_minima(const typename P::acc_t *q, int deg, typename P::mag_t &m1,
                                           typename P::mag_t &m2, uint32_t &sx)
{
    if constexpr (std::is_same<P, F32>::value && UNIFORM && DC >= 2) {
        float m1s;
        two_smallest_signed<DC>(q, m1s, m2);
        m1 = fabsf(m1s);
        sx = __float_as_uint(m1s);
    } else {
        sx = 0;
#pragma unroll
        for (int j = 0; j < DC; ++j)
            if (UNIFORM || j < deg) sx ^= P::sign_word(q[j]);
        two_smallest<P, DC, UNIFORM>(q, deg, m1, m2);
    }
}

// r of each message of a row from its two smallest magnitudes and negall = [(-1)^{s_m} prod of all signs < 0].
// FP32 forms it from other_min; the fixed-point forms scale the two magnitudes first (a floor each).
template <class P>
struct RowOut {
    typename P::mag_t m1, r1, r2;
    __device__ __forceinline__ RowOut(typename P::mag_t a1, typename P::mag_t a2, uint32_t negall, const LaunchParams &p)
        : m1(a1), r1(P::presign(P::scale(a1, p), negall)), r2(P::presign(P::scale(a2, p), negall)) {}
    __device__ __forceinline__ typename P::acc_t operator()(typename P::acc_t q, const LaunchParams &) const
    {
        return P::apply_sign(P::mag(q) == m1 ? r2 : r1, q);
    }
};
template <>
struct RowOut<F32> {
    float m2;
    uint32_t sum;
    __device__ __forceinline__ RowOut(float a1, float a2, uint32_t negall, const LaunchParams &)
        : m2(a2), sum(other_sum(a1, a2, negall << 31)) {}
    __device__ __forceinline__ float operator()(float q, const LaunchParams &p, float scale) const
    {
        return __fmul_rn(scale, other_min(q, m2, sum));
    }
    __device__ __forceinline__ float operator()(float q, const LaunchParams &p) const { return (*this)(q, p, p.alpha); }
};

// ---------------------------------------------------------------------------------------------
// Check-node step (Alg. 1, CN processing) of one check, fused with the stop test of the previous
// decisions.  Returns 1 iff the check's parity word says s_m is satisfied.
// UNIFORM: every row has exactly DC edges; otherwise deg <= DC.
// ---------------------------------------------------------------------------------------------
// LEARNED (FP32 only): when w is non-null the scale is the learned weight of each edge,
// r = sign * (w_{m,n} * min_{j != n} |q_j|), w = this iteration's weights in groups of four edges (train_edge_at), read
// with one 16-byte load a group before the messages, so that their way from L2 overlaps the minima (16384 shots of
// LP-1054, 20 learned iterations, then the plain ones: 603 us with a 4-byte load where a weight is used -> 549 us).
// Rows of more than 16 edges read them after the minima, a group at a time: 32 weights beside 32 messages spill (120 rows
// of 24, two error rates together, us before | after the minima: one shot 276 | 203, 600 shots 971 | 649, 16384 shots
// 4090 | 3288; rows of 12 lose by it, 16384 shots 1910 | 2036).
template <class P, int DC, bool UNIFORM, bool LEARNED = false>
__device__ __forceinline__ int check_step(int c, int M, int deg, uint32_t pw, bool update,
                                          typename P::msg_t *__restrict__ slots, const LaunchParams &p,
                                          const float *__restrict__ w = nullptr)
{
    using acc_t = typename P::acc_t;
    using mag_t = typename P::mag_t;
    if (update) {
        acc_t q[DC];
        constexpr bool kWeightsFirst = LEARNED && DC <= 16;
        float scale[kWeightsFirst ? (DC + 3) / 4 * 4 : 1];
        if constexpr (kWeightsFirst) {
#pragma unroll
            for (int j = 0; j < DC; j += 4) {
                float4 v = make_float4(p.alpha, p.alpha, p.alpha, p.alpha);
                if (w && (UNIFORM || j < deg)) v = __ldg(reinterpret_cast<const float4 *>(w + train_edge_at(4, c, j, M)));
                scale[j] = v.x;
                scale[j + 1] = v.y;
                scale[j + 2] = v.z;
                scale[j + 3] = v.w;
            }
        }
#pragma unroll
        for (int j = 0; j < DC; ++j)
            if (UNIFORM || j < deg) q[j] = load_msg<P>(slots, uint32_t(j * M + c));
        mag_t m1, m2;
        uint32_t sx;                               // bit 31: parity of the signs
        row_minima<P, DC, UNIFORM>(q, deg, m1, m2, sx);
        const uint32_t negall = ((pw >> 1) ^ (sx >> 31)) & 1u;   // (-1)^{s_m} * prod of all signs
        const RowOut<P> out(m1, m2, negall, p);
        if constexpr (LEARNED && !kWeightsFirst) {
            if (w) {
#pragma unroll
                for (int j = 0; j < DC; j += 4) {
                    if (UNIFORM || j < deg) {
                        const float4 v = __ldg(reinterpret_cast<const float4 *>(w + train_edge_at(4, c, j, M)));
                        const float x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                        for (int i = 0; i < 4 && j + i < DC; ++i)
                            if (UNIFORM || j + i < deg) slots[(j + i) * M + c] = out(q[j + i], p, x[i]);
                    }
                }
                return (pw & 1u) == 0;
            }
        }
#pragma unroll
        for (int j = 0; j < DC; ++j) {
            if (UNIFORM || j < deg) {
                if constexpr (kWeightsFirst)
                    slots[j * M + c] = out(q[j], p, scale[j]);
                else
                    slots[j * M + c] = typename P::msg_t(out(q[j], p));
            }
        }
    }
    return (pw & 1u) == 0;
}

// ---------------------------------------------------------------------------------------------
// Variable-node step (Alg. 1, VN processing + a-posteriori LLR + tentative decision) of a
// variable of degree exactly D whose edges are e[0..D).  q_k = gamma + sum_{i != k} r_i in
// ascending order: q_k = ((pre_k + r_{k+1}) + r_{k+2}) + ...  with pre_k = ((gamma + r_0) + r_1)
// + ... + r_{k-1}.  Stores every q_k, flips the parity bit of its checks when the decision
// [Q < 0] differs from `prev`, and returns Q.
// ---------------------------------------------------------------------------------------------
// BYTES: sl holds byte offsets into slots instead of slot indices (lane_slots).
template <class P, int D, bool BYTES = false>
__device__ __forceinline__ typename P::acc_t var_step_exact(const uint32_t *sl, const CheckOf &ck, typename P::acc_t gamma,
                                                            bool prev, typename P::msg_t *__restrict__ slots,
                                                            uint32_t *__restrict__ parity)
{
    using acc_t = typename P::acc_t;
    if constexpr (D == 0) {
        return gamma;
    } else {
        acc_t r[D];
#pragma unroll
        for (int k = 0; k < D; ++k) r[k] = typename P::acc_t(BYTES ? *at_bytes(slots, sl[k]) : slots[sl[k]]);
        acc_t pre[D + 1];
        pre[0] = gamma;
#pragma unroll
        for (int k = 0; k < D; ++k) pre[k + 1] = P::add(pre[k], r[k]);
        const acc_t Q = pre[D];
#pragma unroll
        for (int k = 0; k < D; ++k) {
            acc_t q = pre[k];
#pragma unroll
            for (int i = k + 1; i < D; ++i) q = P::add(q, r[i]);
            (BYTES ? *at_bytes(slots, sl[k]) : slots[sl[k]]) = P::to_msg(q);
        }
        if (P::neg(Q) != prev) {
#pragma unroll
            for (int k = 0; k < D; ++k) flip_check(parity, ck(BYTES ? sl[k] / sizeof(typename P::msg_t) : sl[k]));
        }
        return Q;
    }
}

#define QLDPC_DEG_CASES(X) X(0) X(1) X(2) X(3) X(4) X(5) X(6) X(7) X(8) X(9) X(10) X(11) X(12) X(13) X(14) X(15) X(16)

// f(D, u) for this thread's variable lanes u = tid, tid + T, ... with their degree D a compile-time constant
// (lanes come in classes of one degree, walked in order; reading each lane's degree and branching on it costs
// a tenth of a decode).
template <int DV, class F>
__device__ __forceinline__ void for_lanes(const DeviceGraph &G, int tid, int T, F f)
{
    int u = tid;
    for (int cl = 0; cl < G.ncls && u < G.nv; ++cl) {
        const int u1 = G.cls_end[cl];
        auto run = [&](auto deg) {
#pragma unroll 1
            for (; u < u1; u += T) f(deg, u);
        };
        switch (G.cls_deg[cl]) {
#define QLDPC_CASE(DD)                                                                          \
    case DD:                                                                                    \
        if constexpr (DD <= DV) run(std::integral_constant<int, DD>{});                         \
        break;
            QLDPC_DEG_CASES(QLDPC_CASE)
#undef QLDPC_CASE
        default:   // a degree above the variant's bucket (the host never launches one)
            while (u < u1) u += T;
            break;
        }
    }
}

// The edge slots of lane u as byte offsets into words of WORD bytes, from the 16-bit lists (vslot16): four slots come with
// one load, and one two-way dot product takes a slot out of its register and scales it.  The variable steps are short of
// load instructions (a slot a load: 16384 learned shots of LP-1054 550 -> 531 us, 8191 of its 465 x 1519 data-syndrome
// graph 746 -> 714, 4096 in INT16 212 -> 204; the paired FP32 kernel, which waits on its 8-byte slots, 3631 -> 3619).
template <int D, int WORD>
__device__ __forceinline__ void lane_slots(const uint16_t *__restrict__ list, int NV, int u, uint32_t (&o)[D > 0 ? D : 1])
{
#pragma unroll
    for (int k = 0; k < D; k += 4) {
        const uint16_t *at = list + (size_t(k / 4) * NV + u) * 4;
        uint2 v = make_uint2(0u, 0u);
        if (D - k > 2)
            v = __ldg(reinterpret_cast<const uint2 *>(at));
        else if (D - k == 2)
            v.x = __ldg(reinterpret_cast<const unsigned *>(at));
        else
            v.x = __ldg(at);
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (k + i < D) o[k + i] = __dp2a_lo(i < 2 ? v.x : v.y, unsigned(i & 1 ? WORD << 8 : WORD), 0u);
    }
}

// The same from the 32-bit lists on a graph with more slots than 16 bits index (no such graph fits a block in FP32).
template <int D, int WORD, bool WIDE>
__device__ __forceinline__ void lane_edges(const DeviceGraph &g, int u, uint32_t (&o)[D > 0 ? D : 1])
{
    if constexpr (WIDE) {
#pragma unroll
        for (int k = 0; k < D; ++k) o[k] = __ldg(g.vslot + size_t(k) * g.nv + u) * WORD;
    } else {
        lane_slots<D, WORD>(g.vslot16, g.nv, u, o);
    }
}

// ---------------------------------------------------------------------------------------------
// Throughput kernel
// ---------------------------------------------------------------------------------------------
// Initialization (Alg. 1) of one shot: q^(0) = gamma on every edge; the parity words start at s_m
// and take the decisions of the prior.  Ends with a barrier.
template <class P, int DV, bool WIDE>
__device__ __forceinline__ void batch_init_shot(const DeviceGraph &g, const uint8_t *s, int tid, int T,
                                                const typename P::acc_t *gam, typename P::acc_t *Qs,
                                                uint32_t *parity, typename P::msg_t *slots)
{
    for (int c = tid; c < g.m; c += T) parity[c] = (s[c] & 1u) * 3u;
    __syncthreads();
    const CheckOf ck(g);
    for_lanes<DV>(g, tid, T, [&](auto deg, int u) {
        constexpr int D = decltype(deg)::value;
        uint32_t e[D > 0 ? D : 1];
        lane_edges<D, sizeof(typename P::msg_t), WIDE>(g, u, e);
        const typename P::acc_t x = gam[u];
        const bool d = P::neg(x);
#pragma unroll
        for (int k = 0; k < D; ++k) {
            *at_bytes(slots, e[k]) = P::to_msg(x);
            if (d) flip_check(parity, ck(e[k] / sizeof(typename P::msg_t)));
        }
        Qs[u] = x;
    });
    __syncthreads();
}

// LEARNED: iterations 1..learned_iters use the learned weights; a shot whose syndrome is still not
// met then restarts from its prior with plain min-sum (alpha) for up to max_iter iterations, and
// reports learned_iters + the plain iterations.  Learned launches always stop early.
template <class P, int DC, bool UNIFORM, int DV, bool LEARNED, bool WIDE>
__device__ __forceinline__ void batch_decode(const LaunchParams &p)
{
    using acc_t = typename P::acc_t;
    using msg_t = typename P::msg_t;

    const Problem pr = blockIdx.y == 0 ? p.prob[0] : p.prob[1];
    const DeviceGraph &G = p.prob[blockIdx.y].g;   // read in place (the class tables are indexed at run time)
    const int M = pr.g.m, N = pr.g.n, NV = pr.g.nv;   // checks, variables, variable lanes
    const int T = blockDim.x, tid = threadIdx.x;

    extern __shared__ __align__(16) unsigned char smem[];
    const SmemLayout L = smem_layout(M, NV, pr.g.dc_max, int(sizeof(msg_t)));
    acc_t *Qs = reinterpret_cast<acc_t *>(smem + L.q_off);
    acc_t *gam = reinterpret_cast<acc_t *>(smem + L.g_off);
    uint32_t *parity = reinterpret_cast<uint32_t *>(smem + L.par_off);
    msg_t *slots = reinterpret_cast<msg_t *>(smem + L.slot_off);

    // Prior LLRs: loaded once per block, shared by all its shots (idle lanes: 0, no edges).
    int bad = 0;
    for (int u = tid; u < NV; u += T) {
        const uint32_t v = __ldg(pr.g.vperm + u);
        const float g = v < uint32_t(N) ? pr.prior[v] : 0.0f;
        bad |= !isfinite(g);
        gam[u] = P::quantize(g);
    }
    bad = __syncthreads_or(bad);

    const bool early = LEARNED || (p.flags & kFlagNoEarlyStop) == 0;
    const size_t wstride = learned_stride(pr.g.dc_max, M);   // learned weights of one iteration
    // Shots are claimed one at a time from a per-launch counter, so blocks that draw slowly
    // converging shots take fewer of them (or taken statically when no counter is given).
    // (Two claim words alternate: a thread reads word k&1 after claim k's barrier, and the word is
    // rewritten only after claim k+1's barrier, which every thread reaches after its read.)
    __shared__ int s_shot[2];
    int claim = 0;
    for (int b = blockIdx.x;; b += gridDim.x) {
        if (p.next_shot) {
            if (tid == 0) s_shot[claim] = atomicAdd(p.next_shot + blockIdx.y, 1);
            __syncthreads();
            b = s_shot[claim];
            claim ^= 1;
        }
        if (b >= p.batch) break;
        uint8_t *err = pr.err + size_t(b) * N;
        if (bad) {   // non-finite prior: report the shot as not decoded
            for (int v = tid; v < N; v += T) {
                err[v] = 0;
                if (pr.post) pr.post[size_t(b) * N + v] = __int_as_float(0x7fc00000);
            }
            if (tid == 0) {
                pr.iters[b] = -1;
                pr.ok[b] = 0;
            }
            continue;
        }
        const uint8_t *s = pr.syn + size_t(b) * M;
        batch_init_shot<P, DV, WIDE>(G, s, tid, T, gam, Qs, parity, slots);

        int k = 0, all = 0;
        bool learned = LEARNED;
        int end = LEARNED ? pr.learned_iters : p.max_iter;   // k at which the current phase ends
        for (;;) {
            const bool last = k >= end;
            const float *wk = nullptr;
            if constexpr (LEARNED) wk = (learned && !last) ? pr.weights + size_t(k) * wstride : nullptr;
            int ok = 1;
            for (int c = tid; c < M; c += T) {
                const int deg = UNIFORM ? DC : int(__ldg(pr.g.rdeg + c));
                ok &= check_step<P, DC, UNIFORM, LEARNED>(c, M, deg, parity[c], !last, slots, p, wk);
            }
            all = __syncthreads_and(ok);
            if (early && all) break;
            if (last) {
                if (!LEARNED || !learned) break;
                learned = false;                  // fallback: plain min-sum from the prior
                end = k + p.max_iter;
                batch_init_shot<P, DV, WIDE>(G, s, tid, T, gam, Qs, parity, slots);
                continue;
            }
            const CheckOf ck(pr.g);
            for_lanes<DV>(G, tid, T, [&](auto deg, int u) {
                constexpr int D = decltype(deg)::value;
                uint32_t e[D > 0 ? D : 1];
                lane_edges<D, sizeof(msg_t), WIDE>(G, u, e);
                Qs[u] = var_step_exact<P, D, true>(e, ck, gam[u], P::neg(Qs[u]), slots, parity);
            });
            __syncthreads();
            ++k;
        }

        for (int v = tid; v < N; v += T) {   // in variable order: a warp's stores are adjacent
            const acc_t q = Qs[__ldg(pr.g.vlane + v)];
            err[v] = P::neg(q) ? 1 : 0;
            if (pr.post) pr.post[size_t(b) * N + v] = P::post(q);
        }
        if (tid == 0) {
            pr.iters[b] = k;
            pr.ok[b] = all ? 1 : 0;
        }
        __syncthreads();   // the next shot reuses shared memory
    }
}

template <class P, int DC, bool UNIFORM, int DV, bool LEARNED = false>
__global__ void __launch_bounds__(1024, 1) msa_batch_kernel(const __grid_constant__ LaunchParams p)
{
    if constexpr (sizeof(typename P::msg_t) < 4)
        if (!p.prob[blockIdx.y].g.vslot16) {
            batch_decode<P, DC, UNIFORM, DV, LEARNED, true>(p);
            return;
        }
    batch_decode<P, DC, UNIFORM, DV, LEARNED, false>(p);
}

// ---------------------------------------------------------------------------------------------
// Latency kernel: one block per shot, everything a thread needs across iterations in registers.
// ---------------------------------------------------------------------------------------------
constexpr int kLatCnPerThread = kLatencyCnPerThread;   // checks per thread: M <= 2*blockDim
constexpr int kLatVnPerThread = kLatencyVnPerThread;   // variables per thread: N <= 2*blockDim

template <class P, int DV>
__device__ __forceinline__ typename P::acc_t var_step_regs(int deg, const uint32_t *e, const CheckOf &ck,
                                                           typename P::acc_t gamma, bool prev,
                                                           typename P::msg_t *slots, uint32_t *parity)
{
    switch (deg) {
#define QLDPC_CASE(D)                                                                           \
    case D:                                                                                     \
        if constexpr (D <= DV) return var_step_exact<P, D>(e, ck, gamma, prev, slots, parity); \
        break;
        QLDPC_DEG_CASES(QLDPC_CASE)
#undef QLDPC_CASE
    default: break;
    }
    return gamma;
}

// PT: checks and variable lanes per thread, 1 where a block of at most kLatencyMaxThreads covers both, else 2.  With
// one of each a thread needs 48 to 64 registers instead of 72 to 94, so two to eight blocks share an SM: 65536 shots of
// the 144 x 288 code FP32 861 -> 690 us (and INT16 with 4-byte slots 1322 -> 794), 6400 of the 192 x 400 code 352 -> 338.
template <class P, int DC, bool UNIFORM, int DV, int PT, bool LEARNED = false>
__global__ void __launch_bounds__(kLatencyMaxThreads, 1) msa_latency_kernel(const LaunchParams p)
{
    using acc_t = typename P::acc_t;
    using msg_t = typename P::msg_t;

    const Problem pr = blockIdx.y == 0 ? p.prob[0] : p.prob[1];
    const int M = pr.g.m, N = pr.g.n, NV = pr.g.nv;
    const int T = blockDim.x, tid = threadIdx.x;
    extern __shared__ __align__(16) unsigned char smem[];
    const LatencyLayout L = latency_layout(M, pr.g.dc_max, int(sizeof(msg_t)));
    uint32_t *parity = reinterpret_cast<uint32_t *>(smem + L.par_off);
    msg_t *slots = reinterpret_cast<msg_t *>(smem + L.slot_off);

    // Checks c = tid + i*T: degree in registers.
    int cdeg[PT];
#pragma unroll
    for (int i = 0; i < PT; ++i) {
        const int c = tid + i * T;
        cdeg[i] = c < M ? (UNIFORM ? DC : int(__ldg(pr.g.rdeg + c))) : -1;
    }
    // Variable lanes u = tid + i*T (heaviest first, so the few second-pass variables are the
    // lightest): edge lists, degree and prior in registers; vid = original index for the outputs.
    uint32_t ev[PT][DV];
    int vdeg[PT], vid[PT];
    acc_t gam[PT];
    int bad = 0;
#pragma unroll
    for (int i = 0; i < PT; ++i) {
        const int u = tid + i * T;
        const int v = u < NV ? int(__ldg(pr.g.vperm + u)) : N;   // N: idle lane
        vid[i] = v;
        vdeg[i] = u < NV ? int(__ldg(pr.g.vdeg + u)) : -1;
#pragma unroll
        for (int k = 0; k < DV; ++k)
            ev[i][k] = (k < vdeg[i]) ? __ldg(pr.g.vslot + size_t(k) * NV + u) : 0u;
        const float g = v < N ? pr.prior[v] : 0.0f;
        bad |= !isfinite(g);
        gam[i] = P::quantize(g);
    }
    bad = __syncthreads_or(bad);

    const bool early = LEARNED || (p.flags & kFlagNoEarlyStop) == 0;
    const size_t wstride = learned_stride(pr.g.dc_max, M);
    __shared__ int s_shot[2];   // alternating claim words, as in the batch kernel
    int claim = 0;
    for (int b = blockIdx.x;; b += gridDim.x) {
        if (p.next_shot) {      // more shots than blocks
            if (tid == 0) s_shot[claim] = atomicAdd(p.next_shot + blockIdx.y, 1);
            __syncthreads();
            b = s_shot[claim];
            claim ^= 1;
        }
        if (b >= p.batch) break;
        uint8_t *err = pr.err + size_t(b) * N;
        if (bad) {
#pragma unroll
            for (int i = 0; i < PT; ++i) {
                const int v = vid[i];
                if (v < N) {
                    err[v] = 0;
                    if (pr.post) pr.post[size_t(b) * N + v] = __int_as_float(0x7fc00000);
                }
            }
            if (tid == 0) {
                pr.iters[b] = -1;
                pr.ok[b] = 0;
            }
            continue;
        }
        const uint8_t *s = pr.syn + size_t(b) * M;
        acc_t Q[PT];
        // Initialization (Alg. 1), also the restart of the plain fallback; ends with a barrier.
        auto init_shot = [&]() {
#pragma unroll
            for (int i = 0; i < PT; ++i)
                if (cdeg[i] >= 0) parity[tid + i * T] = (s[tid + i * T] & 1u) * 3u;
            __syncthreads();
#pragma unroll
            for (int i = 0; i < PT; ++i) {
                Q[i] = gam[i];
                const bool d = P::neg(gam[i]);
#pragma unroll
                for (int k = 0; k < DV; ++k) {
                    if (k < vdeg[i]) {
                        slots[ev[i][k]] = P::to_msg(gam[i]);
                        if (d) flip_check(parity, CheckOf(pr.g)(ev[i][k]));
                    }
                }
            }
            __syncthreads();
        };
        init_shot();

        int k = 0, all = 0;
        bool learned = LEARNED;
        int end = LEARNED ? pr.learned_iters : p.max_iter;
        for (;;) {
            const bool last = k >= end;
            const float *wk = nullptr;
            if constexpr (LEARNED) wk = (learned && !last) ? pr.weights + size_t(k) * wstride : nullptr;
            int ok = 1;
#pragma unroll
            for (int i = 0; i < PT; ++i)
                if (cdeg[i] >= 0)
                    ok &= check_step<P, DC, UNIFORM, LEARNED>(tid + i * T, M, cdeg[i], parity[tid + i * T], !last,
                                                              slots, p, wk);
            all = __syncthreads_and(ok);
            if (early && all) break;
            if (last) {
                if (!LEARNED || !learned) break;
                learned = false;                  // fallback: plain min-sum from the prior
                end = k + p.max_iter;
                init_shot();
                continue;
            }
#pragma unroll
            for (int i = 0; i < PT; ++i)
                if (vdeg[i] >= 0)
                    Q[i] = var_step_regs<P, DV>(vdeg[i], ev[i], CheckOf(pr.g), gam[i], P::neg(Q[i]), slots, parity);
            __syncthreads();
            ++k;
        }

#pragma unroll
        for (int i = 0; i < PT; ++i) {
            const int v = vid[i];
            if (v < N) {
                err[v] = P::neg(Q[i]) ? 1 : 0;
                if (pr.post) pr.post[size_t(b) * N + v] = P::post(Q[i]);
            }
        }
        if (tid == 0) {
            pr.iters[b] = k;
            pr.ok[b] = all ? 1 : 0;
        }
        __syncthreads();   // the next shot reuses shared memory
    }
}

}  // namespace kern

// ---------------------------------------------------------------------------------------------
// Instantiation tables for one precision policy: uniform row degree 6, 7, 8, 9 (exact; 9 is a
// degree-8 code's row on the data-syndrome graph [H | I]) or any degree up to 8, 16, 32;
// column-degree bucket 4, 8, 16; for each, the batch and the latency kernel.
// ---------------------------------------------------------------------------------------------
#define QLDPC_DV_LIST(X, A, B) X(A, B, 4) X(A, B, 8) X(A, B, 16)
#define QLDPC_VARIANTS(X)                                                                       \
    QLDPC_DV_LIST(X, 6, true) QLDPC_DV_LIST(X, 7, true) QLDPC_DV_LIST(X, 8, true)               \
    QLDPC_DV_LIST(X, 9, true) QLDPC_DV_LIST(X, 8, false) QLDPC_DV_LIST(X, 16, false) QLDPC_DV_LIST(X, 32, false)

template <class P, bool LEARNED = false>
const void *kernel_table(const KernelChoice &kc)
{
#define QLDPC_K(DCV, UNI, DVV)                                                                  \
    if (kc.dc == DCV && kc.uniform == UNI && kc.dvb == DVV)                                     \
        return !kc.latency      ? reinterpret_cast<const void *>(&kern::msa_batch_kernel<P, DCV, UNI, DVV, LEARNED>) \
               : kc.one_pass    ? reinterpret_cast<const void *>(&kern::msa_latency_kernel<typename kern::WideSlots<P, DCV>::type, DCV, UNI, DVV, 1, LEARNED>) \
                                : reinterpret_cast<const void *>(&kern::msa_latency_kernel<typename kern::WideSlots<P, DCV>::type, DCV, UNI, DVV, 2, LEARNED>);
    QLDPC_VARIANTS(QLDPC_K)
#undef QLDPC_K
    return nullptr;
}

template <class P, bool LEARNED = false>
cudaError_t launch_table(const LaunchParams &p, const KernelChoice &kc, dim3 grid, int threads,
                         size_t smem, cudaStream_t stream)
{
    const void *k = kernel_table<P, LEARNED>(kc);
    if (!k) return cudaErrorInvalidValue;
    void *args[] = {const_cast<LaunchParams *>(&p)};
    const cudaError_t e = cudaLaunchKernel(k, grid, dim3(unsigned(threads)), args, smem, stream);
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace qldpc
