// The two ends of the loop that measures a logical error rate, for sm_103a: the seeded error sampler
// (errors and their syndromes) and the test of decoded shots against the logical operators.
#include <algorithm>
#include <cstdint>

#include <cuda_runtime.h>

#include "msa_launch.h"

namespace qldpc {
namespace kern {

constexpr int kSampleThreads = 256;
constexpr int kSampleShots = 32;      // shots of a tile: one per lane
constexpr int kSegMax = 1280;         // qubits (or checks) of a tile's rows held as bytes at a time, at most

// Columns of a tile of rows of n bytes: rows split evenly into segments of a multiple of 16, at most kSegMax.
__host__ __device__ inline int seg_bytes(int n)
{
    const int parts = (n + kSegMax - 1) / kSegMax;
    return ((n + parts - 1) / parts + 15) / 16 * 16;
}
// Words of a tile row: odd (32 rows fall in 32 banks) and one word past the segment, which an unaligned
// 16-byte chunk reads.
__host__ __device__ inline int seg_stride(int seg) { return seg / 4 + 1; }

// SplitMix64 (Steele, Lea and Flood, OOPSLA 2014): the output of one step from state x.
__device__ __forceinline__ uint64_t splitmix64(uint64_t x)
{
    uint64_t z = x + 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// Rows 0..ns of `len` bytes, n apart in memory, from their tile rows (4-byte words, byte 0 of word 0 first) to
// dst, any alignment: the 16-byte blocks inside a row as vector stores, the bytes before and after them
// singly (block-wide: a row's 66 blocks would leave most of a warp's third pass idle).
__device__ __forceinline__ void store_rows(uint8_t *__restrict__ dst, size_t n, int len, int ns,
                                           const uint32_t *__restrict__ tile, int stride, int tid)
{
    const int per_row = len >> 4;                          // blocks inside a row: this many, or one fewer
    const uint32_t inv = per_row ? 0xffffffffu / uint32_t(per_row) + 1u : 0u;   // x / per_row for x < 2^16
    for (int x = tid; x < ns * per_row; x += kSampleThreads) {
        const int s = per_row == 1 ? x : int(__umulhi(uint32_t(x), inv)), i = x - s * per_row;
        uint8_t *d = dst + size_t(s) * n;
        const int head = int((0u - uint32_t(reinterpret_cast<uintptr_t>(d))) & 15u), at = head + 16 * i;
        if (at + 16 > len) continue;
        const uint32_t *row = tile + s * stride + (at >> 2);
        const int sh = 8 * (head & 3);
        uint32_t w[5];
#pragma unroll
        for (int t = 0; t < 5; ++t) w[t] = row[t];
        uint4 o;
        o.x = __funnelshift_r(w[0], w[1], sh);
        o.y = __funnelshift_r(w[1], w[2], sh);
        o.z = __funnelshift_r(w[2], w[3], sh);
        o.w = __funnelshift_r(w[3], w[4], sh);
        *reinterpret_cast<uint4 *>(d + at) = o;
    }
    for (int x = tid; x < ns * 32; x += kSampleThreads) {  // up to 15 bytes at either end of each row
        const int s = x >> 5, k = x & 15;
        uint8_t *d = dst + size_t(s) * n;
        const int head = min(len, int((0u - uint32_t(reinterpret_cast<uintptr_t>(d))) & 15u)), tail = (len - head) & 15;
        const bool front = (x & 16) == 0;
        const int at = front ? k : len - tail + k;
        if (k < (front ? head : tail)) d[at] = uint8_t(tile[s * stride + (at >> 2)] >> (8 * (at & 3)));
    }
}

// A shot's key and its threshold for the hash: u(q) < p_shot as the comparison x <= limit of the 64-bit hash
// x with ceil(p 2^53) 2^11 - 1, exact because u 2^53 = x >> 11 is a whole number.  any: p_shot > 0.
struct ShotRate {
    uint64_t key, limit;
    bool any;
};
__device__ __forceinline__ ShotRate shot_rate(uint64_t k_seed, uint64_t shot, int N, double p_lo, double p_span)
{
    const uint64_t key = splitmix64(k_seed + shot);
    const double un = double(splitmix64(key + uint64_t(N)) >> 11) * 1.1102230246251565e-16;   // 2^-53
    const double thr = __dmul_rn(__dadd_rn(p_lo, __dmul_rn(p_span, un)), 9007199254740992.0); // p * 2^53
    const uint64_t c = __double2ull_ru(thr);                                                  // <= 2^53
    return ShotRate{key, (c << 11) - 1, c != 0};   // (c = 2^53 wraps to all ones: every hash)
}

// Errors at a per-shot rate and their syndromes.  Counter-based keying (seed, shot, qubit):
// u = top 53 bits of mix(mix(mix(seed) + shot) + qubit) / 2^53; p_shot = p_lo + p_span * u(qubit n);
// e_q = [u(q) < p_shot]; s_i = XOR of e over row i.
//
// A block takes tiles of 32 shots, a lane per shot.  FP64 is left to one rate per shot (a conversion and a
// comparison in FP64 for every qubit kept that pipe 82 % busy and set the time).  A warp's ballot
// is the qubit's error bit in 32 shots, so a check's syndrome bit in all of them is the XOR of its row's
// ballots: one row walk for 32 shots.  Bytes are staged in shared memory and leave as 16-byte stores.
// What bounds it: the hash, 36 clocks of an SM quarter per warp (its 64-bit shifts and XORs sit on the ALU
// pipe; shifts by 64-bit multiply-add took 48).  65536 shots of 1054 qubits: 440 -> 112 us, of which the
// hash alone is 68.
__global__ void __launch_bounds__(kSampleThreads)
    sample_kernel(const DeviceGraph g, uint64_t seed, int64_t first_shot, int32_t batch, double p_lo, double p_span,
                  uint8_t *__restrict__ err, uint8_t *__restrict__ syn)
{
    extern __shared__ __align__(16) uint32_t sm[];
    const int M = g.m, N = g.n, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int T = kSampleThreads, nwarp = T / 32;
    const int nseg = seg_bytes(N), mseg = seg_bytes(M), nstr = seg_stride(nseg), mstr = seg_stride(mseg);
    uint32_t *tile = sm;                                            // [32][stride]
    uint32_t *ew = sm + kSampleShots * max(nstr, mstr);             // [N rounded up to 4] ballots of the qubits
    uint32_t *sw = ew + ((N + 3) & ~3);                             // [M rounded up to 4] syndrome bits of the checks
    __shared__ uint64_t s_key[kSampleShots], s_lim[kSampleShots];
    __shared__ uint32_t s_some;                                     // the shots with a rate above 0
    const uint64_t k_seed = splitmix64(seed);
    const int64_t tiles = (int64_t(batch) + kSampleShots - 1) / kSampleShots;
    for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        const int64_t b0 = t * kSampleShots;
        const int ns = int(min(int64_t(kSampleShots), int64_t(batch) - b0));
        if (warp == 0) {
            const ShotRate r = shot_rate(k_seed, uint64_t(first_shot + b0 + lane), N, p_lo, p_span);
            s_key[lane] = r.key;
            s_lim[lane] = r.limit;
            const uint32_t some = __ballot_sync(0xffffffffu, r.any && lane < ns);
            if (lane == 0) s_some = some;
        }
        __syncthreads();
        const uint64_t key = s_key[lane], lim = s_lim[lane];
        const uint32_t some = s_some, mine = 0u - ((some >> lane) & 1u);
        for (int q0 = 0; q0 < N; q0 += nseg) {
            const int len = min(nseg, N - q0);
            const uint64_t base = key + uint64_t(q0);
            for (int i = warp; 4 * i < len; i += nwarp) {
                uint32_t bytes = 0, w[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const bool e = splitmix64(base + uint32_t(4 * i + j)) <= lim;
                    w[j] = __ballot_sync(0xffffffffu, e) & some;
                    if (e) bytes |= 1u << (8 * j);
                }
                tile[lane * nstr + i] = bytes & mine;         // (bytes past the last qubit are not stored)
                if (lane == 0) *reinterpret_cast<uint4 *>(ew + q0 + 4 * i) = make_uint4(w[0], w[1], w[2], w[3]);
            }
            __syncthreads();
            store_rows(err + size_t(b0) * N + q0, size_t(N), len, ns, tile, nstr, tid);
            __syncthreads();
        }
        for (int c = tid; c < M; c += T) {
            const int deg = __ldg(g.rdeg + c);
            uint32_t par = 0;
            for (int j = 0; j < deg; ++j) par ^= ew[__ldg(g.ecol + size_t(j) * M + c)];
            sw[c] = par;
        }
        __syncthreads();
        for (int c0 = 0; c0 < M; c0 += mseg) {
            const int len = min(mseg, M - c0);
            for (int i = warp; 4 * i < len; i += nwarp) {
                uint32_t bytes = 0;
#pragma unroll
                for (int j = 0; j < 4; ++j)                         // (past the last check: never stored)
                    bytes |= ((sw[c0 + 4 * i + j] >> lane) & 1u) << (8 * j);
                tile[lane * mstr + i] = bytes;
            }
            __syncthreads();
            store_rows(syn + size_t(b0) * M + c0, size_t(M), len, ns, tile, mstr, tid);
            __syncthreads();
        }
    }
}

// One shot per block at a time: batches too small to give every SM a tile of 32 (1000 shots of 1054
// qubits would keep 32 of 152 SMs busy: 18 us against 12 in this form; at 2400 shots 19 and 15).
__global__ void __launch_bounds__(kSampleThreads)
    sample_shot_kernel(const DeviceGraph g, uint64_t seed, int64_t first_shot, int32_t batch, double p_lo, double p_span,
                       uint8_t *__restrict__ err, uint8_t *__restrict__ syn)
{
    extern __shared__ __align__(16) unsigned char es[];
    const int M = g.m, N = g.n, T = kSampleThreads, tid = threadIdx.x;
    __shared__ ShotRate s_rate;
    const uint64_t k_seed = splitmix64(seed);
    for (int b = blockIdx.x; b < batch; b += gridDim.x) {
        if (tid == 0) s_rate = shot_rate(k_seed, uint64_t(first_shot + b), N, p_lo, p_span);
        __syncthreads();
        const ShotRate r = s_rate;
        for (int q = tid; q < N; q += T) {
            const uint8_t e = splitmix64(r.key + uint64_t(q)) <= r.limit && r.any ? 1 : 0;
            es[q] = e;
            err[size_t(b) * N + q] = e;
        }
        __syncthreads();
        for (int c = tid; c < M; c += T) {
            const int deg = __ldg(g.rdeg + c);
            uint32_t par = 0;
            for (int j = 0; j < deg; ++j) par ^= es[__ldg(g.ecol + size_t(j) * M + c)];
            syn[size_t(b) * M + c] = uint8_t(par);
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------------------------
// Logical test: fail_b = !ok_b OR some logical operator has odd overlap with e_b XOR e_hat_b.
// ---------------------------------------------------------------------------------------------
constexpr int kLogicalThreads = 256;
constexpr int kDirectWords = 64;      // residual words of a tile tested straight from the operators' bytes
constexpr int kDirectOps = 512;       // ... for at most so many operators

// The low bit of each byte of w (lowest byte first) as 4 bits; w has no other bits set.
__device__ __forceinline__ uint32_t pack4(uint32_t w) { return (w * 0x01020408u) >> 24; }
__device__ __forceinline__ uint32_t nonzero4(uint32_t w)    // 1 in each byte that is not 0
{
    return ((((w & 0x7f7f7f7fu) + 0x7f7f7f7fu) | w) >> 7) & 0x01010101u;
}
// pack(a.x..w): the marked bytes of 16 as 16 bits
__device__ __forceinline__ uint32_t pack16(uint32_t x, uint32_t y, uint32_t z, uint32_t w)
{
    return pack4(x) | pack4(y) << 4 | pack4(z) << 8 | pack4(w) << 12;
}
// 16 bytes at p, of which `count` exist
__device__ __forceinline__ uint4 load_some(const uint8_t *p, int count)
{
    uint32_t w[4] = {0, 0, 0, 0};
#pragma unroll
    for (int i = 0; i < 16; ++i)
        if (i < count) w[i >> 2] |= uint32_t(__ldg(p + i)) << (8 * (i & 3));
    return make_uint4(w[0], w[1], w[2], w[3]);
}
// Bytes [0, count) as flat bits, chunk(i, aligned, left) giving the 16 bits of bytes [16 i, 16 i + left)
template <class Chunk>
__device__ __forceinline__ void pack_flat(uint16_t *out, int count, bool aligned, int tid, int T, Chunk chunk)
{
    const int full = aligned ? count >> 4 : 0;
#pragma unroll 4
    for (int i = tid; i < full; i += T) out[i] = uint16_t(chunk(i, true, 16));
    for (int i = full + tid; 16 * i < count; i += T) out[i] = uint16_t(chunk(i, false, min(16, count - 16 * i)));
}
// `bits` bits of the flat bit array `flat` from bit `at` (at most 32)
__device__ __forceinline__ uint32_t bits_at(const uint32_t *flat, uint32_t at, int bits)
{
    const uint32_t w = __funnelshift_r(flat[at >> 5], flat[(at >> 5) + 1], at & 31u);
    return bits < 32 ? w & ((1u << bits) - 1u) : w;
}

// 2^log_shots shots per block at a time.  The bytes of a tile's rows, which lie one after another in memory, are
// read as one flat array with 16-byte loads and packed 16 bytes to 16 bits; row words are then cut out
// of the flat bits.  A shot that was not decoded has failed whatever its residual, and the others' residuals
// are mostly 0, so the words that are not 0 are listed:
//   * few in the tile: one warp per word reads, for each of its bits, that qubit's byte of 32 operators at
//     a time; their ballot is XORed into the shot's overlap parities;
//   * many: the operators are packed into words (once per block, when first needed) and a warp tests 32 of
//     them against eight shots, an operator's word read once for the eight and one logic operation for
//     each word of a shot.
// Packing first in every block cost more than the test itself (140 operators of 1054 qubits): 65536 shots
// 490 -> 60 us at 0.1 residual bits a shot, 485 -> 92 with dense residuals; 1000 shots 272 -> 15.  Bound by the
// reads of errors and decisions (46 us with no residual bits at all, 20 at the copy bandwidth).
// `logicals` bytes count as 1 when not 0, error and decision bytes by their low bit.
__global__ void __launch_bounds__(kLogicalThreads, 5)
    logical_kernel(const uint8_t *__restrict__ logicals, int32_t K, int32_t N, const uint8_t *__restrict__ err,
                   const uint8_t *__restrict__ dec, const uint8_t *__restrict__ ok, int32_t batch, int log_shots,
                   uint8_t *__restrict__ fail)
{
    extern __shared__ __align__(16) uint32_t sm[];
    const int W = (N + 31) / 32, Ws = W | 1, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int T = kLogicalThreads, nwarp = T / 32;
    const int shots = 1 << log_shots;
    uint32_t *lw = sm;                                              // [K][Ws]: odd stride, no bank conflicts
    uint32_t *rw = sm + ((K * Ws + 3) & ~3);                        // [W][shots] residual words
    uint32_t *flat = rw + W * shots;                                // flat bits of the tile
    uint32_t *lflat = rw;                                           // flat bits of the operators (while packing)
    __shared__ uint32_t s_odd[2], s_par[64 * (kDirectOps / 32)];
    __shared__ uint16_t s_list[kDirectWords];
    __shared__ int s_count;
    const bool al = ((reinterpret_cast<uintptr_t>(err) | reinterpret_cast<uintptr_t>(dec)) & 15u) == 0;
    const int groups = (K + 31) / 32, eights = shots / 8;
    const int my = tid & (shots - 1);                               // the shot whose words this thread cuts
    const int64_t tiles = (int64_t(batch) + shots - 1) / shots;
    bool packed = false;
    for (int64_t t = blockIdx.x; t < tiles;) {
        const int64_t b0 = t * shots;
        const int ns = int(min(int64_t(shots), int64_t(batch) - b0));
        const uint8_t *e = err + size_t(b0) * N, *d = dec + size_t(b0) * N;   // shots * N is a multiple of 16
        const bool live = my < ns && ok[b0 + my] != 0;
        if (tid < 2) s_odd[tid] = 0u;
        if (tid == 0) s_count = 0;
        pack_flat(reinterpret_cast<uint16_t *>(flat), ns * N, al, tid, T, [&](int i, bool whole, int left) {
            const uint4 a = whole ? __ldg(reinterpret_cast<const uint4 *>(e) + i) : load_some(e + 16 * i, left);
            const uint4 b = whole ? __ldg(reinterpret_cast<const uint4 *>(d) + i) : load_some(d + 16 * i, left);
            return pack16((a.x ^ b.x) & 0x01010101u, (a.y ^ b.y) & 0x01010101u, (a.z ^ b.z) & 0x01010101u,
                          (a.w ^ b.w) & 0x01010101u);
        });
        __syncthreads();
        for (int i = tid; i < W * shots; i += T) {
            const int wd = i >> log_shots;
            const uint32_t w = live ? bits_at(flat, uint32_t(my) * uint32_t(N) + 32u * uint32_t(wd), N - 32 * wd) : 0u;
            rw[i] = w;
            if (w) {
                const int at = atomicAdd(&s_count, 1);
                if (at < kDirectWords) s_list[at] = uint16_t(i);
            }
        }
        __syncthreads();
        const int count = s_count;
        if (count > 0 && count <= kDirectWords && K <= kDirectOps) {
            for (int i = tid; i < shots * groups; i += T) s_par[i] = 0u;
            __syncthreads();
            for (int it = warp; it < count; it += nwarp) {
                const int i = s_list[it], s = i & (shots - 1), q0 = 32 * (i >> log_shots);
                const uint32_t word = rw[i];
                for (int g0 = 0; g0 < groups; g0 += 8) {   // the bytes of a qubit in 256 operators, loaded together
                    uint32_t odd = 0;
                    for (uint32_t w = word; w; w &= w - 1) {
                        const uint8_t *col = logicals + (q0 + __ffs(int(w)) - 1);
                        uint32_t v[8];
#pragma unroll
                        for (int u = 0; u < 8; ++u) {
                            const int l = 32 * (g0 + u) + lane;
                            v[u] = l < K ? uint32_t(__ldg(col + size_t(l) * N)) : 0u;
                        }
#pragma unroll
                        for (int u = 0; u < 8; ++u) odd ^= (v[u] != 0 ? 1u : 0u) << u;
                    }
                    for (int u = 0; u < 8 && g0 + u < groups; ++u) {
                        const uint32_t par = __ballot_sync(0xffffffffu, (odd >> u) & 1u);
                        if (lane == 0 && par) atomicXor(&s_par[s * groups + g0 + u], par);
                    }
                }
            }
            __syncthreads();
            for (int i = tid; i < shots * groups; i += T)
                if (s_par[i]) atomicOr(&s_odd[(i / groups) >> 5], 1u << ((i / groups) & 31));
            __syncthreads();
        } else if (count > 0) {
            if (!packed) {   // pack the operators over this tile's words, then take the tile again
                packed = true;
                const bool lal = (reinterpret_cast<uintptr_t>(logicals) & 15u) == 0;
                pack_flat(reinterpret_cast<uint16_t *>(lflat), K * N, lal, tid, T, [&](int i, bool whole, int left) {
                    const uint4 v = whole ? __ldg(reinterpret_cast<const uint4 *>(logicals) + i) : load_some(logicals + 16 * i, left);
                    return pack16(nonzero4(v.x), nonzero4(v.y), nonzero4(v.z), nonzero4(v.w));
                });
                __syncthreads();
                for (int i = tid; i < K * W; i += T) {
                    const int l = i / W, wd = i - l * W;
                    lw[l * Ws + wd] = bits_at(lflat, uint32_t(l) * uint32_t(N) + 32u * uint32_t(wd), N - 32 * wd);
                }
                __syncthreads();
                continue;
            }
            for (int it = warp; it < groups * eights; it += nwarp) {
                const int o = it & (eights - 1), l = (it >> (log_shots - 3)) * 32 + lane;
                const uint32_t *lrow = lw + (l < K ? l : 0) * Ws;
                uint32_t acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll 2
                for (int wd = 0; wd < W; ++wd) {
                    const uint32_t a = lrow[wd];
                    const uint4 r0 = *reinterpret_cast<const uint4 *>(rw + wd * shots + 8 * o);
                    const uint4 r1 = *reinterpret_cast<const uint4 *>(rw + wd * shots + 8 * o + 4);
                    acc[0] ^= a & r0.x;
                    acc[1] ^= a & r0.y;
                    acc[2] ^= a & r0.z;
                    acc[3] ^= a & r0.w;
                    acc[4] ^= a & r1.x;
                    acc[5] ^= a & r1.y;
                    acc[6] ^= a & r1.z;
                    acc[7] ^= a & r1.w;
                }
                uint32_t odd = 0;
#pragma unroll
                for (int i = 0; i < 8; ++i) odd |= (uint32_t(__popc(acc[i])) & 1u) << i;
                odd = __reduce_or_sync(0xffffffffu, odd);
                if (lane == 0 && odd) atomicOr(&s_odd[o >> 2], odd << (8 * (o & 3)));
            }
            __syncthreads();
        }
        if (tid < ns) fail[b0 + tid] = (!live || ((s_odd[tid >> 5] >> (tid & 31)) & 1u)) ? 1 : 0;   // (my = tid here)
        __syncthreads();   // s_odd and the tile's words are rewritten next
        t += gridDim.x;
    }
}

// One shot per block at a time, for codes too long for a tile of the kernel above.
__global__ void logical_long_kernel(const uint8_t *__restrict__ logicals, int32_t K, int32_t N,
                                    const uint8_t *__restrict__ err, const uint8_t *__restrict__ dec,
                                    const uint8_t *__restrict__ ok, int32_t batch, uint8_t *__restrict__ fail)
{
    extern __shared__ __align__(16) uint32_t lw[];
    const int W = (N + 31) / 32, T = blockDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nwarp = (T + 31) / 32;
    uint32_t *rw = lw + size_t(K) * W;
    for (int idx = warp; idx < K * W; idx += nwarp) {   // pack L row by row, 32 qubits per word
        const int l = idx / W, wd = idx - l * W, q = wd * 32 + lane;
        const uint32_t bits = __ballot_sync(0xffffffffu, q < N && logicals[size_t(l) * N + q]);
        if (lane == 0) lw[idx] = bits;
    }
    for (int b = blockIdx.x; b < batch; b += gridDim.x) {
        __syncthreads();
        for (int wd = warp; wd < W; wd += nwarp) {
            const int q = wd * 32 + lane;
            const bool r = q < N && ((err[size_t(b) * N + q] ^ dec[size_t(b) * N + q]) & 1u);
            const uint32_t bits = __ballot_sync(0xffffffffu, r);
            if (lane == 0) rw[wd] = bits;
        }
        __syncthreads();
        int odd = 0;
        for (int l = tid; l < K; l += T) {
            uint32_t par = 0;
            for (int wd = 0; wd < W; ++wd) par ^= uint32_t(__popc(lw[l * W + wd] & rw[wd]));
            odd |= int(par & 1u);
        }
        odd = __syncthreads_or(odd);
        if (tid == 0) fail[b] = (ok[b] == 0 || odd) ? 1 : 0;
    }
}

}  // namespace kern

size_t sample_smem(int32_t m, int32_t n)
{
    const int stride = std::max(kern::seg_stride(kern::seg_bytes(n)), kern::seg_stride(kern::seg_bytes(m)));
    return (size_t(kern::kSampleShots) * stride + size_t((n + 3) & ~3) + size_t((m + 3) & ~3)) * 4;
}

const void *sample_kernel_ptr() { return reinterpret_cast<const void *>(&kern::sample_kernel); }

cudaError_t launch_sample(const DeviceGraph &g, uint64_t seed, int64_t first_shot, int32_t batch, double p_lo,
                          double p_hi, uint8_t *err, uint8_t *syn, int sm_count, cudaStream_t stream)
{
    const int64_t tiles = (int64_t(batch) + kern::kSampleShots - 1) / kern::kSampleShots;
    if (2 * tiles <= sm_count)   // (a graph that fits on chip has fewer than 48 K variables)
        kern::sample_shot_kernel<<<std::min(batch, sm_count * 8), kern::kSampleThreads, size_t(g.n), stream>>>(
            g, seed, first_shot, batch, p_lo, p_hi - p_lo, err, syn);
    else   // a block a tile: the last wave fills best
        kern::sample_kernel<<<unsigned(tiles), kern::kSampleThreads, sample_smem(g.m, g.n), stream>>>(
            g, seed, first_shot, batch, p_lo, p_hi - p_lo, err, syn);
    return cudaGetLastError();
}

// Shots of a tile: as many as keep it near 33 KB of input bytes and its words small; at 8192 qubits the
// 16 shots of a tile still fit beside the operators.
LogicalPlan plan_logical(int32_t k, int32_t n)
{
    const size_t W = size_t((n + 31) / 32), Ws = W | 1;
    if (n > 8192) return LogicalPlan{0, (size_t(k) + 1) * W * 4, reinterpret_cast<const void *>(&kern::logical_long_kernel)};
    const int shots = n <= 512 ? 64 : n <= 2048 ? 32 : 16;
    const size_t tile = W * size_t(shots) + (size_t(shots) * size_t(n) + 31) / 32 + 2;   // words | flat bits (and one word read past them)
    const size_t lflat = (size_t(k) * size_t(n) + 31) / 32 + 2;
    const size_t words = ((size_t(k) * Ws + 3) & ~size_t(3)) + std::max(tile, lflat);
    return LogicalPlan{shots, words * 4, reinterpret_cast<const void *>(&kern::logical_kernel)};
}

cudaError_t launch_logical(const LogicalPlan &pl, const uint8_t *logicals, int32_t k, int32_t n, const uint8_t *err,
                           const uint8_t *dec, const uint8_t *ok, int32_t batch, uint8_t *fail, int sm_count,
                           cudaStream_t stream)
{
    if (pl.shots == 0) {
        const int grid = int(std::min<int64_t>(batch, int64_t(sm_count) * 8));
        kern::logical_long_kernel<<<grid, 128, pl.smem, stream>>>(logicals, k, n, err, dec, ok, batch, fail);
        return cudaGetLastError();
    }
    const int64_t tiles = (int64_t(batch) + pl.shots - 1) / pl.shots, most = int64_t(sm_count) * 5;
    const int64_t rounds = (tiles + most - 1) / most;
    const int grid = int((tiles + rounds - 1) / rounds);
    const int log_shots = pl.shots == 64 ? 6 : pl.shots == 32 ? 5 : 4;
    kern::logical_kernel<<<grid, kern::kLogicalThreads, pl.smem, stream>>>(logicals, k, n, err, dec, ok, batch, log_shots,
                                                                           fail);
    return cudaGetLastError();
}

}  // namespace qldpc
