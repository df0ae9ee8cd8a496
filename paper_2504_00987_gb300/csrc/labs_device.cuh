// labs_device.cuh -- device primitives of the LABS solver (sm_103a).
//
// Sequences live in registers as NW 32-bit words, at least ceil(N/32) (which
// counts a kernel has stands at its dispatch), bit i of the vector (word i / 32,
// bit i % 32) holding spin s_{i+1} (1 <-> +1).  A warp owns one sequence; every
// lane keeps an identical copy of the words ("warp-uniform") and lane l owns the
// indices l + 32q, q = 0 .. NW-1, of the per-index arrays (key, tabu expiry and
// spin of neighbour j).
#pragma once

#include <cstdint>

#include "labs.h"

namespace lgpu {

constexpr uint32_t kFull = 0xFFFFFFFFu;

// Philox counter word 3 (purpose) of the RNG contract in labs.h.
constexpr uint32_t kPurposeInit = 1u;
constexpr uint32_t kPurposeGen = 2u;
constexpr uint32_t kPurposeMut = 3u;
constexpr uint32_t kPurposeStep = 4u;
constexpr uint32_t kPurposeCross = 5u;

// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): ten rounds of two
// 32x32->64 multiplications by fixed odd constants with a Weyl-sequence key
// schedule; round r uses key + r * (golden-ratio, sqrt(3)-1) constants.
__device__ __forceinline__ uint4 philox4x32_10(uint4 x, uint2 k) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r > 0) {
            k.x += 0x9E3779B9u;
            k.y += 0xBB67AE85u;
        }
        const uint32_t lo0 = 0xD2511F53u * x.x;
        const uint32_t hi0 = __umulhi(0xD2511F53u, x.x);
        const uint32_t lo1 = 0xCD9E8D57u * x.z;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, x.z);
        x = make_uint4(hi1 ^ x.y ^ k.x, lo1, hi0 ^ x.w ^ k.y, lo0);
    }
    return x;
}

__device__ __forceinline__ uint2 philox_key(uint64_t seed) {
    return make_uint2(static_cast<uint32_t>(seed), static_cast<uint32_t>(seed >> 32));
}

__device__ __forceinline__ uint4 draw4(uint2 key, uint32_t instance, uint32_t a, uint32_t b,
                                       uint32_t purpose) {
    return philox4x32_10(make_uint4(instance, a, b, purpose), key);
}

// randInt(lo, hi) inclusive: lo + floor(u * (hi - lo + 1) / 2^32).
__device__ __forceinline__ int32_t rand_int(int32_t lo, int32_t hi, uint32_t u) {
    const uint64_t span = static_cast<uint64_t>(static_cast<int64_t>(hi) - lo + 1);
    return lo + static_cast<int32_t>((static_cast<uint64_t>(u) * span) >> 32);
}

// A value every lane of the warp holds already, in a form the compiler knows to
// be the same in every lane (the result of a warp reduction): branches on it
// need no reconvergence.  A service warp whose request index and fields came
// through loads took 382 cycles a step at N = 64, 230 with this; the step has
// the same instructions but for its branches.  The batch kernel, whose requests
// come through a shuffle, took 3 % more time with it and does without.
__device__ __forceinline__ int32_t warp_uniform(int32_t x) { return __reduce_min_sync(kFull, x); }

// Bits [0, n) of 32-bit word v (n may lie outside the word).
__device__ __forceinline__ uint32_t word_lowmask(int v, int n) {
    const int hi = n - 32 * v;
    return hi >= 32 ? kFull : (hi <= 0 ? 0u : ((1u << hi) - 1u));
}

// out = in >> s for an NW-word vector and a warp-uniform runtime shift
// 0 <= s < 32*NW: word moves by a log-depth select network, then one funnel
// shift per word.  No dynamic register indexing.
template <int NW>
__device__ __forceinline__ void shr_uniform(const uint32_t (&in)[NW], int s, uint32_t (&out)[NW]) {
    uint32_t a[NW];
#pragma unroll
    for (int w = 0; w < NW; ++w) a[w] = in[w];
    const int ws = s >> 5;
#pragma unroll
    for (int step = 1; step < NW; step <<= 1) {
        const bool take = (ws & step) != 0;
#pragma unroll
        for (int w = 0; w < NW; ++w) a[w] = take ? (w + step < NW ? a[w + step] : 0u) : a[w];
    }
    const int bs = s & 31;
#pragma unroll
    for (int w = 0; w < NW; ++w) out[w] = __funnelshift_r(a[w], w + 1 < NW ? a[w + 1] : 0u, bs);
}

// Full-width reversal: bit (32*NW - 1 - i) of out = bit i of in.
template <int NW>
__device__ __forceinline__ void reverse_bits(const uint32_t (&in)[NW], uint32_t (&out)[NW]) {
#pragma unroll
    for (int w = 0; w < NW; ++w) out[w] = __brev(in[NW - 1 - w]);
}

// Skew-symmetric completion of an odd-length sequence (Sec. II.C): with
// centre c = (N-1)/2, s_{c+i} = (-1)^i s_{c-i} for i = 1..c, i.e.
// b_{c+i} = b_{c-i} xor (i odd).  Bits [0, c] are kept, bits >= N cleared.
template <int NW>
__device__ __forceinline__ void skew_complete(uint32_t (&B)[NW], int N) {
    constexpr int NB = 32 * NW;
    const int c = (N - 1) >> 1;
    uint32_t RL[NW], RN[NW];
    reverse_bits<NW>(B, RL);
    shr_uniform<NW>(RL, NB - N, RN);                            // bit m of RN = b_{N-1-m}
    const uint32_t alt = (c & 1) ? 0x55555555u : 0xAAAAAAAAu;  // bit m set iff m - c odd
#pragma unroll
    for (int w = 0; w < NW; ++w) {
        const uint32_t keep = word_lowmask(w, c + 1);
        B[w] = (B[w] & keep) | ((RN[w] ^ alt) & word_lowmask(w, N) & ~keep);
    }
}

}  // namespace lgpu
