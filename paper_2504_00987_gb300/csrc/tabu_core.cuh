// tabu_core.cuh -- one warp runs one tabu search (Algorithm 2 / Algorithm 4).
//
// Neighbour scoring (Sec. III.C, Table I).  Flipping s_j changes C_k by
// delta_k(j) = -2 s_j (s_{j+k} + s_{j-k}) (terms outside 1..N dropped), so
//   E_j = E + sum_k delta_k (2 C_k + delta_k)
//       = E + 4(N-1) + 8 M_j - 4 s_j R_j,
// with M_j = sum_{k>=1} s_{j+k} s_{j-k} and R_j = sum_k C_k (s_{j+k} + s_{j-k}),
// which search_setup computes once per search.  After every move each
// neighbour's energy change is updated exactly in O(1) from C_k and the
// self-convolution V_m of the spins (the identity stands above tabu_search),
// so a step never goes back to the bits.  Arithmetic is exact int32.
//
// Work split: lane l owns the neighbours j = l + 32q: their keys (energy
// change, index and spin in one int), tabu expiry and spins in registers; V,
// C and the spins also in the warp's slice of shared memory, where the move
// shifts them against each other.  The admissible minimum is one
// redux.sync.min over the keys; ballots resolve a tie only where there is one.
#pragma once

#include <climits>
#include <type_traits>

#include "kernels.h"
#include "labs_device.cuh"

namespace lgpu {

// f(integral_constant<int, 0>) .. f(integral_constant<int, n - 1>).
template <int n, int i = 0, class F>
__device__ __forceinline__ void for_each_index(F&& f) {
    if constexpr (i < n) {
        f(std::integral_constant<int, i>{});
        for_each_index<n, i + 1>(f);
    }
}

// sum_i popc(w[i]) * weight with as few popcounts as full adders (two LOP3
// each) leave: a popcount takes the XU pipe 8 cycles a warp, a logic
// instruction the ALU pipe 2, so an adder that saves a popcount is worth it
// where popcounts fill their pipe.
template <int n, int weight = 1>
__device__ __forceinline__ int popc_words(const uint32_t (&w)[n]) {
    if constexpr (n <= 2) {
        int s = 0;
#pragma unroll
        for (int i = 0; i < n; ++i) s += __popc(w[i]);
        return s * weight;
    } else {
        constexpr int f = (n - 1) / 2;
        uint32_t carry[f];
        uint32_t acc = w[0];
#pragma unroll
        for (int i = 0; i < f; ++i) {
            const uint32_t a = acc, b = w[1 + 2 * i], c = w[2 + 2 * i];
            acc = a ^ b ^ c;
            carry[i] = (a & b) | (c & (a | b));
        }
        int s = __popc(acc);
        if constexpr (n - 2 * f == 2) s += __popc(w[n - 1]);
        return s * weight + popc_words<f, 2 * weight>(carry);
    }
}

// Pairs (i, i + l + 32q) of B with unequal bits: `mask[x]` holds the bits of
// word x below N - l, so the pairs end where i + l + 32q does.  The masks are
// those of the last words only, whatever q.
template <int NW, int q>
__device__ __forceinline__ int unequal_pairs(const uint32_t (&B)[NW], const uint32_t (&mask)[NW], int l) {
    uint32_t x[NW - q];
#pragma unroll
    for (int w = 0; w + q < NW; ++w)
        x[w] = (B[w] ^ __funnelshift_r(B[w + q], w + q + 1 < NW ? B[w + q + 1] : 0u, l)) & mask[w + q];
    return popc_words<NW - q>(x);
}

// mask[x] = bits of word x below N - l.  TIGHT: N > 32 (NW - 1), and only the
// last two words can end inside.
template <int NW, bool TIGHT>
__device__ __forceinline__ void pair_masks(int N, int l, uint32_t (&mask)[NW]) {
#pragma unroll
    for (int x = 0; x < NW; ++x) mask[x] = TIGHT && x + 2 < NW ? kFull : word_lowmask(x, N - l);
}

// C_k of the lane's k = lane + 32q (C_0 = N, C_{k >= N} = 0); `mask` as for l = lane.
template <int NW, int q = 0>
__device__ __forceinline__ void lane_correlations(const uint32_t (&s)[NW], const uint32_t (&mask)[NW], int N, int lane,
                                                  int32_t (&c)[NW]) {
    if constexpr (q < NW) {
        c[q] = max(N - lane - 32 * q, 0) - 2 * unequal_pairs<NW, q>(s, mask, lane);
        lane_correlations<NW, q + 1>(s, mask, N, lane, c);
    }
}

template <int NW, bool TIGHT, int q = 0>
__device__ __forceinline__ int32_t sum_squares(const uint32_t (&B)[NW], const uint32_t (&mask)[NW], int N, int l) {
    if constexpr (q == NW) {
        return 0;
    } else {
        const int32_t pairs = N - l - 32 * q;  // below 1 only past the last C_k
        const int32_t Ck = (q + 1 < NW && TIGHT ? pairs : max(pairs, 0)) - 2 * unequal_pairs<NW, q>(B, mask, l);
        return Ck * Ck + sum_squares<NW, TIGHT, q + 1>(B, mask, N, l);
    }
}

// Energy of one sequence computed by a single thread (bits in `B`).
template <int NW, bool TIGHT = false>
__device__ __forceinline__ int32_t thread_energy(const uint32_t (&B)[NW], int N) {
    int32_t E = -N * N;  // k = 0 is summed below
    if constexpr (TIGHT && NW >= 2) {
        // the masks of the last two words as one 64-bit mask, a bit shorter each round
        uint32_t mask[NW];
        pair_masks<NW, true>(N, 0, mask);
        uint64_t last = (static_cast<uint64_t>(mask[NW - 1]) << 32) | mask[NW - 2];
#pragma unroll 2
        for (int l = 0; l < 32; ++l) {
            mask[NW - 2] = static_cast<uint32_t>(last);
            mask[NW - 1] = static_cast<uint32_t>(last >> 32);
            E += sum_squares<NW, true>(B, mask, N, l);
            last >>= 1;
        }
    } else {
        for (int l = 0; l < 32; ++l) {
            uint32_t mask[NW];
            pair_masks<NW, TIGHT>(N, l, mask);
            E += sum_squares<NW, TIGHT>(B, mask, N, l);
        }
    }
    return E;
}

struct TabuOut {
    int64_t steps = 0;
    int32_t E_best = 0;
    bool fault = false;  // the two warps of a replica lost step (a bounded wait ran out)
};

// Two warps of one CTA sharing one replica ("warps per sequence" = 2): each
// runs the whole replica on its own copy of the state and scores half of
// the neighbours; per step they exchange their admissible minima through
// this shared-memory word pair.  Exchange x of a pair uses slot [x & 1] (so
// a warp that runs ahead never overwrites a word its partner has not read:
// it cannot publish x + 2 before the partner published x + 1, which comes
// after the partner read x); a word holds (x mod 2^24) << 40 | value.
struct PairLink {
    unsigned long long slot[2][2];  // [x & 1][half]
};

constexpr uint32_t kPairSpinLimit = 1u << 22;  // ~10^8 cycles, far beyond one step's skew

// Publishes this warp's value v (< 2^40) of exchange x and returns the
// partner's in `other`.  Lane 0 spins on the partner's word with a bounded
// number of polls; false if they run out (the caller stops the replica).
__device__ __forceinline__ bool pair_exchange(PairLink* link, int half, uint32_t x, uint64_t v,
                                              uint64_t& other, int lane) {
    const uint64_t tag = static_cast<uint64_t>(x & 0xFFFFFFu) << 40;
    bool ok = true;
    uint64_t w = 0;
    if (lane == 0) {
        volatile unsigned long long* mine = &link->slot[x & 1u][half];
        volatile unsigned long long* theirs = &link->slot[x & 1u][half ^ 1];
        *mine = tag | v;
        for (uint32_t it = 0;; ++it) {
            w = *theirs;
            if ((w >> 40) == (x & 0xFFFFFFu)) break;
            if (it >= kPairSpinLimit) {
                ok = false;
                break;
            }
        }
    }
    ok = __shfl_sync(kFull, ok ? 1 : 0, 0) != 0;
    other = __shfl_sync(kFull, static_cast<unsigned long long>(w), 0) & ((1ull << 40) - 1);
    return ok;
}

// Scratch of one warp's tabu search (ints): what the launches leave room for
// (tabu_scratch_bytes).
template <int NW>
constexpr int kTabuScratchInts = static_cast<int>(tabu_scratch_bytes(NW) / sizeof(int32_t));

// V_m = sum_a x_a x_{m-a} for m = lane + 32i <= N - 1, stored at V[m] (or at
// V[2N - 2 - m], MIRROR, where X is the sequence reversed): bits X and their
// full-width reversal XL.  a runs over 0..m, so only the last word is cut.
template <int NW, bool MIRROR>
__device__ __forceinline__ void store_self_convolution(const uint32_t (&X)[NW], const uint32_t (&XL)[NW], int N,
                                                       int lane, int32_t* __restrict__ V) {
    uint32_t Y[NW];  // word w + NW - 1 - i: bit a of word w is x_{m-a}
#pragma unroll
    for (int x = 0; x < NW; ++x) Y[x] = __funnelshift_r(XL[x], x + 1 < NW ? XL[x + 1] : 0u, 31 - lane);
    const uint32_t low_l = 0xFFFFFFFFu >> (31 - lane);  // bits 0..lane
    auto one = [&](auto I) {
        constexpr int i = decltype(I)::value;
        uint32_t diff[i + 1];
#pragma unroll
        for (int w = 0; w <= i; ++w) diff[w] = (X[w] ^ Y[w + NW - 1 - i]) & (w == i ? low_l : kFull);
        const int m = lane + 32 * i;
        if (m <= N - 1) V[MIRROR ? 2 * N - 2 - m : m] = m + 1 - 2 * popc_words<i + 1>(diff);
    };
    for_each_index<NW>(one);
}

// Tie and tenure draws (x, y) of tabu step t.
__device__ __forceinline__ uint2 step_draws(uint2 key, uint32_t inst, uint32_t g, int t) {
    const uint4 r = draw4(key, inst, g, static_cast<uint32_t>(t), kPurposeStep);
    return make_uint2(r.x, r.y);
}

// The scratch's parts: V_m, m = 0 .. 2 NB - 1; C_d at C[d] and C[-d]; -2 s~_i
// at S[i], i = -NB .. 2 NB - 1.
template <int NW>
struct TabuScratch {
    static_assert(4 * (2 * 32 * NW) + 4 * (2 * 32 * NW) + 3 * 32 * NW == tabu_scratch_bytes(NW) &&
                      tabu_scratch_bytes(NW) % 16 == 0,
                  "V, C and the spins take the scratch");
    int32_t* V;
    int32_t* C;
    int8_t* S;
    __device__ __forceinline__ explicit TabuScratch(int32_t* base)
        : V(base), C(base + 3 * 32 * NW), S(reinterpret_cast<int8_t*>(base + 4 * 32 * NW) + 32 * NW) {}
};

// Fills the scratch for a search from `seq` and returns its energy; s[q] is
// the spin (0 for j >= N) and d4[q] the energy change D_j / 4 of the lane's
// j = lane + 32q (unset for j >= N).
//
// R_j = sum_i s_i C_{|i-j|} are NB^2 products of small integers: four to an
// instruction as bytes (__dp4a).  The bytes of C, at both signs of the index,
// stand in V's place until V is made; a lane reads the aligned words around
// its own offset -lane once, shifts each pair into place once, and uses the
// result for all its j = lane + 32q, whose windows lie 8 words apart.  C_k
// fits a byte for N <= 128 and in nearly every longer sequence; where it does
// not, the high bits (C_k >> 1) and the low bit go one after the other.
template <int NW>
__device__ __forceinline__ int32_t search_setup(const uint32_t (&seq)[NW], int N, int lane,
                                                int32_t* __restrict__ Cs, int32_t (&s)[NW], int32_t (&d4)[NW]) {
    constexpr int NB = 32 * NW;
    const TabuScratch<NW> sh(Cs);
    int32_t c[NW];
    {
        uint32_t mask[NW];
        pair_masks<NW, false>(N, lane, mask);
        lane_correlations<NW>(seq, mask, N, lane, c);
    }
    if (lane == 0) c[0] = 0;
    int32_t sq = 0;
    bool large = false;
#pragma unroll
    for (int q = 0; q < NW; ++q) {
        const int j = lane + 32 * q;
        sq += c[q] * c[q];
        large = large || abs(c[q]) > 127;
        s[q] = j < N ? 2 * static_cast<int32_t>((seq[q] >> lane) & 1u) - 1 : 0;
        sh.C[j] = c[q];
        sh.C[-j] = c[q];
        sh.S[j] = static_cast<int8_t>(-2 * s[q]);
        sh.S[j - NB] = 0;
        sh.S[j + NB] = 0;
    }
    const int32_t E = __reduce_add_sync(kFull, sq);
    const bool split = NW > 4 && __any_sync(kFull, large);
    int32_t acc[NW];  // -2 R_j
#pragma unroll
    for (int q = 0; q < NW; ++q) acc[q] = 0;
    int8_t* const G = reinterpret_cast<int8_t*>(sh.V) + NB;  // C_{|x|} as a byte at G[x], -NB < x < NB
    const int32_t* const Gw = reinterpret_cast<const int32_t*>(G) + ((-lane) >> 2);
    const int32_t* const Sw = reinterpret_cast<const int32_t*>(sh.S);
    const int bits = 8 * (-lane & 3);
#pragma unroll 1
    for (int part = split ? 1 : 0; part >= 0; --part) {
#pragma unroll
        for (int q = 0; q < NW; ++q) {
            const int j = lane + 32 * q;
            const int8_t byte = static_cast<int8_t>(!split ? c[q] : part ? c[q] >> 1 : c[q] & 1);
            G[j] = byte;
            G[-j] = byte;
            acc[q] *= 2;
        }
        __syncwarp();
        int32_t sw[8 * NW];
#pragma unroll
        for (int n = 0; n < 8 * NW; ++n) sw[n] = Sw[n];
        uint32_t lo = Gw[-8 * (NW - 1)];
#pragma unroll
        for (int x = -8 * (NW - 1); x < 8 * NW; ++x) {
            const uint32_t hi = Gw[x + 1];
            const int32_t u = static_cast<int32_t>(__funnelshift_r(lo, hi, bits));  // C_{|i-j|}, i = 4 (x + 8q) ..
            lo = hi;
#pragma unroll
            for (int q = 0; q < NW; ++q)
                if (x + 8 * q >= 0 && x + 8 * q < 8 * NW) acc[q] = __dp4a(sw[x + 8 * q], u, acc[q]);
        }
        __syncwarp();
    }
    {
        uint32_t RL[NW], RN[NW], BL[NW];
        reverse_bits<NW>(seq, RL);
        store_self_convolution<NW, false>(seq, RL, N, lane, sh.V);
        shr_uniform<NW>(RL, NB - N, RN);  // bit x = b_{N-1-x}
        reverse_bits<NW>(RN, BL);
        store_self_convolution<NW, true>(RN, BL, N, lane, sh.V);
    }
    __syncwarp();
    // D_j / 4 = N - 1 + 2 M_j - s_j R_j, 2 M_j = V_{2j} - 1
#pragma unroll
    for (int q = 0; q < NW; ++q) d4[q] = N - 2 + sh.V[2 * (lane + 32 * q)] + s[q] * (acc[q] >> 1);
    __syncwarp();
    return E;
}

// One tabu search from `seq` (warp-uniform).  On return `seq` holds
// bestSeqTS.  Draws: step t uses Philox(instance, g, t, 4): x tie, y tenure;
// `draws` are the lane's of step 1 + lane (step_draws).
// FIX_FIRST: bit 0 (s_1) is never a candidate move.
// `Cs` is warp-private shared scratch of kTabuScratchInts<NW> ints.
// With TRACE, `trace` receives {g, t, j, E} per step while trace_len <
// trace_cap.
//
// Every neighbour's energy change D_j = E_j - E is kept between steps, and a
// step costs O(N) for the whole neighbourhood.  With s~_i = s_i inside
// 0..N-1 (0 outside), C_k = sum_i s~_i s~_{i+k} and V_m = sum_a s~_a s~_{m-a},
// the move p (s_p before it, sigma = s_p s_j) changes
//   D'_j = D_j + 8 sigma (2 C_{|j-p|} + V_{p+j}) - 16 (s_p s~_{2j-p} + s_j s~_{2p-j}) - 32
//   V'_{p+j} = V_{p+j} - 4 sigma,   C'_{|j-p|} = C_{|j-p|} - 2 sigma - 2 s_p s~_{2p-j}   (j != p)
//   D'_p = -D_p,                    V'_{2p} = V_{2p}
// (C and V on the right before the move; no other V_m or C_k changes).
// Derivation: D_j = 4(N-1) + 8 M_j - 4 s_j R_j with M_j = sum_{k>=1}
// s~_{j+k} s~_{j-k} and R_j = sum_k C_k (s~_{j+k} + s~_{j-k}).  M_j has one
// product with s_p, at the mirror position 2j - p.  R'_j - R_j is -2 s_p C_d
// (d = |j-p|, the two terms j +- k = p) plus sum_k delta_k(p) (s~'_{j+k} +
// s~'_{j-k}) with delta_k(p) = -2 s_p (s~_{p+k} + s~_{p-k}), s~' after the
// move: its pairs (p+-k, j+-k) of one direction make C'_d without the
// product s'_p s'_j, and its crossed pairs (p+k, j-k) all have the index sum
// p + j, so they make V_{p+j} but for the products of s_p and s_j.
// With c' = C'_{|j-p|} the same change reads, in units of 4,
//   D'_j / 4 = D_j / 4 + 2 s_p (s_j (C_{|j-p|} + c' + V_{p+j}) - 2 s~_{2j-p}) - 4,
// six multiply-adds a neighbour with the updates of C and V.
//
// Lane l owns j = l + 32q: key K_j, tabu expiry and s_j in registers.  Keys
// are D_j / 4 << 9 | j << 1 | (s_j == +1): D_j is a multiple of 4 below 2^23
// in magnitude for N <= 256, one redux.sync.min gives the least change, its
// lowest index and that spin.  In shared memory: V; C at both +d and -d, so
// that C_{|j-p|} of consecutive lanes is consecutive words and needs no
// absolute value; -2 s~ as bytes with NB zeros on either side.  Lanes with
// j >= N hold s_j = 0 and a key that never changes.
//
// What bounds it: one warp's steps are a serial chain (test the keys, reduce,
// load what the move shifts, update, next test).  On GB300 redux.sync.min
// takes 18 cycles, a shared load 29, a multiply-add 5, a compare whose
// predicate is used at once 14, a vote with a branch on it 37.  So the keys
// are tested through selects and a minimum tree (predicated minima made a
// chain that cost 70 cycles more at N = 64 and 250 at N = 120), and the move
// of the lowest minimiser is scored before the vote on ties is looked at and
// scored again in the rarer case that another one is drawn (36 cycles less at
// N = 64, 72 at N = 120).  A ballot and a popcount per 32 neighbours in place
// of that one vote took 14 cycles more at N = 64 and 37 at N = 120; keeping
// the best sequence without a branch, 21 and 1 more.
// Measured, cycles a step, one warp / two / four on an SM sub-partition:
// N = 24 174 / 225 / 379, N = 64 191 / 276 / 497, N = 120 331 / 442 / 752,
// N = 160 366 / 503 / 868; about 23 instructions per 32 neighbours and 60
// besides, so four warps issue in 80 % of the cycles (two
// popcounts of windows per neighbour and word, before: one launch of 1,024
// replicas x 10^5 steps at N = 64 took 559 cycles a step).
//
// WPS = 2 (two warps per replica, HALF = which one): the warp keeps the keys
// of its half of q and its own copy of V, C and the spins; the two minima
// meet through `link`; the lower half's neighbours come first in ascending j
// for the tie pick.  Both warps take every decision from the same values, so
// they run the same steps; `xseq` counts the pair's exchanges.  A bounded
// wait that runs out ends the search with fault set.
template <int NW, bool TRACE, bool FIX_FIRST = false, int WPS = 1, int HALF = 0>
__device__ TabuOut tabu_search(uint32_t (&seq)[NW], const int N, const uint2 key,
                               const uint32_t inst, const uint32_t g, const int max_iter,
                               const int64_t budget, uint2 draws, int32_t* __restrict__ Cs,
                               int4* __restrict__ trace, const int64_t trace_cap,
                               int64_t& trace_len, const int lane, PairLink* link = nullptr,
                               uint32_t* xseq = nullptr) {
    static_assert(WPS == 1 || (WPS == 2 && NW % 2 == 0 && HALF >= 0 && HALF < 2), "warps per sequence");
    constexpr int QB = HALF * (NW / WPS), QE = (HALF + 1) * (NW / WPS);  // this warp's q
    // A drawn tie is scored by a second copy of the scoring code at three and
    // four words, and through the loop of the first at the others, where the copy
    // costs registers (cycles a step, with / without the copy, one warp alone on
    // a sub-partition and four: N = 64 231 / 190 and 525 / 497, N = 92 297 / 273
    // and 650 / 608, N = 120 331 / 311 and 751 / 756, N = 160 367 / 366 and 868 /
    // 867, N = 256 503 / 487 and 1,369 / 1,356).  The line was drawn when the copy
    // was ahead at N = 120 (343 / 355); as the step is now it only pays there with
    // four warps on a sub-partition, and at three words not at all.
    constexpr bool kRecompute = NW <= 4 && NW > 2;
    constexpr int32_t kLow = 511;  // key bits below the energy change
    constexpr int32_t kNone = INT_MAX & ~kLow;  // no candidate: above every key, low bits those of j = 0
    const TabuScratch<NW> sh(Cs);
    int32_t* const Vs = sh.V;
    int32_t* const C0 = sh.C;
    int8_t* const S0 = sh.S;
    int32_t s[NW], K[NW], tabu[NW];
    int32_t E_best = search_setup<NW>(seq, N, lane, Cs, s, K);
#pragma unroll
    for (int q = QB; q < QE; ++q) {
        const int j = lane + 32 * q;
        K[q] = j < N ? K[q] * (kLow + 1) + 2 * j + (s[q] > 0 ? 1 : 0) : kNone;
        tabu[q] = 0;
    }
    uint32_t Bb[NW];
#pragma unroll
    for (int w = 0; w < NW; ++w) Bb[w] = seq[w];
    const int min_t = max_iter / 10;
    const int max_t = (12 * max_iter) / 100;
    int nsteps = static_cast<int>(budget < 0 ? max_iter : (budget < max_iter ? budget : max_iter));
    // Up to two words the loop's bounds as a uniform value take a tenth off a lone
    // warp's step (N = 64 211 -> 191 cycles); at four words the same hint cost
    // 2.5 % with four warps on a sub-partition.
    if constexpr (NW <= 2) nsteps = warp_uniform(nsteps);
    // Every D_j / 4 loses 4 per move besides the terms below; the keys leave
    // that out, so a stored key is the true one + off, off = 4 << 9 per move
    // since the last multiple of 32.  thr (stored likewise): a key below it is
    // a move to below E_best, (E_best - E) / 4 << 9.
    constexpr int32_t kDrift = 4 * (kLow + 1);
    int32_t off = 0, thr = 0;
    int t = 0;  // moves made; this step is t + 1
    bool fault = false, stuck = false;
    const int32_t* const Vl = Vs + lane;
    const int32_t* const Cl = C0 + lane;
    const int8_t* const Al = S0 + 2 * lane;
    const int8_t* const Bl = S0 - lane;
    const uint32_t low_lanes = (1u << lane) - 1u;

    while (t < nsteps && !fault && !stuck) {
        // draws of steps t+1 .. t+32, one per lane: tie pick, and expiry of the move's tabu
        if (t > 0) draws = step_draws(key, inst, g, t + 1 + lane);
        const uint32_t u_tie_l = draws.x;
        const int32_t expiry_l = t + 1 + lane + rand_int(min_t, max_t, draws.y);
#pragma unroll
        for (int q = QB; q < QE; ++q)
            if (K[q] != kNone) K[q] -= off;
        thr -= off;
        off = 0;
        const int tend = min(t + 32, nsteps);
#pragma unroll 1
        for (; t < tend; ++t) {
            // ---- admissible minimum
            int32_t cand[NW];
            int32_t kmin_l = kNone;
#pragma unroll
            for (int q = QB; q < QE; ++q) {
                bool adm = tabu[q] <= t || K[q] < thr;
                if (FIX_FIRST && q == 0) adm = adm && lane != 0;
                cand[q] = adm ? K[q] : kNone;
                kmin_l = min(kmin_l, cand[q]);
            }
            const int32_t kmin_w = __reduce_min_sync(kFull, kmin_l);
            int32_t kmin = kmin_w;
            bool tie = false;  // another admissible move is as good
            int count_w = 0, count = 0, count_lo = 0;  // count_lo: minimisers of the lower half (WPS = 2)
            if constexpr (WPS == 1) {
                // least distance above the minimum itself; the same energy within kLow
                uint32_t above = 0xFFFFFFFFu;
#pragma unroll
                for (int q = 0; q < NW; ++q)
                    above = min(above, static_cast<uint32_t>(cand[q]) - static_cast<uint32_t>(kmin_w) - 1u);
                tie = __any_sync(kFull, above < static_cast<uint32_t>(kLow - (kmin_w & kLow))) || kmin_w == kNone;
            } else {
#pragma unroll
                for (int q = QB; q < QE; ++q) count_w += __popc(__ballot_sync(kFull, cand[q] <= (kmin_w | kLow)));
                // a key is above -2^30: shifted, it fits 31 bits beside the count
                const uint32_t kx = kmin_w == kNone ? 0x7FFFFFFFu : static_cast<uint32_t>(kmin_w + (1 << 30));
                uint64_t o = 0;
                if (!pair_exchange(link, HALF, (*xseq)++, (static_cast<uint64_t>(count_w) << 31) | kx, o, lane)) {
                    fault = true;
                    break;
                }
                const uint32_t ko = static_cast<uint32_t>(o & 0x7FFFFFFFu);
                const int32_t kmin_o = ko == 0x7FFFFFFFu ? kNone : static_cast<int32_t>(ko) - (1 << 30);
                const int count_o = static_cast<int>(o >> 31);
                kmin = min(kmin_w, kmin_o);
                // minimisers of either half: the same energy, whatever their index
                const int cw = kmin_w <= (kmin | kLow) ? count_w : 0;
                const int co = kmin_o <= (kmin | kLow) ? count_o : 0;
                count = cw + co;
                count_lo = HALF == 0 ? cw : co;
                tie = count > 1;
            }
            int klow = kmin & kLow;  // 2p + (s_p == +1), p the lowest admissible minimiser
            // ---- the move's V, C and mirror spins (times -2), and what they
            // make of the keys, V and C, for the lowest minimiser: done before
            // the ties are looked at, and again if one of the others is taken
            int32_t kn[NW], vn[NW], cn[NW];
            auto score_move = [&](const int klow) {
                const int p = klow >> 1;
                const int32_t sp = 2 * (klow & 1) - 1;
#pragma unroll
                for (int q = 0; q < NW; ++q) {
                    const int32_t v = Vl[p + 32 * q];
                    const int32_t cd = Cl[32 * q - p];
                    const int32_t sb = Bl[2 * p - 32 * q];
                    cn[q] = cd + sp * (sb - 2 * s[q]);
                    vn[q] = v - 4 * sp * s[q];
                    if (q >= QB && q < QE)
                        kn[q] = K[q] + (2 * (kLow + 1) * sp) * (s[q] * (cd + cn[q] + v) + Al[64 * q - p]);
                }
            };
            const int32_t expiry = __shfl_sync(kFull, expiry_l, t);
            bool again;
            do {
                again = false;
                score_move(klow);
                if (tie) {
                    tie = false;
                    // Every move tabu and none aspirating: the search has no admissible
                    // move and stops.  The default maxIter keeps maxTabu below N, so only a
                    // user maxIter of about 8N or more (maxTabu >= N) gets here.
                    if (kmin == kNone) {
                        stuck = true;
                        break;
                    }
                    int rank[NW];  // minimisers of this warp before the lane's own, in ascending j
                    int below = 0;
#pragma unroll
                    for (int q = QB; q < QE; ++q) {
                        const uint32_t tb = __ballot_sync(kFull, cand[q] <= (kmin | kLow));
                        rank[q] = below + __popc(tb & low_lanes);
                        below += __popc(tb);
                    }
                    if constexpr (WPS == 1) count = below;
                    const uint32_t u_tie = __shfl_sync(kFull, u_tie_l, t);
                    int idx = static_cast<int>((static_cast<uint64_t>(u_tie) * count) >> 32);
                    if (idx > 0) {  // the idx-th minimiser in ascending j
                        bool mine = true;  // WPS = 2: the warp holding it finds it, then tells the other
                        if constexpr (WPS == 2) {
                            mine = HALF == 0 ? idx < count_lo : idx >= count_lo;
                            if (HALF == 1) idx -= count_lo;
                        }
                        if (mine) {  // its key tells its index and spin
                            int32_t pick = kNone;
#pragma unroll
                            for (int q = QB; q < QE; ++q)
                                if (cand[q] <= (kmin | kLow) && rank[q] == idx) pick = cand[q];
                            klow = __reduce_min_sync(kFull, pick) & kLow;
                        }
                        if constexpr (WPS == 2) {
                            uint64_t o = 0;
                            if (!pair_exchange(link, HALF, (*xseq)++, mine ? static_cast<uint64_t>(klow) : 0u, o, lane)) {
                                fault = true;
                                break;
                            }
                            if (!mine) klow = static_cast<int>(o);
                        }
                        if constexpr (kRecompute)
                            score_move(klow);
                        else
                            again = true;
                    }
                }
            } while (again);
            if (stuck || fault) break;
            __syncwarp();  // every lane has read what the stores below change
            // ---- apply the move
            const int p = klow >> 1;
            const int32_t sp = 2 * (klow & 1) - 1;
            const int32_t dk = kmin & ~kLow;
            off += kDrift;
            {
                int32_t* const vp = Vs + lane + p;
                int32_t* const cp = C0 + lane - p;
                int32_t* const cm = C0 - lane + p;
                // D'_p = -D_p and s'_p = -s_p: (off - kDrift - dk) + off, the spin bit flipped
                const int32_t kp = 2 * off - kDrift - dk + (klow ^ 1);
#pragma unroll
                for (int q = 0; q < NW; ++q) {
                    const bool own = p - lane == 32 * q;
                    if (q >= QB && q < QE) {
                        K[q] = own ? kp : kn[q];
                        tabu[q] = own ? expiry : tabu[q];
                    }
                    if (!own) vp[32 * q] = vn[q];
                    cp[32 * q] = cn[q];
                    cm[-32 * q] = cn[q];
                    if (own) s[q] = -s[q];
                }
                S0[p] = static_cast<int8_t>(2 * sp);  // every lane the same byte
            }
            __syncwarp();
            const int32_t gain = thr - dk;  // (E_best - E') / 4 << 9
            thr = min(gain, 0) + off;
            if (gain > 0) {
                E_best -= gain >> 7;  // 4 (E_best - E') / 4
#pragma unroll
                for (int w = 0; w < NW; ++w) Bb[w] = __ballot_sync(kFull, s[w] > 0);
            }
            if constexpr (TRACE) {
                if (trace_len < trace_cap) {
                    // E' = E_best - (E_best - E')
                    if (lane == 0 && HALF == 0)
                        trace[trace_len] = make_int4(static_cast<int>(g), t + 1, p, E_best - (min(gain, 0) >> 7));
                    ++trace_len;
                }
            }
        }
    }
    __syncwarp();  // the scratch is reused by the caller
#pragma unroll
    for (int w = 0; w < NW; ++w) seq[w] = Bb[w];
    TabuOut out;
    out.steps = t;
    out.E_best = E_best;
    out.fault = fault;
    return out;
}

}  // namespace lgpu
