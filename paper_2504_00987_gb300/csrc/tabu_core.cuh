// tabu_core.cuh -- one warp runs one tabu search (Algorithm 2 / Algorithm 4).
//
// Neighbour scoring (Sec. III.C, Table I).  Flipping s_j changes C_k by
// delta_k(j) = -2 s_j (s_{j+k} + s_{j-k}) (terms outside 1..N dropped), so
//   E_j = E + sum_k delta_k (2 C_k + delta_k)
//       = E + 4(N-1) + 8 M_j - 4 s_j R_j,
// with M_j = sum_{k>=1} s_{j+k} s_{j-k} (a masked popcount of the XOR of the
// two windows of j) and R_j = sum_k C_k (s_{j+k} + s_{j-k}).  R_j is set up
// once per search on bit planes (0-based bits b_i, s_i = 2 b_i - 1):
//   R_j = 2 S_j - T_j,  S_j = sum_k C_k (b_{j+k} + b_{j-k}),
//   T_j = sum_{k<=j} C_k + sum_{k<=N-1-j} C_k,
// where S_j = sum_m w_m [popc(t_m & X_j) + popc(t_m & Y_j)] over the
// two's-complement planes t_m of C_k (from warp ballots), X_j = pivot >> j
// (bit k = b_{j+k}) and Y_j the mirrored window (bit k = b_{j-k}); T_j comes
// from prefix sums of C_k.  After every move each neighbour's energy change
// is updated exactly in O(1) from C_k and the self-convolution V_m of the
// spins (the identity stands above tabu_search), so a step never goes back to
// the bits.  Arithmetic is exact int32.
//
// Work split: lane l owns the neighbours j = l + 32q: their keys (energy
// change, index and spin in one int), tabu expiry and spins in registers; V,
// C and the spins also in the warp's slice of shared memory, where the move
// shifts them against each other.  The admissible minimum is one
// redux.sync.min over the keys; ballots resolve a tie only where there is one.
#pragma once

#include <climits>

#include "labs_device.cuh"

namespace lgpu {

// C_k = (N - k) - 2 popc(b_i xor b_{i+k} over i < N-k) for the lane's
// k = lane + 32q (C_0 and C_{k >= N} are 0).
template <int NW>
__device__ __forceinline__ void correlations(const uint32_t (&B)[NW], int N, int lane,
                                             int32_t (&c)[NW]) {
#pragma unroll
    for (int q = 0; q < NW; ++q) {
        const int k = lane + 32 * q;
        int cnt = 0;
#pragma unroll
        for (int w = 0; w + q < NW; ++w) {
            const uint32_t xk = __funnelshift_r(B[w + q], (w + q + 1 < NW) ? B[w + q + 1] : 0u, lane);
            cnt += __popc((B[w] ^ xk) & word_lowmask(w, N - k));
        }
        c[q] = (k >= 1 && k <= N - 1) ? (N - k) - 2 * cnt : 0;
    }
}

// Energy of the warp-uniform sequence B (all lanes return it).
template <int NW>
__device__ __forceinline__ int32_t warp_energy(const uint32_t (&B)[NW], int N, int lane) {
    int32_t c[NW];
    correlations<NW>(B, N, lane, c);
    int32_t sq = 0;
#pragma unroll
    for (int q = 0; q < NW; ++q) sq += c[q] * c[q];
    return __reduce_add_sync(kFull, sq);
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

// Bit-plane count bound: |C_k| <= N - 1 < 32*NW, so C_k fits in
// bitlen(32*NW - 1) + 1 two's-complement bits.
template <int NW>
struct PlaneMax {
    static constexpr int value = (NW == 2) ? 7 : (NW <= 4) ? 8 : 9;
};

// sum_i popc(w[i]) * weight for n words, carry-save compressed: full
// adders (sum = a^b^c, carry = maj(a,b,c), one LOP3 each) fold three words
// of one weight into one word of that weight and one of twice the weight,
// so n words cost about n/2 + log n popcounts instead of n.  The adders
// trade popcounts (XU pipe) for logic (ALU pipe), which pays while the
// step has registers to spare: for 7 or more words (six- and eight-word
// sequences, N > 160) plain popcounts measured 14-21 % faster on GB300
// and 2-16 % slower below; five-word sequences (6 words) count plainly as
// well.  Five words (four-word sequences) take one full adder and two plain
// popcounts, about 1 % faster than two adders.
template <int n, int weight>
__device__ __forceinline__ int csa_popc(const uint32_t (&w)[n]) {
    if constexpr (weight == 1 && n == 5) {
        const uint32_t a = w[0], b = w[1], c = w[2];
        return __popc(a ^ b ^ c) + 2 * __popc((a & b) | (c & (a | b))) + __popc(w[3]) + __popc(w[4]);
    } else if constexpr (n <= 2 || (weight == 1 && n >= 6)) {
        int s = 0;
#pragma unroll
        for (int i = 0; i < n; ++i) s += __popc(w[i]);
        return s * weight;
    } else {
        constexpr int f = (n - 1) / 2;  // full adders at this weight
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
        return s * weight + csa_popc<f, 2 * weight>(carry);
    }
}

// S[q] += sum over planes m < P of w_m [popc(t_m & X_q) + popc(t_m & Y_q)],
// plane 0 being the constant parity pattern of C_k (C_k = N - k mod 2) and
// plane P-1 the sign plane (weight -2^(P-1)).  Fully unrolled for a
// compile-time P so every ballot and popcount of the step can overlap.
template <int NW, int P>
__device__ __forceinline__ void score_planes(const int32_t (&c)[NW], const uint32_t (&par)[NW],
                                             const uint32_t (&X)[NW][NW],
                                             const uint32_t (&Y)[NW][NW], int32_t (&S)[NW]) {
#pragma unroll
    for (int m = 0; m < P; ++m) {
        uint32_t tp[NW];
#pragma unroll
        for (int w = 0; w < NW; ++w) tp[w] = (m == 0) ? par[w] : __ballot_sync(kFull, (c[w] >> m) & 1);
        constexpr int32_t one = 1;
        const int32_t wm = (m == P - 1) ? -(one << m) : (one << m);
#pragma unroll
        for (int q = 0; q < NW; ++q) {
            uint32_t words[NW + 1];  // (NW - q) words of X_j and (q + 1) of Y_j
#pragma unroll
            for (int w = 0; w + q < NW; ++w) words[w] = tp[w] & X[q][w];
#pragma unroll
            for (int w = 0; w <= q; ++w) words[NW - q + w] = tp[w] & Y[q][w];
            S[q] += csa_popc<NW + 1, 1>(words) * wm;
        }
    }
}

// Inclusive prefix sums of C at the lane's own indices: pc[q] = PC(l + 32q),
// PC(n) = sum_{k=1}^{n} C_k (C_0 = 0).  Two chunks share one packed 32-bit
// shuffle scan (low and high 16-bit halves; every within-chunk prefix is
// bounded by 32 (N-1) < 2^15).  Used once per search; afterwards the sums
// are updated incrementally per move.
template <int NW>
__device__ __forceinline__ void prefix_own(const int32_t (&c)[NW], int lane, int32_t (&pc)[NW]) {
    constexpr int NP = NW & ~1;  // chunks scanned in pairs
    int32_t carry = 0;
#pragma unroll
    for (int q = 0; q < NP; q += 2) {
        int32_t v = c[q] + c[q + 1] * 65536;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t n = __shfl_up_sync(kFull, v, o);
            if (lane >= o) v += n;
        }
        const int32_t last = __shfl_sync(kFull, v, 31);
        const int32_t lo = static_cast<int32_t>(static_cast<int16_t>(v & 0xFFFF));
        const int32_t hi = (v - lo) / 65536;
        const int32_t lo31 = static_cast<int32_t>(static_cast<int16_t>(last & 0xFFFF));
        const int32_t hi31 = (last - lo31) / 65536;
        pc[q] = carry + lo;
        pc[q + 1] = carry + lo31 + hi;
        carry += lo31 + hi31;
    }
    if constexpr (NW & 1) {  // an odd word count leaves one chunk, scanned alone
        int32_t v = c[NW - 1];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t n = __shfl_up_sync(kFull, v, o);
            if (lane >= o) v += n;
        }
        pc[NW - 1] = carry + v;
    }
}

// T_j = PC(j) + PC(N-1-j) for the lane's j = l + 32q: its own prefix plus
// the mirror index's prefix, read back through the warp's shared scratch.
template <int NW>
__device__ __forceinline__ void mirror_terms(const int32_t (&pc)[NW], int N, int lane,
                                             int32_t* __restrict__ Cs, int32_t (&T)[NW]) {
#pragma unroll
    for (int q = 0; q < NW; ++q) Cs[lane + 32 * q] = pc[q];
    __syncwarp();
#pragma unroll
    for (int q = 0; q < NW; ++q) {
        const int j = lane + 32 * q;
        T[q] = pc[q] + Cs[j < N ? N - 1 - j : 0];
    }
    __syncwarp();
}

// Scores S_j with P bit planes, where P >= the planes C_k needs (extra
// planes only repeat the sign and leave the sum exact).  Three fully
// unrolled widths keep the code small enough for the instruction cache
// (a jump table over every width measured several hundred cycles slower).
template <int NW>
__device__ __forceinline__ void score_dispatch(int P, const int32_t (&c)[NW], const uint32_t (&par)[NW],
                                               const uint32_t (&X)[NW][NW], const uint32_t (&Y)[NW][NW],
                                               int32_t (&S)[NW]) {
#pragma unroll
    for (int q = 0; q < NW; ++q) S[q] = 0;
    if (P <= 5)
        score_planes<NW, 5>(c, par, X, Y, S);
    else if (P <= 6)
        score_planes<NW, 6>(c, par, X, Y, S);
    else
        score_planes<NW, PlaneMax<NW>::value>(c, par, X, Y, S);
}

// Number of two's-complement planes that hold every C_k of the warp:
// bit length of max |C_k| plus the sign bit.
template <int NW>
__device__ __forceinline__ int plane_count(const int32_t (&c)[NW]) {
    uint32_t mx = 0;
#pragma unroll
    for (int q = 0; q < NW; ++q) mx = max(mx, static_cast<uint32_t>(abs(c[q])));
    return 33 - __clz(__reduce_max_sync(kFull, mx));
}

// The lane's windows of an NW-word vector: XB[i] = word i of B >> lane and
// YB[i] = word i of RL >> (31 - lane).  For j = lane + 32q, word w of the
// forward window X_j (bit k = b_{j+k}) is XB[q + w] and word w of the
// backward window Y_j (bit k = b_{j-k}) is YB[w + NW - 1 - q]; both are zero
// past the ends of the sequence.
template <int NW>
__device__ __forceinline__ void pivot_windows(const uint32_t (&B)[NW], const uint32_t (&RL)[NW],
                                              int lane, uint32_t (&XB)[NW], uint32_t (&YB)[NW]) {
#pragma unroll
    for (int i = 0; i < NW; ++i) {
        XB[i] = __funnelshift_r(B[i], i + 1 < NW ? B[i + 1] : 0u, lane);
        YB[i] = __funnelshift_r(RL[i], i + 1 < NW ? RL[i + 1] : 0u, 31 - lane);
    }
}

// Scratch of one warp's tabu search (ints): V (2 NB), C (2 NB), spins (3 NB
// bytes), NB = 32 NW; a multiple of 16 bytes.
template <int NW>
constexpr int kTabuScratchInts = 128 * NW + 24 * NW;

// V_m = sum_a s_a s_{m-a} (terms outside 0..N-1 dropped) for m = lane + 32i,
// i < 2 NW, from the bits of the sequence and its mirror image.
template <int NW>
__device__ __forceinline__ void store_self_convolution(const uint32_t (&B)[NW], const uint32_t (&RL)[NW], int N,
                                                       int lane, int32_t* __restrict__ Vs) {
    // Z[x + 1] = word x of RL >> (31 - lane), x = -1 .. NW-1: bit i of word
    // w + NW - 1 - i' is b_{m-a} for m = lane + 32 i', a = 32 w + i
    uint32_t Z[NW + 1];
    Z[0] = __funnelshift_r(0u, RL[0], 31 - lane);
#pragma unroll
    for (int x = 0; x < NW; ++x) Z[x + 1] = __funnelshift_r(RL[x], x + 1 < NW ? RL[x + 1] : 0u, 31 - lane);
#pragma unroll
    for (int i = 0; i < 2 * NW; ++i) {
        const int m = lane + 32 * i;
        const int lo = max(0, m - N + 1), hi = min(m, N - 1);  // a in [lo, hi]
        int diff = 0;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            const int x = w + NW - 1 - i;  // compile-time
            if (x >= -1 && x < NW)
                diff += __popc((B[w] ^ Z[x + 1]) & word_lowmask(w, hi + 1) & ~word_lowmask(w, lo));
        }
        Vs[m] = max(hi - lo + 1, 0) - 2 * diff;
    }
}

// The scratch's parts: V_m, m = 0 .. 2 NB - 1; C_d at C[d] and C[-d]; -2 s~_i
// at S[i], i = -NB .. 2 NB - 1.
template <int NW>
struct TabuScratch {
    int32_t* V;
    int32_t* C;
    int8_t* S;
    __device__ __forceinline__ explicit TabuScratch(int32_t* base)
        : V(base), C(base + 3 * 32 * NW), S(reinterpret_cast<int8_t*>(base + 4 * 32 * NW) + 32 * NW) {}
};

// Fills the scratch for a search from `seq` and returns its energy; s[q] is
// the spin (0 for j >= N) and d4[q] the energy change D_j / 4 of the lane's
// j = lane + 32q (unset for j >= N).
template <int NW>
__device__ __forceinline__ int32_t search_setup(const uint32_t (&seq)[NW], int N, int lane,
                                                int32_t* __restrict__ Cs, int32_t (&s)[NW], int32_t (&d4)[NW]) {
    constexpr int NB = 32 * NW;
    const TabuScratch<NW> sh(Cs);
    int32_t c[NW];
    correlations<NW>(seq, N, lane, c);
    int32_t sq = 0;
#pragma unroll
    for (int q = 0; q < NW; ++q) sq += c[q] * c[q];
    const int32_t E = __reduce_add_sync(kFull, sq);
    // R_j = 2 S_j - T_j from the bit planes of C_k (S_j) and the prefix sums
    // of C_k (T_j = PC(j) + PC(N-1-j))
    uint32_t RL[NW], XB[NW], YB[NW], par[NW];
    reverse_bits<NW>(seq, RL);
    pivot_windows<NW>(seq, RL, lane, XB, YB);
#pragma unroll
    for (int w = 0; w < NW; ++w) {
        const uint32_t alt = ((N - 32 * w) & 1) ? 0x55555555u : 0xAAAAAAAAu;  // (N - k) odd
        par[w] = alt & word_lowmask(w, N) & (w == 0 ? ~1u : kFull);
    }
    uint32_t X[NW][NW], Y[NW][NW];
#pragma unroll
    for (int q = 0; q < NW; ++q) {
#pragma unroll
        for (int w = 0; w + q < NW; ++w) X[q][w] = XB[q + w];
#pragma unroll
        for (int w = 0; w <= q; ++w) Y[q][w] = YB[w + NW - 1 - q];
    }
    int32_t S[NW], pc[NW], T[NW];
    score_dispatch<NW>(plane_count<NW>(c), c, par, X, Y, S);
    prefix_own<NW>(c, lane, pc);
    mirror_terms<NW>(pc, N, lane, Cs, T);
    store_self_convolution<NW>(seq, RL, N, lane, sh.V);
#pragma unroll
    for (int q = 0; q < NW; ++q) {
        const int j = lane + 32 * q;
        s[q] = j < N ? ((XB[q] & 1u) ? 1 : -1) : 0;
        sh.C[j] = c[q];
        sh.C[-j] = c[q];
        sh.S[j] = static_cast<int8_t>(-2 * s[q]);
        sh.S[j - NB] = 0;
        sh.S[j + NB] = 0;
    }
    __syncwarp();
    // D_j / 4 = N - 1 + 2 M_j - s_j R_j, 2 M_j = V_{2j} - 1
#pragma unroll
    for (int q = 0; q < NW; ++q) d4[q] = N - 2 + sh.V[2 * (lane + 32 * q)] - s[q] * (2 * S[q] - T[q]);
    __syncwarp();
    return E;
}

// One tabu search from `seq` (warp-uniform).  On return `seq` holds
// bestSeqTS.  Draws: step t uses Philox(instance, g, t, 4): x tie, y tenure.
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
// N = 64 217 / 295 / 510, N = 120 343 / 453 / 758, N = 192 414 / 574 (two
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
                               const int64_t budget, int32_t* __restrict__ Cs,
                               int4* __restrict__ trace, const int64_t trace_cap,
                               int64_t& trace_len, const int lane, PairLink* link = nullptr,
                               uint32_t* xseq = nullptr) {
    static_assert(WPS == 1 || (WPS == 2 && NW % 2 == 0 && HALF >= 0 && HALF < 2), "warps per sequence");
    constexpr int NB = 32 * NW;
    constexpr int QB = HALF * (NW / WPS), QE = (HALF + 1) * (NW / WPS);  // this warp's q
    // A drawn tie is scored by a second copy of the scoring code from three
    // words on, and through the loop of the first where two words make that
    // copy as long as the rest of the step (cycles a step, one warp alone:
    // N = 64 232 with the copy, 217 without; N = 120 343 and 355; N = 192 414
    // and 443).
    constexpr bool kRecompute = NW <= 4 ? NW > 2 : true;
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
    const int nsteps = static_cast<int>(budget < 0 ? max_iter : (budget < max_iter ? budget : max_iter));
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

    while (t < nsteps && !fault && !stuck) {
        // draws of steps t+1 .. t+32, one per lane: tie pick, and expiry of the move's tabu
        const uint4 r = draw4(key, inst, g, static_cast<uint32_t>(t + 1 + lane), kPurposeStep);
        const uint32_t u_tie_l = r.x;
        const int32_t expiry_l = t + 1 + lane + rand_int(min_t, max_t, r.y);
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
                    uint32_t tb[NW];
    #pragma unroll
                    for (int q = QB; q < QE; ++q) {
                        tb[q] = __ballot_sync(kFull, cand[q] <= (kmin | kLow));
                        if constexpr (WPS == 1) count += __popc(tb[q]);
                    }
                    const uint32_t u_tie = __shfl_sync(kFull, u_tie_l, t);
                    int idx = static_cast<int>((static_cast<uint64_t>(u_tie) * count) >> 32);
                    if (idx > 0) {  // the idx-th minimiser in ascending j
                        int p = 0;
                        bool mine = true;  // WPS = 2: the warp holding it finds it, then tells the other
                        if constexpr (WPS == 2) {
                            mine = HALF == 0 ? idx < count_lo : idx >= count_lo;
                            if (HALF == 1) idx -= count_lo;
                        }
                        if (mine) {
                            bool found = false;
    #pragma unroll
                            for (int q = QB; q < QE; ++q) {
                                const int pc_q = __popc(tb[q]);
                                if (!found) {
                                    if (idx < pc_q) {
                                        p = 32 * q + nth_set_bit(tb[q], idx);
                                        found = true;
                                    } else {
                                        idx -= pc_q;
                                    }
                                }
                            }
                        }
                        if constexpr (WPS == 2) {
                            uint64_t o = 0;
                            if (!pair_exchange(link, HALF, (*xseq)++, mine ? static_cast<uint64_t>(p) : 0u, o, lane)) {
                                fault = true;
                                break;
                            }
                            if (!mine) p = static_cast<int>(o);
                        }
                        klow = 2 * p + (S0[p] < 0 ? 1 : 0);
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
