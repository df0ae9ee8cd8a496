// tabu_skew.cuh -- the tabu search restricted to skew-symmetric sequences
// (Sec. II.C), one warp per search.
//
// For odd N with centre c = (N-1)/2, move i (0 <= i <= c) flips b_i and, for
// i < c, its partner b_j, j = N-1-i, so a skew-symmetric pivot stays
// skew-symmetric.  The energy of move i < c comes from the single-flip
// energies E_i, E_j:
//   E_{ij} = E_i + E_j - E + 16 s_i s_j C_d + 8 s_i s_j R - 32
//            - 16 (s_j s_{i-d} + s_i s_{j+d})        (terms outside 0..N-1 dropped)
// with d = j - i and R = sum_m s_m s_{N-1-m}.  Derivation: flipping {i, j}
// changes C_k by delta_k(i) + delta_k(j), plus 4 s_i s_j at k = d (both
// deltas negate the product s_i s_j, which keeps its sign); in
// sum_k (C_k + delta_k)^2 the cross sum sum_k delta_k(i) delta_k(j) is
// 4 s_i s_j (C_d + R - 2 s_i s_j), because the products s_{i+k} s_{j+k} and
// s_{i-k} s_{j-k} tile C_d without the pair (i, j), and s_{i+k} s_{j-k},
// s_{i-k} s_{j+k} tile R without it; the k = d correction leaves
// 8 s_i s_j (C_d + delta_d(i) + delta_d(j)) + 16.
// Skew symmetry, s_j = x_i s_i with x_i = (-1)^(c-i), shortens it: reversal
// with alternating signs maps the pivot to itself up to its sign and keeps
// energies, so E_j = E_i; and s_{j+d} = x_i s_{i-d}, since d is even.  With
// D_i = E_i - E,
//   E_{ij} - E = 2 D_i + x_i (16 C_d + 8 R - 32 s_i s~_{i-d}) - 32.
// R is unchanged by every move (s_i s_j and s_c^2 keep their signs), so it is
// computed once per search.  Move c is the single flip, D_c.
//
// Per step: the moves' energies from the kept D_i, the admissible minimum
// over the n = c + 1 moves with the same tabu, aspiration, tie and draw
// rules, and one O(N) update of D, C, V and the spins per flipped bit, as in
// tabu_search.  The lanes keep D_i for the free half only, and the spins of
// all bits.
//
// What bounds it: like tabu_search, the serial chain of a step, here with two
// dependent updates in it.  Two warps on a sub-partition, N = 101, 1,216
// replicas x 10^4 steps: 3.73 ms on GB300 (scoring every step from the bit
// planes of C_k: 17.28 ms).
#pragma once

#include "tabu_core.cuh"

namespace lgpu {

template <int NW, bool TRACE, bool FIX_FIRST>
__device__ TabuOut tabu_search_skew(uint32_t (&seq)[NW], const int N, const uint2 key,
                                    const uint32_t inst, const uint32_t g, const int max_iter,
                                    const int64_t budget, uint2 draws, int32_t* __restrict__ Cs,
                                    int4* __restrict__ trace, const int64_t trace_cap,
                                    int64_t& trace_len, const int lane) {
    constexpr int NH = (NW + 1) / 2;  // words of the free half: c < 16 NW
    constexpr int32_t kLow = 511;     // key bits below the energy change, as in tabu_search
    constexpr int32_t kNone = INT_MAX & ~kLow;
    const int c = (N - 1) >> 1;
    const TabuScratch<NW> sh(Cs);
    int32_t s[NW], d4[NW];  // d4: D_i / 4 (q < NH)
    int32_t E_best = search_setup<NW>(seq, N, lane, Cs, s, d4);
    uint32_t Bb[NW];
#pragma unroll
    for (int w = 0; w < NW; ++w) Bb[w] = seq[w];
    const int32_t R = sh.V[N - 1];
    // (E_{ij} - E) / 4 = mul D_i / 4 + x4 (C_d + s_i (-2 s~_{i-d})) + add
    int32_t tabu[NH], mul[NH], x4[NH], add[NH];
    const int32_t* Cd[NH];
    const int8_t* Sd[NH];
    bool movable[NH];
#pragma unroll
    for (int q = 0; q < NH; ++q) {
        const int i = lane + 32 * q;
        const int x = ((c - i) & 1) ? -1 : 1;
        tabu[q] = 0;
        movable[q] = i <= c && !(FIX_FIRST && i == 0);
        mul[q] = i < c ? 2 : (i == c ? 1 : 0);
        x4[q] = i < c ? 4 * x : 0;
        add[q] = i < c ? 2 * x * R - 8 : 0;
        Cd[q] = sh.C + (i < c ? 2 * (c - i) : 0);
        Sd[q] = sh.S + (i < c ? i - 2 * (c - i) : 0);
    }
    const int min_t = max_iter / 10;
    const int max_t = (12 * max_iter) / 100;
    const int nsteps = static_cast<int>(budget < 0 ? max_iter : (budget < max_iter ? budget : max_iter));
    const uint32_t low_lanes = (1u << lane) - 1u;
    int32_t thr = 0;  // a key below this is a move to below E_best
    int t = 0;        // moves made; this step is t + 1
    bool stuck = false;

    // Flips bit p (sp its spin before): one update of tabu_search.
    auto flip = [&](const int p, const int32_t sp) {
        int32_t* const vp = sh.V + lane + p;
        int32_t* const cp = sh.C + lane - p;
        int32_t* const cm = sh.C - lane + p;
        const int8_t* const ap = sh.S + 2 * lane - p;
        const int8_t* const bp = sh.S - lane + 2 * p;
        int32_t v[NW], cd[NW], cn[NW];
#pragma unroll
        for (int q = 0; q < NW; ++q) {
            v[q] = vp[32 * q];
            cd[q] = cp[32 * q];
            cn[q] = cd[q] + sp * (bp[-32 * q] - 2 * s[q]);
            if (q < NH) {
                const int32_t up = 2 * sp * (s[q] * (cd[q] + cn[q] + v[q]) + ap[64 * q]) - 4;
                d4[q] = lane + 32 * q == p ? -d4[q] : d4[q] + up;
            }
        }
        __syncwarp();  // every lane has read what the stores below change
#pragma unroll
        for (int q = 0; q < NW; ++q) {
            const bool own = lane + 32 * q == p;
            if (!own) vp[32 * q] = v[q] - 4 * sp * s[q];
            cp[32 * q] = cn[q];
            cm[-32 * q] = cn[q];
            if (own) s[q] = -s[q];
        }
        sh.S[p] = static_cast<int8_t>(2 * sp);  // every lane the same byte
        __syncwarp();
    };

    while (t < nsteps && !stuck) {
        // draws of steps t+1 .. t+32, one per lane: tie pick, and expiry of the move's tabu
        if (t > 0) draws = step_draws(key, inst, g, t + 1 + lane);
        const uint32_t u_tie_l = draws.x;
        const int32_t expiry_l = t + 1 + lane + rand_int(min_t, max_t, draws.y);
        const int tend = min(t + 32, nsteps);
#pragma unroll 1
        for (; t < tend; ++t) {
            // ---- move energies and the admissible minimum
            int32_t cand[NH];
            int32_t kmin_l = kNone;
#pragma unroll
            for (int q = 0; q < NH; ++q) {
                const int32_t e4 = mul[q] * d4[q] + (x4[q] * (*Cd[q] + s[q] * *Sd[q]) + add[q]);
                const int32_t k = e4 * (kLow + 1) + 2 * (lane + 32 * q) + (s[q] > 0 ? 1 : 0);
                cand[q] = movable[q] && (tabu[q] <= t || k < thr) ? k : kNone;
                kmin_l = min(kmin_l, cand[q]);
            }
            const int32_t kmin = __reduce_min_sync(kFull, kmin_l);
            int klow = kmin & kLow;  // 2p + (s_p == +1), p the lowest admissible minimiser
            uint32_t above = 0xFFFFFFFFu;  // least distance above the minimum itself
#pragma unroll
            for (int q = 0; q < NH; ++q)
                above = min(above, static_cast<uint32_t>(cand[q]) - static_cast<uint32_t>(kmin) - 1u);
            const int32_t expiry = __shfl_sync(kFull, expiry_l, t);
            if (__any_sync(kFull, above < static_cast<uint32_t>(kLow - klow)) || kmin == kNone) {
                if (kmin == kNone) {  // no admissible move: needs a user maxIter that lets maxTabu reach n
                    stuck = true;
                    break;
                }
                int rank[NH];  // minimisers before the lane's own, in ascending i
                int count = 0;
#pragma unroll
                for (int q = 0; q < NH; ++q) {
                    const uint32_t tb = __ballot_sync(kFull, cand[q] <= (kmin | kLow));
                    rank[q] = count + __popc(tb & low_lanes);
                    count += __popc(tb);
                }
                const uint32_t u_tie = __shfl_sync(kFull, u_tie_l, t);
                const int idx = static_cast<int>((static_cast<uint64_t>(u_tie) * count) >> 32);
                if (idx > 0) {  // the idx-th minimiser in ascending i: its key tells its index and spin
                    int32_t pick = kNone;
#pragma unroll
                    for (int q = 0; q < NH; ++q)
                        if (cand[q] <= (kmin | kLow) && rank[q] == idx) pick = cand[q];
                    klow = __reduce_min_sync(kFull, pick) & kLow;
                }
            }
            // ---- apply: flip b_p and its partner, tenure, bestSeqTS
            const int p = klow >> 1;
            const int32_t sp = 2 * (klow & 1) - 1;
            flip(p, sp);
            if (p < c) flip(N - 1 - p, ((c - p) & 1) ? -sp : sp);
#pragma unroll
            for (int q = 0; q < NH; ++q)
                if (lane + 32 * q == p) tabu[q] = expiry;
            const int32_t gain = thr - (kmin & ~kLow);  // (E_best - E') / 4 << 9
            thr = min(gain, 0);
            if (gain > 0) {
                E_best -= gain >> 7;  // 4 (E_best - E') / 4
#pragma unroll
                for (int w = 0; w < NW; ++w) Bb[w] = __ballot_sync(kFull, s[w] > 0);
            }
            if constexpr (TRACE) {
                if (trace_len < trace_cap) {
                    if (lane == 0) trace[trace_len] = make_int4(static_cast<int>(g), t + 1, p, E_best - (thr >> 7));
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
    out.fault = false;  // one warp per search: nothing to lose step with
    return out;
}

}  // namespace lgpu
