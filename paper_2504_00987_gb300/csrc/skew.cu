// skew.cu -- labs_skew_deviation_batch: the deviation from skew-symmetry
// d(S) of Appendix A (Eqs. 5-9) for a batch of sequences.
//
// For a sequence T of odd length L = 2n - 1 (bits t_0 .. t_{L-1}, centre
// c = n - 1), Eq. 5 counts the i in 1..n-1 with s_{n+i} != (-1)^i s_{n-i};
// in bits that is t_{c+i} xor t_{c-i} xor [i odd], so
//   n_non-skew(T) = popc((R ^ Lr ^ ALT) & bits[1, n-1]),
// with R bit i = t_{c+i}, Lr bit i = t_{c-i} and ALT the odd positions.
// d(S) is the minimum of n_non-skew over the rotations Rot(S; r) (Eq. 6) for
// odd N, and over the rotations followed by one deletion Del(.; i) (Eq. 8)
// for even N (the reading that reproduces the d column of Table II).
//
// Let D be the sequence repeated, u_m = D[r + m] rotation r, and for even N let
// u_d be deleted (L = N - 1, c = (N - 2) / 2).  Moving d outwards from the
// centre by one changes one pair, so the N deletions of a rotation are two
// walks from a common start: with
//   A_i = u_{c+i} ^ u_{c-i} ^ [i odd],  B_i = u_{c+i+1} ^ u_{c-i} ^ [i odd],
//   G_i = u_{c+i+1} ^ u_{c-i+1} ^ [i odd],
// the mismatches are sum_i B_i + sum_{i<=t} (A_i - B_i) for d = c + 1 + t and
// sum_i B_i + sum_{i<=t} (G_i - B_i) for d = c - t, t = 0 .. n-1.
//
// A lane takes 32 rotations at once, one per bit: for fixed i the words
// D[32w + c + i ..] and D[32w + c - i ..] hold u_{c+i} and u_{c-i} of 32
// rotations, the counts are bit-sliced (plane k holds bit k of the 32 counts;
// every count is at most n - 1 < 128), a step of a walk is a ripple of full
// adders, one LOP3 per sum and carry, and the running minimum a borrow chain
// and a select: about 60 logic instructions per i for 64 of the N^2
// candidates.  ceil(N / 32) lanes share a sequence.  What bounds it: the
// logic instructions, at half the issue rate (no traffic to speak of).
// 100,000 sequences of N = 120 take 94 us on GB300 (one warp per sequence
// that rescored all words for every deletion: 3,769 us); 60,000 of N = 64,
// 128, 160, 256: 19, 63, 113, 258 us.
#include <cuda_runtime.h>

#include <climits>

#include "capi_util.h"
#include "kernels.h"
#include "labs_device.cuh"

namespace lgpu {

constexpr int kSkewWarps = 4;
constexpr int kSkewWords = 160;  // words of D of one warp's sequences (at most 5 for each of 32)

// sum and carry of three bit-sliced bits
__device__ __forceinline__ uint32_t xor3(uint32_t a, uint32_t b, uint32_t c) { return a ^ b ^ c; }
__device__ __forceinline__ uint32_t maj3(uint32_t a, uint32_t b, uint32_t c) { return (a & b) | (c & (a | b)); }

// cur += (x ? (dec ? -1 : +1) : 0) in every bit lane.
template <int P>
__device__ __forceinline__ void step_count(uint32_t (&cur)[P], uint32_t x, uint32_t dec) {
    uint32_t carry = cur[0] & x;
    cur[0] ^= x;
#pragma unroll
    for (int k = 1; k < P; ++k) {
        const uint32_t s = cur[k];
        cur[k] = xor3(s, dec, carry);
        carry = maj3(s, dec, carry);
    }
}

// best = min(best, cur) in every bit lane.
template <int P>
__device__ __forceinline__ void take_min(uint32_t (&best)[P], const uint32_t (&cur)[P]) {
    uint32_t less = 0;  // borrow of cur - best
#pragma unroll
    for (int k = 0; k < P; ++k) less = maj3(~cur[k], best[k], less);
#pragma unroll
    for (int k = 0; k < P; ++k) best[k] = (cur[k] & less) | (best[k] & ~less);
}

// Bits [start, start + 64) of the bit string V, start >= 0.
__device__ __forceinline__ void window64(const uint32_t* V, int start, uint32_t& lo, uint32_t& hi) {
    const int o = start >> 5, b = start & 31;
    lo = __funnelshift_r(V[o], V[o + 1], b);
    hi = __funnelshift_r(V[o + 1], V[o + 2], b);
}

// P: planes of a count, 2^P >= n.  lps = ceil(N / 32) lanes per sequence,
// stride = words of shared memory per sequence (skew_words).
template <int P>
__global__ void __launch_bounds__(kSkewWarps * 32) skew_kernel(const uint64_t* __restrict__ seqs, int N,
                                                               int64_t B, int lps, int stride,
                                                               int32_t* __restrict__ out) {
    __shared__ uint32_t Dsh[kSkewWarps][kSkewWords];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int spw = 32 / lps;  // sequences per warp
    const int group = min(lane / lps, spw - 1);
    const int w = min(lane - group * lps, lps - 1);  // lanes left over repeat the last word
    const int64_t first = (static_cast<int64_t>(blockIdx.x) * kSkewWarps + warp) * spw;
    if (first >= B) return;
    const int64_t b = min(first + group, B - 1);  // groups past the end repeat the last sequence
    const bool odd = (N & 1) != 0;
    const int c = ((odd ? N : N - 1) - 1) / 2;  // centre index of the candidates
    const int n = c + 1;
    // Dp[0] pads the words before D; word k of D (bits 32k ..) at Dp[1 + k]
    uint32_t* const Dp = Dsh[warp] + group * stride;
    const uint32_t* const S = reinterpret_cast<const uint32_t*>(seqs + b * ((N + 63) / 64));
    const int W32 = (N + 31) / 32;
    if (w == 0) Dp[0] = 0u;
    if (N < 32) {
        // A word holds several repeats: doubled up to 64 bits once, then shifted
        // (a call of 100 sequences repeat by repeat / so: N = 3 3.2 / 1.5 us,
        // N = 16 2.8 / 2.3; one warp per sequence, before the walks, 2.4 and 5.5).
        uint64_t rep = __ldg(S) & word_lowmask(0, N);
        for (int len = N; len < 64; len *= 2) rep |= rep << len;
        const int step = 32 % N;
        int p = 0;  // 32 k mod N; one lane per sequence, so k goes up by one
        for (int k = 0; k < stride - 1; ++k) {
            Dp[1 + k] = static_cast<uint32_t>(rep >> p);
            p += step;
            if (p >= N) p -= N;
        }
    } else {
        for (int k = w; k < stride - 1; k += lps) {
            uint32_t v = 0;
            int p = (32 * k) % N;
            for (int have = 0; have < 32;) {
                const int o = p >> 5;
                const uint32_t x = __funnelshift_r(__ldg(S + o), o + 1 < W32 ? __ldg(S + o + 1) : 0u, p & 31);
                const int take = min(N - p, 32 - have);
                v |= (x & word_lowmask(0, take)) << have;
                have += take;
                p = p + take == N ? 0 : p + take;
            }
            Dp[1 + k] = v;
        }
    }
    __syncwarp();
    const int at = 32 * (w + 1) + c;  // bit of Dp at which u_c of the lane's rotations starts
    uint32_t best[P], cur[P], cur2[P];
#pragma unroll
    for (int k = 0; k < P; ++k) best[k] = 0u;
    // sum of A_i (odd N) or B_i (even N), four terms per ripple
    for (int i0 = 1; i0 < n; i0 += 32) {
        uint32_t ulo, uhi, dlo, dhi;
        window64(Dp, at + i0 + (odd ? 0 : 1), ulo, uhi);
        window64(Dp, at - i0 - 31, dlo, dhi);
        const int m = min(32, n - i0);
        for (int j = 0; j < m; j += 4) {
            uint32_t x[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const uint32_t v = __funnelshift_r(ulo, uhi, j + e) ^ __funnelshift_r(dlo, dhi, 31 - j - e);
                x[e] = j + e < m ? ((e & 1) ? v : ~v) : 0u;  // i0 + j + e is odd for even e
            }
            const uint32_t c1 = maj3(best[0], x[0], x[1]);
            best[0] = xor3(best[0], x[0], x[1]);
            const uint32_t c2 = maj3(best[0], x[2], x[3]);
            best[0] = xor3(best[0], x[2], x[3]);
            if constexpr (P > 1) {
                uint32_t carry = maj3(best[1], c1, c2);
                best[1] = xor3(best[1], c1, c2);
#pragma unroll
                for (int k = 2; k < P; ++k) {
                    const uint32_t s = best[k];
                    best[k] = s ^ carry;
                    carry &= s;
                }
            }
        }
    }
    if (!odd) {
#pragma unroll
        for (int k = 0; k < P; ++k) cur[k] = cur2[k] = best[k];
        uint32_t up, uhi, down, dhi;  // u_{c+i} and u_{c-i+1} of this i
        window64(Dp, at + 1, up, uhi);
        window64(Dp, at, down, dhi);
        for (int i0 = 1; i0 < n; i0 += 32) {
            uint32_t ulo, dlo;
            window64(Dp, at + i0 + 1, ulo, uhi);
            window64(Dp, at - i0 - 31, dlo, dhi);
            const int m = min(32, n - i0);
#pragma unroll 2
            for (int j = 0; j < m; ++j) {
                const uint32_t nx = __funnelshift_r(ulo, uhi, j);       // u_{c+i+1}
                const uint32_t dn = __funnelshift_r(dlo, dhi, 31 - j);  // u_{c-i}
                const uint32_t alt = (j & 1) ? 0u : kFull;
                const uint32_t Bi = nx ^ dn ^ alt;
                step_count<P>(cur, up ^ nx, Bi & ~(up ^ dn ^ alt));
                take_min<P>(best, cur);
                step_count<P>(cur2, down ^ dn, Bi & ~(nx ^ down ^ alt));
                take_min<P>(best, cur2);
                up = nx;
                down = dn;
            }
        }
    }
    // the least of the lane's counts: keep the rotations with a 0 in each plane, highest first
    uint32_t alive = word_lowmask(w, N);
    int least = 0;
#pragma unroll
    for (int k = P - 1; k >= 0; --k) {
        const uint32_t zero = alive & ~best[k];
        if (zero == 0u)
            least |= 1 << k;
        else
            alive = zero;
    }
    for (int k = 1; k < lps; ++k) {  // lane `group * lps` collects its group
        const int o = __shfl_sync(kFull, least, min(group * lps + k, 31));
        if (w == 0) least = min(least, o);
    }
    if (lane == group * lps && first + group < B) out[first + group] = least;
}

// Words of shared memory per sequence: one in front, and D as far as the last
// 64-bit window of the last lane reaches.
inline int skew_words(int N, int lps) {
    const int c = (((N & 1) ? N : N - 1) - 1) / 2;
    return 1 + ((32 * (lps - 1) + 2 * c + 2) >> 5) + 3;
}

cudaError_t launch_skew(const uint64_t* d_seqs, int N, int64_t B, int32_t* d_out, cudaStream_t stream) {
    const int lps = (N + 31) / 32, spw = 32 / lps;
    const int stride = skew_words(N, lps);
    if (stride * spw > kSkewWords) return cudaErrorInvalidValue;
    const int64_t per_block = static_cast<int64_t>(kSkewWarps) * spw;
    const unsigned blocks = static_cast<unsigned>((B + per_block - 1) / per_block);
    if (N <= 64)
        skew_kernel<5><<<blocks, kSkewWarps * 32, 0, stream>>>(d_seqs, N, B, lps, stride, d_out);
    else if (N <= 128)
        skew_kernel<6><<<blocks, kSkewWarps * 32, 0, stream>>>(d_seqs, N, B, lps, stride, d_out);
    else
        skew_kernel<7><<<blocks, kSkewWarps * 32, 0, stream>>>(d_seqs, N, B, lps, stride, d_out);
    return cudaGetLastError();
}

}  // namespace lgpu

extern "C" int32_t labs_skew_deviation_batch(const uint64_t* d_seqs, int32_t N, int64_t B, int32_t* d_d,
                                             labs_stream_t stream) {
    using namespace lcapi;
    if (N < 3 || N > LABS_MAX_N) return fail(LABS_EINVAL, "N=%d outside 3..%d", N, LABS_MAX_N);
    if ((N & 1) == 0 && N < 4) return fail(LABS_EINVAL, "even N must be >= 4");
    if (B < 0) return fail(LABS_EINVAL, "B < 0");
    if (B == 0) return ok();
    if (B > (int64_t{1} << 33)) return fail(LABS_EINVAL, "B too large");
    LABS_TRY(check_dev(d_seqs, 8, "d_seqs", false));
    LABS_TRY(check_dev(d_d, 4, "d_d", false));
    const cudaError_t e = lgpu::launch_skew(d_seqs, N, B, d_d, static_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) return cuda_fail(e, "skew kernel launch");
    return ok();
}
