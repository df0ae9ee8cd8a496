// energy.cu -- labs_energy_batch: C_k (Eq. 1) and E (Eq. 2) of B packed
// sequences.  C_k = (N - k) - 2 popc(b_i xor b_{i+k}, i < N - k): one
// funnel-shifted window, an xor and a popcount per 32 products.
//  - E only, many sequences: one thread per sequence (NW words in registers).
//  - E and C, or few sequences: one warp per sequence, lane l computes C_k for
//    k = l + 32q, so each row of C is written by consecutive lanes
//    (coalesced); the masks of a lane are those of every sequence, so a warp of
//    a large batch keeps them and takes one group of sequences after the other.
// What bounds them: popcounts, 8 cycles of the XU pipe a warp and 8 of them per
// 32 values of k at N = 120 after the full adders (10 words), 51 us for 10^6
// sequences; with C, instructions (82 a warp and sequence at N = 127, issued in
// 65 % of the cycles, the ALU pipe as full) and too few warps to cover the rows'
// loads, not the rows' stores (a fill of as many bytes takes 22.6 us of its 34.8;
// 16-byte stores through shared memory took 35 us where these take 33).  On
// GB300, N = 120: 10^6 energies 57 us (masks rebuilt for every word and round, no
// adders: 151), 300,000 with C 33 us (57); 100 energies 1.5 us on the device (8.6).
#include <cuda_runtime.h>

#include <algorithm>

#include "capi_util.h"
#include "kernels.h"
#include "tabu_core.cuh"

namespace lgpu {

constexpr int kEnergyThreads = 256;

// Words per row in memory: whole 64-bit words.
template <int NW>
constexpr int kRowWords = (NW + 1) & ~1;

template <int NW>
__device__ __forceinline__ void load_row(const uint32_t* __restrict__ seqs, int64_t b, int N, uint32_t (&s)[NW]) {
    const uint2* src = reinterpret_cast<const uint2*>(seqs + b * kRowWords<NW>);  // 8-byte aligned rows
#pragma unroll
    for (int v = 0; v < kRowWords<NW> / 2; ++v) {
        const uint2 x = __ldg(src + v);
        s[2 * v] = x.x;
        if (2 * v + 1 < NW) s[2 * v + 1] = x.y;
    }
    s[NW - 1] &= word_lowmask(NW - 1, N);  // bits >= N are ignored
}

template <int NW>
__global__ void __launch_bounds__(kEnergyThreads) energy_thread_kernel(const uint32_t* __restrict__ seqs, int N,
                                                                       int64_t B, int32_t* __restrict__ E) {
    const int64_t b = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (b >= B) return;
    uint32_t s[NW];
    load_row<NW>(seqs, b, N, s);
    E[b] = thread_energy<NW, true>(s, N);
}

// A warp takes ROWS consecutive sequences at a time, so that one's loads and
// reduction overlap the others' work.  ROWS = 1: each warp has one sequence, and
// the kernel no loop, whose bounds took a fifth of a small call (E and C, 4,000
// sequences of N = 64 2.15 / 1.67 us with / without it).
template <int NW, int ROWS>
__global__ void __launch_bounds__(kEnergyThreads) energy_warp_kernel(const uint32_t* __restrict__ seqs, int N,
                                                                     int64_t B, int32_t* __restrict__ E,
                                                                     int32_t* __restrict__ C) {
    const int lane = threadIdx.x & 31;
    const int64_t warps = static_cast<int64_t>(gridDim.x) * (kEnergyThreads / 32);
    const int64_t warp = (static_cast<int64_t>(blockIdx.x) * kEnergyThreads + threadIdx.x) >> 5;
    uint32_t mask[NW];
    pair_masks<NW, false>(N, lane, mask);
    for (int64_t b0 = warp * ROWS; b0 < B; b0 += warps * ROWS) {
        const int rows = ROWS == 1 ? 1 : static_cast<int>(min(static_cast<int64_t>(ROWS), B - b0));
        int32_t sq[ROWS];
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            uint32_t s[NW];
            load_row<NW>(seqs, ROWS == 1 ? b0 : min(b0 + r, B - 1), N, s);
            int32_t c[NW];
            lane_correlations<NW>(s, mask, N, lane, c);
            sq[r] = lane >= 1 ? c[0] * c[0] : 0;  // C_0 does not count
#pragma unroll
            for (int q = 1; q < NW; ++q) sq[r] += c[q] * c[q];
            if (C != nullptr && r < rows) {
#pragma unroll
                for (int q = 0; q < NW; ++q) {
                    const int k = lane + 32 * q;
                    if (k >= 1 && k <= N - 1) C[(b0 + r) * (N - 1) + k - 1] = c[q];
                }
            }
        }
        int32_t e = 0;
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            const int32_t t = __reduce_add_sync(kFull, sq[r]);
            e = lane == r ? t : e;
        }
        if (lane < rows) E[b0 + lane] = e;
        if constexpr (ROWS == 1) break;
    }
}

template <int NW, int ROWS>
static void launch_energy_warps(const uint32_t* seqs, int N, int64_t B, int32_t* d_E, int32_t* d_C,
                                cudaStream_t stream) {
    constexpr int per_block = kEnergyThreads / 32 * ROWS;
    int64_t blocks = (B + per_block - 1) / per_block;
    if (ROWS > 1) blocks = std::min(blocks, static_cast<int64_t>(lcapi::sm_count()) * 8);  // 64 warps on every SM
    energy_warp_kernel<NW, ROWS><<<static_cast<unsigned>(blocks), kEnergyThreads, 0, stream>>>(seqs, N, B, d_E, d_C);
}

// E alone takes a thread per sequence from 8 NW^2 sequences per SM on: a
// thread's chain grows with NW^2, and below that it outlasts the warps'
// (us, warps / threads: N = 64 1.8 / 2.4 at B = 4,000, 3.0 / 2.5 at 20,000;
// N = 120 2.9 / 3.8 at 10,000, 5.5 / 5.9 at 40,000, 24 / 18 at 300,000;
// N = 256 12 / 17 at 40,000, 25 / 24 at 100,000).  A warp takes one sequence
// up to 48 per SM, at seven and eight words up to 192, and four at a time from
// there (E and C, one / four: N = 64 1.94 / 2.05 at B = 6,000, 2.17 / 2.06 at
// 9,728; N = 128 2.35 / 2.60 and 2.89 / 2.69; N = 256 3.57 / 4.62 at 6,000,
// 8.1 / 8.7 at 20,000, 11.4 / 11.6 at 30,000, 21.0 / 20.0 at 60,000).
template <int NW>
static cudaError_t launch_energy_w(const uint64_t* d_seqs, int N, int64_t B, int32_t* d_E,
                                   int32_t* d_C, cudaStream_t stream) {
    const uint32_t* seqs = reinterpret_cast<const uint32_t*>(d_seqs);
    const int64_t sms = lcapi::sm_count();
    if (d_C == nullptr && B > sms * 8 * NW * NW) {
        const int64_t blocks = (B + kEnergyThreads - 1) / kEnergyThreads;
        energy_thread_kernel<NW><<<static_cast<unsigned>(blocks), kEnergyThreads, 0, stream>>>(seqs, N, B, d_E);
    } else if (B <= sms * (NW >= 7 ? 192 : 48)) {
        launch_energy_warps<NW, 1>(seqs, N, B, d_E, d_C, stream);
    } else {
        launch_energy_warps<NW, 4>(seqs, N, B, d_E, d_C, stream);
    }
    return cudaGetLastError();
}

cudaError_t launch_energy(const uint64_t* d_seqs, int N, int64_t B, int32_t* d_E, int32_t* d_C,
                          cudaStream_t stream) {
    switch ((N + 31) / 32) {
        case 1: return launch_energy_w<1>(d_seqs, N, B, d_E, d_C, stream);
        case 2: return launch_energy_w<2>(d_seqs, N, B, d_E, d_C, stream);
        case 3: return launch_energy_w<3>(d_seqs, N, B, d_E, d_C, stream);
        case 4: return launch_energy_w<4>(d_seqs, N, B, d_E, d_C, stream);
        case 5: return launch_energy_w<5>(d_seqs, N, B, d_E, d_C, stream);
        case 6: return launch_energy_w<6>(d_seqs, N, B, d_E, d_C, stream);
        case 7: return launch_energy_w<7>(d_seqs, N, B, d_E, d_C, stream);
        default: return launch_energy_w<8>(d_seqs, N, B, d_E, d_C, stream);
    }
}

}  // namespace lgpu
