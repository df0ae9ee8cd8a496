// mts_kernels.cuh -- Memetic-Tabu (Algorithm 1 / Algorithm 3) and batched
// tabu search (Algorithm 2 / Algorithm 4) kernels, templated on the word
// count, tracing and the skew-symmetric restriction (Sec. II.C).  One warp
// runs one replica: its population lives in the warp's slice of shared
// memory (K packed sequences and their energies), followed by its tabu search's
// correlations, self-convolution and spins; the neighbours' keys and the tabu
// list are in registers.  Replicas never synchronise with each other;
// the only cross-replica state is the optional global termination flag.
// mts.cu instantiates the unrestricted kernels, mts_skew.cu the restricted
// ones and mts_resume.cu the resumable ones (both kinds), so each
// translation unit compiles one family.
#pragma once

#include <cuda_runtime.h>

#include "capi_util.h"
#include "kernels.h"
#include "replica.cuh"

namespace lgpu {

// One warp per CTA: replicas and searches share nothing, so a CTA's end should
// free no more than its own slot, and few of them spread over the SMs (a lone
// search of N = 201 takes 73 us on an SM of its own and 87 us beside three
// others; 5,000 of them, of uneven length, 331 us instead of 394).
// Sixteen CTAs per SM leave 128 registers a thread.  Without a bound the
// compiler aims at more warps than the workloads put on an SM and squeezes the
// short steps, and it takes too many registers for sixteen at six words (cycles
// a step, without / with the bound, one warp alone on a sub-partition and four:
// N = 64 199 / 190 and 502 / 497, N = 92 294 / 297 and 658 / 650, N = 120 411 /
// 331 and 795 / 751, N = 160 363 / 366 and 870 / 868, N = 192 419 / 434 and
// 1,142 / 1,027).
constexpr int kMinBlocks = 16;
// Seven and eight words take up to 255 registers while at most eight replicas
// fall on an SM, which is all those leave room for (128 / 255 registers, one
// GB300: 152 replicas of N = 256 x 20,000 steps 5.95 / 5.12 ms, 608 of N = 200
// 5.85 / 4.69, 1,216 of N = 256 8.11 / 7.41); with more, 16 warps on an SM win
// (a step of 2,432 at N = 256: 1,356 / 1,429 cycles).  Fewer words gain little or
// lose (cycles a step, 128 / 255 registers, a lone warp: N = 192 434 / 426, N = 160
// 366 / 398, N = 120 331 / 334), and so do searches (100 of N = 201 70.5 / 71.8 us,
// 5,000 307 / 322; of N = 256 98 / 93 and 435 / 437): those keep 128.
constexpr int kFewBlocks = 8;
template <int NW>
inline bool few_replicas(int64_t n) {
    return NW >= 7 && n <= static_cast<int64_t>(lcapi::sm_count()) * kFewBlocks;
}

// Grid of n one-warp CTAs (n <= 2^32), and the CTA's index in it.
inline dim3 warp_grid(int64_t n) {
    constexpr int64_t row = int64_t{1} << 30;
    return n <= row ? dim3(static_cast<unsigned>(n)) : dim3(static_cast<unsigned>(row), static_cast<unsigned>((n + row - 1) / row));
}
__device__ __forceinline__ int64_t warp_index() {
    return static_cast<int64_t>(blockIdx.y) * gridDim.x + blockIdx.x;
}

template <int NW, bool TRACE, bool SKEW, int BLOCKS>
__global__ void __launch_bounds__(32, BLOCKS) mts_kernel(const MtsArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x;
    const int64_t r = warp_index();
    if (r >= a.replicas) return;

    uint32_t* pop = reinterpret_cast<uint32_t*>(smem);
    int32_t* popE = reinterpret_cast<int32_t*>(pop + a.K * NW);
    int32_t* Cs = popE + a.K;
    ReplicaCfg cfg;
    cfg.N = a.N;
    cfg.K = a.K;
    cfg.p_comb_u32 = a.p_comb_u32;
    cfg.p_mut_u32 = a.p_mut_u32;
    cfg.replace_policy = a.replace_policy;
    cfg.target_E = a.target_E;
    cfg.max_generations = a.max_generations;
    cfg.max_steps = a.max_steps;
    cfg.max_iter = a.max_iter;
    cfg.variant = a.variant;
    cfg.inst = static_cast<uint32_t>(a.first_instance + static_cast<uint64_t>(r));
    cfg.key = philox_key(a.seed);
    int4* trace = a.d_trace ? a.d_trace + r * a.trace_cap : nullptr;
    replica_run<NW, TRACE, SKEW>(cfg, pop, popE, Cs, trace, a.trace_cap, a.d_glf, a.d_out + r, lane);
}

// Memetic-Tabu with resumable state: each replica starts from its initial
// population or from its record in ra.d_state, runs to its stop condition
// and writes its record back (population, energies, best, counters).  The
// draws are addressed by (instance, generation, index), so a run continued
// from a record at a generation boundary equals the uninterrupted run.  A
// record of another run (N, K, variant, seed or instance) is left untouched
// and the replica reports LABS_RUN_BADSTATE.
template <int NW, bool SKEW, int BLOCKS>
__global__ void __launch_bounds__(32, BLOCKS) mts_resume_kernel(const ResumeArgs ra) {
    extern __shared__ __align__(16) unsigned char smem[];
    const MtsArgs& a = ra.m;
    const int lane = threadIdx.x;
    const int64_t r = warp_index();
    if (r >= a.replicas) return;

    uint32_t* pop = reinterpret_cast<uint32_t*>(smem);
    int32_t* popE = reinterpret_cast<int32_t*>(pop + a.K * NW);
    int32_t* Cs = popE + a.K;
    ReplicaCfg cfg;
    cfg.N = a.N;
    cfg.K = a.K;
    cfg.p_comb_u32 = a.p_comb_u32;
    cfg.p_mut_u32 = a.p_mut_u32;
    cfg.replace_policy = a.replace_policy;
    cfg.target_E = a.target_E;
    cfg.max_generations = a.max_generations;
    cfg.max_steps = a.max_steps;
    cfg.max_iter = a.max_iter;
    cfg.variant = a.variant;
    cfg.inst = static_cast<uint32_t>(a.first_instance + static_cast<uint64_t>(r));
    cfg.key = philox_key(a.seed);

    unsigned char* rec = ra.d_state + static_cast<size_t>(r) * ra.state_bytes;
    ResumeHeader* h = reinterpret_cast<ResumeHeader*>(rec);
    uint32_t* hpop = reinterpret_cast<uint32_t*>(rec + sizeof(ResumeHeader));
    int32_t* hpopE = reinterpret_cast<int32_t*>(hpop + a.K * NW);
    ReplicaState<NW> st;
    if (ra.resume) {
        const bool match = h->N == a.N && h->K == a.K && h->variant == a.variant &&
                           h->instance == cfg.inst && h->seed == a.seed;
        if (!match) {
            if (lane == 0) {
                labs_device_result* o = a.d_out + r;
                for (int w = 0; w < LABS_MAX_W; ++w) o->seq[w] = 0;
                o->E = -1;
                o->status = LABS_RUN_BADSTATE;
                o->generations = 0;
                o->steps = 0;
                o->trace_len = 0;
            }
            return;
        }
        for (int x = lane; x < a.K * NW; x += 32) pop[x] = hpop[x];
        for (int x = lane; x < a.K; x += 32) popE[x] = hpopE[x];
#pragma unroll
        for (int w = 0; w < NW; ++w) st.best[w] = h->best[w];
        st.E_best = h->E_best;
        st.status = LABS_RUN_BUDGET;
        st.g = h->g;
        st.steps = h->steps;
        __syncwarp();
    } else {
        replica_init<NW, SKEW>(cfg, pop, popE, st, lane);
    }
    int64_t trace_len = 0;
    while (!replica_should_stop<NW>(cfg, st, a.d_glf))
        replica_generation<NW, false, SKEW>(cfg, st, pop, popE, Cs, nullptr, 0, trace_len, a.d_glf, lane);
    replica_store_result<NW>(st, 0, a.d_out + r, lane);
    __syncwarp();
    for (int x = lane; x < a.K * NW; x += 32) hpop[x] = pop[x];
    for (int x = lane; x < a.K; x += 32) hpopE[x] = popE[x];
    if (lane < 2 * LABS_MAX_W) {
        uint32_t v = 0;
#pragma unroll
        for (int w = 0; w < NW; ++w) v = (lane == w) ? st.best[w] : v;
        h->best[lane] = v;
    }
    if (lane == 0) {
        h->E_best = st.E_best;
        h->status = st.status;
        h->g = st.g;
        h->steps = st.steps;
        h->N = a.N;
        h->K = a.K;
        h->variant = a.variant;
        h->instance = cfg.inst;
        h->seed = a.seed;
    }
}

template <int NW, bool TRACE, bool SKEW>
__global__ void __launch_bounds__(32, kMinBlocks) tabu_kernel(const TabuArgs a) {
    __shared__ __align__(16) int32_t Cs[kTabuScratchInts<NW>];
    const int lane = threadIdx.x;
    const int64_t b = warp_index();
    if (b >= a.B) return;
    const int N = a.N;
    const uint2 key = philox_key(a.seed);
    const uint32_t inst = static_cast<uint32_t>(a.first_instance + static_cast<uint64_t>(b));
    constexpr int ROW = (NW + 1) & ~1;  // 32-bit words per row: whole 64-bit words
    uint32_t seq[NW];
    load_seq<NW>(reinterpret_cast<const uint32_t*>(a.d_start) + b * ROW, seq);
#pragma unroll
    for (int w = 0; w < NW; ++w) seq[w] &= word_lowmask(w, N);  // bits >= N are ignored
    if constexpr (SKEW) skew_complete<NW>(seq, N);              // the free half decides
    const int nmov = SKEW ? (N + 1) / 2 : N;
    int max_iter = a.max_iter;
    if (max_iter < 0) {
        const uint4 d = draw4(key, inst, a.generation, 1u, kPurposeGen);
        max_iter = nmov / 2 + rand_int(0, nmov, d.w);
    }
    int4* trace = a.d_trace ? a.d_trace + b * a.trace_cap : nullptr;
    int64_t trace_len = 0;
    const bool fix = (a.variant & LABS_VARIANT_FIX_FIRST_SPIN) != 0;
    const uint2 draws = step_draws(key, inst, a.generation, 1 + lane);
    TabuOut to;
    if constexpr (SKEW) {
        to = fix ? tabu_search_skew<NW, TRACE, true>(seq, N, key, inst, a.generation, max_iter, -1, draws,
                                                     Cs, trace, a.trace_cap, trace_len, lane)
                 : tabu_search_skew<NW, TRACE, false>(seq, N, key, inst, a.generation, max_iter, -1, draws,
                                                      Cs, trace, a.trace_cap, trace_len, lane);
    } else {
        to = fix ? tabu_search<NW, TRACE, true>(seq, N, key, inst, a.generation, max_iter, -1, draws,
                                                Cs, trace, a.trace_cap, trace_len, lane)
                 : tabu_search<NW, TRACE, false>(seq, N, key, inst, a.generation, max_iter, -1, draws,
                                                 Cs, trace, a.trace_cap, trace_len, lane);
    }
    if (lane < ROW) {
        uint32_t v = 0;
#pragma unroll
        for (int w = 0; w < NW; ++w) v = (lane == w) ? seq[w] : v;
        reinterpret_cast<uint32_t*>(a.d_best)[b * ROW + lane] = v;
    }
    if (lane == 0) {
        a.d_bestE[b] = to.E_best;
        if (a.d_steps) a.d_steps[b] = to.steps;
    }
}

// The largest population and scratch of one warp fit the dynamic shared memory
// that every launch may take, so the launches below set no limit of their kernels
// (see allow_cta_smem).
static_assert(LABS_MAX_K * (2 * LABS_MAX_W + 1) * 4 + tabu_scratch_bytes(2 * LABS_MAX_W) + 15 <= 48 * 1024,
              "a warp's shared memory");

template <int NW, bool TRACE, bool SKEW, int BLOCKS>
cudaError_t launch_mts_b(const MtsArgs& a, cudaStream_t stream) {
    mts_kernel<NW, TRACE, SKEW, BLOCKS><<<warp_grid(a.replicas), 32, a.smem_per_warp, stream>>>(a);
    return cudaGetLastError();
}

template <int NW, bool TRACE, bool SKEW>
cudaError_t launch_mts_t(const MtsArgs& a, cudaStream_t stream) {
    if constexpr (NW >= 7 && !TRACE)
        if (few_replicas<NW>(a.replicas)) return launch_mts_b<NW, TRACE, SKEW, kFewBlocks>(a, stream);
    return launch_mts_b<NW, TRACE, SKEW, kMinBlocks>(a, stream);
}

// 32-bit words per sequence in registers, for launches and searches.  A step's
// work grows with them, so every count has its kernel (one word against two, one
// N = 24 instance of 2,000 generations: 5.72 ms against 6.60; seven against
// eight, 5,000 searches at N = 201: 309 us against 343).
inline int word_count(int N) { return (N + 31) / 32; }

// Words per member of a resumable record, and of the kernels that read it: part
// of the record's layout, so N <= 32 runs two words there and N = 193..224 eight.
inline int record_words(int N) { return N <= 64 ? 2 : N <= 96 ? 3 : N <= 128 ? 4 : N <= 160 ? 5 : N <= 192 ? 6 : 8; }

template <bool SKEW>
cudaError_t launch_mts_family(const MtsArgs& a, cudaStream_t stream) {
    const bool tr = a.d_trace != nullptr;
    switch (word_count(a.N)) {
        case 1: return tr ? launch_mts_t<1, true, SKEW>(a, stream) : launch_mts_t<1, false, SKEW>(a, stream);
        case 2: return tr ? launch_mts_t<2, true, SKEW>(a, stream) : launch_mts_t<2, false, SKEW>(a, stream);
        case 3: return tr ? launch_mts_t<3, true, SKEW>(a, stream) : launch_mts_t<3, false, SKEW>(a, stream);
        case 4: return tr ? launch_mts_t<4, true, SKEW>(a, stream) : launch_mts_t<4, false, SKEW>(a, stream);
        case 5: return tr ? launch_mts_t<5, true, SKEW>(a, stream) : launch_mts_t<5, false, SKEW>(a, stream);
        case 6: return tr ? launch_mts_t<6, true, SKEW>(a, stream) : launch_mts_t<6, false, SKEW>(a, stream);
        case 7: return tr ? launch_mts_t<7, true, SKEW>(a, stream) : launch_mts_t<7, false, SKEW>(a, stream);
        default: return tr ? launch_mts_t<8, true, SKEW>(a, stream) : launch_mts_t<8, false, SKEW>(a, stream);
    }
}

template <int NW, bool SKEW, int BLOCKS>
cudaError_t launch_resume_b(const ResumeArgs& a, cudaStream_t stream) {
    mts_resume_kernel<NW, SKEW, BLOCKS><<<warp_grid(a.m.replicas), 32, a.m.smem_per_warp, stream>>>(a);
    return cudaGetLastError();
}

template <int NW, bool SKEW>
cudaError_t launch_resume_w(const ResumeArgs& a, cudaStream_t stream) {
    if constexpr (NW >= 7)
        if (few_replicas<NW>(a.m.replicas)) return launch_resume_b<NW, SKEW, kFewBlocks>(a, stream);
    return launch_resume_b<NW, SKEW, kMinBlocks>(a, stream);
}

template <bool SKEW>
cudaError_t launch_resume_family(const ResumeArgs& a, cudaStream_t stream) {
    switch (record_words(a.m.N)) {
        case 2: return launch_resume_w<2, SKEW>(a, stream);
        case 3: return launch_resume_w<3, SKEW>(a, stream);
        case 4: return launch_resume_w<4, SKEW>(a, stream);
        case 5: return launch_resume_w<5, SKEW>(a, stream);
        case 6: return launch_resume_w<6, SKEW>(a, stream);
        default: return launch_resume_w<8, SKEW>(a, stream);
    }
}

template <int NW, bool SKEW>
cudaError_t launch_tabu_w(const TabuArgs& a, cudaStream_t stream) {
    if (a.d_trace)
        tabu_kernel<NW, true, SKEW><<<warp_grid(a.B), 32, 0, stream>>>(a);
    else
        tabu_kernel<NW, false, SKEW><<<warp_grid(a.B), 32, 0, stream>>>(a);
    return cudaGetLastError();
}

template <bool SKEW>
cudaError_t launch_tabu_family(const TabuArgs& a, cudaStream_t stream) {
    switch (word_count(a.N)) {
        case 1: return launch_tabu_w<1, SKEW>(a, stream);
        case 2: return launch_tabu_w<2, SKEW>(a, stream);
        case 3: return launch_tabu_w<3, SKEW>(a, stream);
        case 4: return launch_tabu_w<4, SKEW>(a, stream);
        case 5: return launch_tabu_w<5, SKEW>(a, stream);
        case 6: return launch_tabu_w<6, SKEW>(a, stream);
        case 7: return launch_tabu_w<7, SKEW>(a, stream);
        default: return launch_tabu_w<8, SKEW>(a, stream);
    }
}

}  // namespace lgpu
