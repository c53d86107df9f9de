// Stand-alone launch of the weight-streaming GEMM phase (test and measurement hook): the same
// producer / consumer code as the persistent decode kernel, one phase, plain epilogues.
#pragma once

#include "stream.cuh"

namespace ada {

// fp32 activations X[cols][K] -> fragment layout (high/low bf16 split), the last block padded with zeros.
__global__ void k_xfrag_pack(const float *__restrict__ X, int K, int cols, __nv_bfloat16 *__restrict__ out) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= (K + st::KC - 1) / st::KC * st::KC) return;
    for (int c = 0; c < st::MAX_COLS; ++c) st::xfrag_store(out, k, c, c < cols && k < K ? X[(size_t)c * K + k] : 0.f);
}

struct ProbeEpilogue {
    float *Y;
    int ldy, mode, rows;
    __device__ __forceinline__ void pre(int, int, int, int) const {}
    __device__ __forceinline__ void operator()(int, bool act, int tile, int row, int col, float d0, float d1) const {
        const int n = tile * 16 + row;
        if (act && n < rows) Y[(size_t)col * ldy + n] = mode == 0 ? d0 : d0 / (1.0f + expf(-d0)) * d1;
    }
};

// How a launch parks weight stages: at most `most` per warp; the activations are fetched `hold_ns` nanoseconds late, so that as many land before them.
struct ProbeParking {
    int most;
    unsigned long long hold_ns;
};

// mode 0: Y[col][n] = sum_k W[n][k] X[col][k]                       (N rows)
// mode 1: Y[col][n] = silu(g) * u, g = W[n].X, u = W[half + n].X     (half = N/2 rows of each)
// PARK: as the decode kernel of one column tile, with tensor memory for parked stages; err[1] counts them.
template <bool PARK>
__global__ void __launch_bounds__(st::THREADS, 1)
k_gemm_probe(const CUtensorMap *__restrict__ W, int N, int K, int mode, const uint4 *__restrict__ X, float *__restrict__ Y,
             int ldy, int cols, int repeat, int *err, unsigned long long *part, ProbeParking parking, unsigned long long wait_ns) {
    extern __shared__ unsigned char smem_raw[];
    st::Smem *sm = st::smem_base(smem_raw);
    const int warp = threadIdx.x >> 5;
    st::smem_init(sm);
    if (PARK && warp == st::CONS_WARPS) {
        st::park_alloc(sm);
        tc_fence_before();
    }
    __syncthreads();
    if (PARK) tc_fence_after();
    st::Shared S{sm, err, Trace{nullptr, nullptr, 0}, 0, wait_ns};
    const int cta = blockIdx.x, G = gridDim.x;
    st::Gemm g;
    g.N = N; g.K = K; g.pair = mode == 1 ? 2 : 1; g.half = mode == 1 ? N / 2 : 0;
    // tiles split between CTAs need a grid-wide meeting between products: only for a single product
    g.split = repeat == 1 && part != nullptr;
    const st::Plan pl = st::make_plan(g, cta, G);
    const st::Cols cols_used((1u << cols) - 1u);
    st::Rings r;
    if (warp == st::CONS_WARPS) {
        const uint64_t pol = st::policy_evict_first();
        for (int it = 0; it < repeat; ++it) st::gemm_produce_w(S, pl, W, nullptr, g.half, r, pol);
    } else if (warp == st::CONS_WARPS + 1) {
        const uint64_t pol = st::policy_evict_last();
        const auto hold = [&]() {
            if (parking.hold_ns == 0) return;
            const unsigned long long t0 = st::gtime();
            while (st::gtime() - t0 < parking.hold_ns) __nanosleep(100);
            __syncwarp();
        };
        for (int it = 0; it < repeat; ++it) st::gemm_produce_x(S, pl, X, cols_used, r, pol, st::NoHook(), hold);
    } else {
        const ProbeEpilogue epi{Y, ldy, mode, mode == 0 ? N : g.half};
        for (int it = 0; it < repeat; ++it) {
            st::gemm_consume<PARK>(S, pl, cols_used, (1u << cols) - 1u, part, 1u, cta, r, epi, parking.most);
            st::bar_consumers();   // the exchange area is free for the next product
        }
        if (PARK && (threadIdx.x & 31) == 0 && r.parked) atomicAdd(err + 1, r.parked);
    }
    if (PARK) tc_fence_before();
    st::settle_on_abort(S);
    if (PARK && warp == st::CONS_WARPS) {
        __syncwarp();
        tc_fence_after();
        st::park_free(sm);
    }
}

}  // namespace ada
