// Dense products of the prompt pass ("KV cache <- LM(x)", first line of Algorithm 1) on the fifth-generation
// tensor cores of sm_100a: tcgen05.mma over pairs of CTAs (cta_group::2) with the accumulators in tensor memory,
// operands staged in shared memory by TMA, and the operation that follows a product fused into its epilogue.
//
// A block of prompt positions (up to PF_ROWS) goes through a weight matrix in one product
//     Y[m][n] = sum_k X[m][k] W[n][k],   m < rows positions, n < N weight rows.
// X arrives as two bf16 matrices, a high part and a low part (x = hi + lo, as everywhere in this library: fp32
// activations lose nothing), both multiplied into the same fp32 accumulator: 4 m n k floating-point operations.
//
// What bounds it.  From about 128 positions up the tensor cores (the weights of a block are fetched once from
// HBM and then from L2).  A pair of CTAs computes a tile of 256 positions x 256 weight rows: each CTA holds its
// own 128 positions (hi and lo) and half of the weight rows, so a k block of 64 costs a CTA 48 KB of shared-memory
// fill per 1024 tensor-core cycles.  One CTA per tile of 128 x 128 (the previous form) needed 48 KB per 512
// cycles and 2.7 times the L2 traffic per weight byte, and was bound by that.
//
// Accumulation.  The tensor core adds into its fp32 accumulator with truncation, so the error of one accumulator
// grows with the products added to it (1e-3 absolute at K = 14336 with sums of size 10).  A product is therefore cut
// into chunks of 512 k; a chunk accumulates in one of two 256-column tensor-memory buffers while the epilogue warps
// add the other one, already complete, to fp32 registers (round to nearest).  Each buffer sees 64 additions.
//
// Work division.  Tiles in excess of whole waves over the CTA pairs are divided by chunks, not by tiles
// ("stream-K"): every pair gets the same number of chunks (+- 1).  A tile cut between pairs is summed by the pair
// that holds its last chunk, in a fixed order; the others publish their partial sums first thing in the kernel, and
// a pair only ever waits for pairs with a lower number, so no assumption about co-residency is made.  With whole
// tiles a 1024-position block of the 8B shape would fill 83 % of its waves, a 500-position one 60 %.
//
// Roles of a CTA: warp 0 issues the TMA loads, warp 1 allocates the tensor memory and (in the first CTA of the pair)
// issues the MMAs, warps 4..11 read the accumulators and run the epilogue.  Every wait is bounded; on expiry an
// error word is set, the roles leave their loops, the tensor memory is released and the kernel ends.
#pragma once

#include "kernels.cuh"
#include "stream.cuh"

namespace ada {
namespace dg {

using namespace st;

constexpr int PF_ROWS = 2048;  // prompt positions of one block: 32 layers of launches and ragged waves are paid once per
                               // block; activations of a block stay below the size of the L2 cache per product
constexpr int BM = 128;        // positions one CTA of a pair holds (UMMA M = 256 over the pair)
constexpr int BNH = 128;       // weight rows one CTA of a pair holds (UMMA N = 256)
constexpr int TM = 2 * BM, TN = 2 * BNH;
constexpr int BK = 64;         // k elements per stage: one 128-byte swizzle row
constexpr int CK = 8;          // k blocks per accumulator chunk
constexpr int STAGES = 4;
constexpr int GEPI_WARPS = 8;  // epilogue warps: lane quadrant (warp % 4) x half of the tile's columns
constexpr int GTHREADS = 128 + 32 * GEPI_WARPS;
// The register file is divided per warpgroup at launch (168 a thread); the epilogue warps hold 128 sums each and take
// what the first warpgroup (TMA, MMA, two idle warps) gives back: (56 + 224 + 224) x 128 = 168 x 384.
constexpr int GREGS_ISSUE = 40, GREGS_EPI = 232;
constexpr int A_BYTES = BM * BK * 2, B_BYTES = BNH * BK * 2, STAGE_BYTES = 2 * A_BYTES + B_BYTES;
constexpr int TMEM_COLS = 512; // two accumulator buffers of 256 fp32 columns
constexpr unsigned long long DENSE_WAIT_NS = 2000000000ull;
constexpr size_t GPART_WARP = 128 * 32 * sizeof(float);           // partial sums of one epilogue warp
constexpr size_t GPART_CTA = GEPI_WARPS * GPART_WARP;

struct DSmem {   // must start on a 1024-byte boundary (swizzle pattern)
    alignas(1024) unsigned char stage[STAGES][STAGE_BYTES];   // [X.hi 128 x 64 | X.lo 128 x 64 | W 128 x 64], rows of 128 B
    alignas(8) unsigned long long full[STAGES], empty[STAGES], acc_full[2], acc_empty[2];
    uint32_t tmem_base;
    int abort;
};
constexpr size_t DSMEM_BYTES = sizeof(DSmem) + 1024;
static_assert(STAGE_BYTES % 1024 == 0 && A_BYTES % 1024 == 0, "operand tiles must start on 1024-byte boundaries");
static_assert(DSMEM_BYTES <= 232448, "exceeds the 227 KB of shared memory a block may use");

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t map_to_cta(const void *p, uint32_t rank) {   // shared::cluster address of the same object in another CTA
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(s32(p)), "r"(rank));
    return a;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_at(uint32_t cluster_addr) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// TMA load into this CTA's shared memory, completing on a barrier that may live in the other CTA of the pair.
__device__ __forceinline__ void tma_load_2d_pair(void *dst, const CUtensorMap *map, int c0, int c1, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2 [%0], [%1, {%2, %3}], [%4];" ::"r"(s32(dst)),
                 "l"(map), "r"(c0), "r"(c1), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory matrix descriptor of a K-major tile whose rows are 128 bytes, 128-byte swizzled (the layout
// a TMA box of 64 bf16 x rows leaves): start address / 16 in bits 0-13, leading byte offset / 16 in bits
// 16-29 (1: not used by swizzled K-major tiles), stride byte offset / 16 in bits 32-45 (1024 bytes from one
// group of eight rows to the next), descriptor version 1 in bits 46-47, swizzle mode 2 (128 bytes) in bits 61-63.
__device__ __forceinline__ unsigned long long smem_desc(uint32_t saddr) {
    return (unsigned long long)((saddr >> 4) & 0x3fffu) | (1ull << 16) | (64ull << 32) | (1ull << 46) | (2ull << 61);
}
// Instruction descriptor of kind::f16: fp32 accumulator (bits 4-5 = 1), bf16 A and B (bits 7-9 and 10-12 = 1),
// both K-major (bits 15, 16 = 0), N / 8 in bits 17-22, M / 16 in bits 24-28.
template <int M, int N> struct Idesc { static constexpr uint32_t v = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24); };

__device__ __forceinline__ void umma_pair(uint32_t d_tmem, unsigned long long adesc, unsigned long long bdesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(Idesc<TM, TN>::v), "r"(accumulate)
        : "memory");
}
// The barrier at this offset of both CTAs is arrived on once every MMA issued so far by this thread has completed.
__device__ __forceinline__ void umma_commit_pair(unsigned long long *bar) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(s32(bar)), "h"((uint16_t)3)
                 : "memory");
}
// 32 consecutive fp32 columns of this warp's 32 tensor-memory lanes.
__device__ __forceinline__ void tmem_ld32(uint32_t (&v)[32], uint32_t addr) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                   "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
                   "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
                   "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
                 : "r"(addr));
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// 16-byte load from L2 that the compiler keeps in program order (register pressure stays what the source says).
__device__ __forceinline__ float4 ld_cg_inorder(const float4 *p) {
    float4 v;
    asm volatile("ld.global.cg.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p) : "memory");
    return v;
}

template <typename SM> __device__ __forceinline__ bool dwait(SM *sm, int *err, unsigned long long *bar, uint32_t parity) {
    if (mbar_try(bar, parity)) return true;
    unsigned long long t0 = 0;
    for (uint32_t it = 0;; ++it) {
        if (mbar_try(bar, parity)) return true;
        if ((it & 255u) == 0) {
            if (*(volatile int *)&sm->abort) return false;
            const unsigned long long t = gtime();
            if (t0 == 0) t0 = t;
            else if (t - t0 > DENSE_WAIT_NS) {
                atomicCAS(err, 0, ERR_TIMEOUT_MBAR);
                *(volatile int *)&sm->abort = 1;
                return false;
            }
        }
    }
}

// Division of one product's tiles over the CTA pairs (chosen on the host, plan_dense).  Tiles are numbered with the
// position tile fastest, so that the pairs at work at one time share weight rows.  The last sk_tiles tiles are divided
// by chunks over sk_pairs pairs, the others are dealt out whole.
struct GemmPlan { int mt, tiles, chunks, pairs, sk_tiles, sk_pairs; };

struct Seg { int tile, c0, c1; };   // chunks [c0, c1) of a tile
struct Sched {
    GemmPlan g;
    int pair, t_last, t_first, u_end, u_beg, i, phase;   // phase 0: last shared tile, 1: the whole ones between, 2: whole tiles, 3: first shared tile, 4: end
    __device__ __forceinline__ int unit(int p) const { return (int)((long long)g.sk_tiles * g.chunks * p / g.sk_pairs); }
    __device__ __forceinline__ Sched(const GemmPlan &g_, int pair_) : g(g_), pair(pair_), t_last(0), t_first(0), u_end(0), u_beg(0), i(0), phase(2) {
        if (g.sk_tiles > 0 && pair < g.sk_pairs) {
            u_beg = unit(pair);
            u_end = unit(pair + 1);
            if (u_end > u_beg) {
                t_first = u_beg / g.chunks;
                t_last = (u_end - 1) / g.chunks;
                phase = 0;
            }
        }
        if (phase == 2) i = pair;
    }
    // Pieces another pair waits for come first, the piece that waits for others comes last.
    __device__ __forceinline__ bool next(Seg &s) {
        const int base = g.tiles - g.sk_tiles;
        if (phase == 0) {
            phase = 1;
            i = t_last - 1;
            if (t_last != t_first || u_end < (t_last + 1) * g.chunks) {
                s.tile = base + t_last;
                s.c0 = t_last == t_first ? u_beg - t_last * g.chunks : 0;
                s.c1 = u_end - t_last * g.chunks;
                return true;
            }
        }
        if (phase == 1) {
            if (i > t_first) {
                s.tile = base + i--;
                s.c0 = 0;
                s.c1 = g.chunks;
                return true;
            }
            phase = 2;
            i = pair;
        }
        if (phase == 2) {
            if (i < base) {
                s.tile = i;
                s.c0 = 0;
                s.c1 = g.chunks;
                i += g.pairs;
                return true;
            }
            phase = 3;
        }
        if (phase == 3) {
            phase = 4;
            if (u_end > u_beg && (t_first != t_last || u_end == (t_last + 1) * g.chunks)) {
                s.tile = base + t_first;
                s.c0 = u_beg - t_first * g.chunks;
                s.c1 = g.chunks;
                return true;
            }
        }
        return false;
    }
};

constexpr int EPI_STORE = 0, EPI_ADD = 1, EPI_QKV = 2, EPI_SWIGLU = 3;
struct GemmArgs {
    GemmPlan plan;
    int rows, K;
    int nw[3], nt[3];             // weight rows and tile columns of the up to three matrices (QKV: q, k, v; SwiGLU: gate, up)
    float *Y; int ldy;            // STORE, ADD
    __nv_bfloat16 *hi, *lo;       // QKV: scaled queries [rows][nw[0]]; SwiGLU: activations [rows][nw[0]]
    const float *cs;              // QKV: cos, sin [rows][hd / 2][2]
    int layer, seq, pos0;         // QKV: rows are positions pos0 .. of sequence seq
    float *part;                  // partial sums of tiles cut between pairs
    unsigned *flag;               // [CTA][epilogue warp]: launch number of the partial sums published last
    unsigned epoch;
    int *err;
};

// a pair of fp32 values as bf16 high parts and low parts
__device__ __forceinline__ void split2(float a, float b, uint32_t &hi, uint32_t &lo) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    const __nv_bfloat162 l = __floats2bfloat162_rn(a - __low2float(h), b - __high2float(h));
    hi = *reinterpret_cast<const uint32_t *>(&h);
    lo = *reinterpret_cast<const uint32_t *>(&l);
}

// Y[m][n] = or += acc (columns [n, n + 128) of row m; ldy a multiple of 4, N arbitrary).
template <bool ADD> __device__ __forceinline__ void epi_rows(const float (&acc)[128], float *__restrict__ y, int left) {
#pragma unroll
    for (int j = 0; j < 128; j += 4) {
        if (j + 4 <= left) {
            float4 o = make_float4(acc[j], acc[j + 1], acc[j + 2], acc[j + 3]);
            float4 *p = reinterpret_cast<float4 *>(y + j);
            if (ADD) { const float4 r = *p; o.x += r.x; o.y += r.y; o.z += r.z; o.w += r.w; }
            *p = o;
        } else {
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (j + e < left) y[j + e] = (ADD ? y[j + e] : 0.f) + acc[j + e];
        }
    }
}

// One row's q, k or v features [n, n + 128) of its matrix: q and k are rotated, q is scaled and split into bf16 high and
// low parts, k and v go to the cache row of the position (16-byte chunks xor-swizzled, see kv_swz).
template <int HD> __device__ __forceinline__ void epi_qkv(const Ctx &c, const GemmArgs &a, float (&acc)[128], int which, int n, int m) {
    const int pos = a.pos0 + m;
#pragma unroll
    for (int h = 0; h < 128 / HD; ++h) {
        if (n + h * HD >= a.nw[which]) break;
        const int head = n / HD + h;
        if (which < 2) {
            const float *cs = a.cs + (size_t)m * HD;
#pragma unroll
            for (int i = 0; i < HD / 2; i += 2) {
                const float4 t = *reinterpret_cast<const float4 *>(cs + 2 * i);
                float &x0 = acc[h * HD + i], &x1 = acc[h * HD + i + HD / 2], &y0 = acc[h * HD + i + 1], &y1 = acc[h * HD + i + 1 + HD / 2];
                const float a0 = x0 * t.x - x1 * t.y, a1 = x1 * t.x + x0 * t.y, b0 = y0 * t.z - y1 * t.w, b1 = y1 * t.z + y0 * t.w;
                x0 = a0; x1 = a1; y0 = b0; y1 = b1;
            }
        }
        if (which == 0) {
            const float scale = rsqrtf((float)HD);
            const size_t o = (size_t)m * a.nw[0] + head * HD;
#pragma unroll
            for (int j = 0; j < HD; j += 8) {
                uint4 hi, lo;
                const float *v = acc + h * HD + j;
                split2(v[0] * scale, v[1] * scale, hi.x, lo.x);
                split2(v[2] * scale, v[3] * scale, hi.y, lo.y);
                split2(v[4] * scale, v[5] * scale, hi.z, lo.z);
                split2(v[6] * scale, v[7] * scale, hi.w, lo.w);
                *reinterpret_cast<uint4 *>(a.hi + o + j) = hi;
                *reinterpret_cast<uint4 *>(a.lo + o + j) = lo;
            }
        } else {
            __nv_bfloat16 *dst = reinterpret_cast<__nv_bfloat16 *>(c.kv_pool) + kv_index(c, a.seq, a.layer, which - 1, head, pos);
#pragma unroll
            for (int j = 0; j < HD; j += 8) {
                uint4 o;
                const float *v = acc + h * HD + j;
                __nv_bfloat162 b[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) b[e] = __floats2bfloat162_rn(v[2 * e], v[2 * e + 1]);
                o = *reinterpret_cast<const uint4 *>(b);
                *reinterpret_cast<uint4 *>(dst + (((j >> 3) ^ (pos & c.kv_swz)) << 3)) = o;
            }
        }
    }
}

// 64 gate and 64 up features of one row -> SwiGLU activation, split into bf16 high and low parts.
__device__ __forceinline__ void epi_swiglu(const float (&acc)[128], __nv_bfloat16 *__restrict__ hi, __nv_bfloat16 *__restrict__ lo) {
#pragma unroll
    for (int j = 0; j < 64; j += 8) {
        float s[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const float g = acc[j + e];
            s[e] = g / (1.0f + expf(-g)) * acc[64 + j + e];
        }
        uint4 h, l;
        split2(s[0], s[1], h.x, l.x);
        split2(s[2], s[3], h.y, l.y);
        split2(s[4], s[5], h.z, l.z);
        split2(s[6], s[7], h.w, l.w);
        *reinterpret_cast<uint4 *>(hi + j) = h;
        *reinterpret_cast<uint4 *>(lo + j) = l;
    }
}

// mapXhi / mapXlo: 2-D maps over the bf16 matrices [rows][K] (box 64 x 128); mapW0..2: over the weight matrices [N][K]
// (box 64 x 128); all 128-byte swizzled, zero fill outside.  K a multiple of 64.  Grid: 2 x plan.pairs CTAs.
template <int EPI, int HD>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(GTHREADS, 1)
k_dense_gemm(const __grid_constant__ CUtensorMap mapXhi, const __grid_constant__ CUtensorMap mapXlo, const __grid_constant__ CUtensorMap mapW0,
             const __grid_constant__ CUtensorMap mapW1, const __grid_constant__ CUtensorMap mapW2, const __grid_constant__ Ctx c,
             const __grid_constant__ GemmArgs a) {
    extern __shared__ unsigned char dsm_raw[];
    DSmem *sm = reinterpret_cast<DSmem *>(dsm_raw + ((1024u - (s32(dsm_raw) & 1023u)) & 1023u));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    const int pair = blockIdx.x >> 1, nkb = a.K / BK;
    if (threadIdx.x == 0) {
        for (int i = 0; i < STAGES; ++i) { mbar_init(&sm->full[i], 1); mbar_init(&sm->empty[i], 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(&sm->acc_full[i], 1); mbar_init(&sm->acc_empty[i], 2 * GEPI_WARPS); }
        sm->abort = 0;
        fence_mbar_init();
        fence_proxy_async();
    }
    __syncthreads();
    if (warp == 1) {   // tensor memory for the accumulators: allocated, and later released, by this warp of both CTAs
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s32(&sm->tmem_base)), "r"(TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();   // the other CTA's barriers exist and its tensor memory is allocated
    tc_fence_after();
    const uint32_t tmem = *(volatile uint32_t *)&sm->tmem_base;

    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(GREGS_ISSUE));
        if (warp == 0 && lane == 0) {
            Sched sch(a.plan, pair);
            Seg s;
            int it = 0;
            bool ok = true;
            while (ok && sch.next(s)) {
                const int tm = s.tile % a.plan.mt, tn = s.tile / a.plan.mt, m0 = tm * TM + (int)rank * BM;
                const CUtensorMap *mw = &mapW0;
                int n0;
                if (EPI == EPI_SWIGLU) {
                    n0 = tn * BNH;
                    if (rank) mw = &mapW1;
                } else {
                    int t = tn;
                    if (EPI == EPI_QKV && t >= a.nt[0]) {
                        t -= a.nt[0];
                        mw = &mapW1;
                        if (t >= a.nt[1]) { t -= a.nt[1]; mw = &mapW2; }
                    }
                    n0 = t * TN + (int)rank * BNH;
                }
                const int kb1 = min(s.c1 * CK, nkb);
                for (int kb = s.c0 * CK; kb < kb1; ++kb, ++it) {
                    const int st = it % STAGES;
                    ok = dwait(sm, a.err, &sm->empty[st], ((it / STAGES) & 1) ^ 1);
                    if (!ok) break;
                    if (rank == 0) mbar_expect_tx(&sm->full[st], 2u * STAGE_BYTES);   // both CTAs' tiles complete on the first CTA's barrier
                    const uint32_t bar = map_to_cta(&sm->full[st], 0);
                    tma_load_2d_pair(sm->stage[st], &mapXhi, kb * BK, m0, bar);
                    tma_load_2d_pair(sm->stage[st] + A_BYTES, &mapXlo, kb * BK, m0, bar);
                    tma_load_2d_pair(sm->stage[st] + 2 * A_BYTES, mw, kb * BK, n0, bar);
                }
            }
        }
        if (warp == 1 && lane == 0 && rank == 0) {
            Sched sch(a.plan, pair);
            Seg s;
            int it = 0, ch = 0;
            bool ok = true;
            while (ok && sch.next(s)) {
                for (int cc = s.c0; ok && cc < s.c1; ++cc, ++ch) {
                    const int b = ch & 1, kb1 = min((cc + 1) * CK, nkb);
                    ok = dwait(sm, a.err, &sm->acc_empty[b], ((ch >> 1) & 1) ^ 1);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t acc = tmem + (uint32_t)(b * TN);
                    uint32_t add = 0;
                    for (int kb = cc * CK; kb < kb1; ++kb, ++it) {
                        const int st = it % STAGES;
                        ok = dwait(sm, a.err, &sm->full[st], (it / STAGES) & 1);
                        if (!ok) break;
                        tc_fence_after();
                        const unsigned long long ahi = smem_desc(s32(sm->stage[st])), alo = smem_desc(s32(sm->stage[st] + A_BYTES)),
                                                 w = smem_desc(s32(sm->stage[st] + 2 * A_BYTES));
#pragma unroll
                        for (int k = 0; k < BK / 16; ++k) {   // 32 bytes further along the swizzled row per K = 16 step
                            umma_pair(acc, ahi + 2 * k, w + 2 * k, add);
                            umma_pair(acc, alo + 2 * k, w + 2 * k, 1u);
                            add = 1u;
                        }
                        umma_commit_pair(&sm->empty[st]);   // the stage is free in both CTAs once these MMAs have read it
                    }
                    umma_commit_pair(&sm->acc_full[b]);
                }
            }
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(GREGS_EPI));
        // epilogue: warp w may read the 32 lanes 32 (w % 4) .. of the tensor memory; lane = position within the CTA's 128
        const int q = warp & 3, h = (warp - 4) >> 2, ew = warp - 4;
        const uint32_t t_lane = tmem + ((uint32_t)(q * 32) << 16);
        Sched sch(a.plan, pair);
        Seg s;
        int ch = 0;
        bool ok = true;
        while (ok && sch.next(s)) {
            const int tm = s.tile % a.plan.mt, tn = s.tile / a.plan.mt;
            const int mw = tm * TM + (int)rank * BM + q * 32, m = mw + lane;   // first row of the warp, row of the lane
            const bool live = mw < a.rows;                                     // the same in every lane, and in the same warp of every pair
            float acc[128];
#pragma unroll
            for (int j = 0; j < 128; ++j) acc[j] = 0.f;
            for (int cc = s.c0; cc < s.c1; ++cc, ++ch) {
                const int b = ch & 1;
                ok = dwait(sm, a.err, &sm->acc_full[b], (ch >> 1) & 1);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                tc_fence_after();
                if (live) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        uint32_t v[32];
                        const int col = EPI == EPI_SWIGLU ? (j >> 1) * BNH + h * 64 + (j & 1) * 32 : h * 128 + j * 32;
                        tmem_ld32(v, t_lane + (uint32_t)(b * TN + col));
                        tmem_ld_wait();
#pragma unroll
                        for (int e = 0; e < 32; ++e) acc[32 * j + e] += __uint_as_float(v[e]);
#pragma unroll
                        for (int e = 0; e < 32; ++e) asm volatile("" : "+f"(acc[32 * j + e]));
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_at(map_to_cta(&sm->acc_empty[b], 0));
            }
            if (!ok || !live) continue;
            if (s.c1 < a.plan.chunks) {   // another pair finishes this tile
                float4 *o = reinterpret_cast<float4 *>(reinterpret_cast<unsigned char *>(a.part) + (size_t)(2 * pair + (int)rank) * GPART_CTA + ew * GPART_WARP) + lane;
#pragma unroll
                for (int j = 0; j < 32; ++j) __stcg(o + 32 * j, make_float4(acc[4 * j], acc[4 * j + 1], acc[4 * j + 2], acc[4 * j + 3]));
                __threadfence();
                __syncwarp();
                if (lane == 0) asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(a.flag + (2 * pair + (int)rank) * GEPI_WARPS + ew), "r"(a.epoch) : "memory");
                continue;
            }
            if (s.c0 > 0) {   // add what the pairs before this one computed of the tile: nearest first
                const int u0 = (s.tile - (a.plan.tiles - a.plan.sk_tiles)) * a.plan.chunks;
                for (int p = pair - 1; ok && p >= 0 && sch.unit(p + 1) > u0; --p) {
                    const int cta = 2 * p + (int)rank;
                    const unsigned *f = a.flag + cta * GEPI_WARPS + ew;
                    unsigned v;
                    const unsigned long long t0 = gtime();
                    for (;;) {
                        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(f) : "memory");
                        if (v == a.epoch) break;
                        if (*(volatile int *)&sm->abort) { ok = false; break; }
                        if (gtime() - t0 > DENSE_WAIT_NS) {
                            atomicCAS(a.err, 0, ERR_TIMEOUT_MBAR);
                            *(volatile int *)&sm->abort = 1;
                            ok = false;
                            break;
                        }
                    }
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                    const float4 *in = reinterpret_cast<const float4 *>(reinterpret_cast<const unsigned char *>(a.part) + (size_t)cta * GPART_CTA + ew * GPART_WARP) + lane;
#pragma unroll
                    for (int j0 = 0; j0 < 32; j0 += 8) {   // eight loads in flight: more would not fit beside the sums
                        float4 r[8];
#pragma unroll
                        for (int j = 0; j < 8; ++j) r[j] = ld_cg_inorder(in + 32 * (j0 + j));
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            const int e = 4 * (j0 + j);
                            acc[e] += r[j].x; acc[e + 1] += r[j].y; acc[e + 2] += r[j].z; acc[e + 3] += r[j].w;
                        }
                    }
                }
                if (!ok) continue;
            }
            if (m >= a.rows) continue;
            if constexpr (EPI == EPI_STORE || EPI == EPI_ADD) {
                const int n = tn * TN + h * 128;
                if (n < a.nw[0]) epi_rows<EPI == EPI_ADD>(acc, a.Y + (size_t)m * a.ldy + n, a.nw[0] - n);
            } else if constexpr (EPI == EPI_QKV) {
                int t = tn, which = 0;
                if (t >= a.nt[0]) {
                    t -= a.nt[0];
                    which = 1;
                    if (t >= a.nt[1]) { t -= a.nt[1]; which = 2; }
                }
                epi_qkv<HD>(c, a, acc, which, t * TN + h * 128, m);
            } else {
                const int n = tn * BNH + h * 64;
                if (n < a.nw[0]) epi_swiglu(acc, a.hi + (size_t)m * a.nw[0] + n, a.lo + (size_t)m * a.nw[0] + n);
            }
        }
    }
    if (*(volatile int *)&sm->abort) {   // copies already issued may still be landing: give them time before the block's memory goes
        const unsigned long long t0 = gtime();
        while (gtime() - t0 < 200000ull) __nanosleep(1000);
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    cluster_sync();   // neither CTA leaves while the other may still signal its barriers or use its tensor memory
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    }
}

// Embeds a block of prompt tokens and tabulates the rotary cos / sin of its positions.  One CTA per row.
__global__ void __launch_bounds__(256) k_pf_embed(Ctx c, const __nv_bfloat16 *__restrict__ embed, float rope_base, int seq, int pos0,
                                                  float *__restrict__ resid, float *__restrict__ cs) {
    const int r = blockIdx.x, pos = pos0 + r, half = c.hd / 2;
    const __nv_bfloat16 *e = embed + (size_t)c.tokens[(size_t)seq * c.max_seq + pos] * c.d;
    for (int i = threadIdx.x * 8; i < c.d; i += 256 * 8) {
        float v[8];
        Vec16<__nv_bfloat16>::load(e + i, v);
        float4 *o = reinterpret_cast<float4 *>(resid + (size_t)r * c.d + i);
        o[0] = make_float4(v[0], v[1], v[2], v[3]);
        o[1] = make_float4(v[4], v[5], v[6], v[7]);
    }
    for (int i = threadIdx.x; i < half; i += 256) {
        double sn, co;
        sincos((double)pos * pow((double)rope_base, -2.0 * i / c.hd), &sn, &co);
        cs[((size_t)r * half + i) * 2] = (float)co;
        cs[((size_t)r * half + i) * 2 + 1] = (float)sn;
    }
}

// The last row of the prompt becomes row 0 of the per-operation buffers, where the LM head reads it.
__global__ void k_pf_last(Ctx c, const float *__restrict__ resid, int row, int seq, int pos) {
    for (int i = threadIdx.x; i < c.d; i += blockDim.x) c.resid[i] = resid[(size_t)row * c.d + i];
    if (threadIdx.x == 0) {
        c.rt->seq[0] = seq; c.rt->pos[0] = pos; c.rt->first_layer[0] = 0;
        c.rt->n_rows = 1;
    }
}

// RMSNorm and split in one pass: x = resid[r] / sqrt(mean(resid[r]^2) + eps) * g -> high and low parts.  One CTA
// (256 threads) per row, four elements per access; K a multiple of 64.
__global__ void __launch_bounds__(256) k_norm_split_rows(const float *__restrict__ X, int K, const __nv_bfloat16 *__restrict__ gain,
                                                         float eps, __nv_bfloat16 *__restrict__ hi, __nv_bfloat16 *__restrict__ lo) {
    const int r = blockIdx.x;
    __shared__ float red[8];
    const float4 *x = reinterpret_cast<const float4 *>(X + (size_t)r * K);
    float ss = 0.f;
    for (int i = threadIdx.x; i < K / 4; i += 256) {
        const float4 v = x[i];
        ss = fmaf(v.x, v.x, fmaf(v.y, v.y, fmaf(v.z, v.z, fmaf(v.w, v.w, ss))));
    }
    ss = warp_sum(ss);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
    __syncthreads();
    float tot = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) tot += red[w];
    const float rstd = 1.0f / sqrtf(tot / K + eps);
    for (int i = threadIdx.x; i < K / 4; i += 256) {
        const float4 v = x[i];
        const uint2 gq = reinterpret_cast<const uint2 *>(gain)[i];
        uint2 h, l;
        split2(v.x * rstd * __uint_as_float(gq.x << 16), v.y * rstd * __uint_as_float(gq.x & 0xffff0000u), h.x, l.x);
        split2(v.z * rstd * __uint_as_float(gq.y << 16), v.w * rstd * __uint_as_float(gq.y & 0xffff0000u), h.y, l.y);
        reinterpret_cast<uint2 *>(hi + (size_t)r * K)[i] = h;
        reinterpret_cast<uint2 *>(lo + (size_t)r * K)[i] = l;
    }
}

// fp32 rows X[r][ldx] (r < rows) -> the two bf16 matrices [128][K] the dense GEMM reads: high part and low part
// (x = hi + lo); rows >= `rows` are zero.  One block per row.
__global__ void k_split_rows(const float *__restrict__ X, int ldx, int rows, int K, __nv_bfloat16 *__restrict__ hi, __nv_bfloat16 *__restrict__ lo) {
    const int r = blockIdx.x;
    for (int k = threadIdx.x; k < K; k += blockDim.x) {
        const float v = r < rows ? X[(size_t)r * ldx + k] : 0.f;
        const __nv_bfloat16 h = __float2bfloat16_rn(v);
        hi[(size_t)r * K + k] = h;
        lo[(size_t)r * K + k] = __float2bfloat16_rn(v - __bfloat162float(h));
    }
}

// Causal attention of a block of prompt rows on the tensor cores (mma.sync m16n8k16, bf16 cache).  One warp owns
// one 16-row query tile: 16 / GROUP consecutive prompt positions x the GROUP q heads of one kv head; a block of
// four warps shares the K and V rows of 64 cache positions at a time, copied into shared memory exactly as the
// cache stores them (16-byte chunks xor-swizzled by position: conflict-free for ldmatrix).  Queries are rotated
// already, scaled and split into bf16 high / low parts (epi_qkv), the probabilities are split in registers, so nothing but the cache itself is rounded to bf16.  Online softmax in position order; the context
// is not split, the result goes straight to the next product's
// input, split into high and low parts.
template <int HD, int GROUP>
__global__ void __launch_bounds__(128) k_pf_attn_mma(Ctx c, int layer, int rows, int seq, int pos0, const __nv_bfloat16 *__restrict__ qhi,
                                                     const __nv_bfloat16 *__restrict__ qlo, __nv_bfloat16 *__restrict__ ohi, __nv_bfloat16 *__restrict__ olo) {
    constexpr int KSQ = HD / 16, NT = HD / 8, PPW = 16 / GROUP, TILE = 64;
    __shared__ __align__(128) unsigned char sK[TILE * HD * 2], sV[TILE * HD * 2];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, kvh = blockIdx.y;
    const int r_blk = blockIdx.x * 4 * PPW, r_w = r_blk + warp * PPW;   // first row of the block / of this warp
    const int pos_blk_max = pos0 + min(r_blk + 4 * PPW, rows) - 1;
    const __nv_bfloat16 *pool = reinterpret_cast<const __nv_bfloat16 *>(c.kv_pool);
    // ---- this lane's parts of the query fragments: rows lane/4 and lane/4 + 8 of the tile
    int lim[2];
    uint32_t ah[KSQ][4], al[KSQ][4];
#pragma unroll
    for (int rh = 0; rh < 2; ++rh) {
        const int row = (lane >> 2) + 8 * rh, r = r_w + row / GROUP, g = row % GROUP;
        const bool live = r < rows;
        lim[rh] = live ? pos0 + r : -1;
        const size_t o = ((size_t)min(r, rows - 1) * c.nq + kvh * GROUP + g) * HD;
#pragma unroll
        for (int ks = 0; ks < KSQ; ++ks)
#pragma unroll
            for (int kh = 0; kh < 2; ++kh) {
                const int j = ks * 16 + kh * 8 + 2 * (lane & 3);
                ah[ks][rh + 2 * kh] = live ? *reinterpret_cast<const uint32_t *>(qhi + o + j) : 0u;
                al[ks][rh + 2 * kh] = live ? *reinterpret_cast<const uint32_t *>(qlo + o + j) : 0u;
            }
    }
    const int lim_w = r_w < rows ? pos0 + min(r_w + PPW, rows) - 1 : -1;   // last position any row of this warp sees (the same in every lane)
    float m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.f, 0.f};
    float o[NT][4];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int i = 0; i < 4; ++i) o[nt][i] = 0.f;
    for (int t0 = 0; t0 <= pos_blk_max; t0 += TILE) {
        __syncthreads();   // the previous tile has been used
        for (int i = threadIdx.x; i < TILE * (HD / 8); i += 128) {
            const int t = i / (HD / 8), ch = i - t * (HD / 8), p = t0 + t;
            uint4 kq = make_uint4(0, 0, 0, 0), vq = kq;
            if (p <= pos_blk_max) {
                kq = *reinterpret_cast<const uint4 *>(pool + kv_index(c, seq, layer, 0, kvh, p) + ch * 8);
                vq = *reinterpret_cast<const uint4 *>(pool + kv_index(c, seq, layer, 1, kvh, p) + ch * 8);
            }
            *reinterpret_cast<uint4 *>(sK + (size_t)t * HD * 2 + ch * 16) = kq;
            *reinterpret_cast<uint4 *>(sV + (size_t)t * HD * 2 + ch * 16) = vq;
        }
        __syncthreads();
        for (int sl = 0; sl < TILE / 16; ++sl) {
            const int p0 = t0 + 16 * sl;
            if (p0 > lim_w) break;   // nothing further in this tile is visible to this warp (uniform per warp)
            // ---- scores of the 16 positions p0 .. p0 + 15
            float sh[2][4], sl_[2][4];
#pragma unroll
            for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                for (int i = 0; i < 4; ++i) { sh[nt][i] = 0.f; sl_[nt][i] = 0.f; }
            const int id = lane >> 3;
            {
                const int pl = 16 * sl + (lane & 7) + 8 * (id >> 1);
                const unsigned char *krow = sK + pl * (HD * 2);
#pragma unroll
                for (int ks = 0; ks < KSQ; ++ks) {
                    uint32_t kf[4];
                    ldmatrix_x4(kf, krow + ((((2 * ks) | (id & 1)) ^ (pl & 7)) << 4));
                    mma16816(sh[0], ah[ks], kf[0], kf[1]);
                    mma16816(sh[1], ah[ks], kf[2], kf[3]);
                    mma16816(sl_[0], al[ks], kf[0], kf[1]);
                    mma16816(sl_[1], al[ks], kf[2], kf[3]);
                }
            }
            float s[2][4];
#pragma unroll
            for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int pos = p0 + 8 * nt + 2 * (lane & 3) + (i & 1);
                    s[nt][i] = pos <= lim[i >> 1] ? sh[nt][i] + sl_[nt][i] : -INFINITY;
                }
            // ---- online softmax
            uint32_t ph[4], plo[4];
#pragma unroll
            for (int rh = 0; rh < 2; ++rh) {
                float mx = fmaxf(fmaxf(s[0][2 * rh], s[0][2 * rh + 1]), fmaxf(s[1][2 * rh], s[1][2 * rh + 1]));
                mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
                mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
                const float mn = fmaxf(m_run[rh], mx);
                float corr = 1.f, p[4] = {0.f, 0.f, 0.f, 0.f};
                if (mn != -INFINITY) {
                    corr = __expf(m_run[rh] - mn);
                    p[0] = __expf(s[0][2 * rh] - mn); p[1] = __expf(s[0][2 * rh + 1] - mn);
                    p[2] = __expf(s[1][2 * rh] - mn); p[3] = __expf(s[1][2 * rh + 1] - mn);
                }
                m_run[rh] = mn;
                l_run[rh] = l_run[rh] * corr + ((p[0] + p[1]) + (p[2] + p[3]));
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) { o[nt][2 * rh] *= corr; o[nt][2 * rh + 1] *= corr; }
                const __nv_bfloat162 h0 = __floats2bfloat162_rn(p[0], p[1]), h1 = __floats2bfloat162_rn(p[2], p[3]);
                const __nv_bfloat162 l0 = __floats2bfloat162_rn(p[0] - __low2float(h0), p[1] - __high2float(h0));
                const __nv_bfloat162 l1 = __floats2bfloat162_rn(p[2] - __low2float(h1), p[3] - __high2float(h1));
                ph[rh] = *reinterpret_cast<const uint32_t *>(&h0);
                ph[2 + rh] = *reinterpret_cast<const uint32_t *>(&h1);
                plo[rh] = *reinterpret_cast<const uint32_t *>(&l0);
                plo[2 + rh] = *reinterpret_cast<const uint32_t *>(&l1);
            }
            // ---- o += P V
            {
                const int pl = 16 * sl + (lane & 7) + 8 * (id & 1);
                const unsigned char *vrow = sV + pl * (HD * 2);
#pragma unroll
                for (int np = 0; np < NT / 2; ++np) {
                    uint32_t vf[4];
                    ldmatrix_x4_trans(vf, vrow + ((((2 * np) | (id >> 1)) ^ (pl & 7)) << 4));
                    mma16816(o[2 * np], ph, vf[0], vf[1]);
                    mma16816(o[2 * np + 1], ph, vf[2], vf[3]);
                    mma16816(o[2 * np], plo, vf[0], vf[1]);
                    mma16816(o[2 * np + 1], plo, vf[2], vf[3]);
                }
            }
        }
    }
#pragma unroll
    for (int rh = 0; rh < 2; ++rh) {
        l_run[rh] += __shfl_xor_sync(0xffffffffu, l_run[rh], 1);
        l_run[rh] += __shfl_xor_sync(0xffffffffu, l_run[rh], 2);
        const int row = (lane >> 2) + 8 * rh, r = r_w + row / GROUP, g = row % GROUP;
        if (r < rows) {
            const size_t o_at = ((size_t)r * c.nq + kvh * GROUP + g) * HD;
            const float inv = 1.0f / l_run[rh];
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                uint32_t h, l;
                split2(o[nt][2 * rh] * inv, o[nt][2 * rh + 1] * inv, h, l);
                *reinterpret_cast<uint32_t *>(ohi + o_at + nt * 8 + 2 * (lane & 3)) = h;
                *reinterpret_cast<uint32_t *>(olo + o_at + nt * 8 + 2 * (lane & 3)) = l;
            }
        }
    }
}

}  // namespace dg
}  // namespace ada
