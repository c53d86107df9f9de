// Weight-streaming primitives of the persistent decode kernel (sm_100a).
//
// The decode step is bound by HBM bandwidth: every weight byte is read once per pass and used
// for a few tokens (eight columns, or 24).  The pieces here keep the memory pipe full:
//   * weights reach shared memory through TMA tensor copies (cp.async.bulk.tensor, one 16 KB box
//     of 16 rows x 512 k per instruction, 128-byte swizzled) issued by a dedicated producer warp
//     into a ring of stages guarded by mbarriers; the producer runs ahead of the consumers across
//     phase boundaries, because the weight sequence of a CTA does not depend on activations.
//     (Sixteen 1 KB untiled bulk copies per stage reached only 3.6 TB/s on B200: the copy engine
//     spends about 40 ns per request whatever its size, so requests have to be large.)
//   * activations arrive through a second, small ring in the register layout the tensor-core
//     instruction wants, already split into a bf16 high part and a bf16 low part, so that
//     fp32 activations lose nothing: W.x = W.hi(x) + W.lo(x) with fp32 accumulation;
//   * eight consumer warps multiply with mma.sync m16n8k16 (weights are the 16-row operand, eight
//     tokens are the columns of a tile).  The tensor cores are used as a cheap way to issue
//     the multiply-adds; the bound stays the memory system.
//   * all CTAs of the persistent grid meet at a counter-based grid barrier between phases.
// Every wait is bounded: on expiry an error word is set and all later waits fall through.
//
// This file and mega.cuh are compiled once per number of token columns: ADA_TILES column tiles of eight, in the namespaces
// ADA_ST and ADA_MG.  One tile (st, mg) is the kernel for up to eight columns; three (st3, mg3) carry several sequences with
// several tokens each over one weight stream.  A column's numbers are formed alike in both.
#ifndef ADA_TILES
#define ADA_TILES 1
#define ADA_ST st
#define ADA_MG mg
#endif
#if (ADA_TILES == 1 && !defined(ADA_STREAM_1)) || (ADA_TILES == 3 && !defined(ADA_STREAM_3))
#if ADA_TILES == 1
#define ADA_STREAM_1
#else
#define ADA_STREAM_3
#endif

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "decode_args.cuh"
#include "tmem.cuh"

namespace ada {
namespace ADA_ST {

constexpr int KC = 512;                          // k elements per stage
constexpr int KSTEPS = KC / 16;                  // mma k-steps per stage
constexpr int TILE_N = 16;                       // weight rows per stage (mma M)
constexpr int KG = KC / 64;                      // 64-element (128-byte) k groups per stage
constexpr int W_STAGE = TILE_N * KC * 2;         // 16384: [k group][row][128 B, 16-byte chunks xor-swizzled by row%8]
constexpr int X_STAGE = KSTEPS * 32 * 16;        // 16384: [column pair][k-step][8 slots][b0.hi b1.hi b0.lo b1.lo]
constexpr int TILES = ADA_TILES;                 // token column tiles
// weight / activation stages in flight per CTA.  (One tile: 10 / 2 measured the same.  Three: a chunk's activations alone may
// take three stages, and the next chunk's must be on their way.)
constexpr int NW = TILES == 1 ? 9 : 6;
constexpr int NX = TILES == 1 ? 3 : 6;
constexpr int CONS_WARPS = 8;
constexpr int CONS_THREADS = CONS_WARPS * 32;
constexpr int THREADS = CONS_THREADS + 64;       // + weight producer warp + activation producer warp
constexpr int MAX_COLS = 8 * TILES;              // tokens per pass (one tile: mma N)
constexpr int MAX_SEQS = 8;                      // sequences per launch
constexpr int RED_BYTES = CONS_WARPS * 2 * TILES * 128 * 4;  // cross-warp reduction scratch (two matrices per warp)
constexpr int X_BLOCK = TILES * X_STAGE;         // activations of one chunk in global memory, all columns
constexpr int SCRATCH_BYTES = 33 * 1024;         // consumers' scratch: GEMM reduction, or the attention phase's buffers

constexpr int ERR_TIMEOUT_MBAR = 1, ERR_TIMEOUT_GRID = 2;
constexpr unsigned long long WAIT_NS_DEFAULT = 2000000000ull;   // a single wait gives up after two seconds unless told otherwise
constexpr unsigned long long SHORT_LIMIT_NS = 1000000ull;       // a limit below this is checked at every poll, not every 64th or 128th

// ---------------------------------------------------------------- GEMM shapes and their division

// One GEMM as seen by the whole grid: Y[n][col] = sum_k W[n][k] X[k][col].
//   pair == 1: N rows, tiles of 16 rows (the last may be ragged).
//   pair == 2: W holds two stacked matrices of `half` rows each (gate over up), or they are two tensors; a tile is rows
//              [16 t, 16 t + 16) of both, and the epilogue sees both accumulators.
// The weights are described by a rank-3 tensor map over the row-major [N][K] matrix, dimensions
// (64 elements, N rows, K/64 groups) with strides (2 B, 2K B, 128 B) and box (64, 16, 8): one box
// is a stage.  Rows past N and k groups past K read as zeros.  K must be a multiple of 64.
struct Gemm {
    int N, K, pair, half;
    int split;   // tiles may be cut between two CTAs (needs an exchange area; see Plan)
    __host__ __device__ __forceinline__ int tiles() const { return pair == 2 ? half / TILE_N : (N + TILE_N - 1) / TILE_N; }
};

__host__ __device__ __forceinline__ void cta_tile_range(int T, int cta, int G, int &t0, int &t1) {
    if (cta >= G) { t0 = t1 = 0; return; }
    t0 = (int)((long long)T * cta / G);
    t1 = (int)((long long)T * (cta + 1) / G);
}
// ---------------------------------------------------------------- unit-balanced split of a GEMM
// With whole tiles some CTAs stream one tile more than the others (7 against 6 in the 8B gate-up
// GEMM) and the phase lasts as long as they do.  When g.split is set the work is instead measured in
// units of (tile, k chunk): CTA c takes the units [U c / C, U (c + 1) / C) of the tile-major order,
// so every CTA streams the same number of stages (+- one).  A tile cut by a CTA boundary is
// computed in two parts.  The CTA with its chunks from 0 (the head part, [0, kb)) meets them early
// in its k loop and publishes its partial sums as soon as they are complete; the CTA with the later
// chunks (the tail part, [ka, nch)) finishes them at the end of its loop, adds the published part
// (own + published, the published k-splits in index order: the sum does not depend on timing) and
// runs the epilogue.  All tiles of a CTA, partial ones included, form one group that shares every
// activation chunk; when the head part ends before the tail part begins they take turns in slot 0.
// GEMMs with fewer units per CTA than chunks per tile, or more tiles per CTA than consumer warps,
// keep whole tiles.  The plan is a function of the GEMM's shape and the grid only.
struct Plan {
    int t0, n;             // tiles t0 .. t0 + n - 1: whole ones, in groups of CONS_WARPS; or (split) one group of n slots, slot s
                           // holding tile t0 + s, except that
    short nch;             // k chunks of the GEMM
    short s0_own_k0;       //   slot 0 multiplies its own tile from chunk s0_own_k0 on (0: a whole tile),
    short s0_pub_k1;       //   and before that the chunks below s0_pub_k1 of tile t0 + n, to publish (0: none);
    short sl_k1;           //   the last slot (if not slot 0) multiplies chunks below sl_k1 only, to publish (nch: a whole tile)
    short ksp;             // split with a tail part: k-splits in which the CTA before publishes its head part
    unsigned char pair, split;
};
// the k-splits of a group of ng slots
__host__ __device__ __forceinline__ int group_ks(int ng) {
    int TS = 1;
    while (TS < ng) TS <<= 1;
    return CONS_WARPS / TS;
}
__host__ __device__ inline Plan make_plan(const Gemm &g, int cta, int C, bool with_ksp = true) {
    Plan p;
    p.pair = (unsigned char)g.pair;
    p.split = 0;
    p.t0 = p.n = 0;
    p.s0_own_k0 = p.s0_pub_k1 = p.ksp = 0;
    const int T = g.tiles(), nch = (g.K + KC - 1) / KC;
    p.nch = p.sl_k1 = (short)nch;
    if (cta < 0 || cta >= C) return p;
    // 32-bit arithmetic throughout (a 64-bit division costs hundreds of cycles); GEMMs whose unit
    // count times the CTA count does not fit keep whole tiles
    const unsigned U = (unsigned)T * (unsigned)nch;
    const bool fits = (unsigned long long)T * nch * (unsigned)(C + 1) < 0x7fffffffull;
    const unsigned L = (U + C - 1) / C;      // most units of one CTA; a run of L units touches <= (L + nch - 2) / nch + 1 tiles
    if (!g.split || !fits || U / C < (unsigned)nch || (L + nch - 2) / nch + 1 > (unsigned)CONS_WARPS) {
        int t1;
        cta_tile_range(T, cta, C, p.t0, t1);
        p.n = t1 - p.t0;
        return p;
    }
    p.split = 1;
    const unsigned u0 = U * (unsigned)cta / C, u1 = U * (unsigned)(cta + 1) / C;
    const int ta = (int)(u0 / nch), tb = (int)((u1 - 1) / nch);
    const int ka = (int)(u0 - ta * nch), kb = (int)((u1 - 1) - tb * nch) + 1;
    const bool has_tail = ka > 0, has_head = kb < nch;
    const bool shared = has_tail && has_head && kb <= ka;
    p.t0 = ta;
    p.n = tb - ta + 1;
    p.s0_own_k0 = (short)ka;
    if (shared) { p.s0_pub_k1 = (short)kb; p.n -= 1; }
    else if (has_head) p.sl_k1 = (short)kb;
    if (ka > 0 && with_ksp) p.ksp = (short)group_ks(make_plan(g, cta - 1, C, false).n);
    return p;
}
// the tile slot s of a split plan multiplies at chunk kc (-1: none)
__host__ __device__ __forceinline__ int plan_tile(const Plan &p, int s, int kc) {
    if (s == 0) return kc < p.s0_pub_k1 ? p.t0 + p.n : (kc >= p.s0_own_k0 ? p.t0 : -1);
    if (s == p.n - 1 && kc >= p.sl_k1) return -1;
    return p.t0 + s;
}

struct Smem {                                    // must start on a 1024-byte boundary (swizzle pattern)
    alignas(1024) unsigned char w[NW][W_STAGE];
    alignas(128) unsigned char x[NX][X_STAGE];
    alignas(16) unsigned char scratch[SCRATCH_BYTES];
    alignas(16) float vec[MAX_COLS];                   // per-column scalars (rstd, ...)
    alignas(8) unsigned long long w_full[NW], w_empty[NW], x_full[NX], x_empty[NX];
    alignas(16) int desc[3][TILES == 1 ? 24 : 44];                  // per-role copy of the step descriptor (persistent decode kernel)
    int abort;
    int bcast[8];
    unsigned trace_n;
    unsigned vec_seq;                             // phase for which vec[] holds the normalisation factors (see vec_wait)
    unsigned w_issued;                            // weight stages issued so far (see w_wait)
    uint32_t tmem;                                // base of this CTA's tensor memory (kernels that park weight stages there)
    unsigned long long t_booked;                  // CTA 0's activation producer: time up to which phases have been booked
    Plan plan[6];                                 // this CTA's share of every product of the program
};

// ---------------------------------------------------------------- PTX wrappers

__device__ __forceinline__ uint32_t s32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(unsigned long long *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(s32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(unsigned long long *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(s32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned long long *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(s32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try(unsigned long long *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(s32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool mbar_test(unsigned long long *bar, uint32_t parity) {   // (does not wait)
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(s32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ unsigned long long gtime() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ uint64_t policy_evict_first() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ uint64_t policy_evict_last() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    return p;
}
// Bulk copy global -> shared of `bytes` (multiple of 16; both addresses 16-byte aligned), completing
// on `bar` with the byte count.
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, unsigned long long *bar, uint64_t pol) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(s32(dst)),
        "l"(src), "r"(bytes), "r"(s32(bar)), "l"(pol)
        : "memory");
}
// TMA tensor copy of one box of a rank-3 map (coordinates innermost first) into shared memory.
__device__ __forceinline__ void tma_load_3d(void *dst, const CUtensorMap *map, int c0, int c1, int c2, unsigned long long *bar,
                                            uint64_t pol) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3, %4}], [%5], %6;" ::"r"(
            s32(dst)),
        "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(s32(bar)), "l"(pol)
        : "memory");
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async;" ::: "memory"); }
__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

__device__ __forceinline__ void ldmatrix_x4(uint32_t (&a)[4], const void *p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3])
                 : "r"(s32(p)));
}
__device__ __forceinline__ void ldmatrix_x4_at(uint32_t (&a)[4], uint32_t p) {   // (shared-memory address)
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]) : "r"(p));
}
__device__ __forceinline__ uint4 lds128(uint32_t p) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(p));
    return v;
}
__device__ __forceinline__ uint2 lds64(uint32_t p) {
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(p));
    return v;
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&a)[4], const void *p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3])
                 : "r"(s32(p)));
}
// d += a (16x16, row) * b (16x8, col), bf16 inputs, fp32 accumulation.
__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void bar_consumers() { asm volatile("bar.sync 1, %0;" ::"n"(CONS_THREADS) : "memory"); }

__device__ __forceinline__ uint32_t ld_acquire(const unsigned *p) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void red_release_add(unsigned *p, unsigned v) {
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// ---------------------------------------------------------------- bounded waits

struct Shared {            // what every role needs to wait safely
    Smem *sm;
    int *err;              // global error word (0 = fine)
    Trace tr;
    int tr_on;             // this block is currently tracing
    unsigned long long wait_ns;   // a single wait gives up after this many nanoseconds
};

constexpr int EV_PHASE_BEGIN = 1, EV_X0 = 2, EV_W0 = 3, EV_MAIN_END = 4, EV_EPI_END = 5, EV_WP_BEGIN = 6, EV_WP_END = 7,
              EV_ITEM = 8, EV_COMBINE = 9, EV_ARRIVE = 10, EV_ATT = 14;

__device__ __forceinline__ void trace(const Shared &S, int ev, int arg) {
    if (S.tr_on && S.tr.buf) {
        const unsigned i = atomicAdd(&S.sm->trace_n, 1u);
        if (i < S.tr.cap) {
            unsigned long long *e = S.tr.buf + 2 * ((size_t)blockIdx.x * S.tr.cap + i);
            e[0] = gtime();
            e[1] = ((unsigned long long)blockIdx.x << 32) | ((unsigned long long)(arg & 0xffff) << 8) | (unsigned)ev;
            S.tr.count[blockIdx.x] = i + 1;
        }
    }
}

__device__ __forceinline__ bool aborted(const Shared &S) { return *(volatile int *)&S.sm->abort != 0; }

__device__ __noinline__ void raise_error(const Shared &S, int code) {
    atomicCAS(S.err, 0, code);
    *(volatile int *)&S.sm->abort = 1;
}

// Wait for an mbarrier phase.  Once an error is raised (here or anywhere in the grid) every wait
// falls through at once: the roles then run to the end of their loops on whatever data is there,
// so that no warp is left behind at a block-level barrier, and the kernel ends.
// Called by whole warps.  The lanes poll for themselves and may leave at different turns, on a satisfied wait or on an error; what
// follows (fragment and tensor-memory loads, multiply-adds, votes) wants them together, so that is where the wait ends.
__device__ __forceinline__ void mbar_wait(const Shared &S, unsigned long long *bar, uint32_t parity) {
    if (!mbar_try(bar, parity)) {
        unsigned long long t0 = 0;
        for (uint32_t it = 0; !mbar_try(bar, parity); ++it) {
            if ((it & 127u) == 0 || S.wait_ns < SHORT_LIMIT_NS) {
                if (aborted(S)) break;
                if (*(volatile int *)S.err != 0) { *(volatile int *)&S.sm->abort = 1; break; }
                unsigned long long t = gtime();
                if (t0 == 0) t0 = t;
                else if (t - t0 > S.wait_ns) { raise_error(S, ERR_TIMEOUT_MBAR); break; }
            }
        }
    }
    __syncwarp();
}

// Epilogue operands are fetched while the weights stream, by 4-byte asynchronous copies into words of
// the scratch area that belong to one thread each (word k of pass p at [p][k][thread]) rather than into registers: a
// value held in a register across the main loop ties up the register file, and wherever the
// compiler has to move it the warp first waits for the load.  Each thread reads back only its own
// words, after cp_async_wait_all().  The exchange of partial sums uses the first 8 KB of the scratch area.
// (Passes beyond the stash, which only three column tiles have, fetch theirs when they need them.)
constexpr int STASH_OFFSET = RED_BYTES, STASH_WORDS = 3, STASH_PASSES = TILES == 1 ? 4 : 3;   // one tile: 8 tiles x 8 columns of 16 rows by 256 threads
static_assert(STASH_OFFSET + STASH_PASSES * STASH_WORDS * CONS_THREADS * 4 <= SCRATCH_BYTES, "stash exceeds the scratch area");
__device__ __forceinline__ uint32_t *stash_of(Smem *sm, int pass) {
    return reinterpret_cast<uint32_t *>(sm->scratch + STASH_OFFSET) + pass * (STASH_WORDS * CONS_THREADS) + threadIdx.x;
}
__device__ __forceinline__ void cp_async4(uint32_t *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(s32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }
// element n of a bf16 vector from the aligned 32-bit word that holds it
__device__ __forceinline__ float bf16_of_word(uint32_t w, int n) { return __uint_as_float((n & 1) ? (w & 0xffff0000u) : (w << 16)); }

// The consumers wait until the activation producer warp has left the per-column factors of phase
// `seq` in vec[] (it computes them while the first weight stages are being multiplied).
__device__ __forceinline__ void vec_wait(const Shared &S, unsigned seq) {
    unsigned long long t0 = 0;
    for (uint32_t it = 0;; ++it) {
        if (*(volatile unsigned *)&S.sm->vec_seq == seq) return;
        if ((it & 127u) == 127u || S.wait_ns < SHORT_LIMIT_NS) {
            if (aborted(S)) return;
            if (*(volatile int *)S.err != 0) { *(volatile int *)&S.sm->abort = 1; return; }
            unsigned long long t = gtime();
            if (t0 == 0) t0 = t;
            else if (t - t0 > S.wait_ns) { raise_error(S, ERR_TIMEOUT_MBAR); return; }
        }
    }
}

// Grid barrier on a monotonically increasing counter: arrive once per CTA, wait for `target`.
__device__ __forceinline__ void grid_arrive(unsigned *ctr) {
    // the release of the reduction orders this thread's earlier writes, and through the block-level
    // barrier before it those of the whole CTA; a separate fence before it only adds its latency.  What bulk copies read of
    // them is ordered by the proxy fence that a producer passes between its acquire -- of this counter, or of the record of a later
    // control point -- and its first copy (one here as well cost 0.2 us a phase).
    red_release_add(ctr, 1u);
}
__device__ __forceinline__ void grid_wait(const Shared &S, const unsigned *ctr, unsigned target) {
    unsigned long long t0 = 0;
    for (uint32_t it = 0;; ++it) {
        if (ld_acquire(ctr) >= target) return;
        if ((it & 63u) == 0 || S.wait_ns < SHORT_LIMIT_NS) {
            if (aborted(S)) return;
            if (*(volatile int *)S.err != 0) { *(volatile int *)&S.sm->abort = 1; return; }
            unsigned long long t = gtime();
            if (t0 == 0) t0 = t;
            else if (t - t0 > S.wait_ns) { raise_error(S, ERR_TIMEOUT_GRID); return; }
        }
        __nanosleep(32);
    }
}

// ---------------------------------------------------------------- activation layout

// Activations for a GEMM of depth K live in global memory as ceil(K/KC) blocks of X_BLOCK bytes.
// A block holds four sub-blocks of 4 KB per column tile, one per pair of token columns; in sub-block p, k-step s,
// slot j (0..7) holds 16 bytes: the mma B fragment (b0, b1) of the bf16 high parts, then of the
// bf16 low parts, for token column 2 p + j/4 and k = 16 s + 2 (j%4) + {0,1} (+8 for b1).  Lane l of
// a warp reads slot l%8 of sub-block l/8.  A pass that carries few tokens fetches only the
// sub-blocks of the column pairs in use: activations go through the same copy engine as the
// weights, and for a CTA holding two weight tiles a full block per chunk would be half as many
// bytes again as the weights.
__device__ __forceinline__ size_t xfrag_index(int k, int col) {   // index in 2-byte units of the high part
    const int chunk = k / KC, ks = (k % KC) >> 4, kk = k & 15;
    const int slot = (col & 1) * 4 + ((kk & 7) >> 1);
    return (((((size_t)chunk * (4 * TILES) + (col >> 1)) * KSTEPS + ks) * 8 + slot) << 3) + ((kk >> 3) << 1) + (kk & 1);
}
__device__ __forceinline__ void xfrag_store(__nv_bfloat16 *X, int k, int col, float v) {
    const __nv_bfloat16 hi = __float2bfloat16_rn(v);
    const __nv_bfloat16 lo = __float2bfloat16_rn(v - __bfloat162float(hi));
    const size_t i = xfrag_index(k, col);
    X[i] = hi;
    X[i + 4] = lo;
}
// two neighbouring elements k (even), k + 1
__device__ __forceinline__ void xfrag_store2(__nv_bfloat16 *X, int k, int col, float a, float b) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    const size_t i = xfrag_index(k, col);
    *reinterpret_cast<__nv_bfloat162 *>(X + i) = h;
    *reinterpret_cast<__nv_bfloat162 *>(X + i + 4) = __floats2bfloat162_rn(a - __low2float(h), b - __high2float(h));
}
__host__ __device__ inline size_t xfrag_bytes(int K) { return (size_t)((K + KC - 1) / KC) * X_BLOCK; }

// ---------------------------------------------------------------- GEMM phase

// The activation columns a pass fetches: column pairs cp0 .. cp0 + ncp - 1.
struct Cols {
    int cp0, ncp;
    __device__ __forceinline__ explicit Cols(unsigned mask) {   // the pairs spanning the columns set in `mask`
        cp0 = mask ? (__ffs(mask) - 1) >> 1 : 0;
        ncp = mask ? ((31 - __clz(mask)) >> 1) - cp0 + 1 : 1;
    }
    // k chunks whose activations share one 16 KB stage: 4 for one column pair, 2 for two, else 1.  (The
    // ring holds three stages; with one chunk per stage a CTA that owns two weight tiles would wait
    // for an activation copy every 96 KB of weights.)
    __device__ __forceinline__ int chunks() const { return ncp == 1 ? 4 : ncp == 2 ? 2 : 1; }   // a power of two
    // column tiles of four pairs, counted from the first pair fetched; each is an activation stage of its own where there are several
    __device__ __forceinline__ int tiles() const { return TILES == 1 ? 1 : (ncp + 3) >> 2; }
    // Up to four columns: one multiply-add takes their high parts as token columns 0..3 and their low parts as 4..7.
    __device__ __forceinline__ bool packed() const { return ncp <= 2; }
};

struct Rings {   // position of one role in the two rings: number of the next weight stage; slot and parity of the next activation stage
    uint32_t w = 0, xs = 0, xp = 0;
    int parked = 0;   // weight stages that this (consumer) warp has parked so far
    __device__ __forceinline__ void next_x() { if (++xs == NX) { xs = 0; xp ^= 1; } }
};

// A plan as a sequence of groups of at most CONS_WARPS slots: a split plan is one group.
struct Groups {
    int g0, left;
    __device__ __forceinline__ explicit Groups(const Plan &p) : g0(p.t0), left(p.n) {}
    __device__ __forceinline__ int slots() const { return min(left, CONS_WARPS); }
    __device__ __forceinline__ void next() { g0 += CONS_WARPS; left -= CONS_WARPS; }
};
// Tile slots over which gemm_consume spreads the elements of a group: log2 (eight where a plan has several groups, so that every
// group is spread alike).
__device__ __forceinline__ int element_shift(int slots) { return slots > CONS_WARPS ? 3 : slots > 1 ? 32 - __clz(slots - 1) : 0; }
__device__ __forceinline__ void st_relaxed_u64(unsigned long long *p, unsigned long long v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// Stages of a group of ng slots in front of chunk kc (in units of the plan's one or two matrices).
__device__ __forceinline__ int stages_before(const Plan &p, int ng, int kc) {
    const int gap = max(0, min(kc, p.s0_own_k0) - p.s0_pub_k1);            // chunks below kc at which slot 0 has none
    const int end = ng > 1 ? max(0, kc - p.sl_k1) : 0;                     // chunks below kc at which the last slot has none any more
    return kc * ng - gap - end;
}

// A weight stage is used, waited for and released by one warp only.  An mbarrier tells phases apart by one parity bit: a warp that
// looks at a slot two fills ahead would take the fill before for its own.  So the producer publishes how many stages it has
// issued: once stage i is among them, the fill before it in the same slot has been released, and the parity is unambiguous.
// (With all eight warps waiting for and releasing every stage each of them walked the whole stream, and a slot was free again
// only when the slowest of them, busy multiplying, had come by.)
__device__ __forceinline__ void w_issued_set(Smem *sm, uint32_t n) { asm volatile("st.release.cta.shared.u32 [%0], %1;" ::"r"(s32(&sm->w_issued)), "r"(n) : "memory"); }
__device__ __forceinline__ uint32_t w_issued_get(Smem *sm) {
    uint32_t n;
    asm volatile("ld.acquire.cta.shared.u32 %0, [%1];" : "=r"(n) : "r"(s32(&sm->w_issued)) : "memory");
    return n;
}
// Wait until stage i has landed; `known`: stages this warp knows to be issued.  (A stage that was not issued when the wait for that ended
// on an error lets the second wait fall through as well.)
__device__ __forceinline__ void w_wait(const Shared &S, uint32_t i, uint32_t &known) {
    if ((int)(known - i) <= 0) {
        unsigned long long t0 = 0;
        for (uint32_t it = 0;; ++it) {
            known = w_issued_get(S.sm);
            if ((int)(known - i) > 0) break;
            if ((it & 127u) == 127u || S.wait_ns < SHORT_LIMIT_NS) {
                if (aborted(S)) break;
                if (*(volatile int *)S.err != 0) { *(volatile int *)&S.sm->abort = 1; break; }
                const unsigned long long t = gtime();
                if (t0 == 0) t0 = t;
                else if (t - t0 > S.wait_ns) { raise_error(S, ERR_TIMEOUT_MBAR); break; }
            }
        }
    }
    mbar_wait(S, &S.sm->w_full[i % NW], (i / NW) & 1);
}

// Weight producer warp: streams this CTA's tiles of the GEMM through the weight ring.  W2: map of the second matrix of a
// pair where the two are separate tensors (null: stacked in W, `half` rows on).
__device__ __forceinline__ void gemm_produce_w(const Shared &S, const Plan &pl, const CUtensorMap *W, const CUtensorMap *W2, int half, Rings &r, uint64_t pol) {
    Smem *sm = S.sm;
    const int lane = threadIdx.x & 31;
    const int nch = pl.nch, pair = pl.pair;
    if (lane == 0) trace(S, EV_WP_BEGIN, 0);
#pragma unroll 1
    for (Groups g(pl); g.left > 0; g.next()) {
        const int ng = g.slots();
#pragma unroll 1
        for (int kc = 0; kc < nch; ++kc)
#pragma unroll 1
            for (int s = 0; s < ng; ++s) {
                const int tile = pl.split ? plan_tile(pl, s, kc) : g.g0 + s;
                if (tile < 0) continue;
#pragma unroll 1
                for (int p = 0; p < pair; ++p) {
                    const uint32_t ws = r.w % NW;
                    mbar_wait(S, &sm->w_empty[ws], ((r.w / NW) & 1) ^ 1);
                    ++r.w;
                    if (lane == 0) {
                        if (!aborted(S)) {
                            mbar_expect_tx(&sm->w_full[ws], (uint32_t)W_STAGE);
                            tma_load_3d(sm->w[ws], (p && W2) ? W2 : W, 0, tile * TILE_N + ((p && !W2) ? half : 0), kc * KG, &sm->w_full[ws], pol);
                        }
                        w_issued_set(sm, r.w);
                    }
                }
            }
    }
    if (lane == 0) trace(S, EV_WP_END, 0);
}

// Activation producer warp: one stage per (tile group, k chunks).
// `after_first` runs once, after the first stage has been issued: work of the phase that is not
// needed before the epilogues (the normalisation factors) and must not delay the first copy.
// `ready` runs once, immediately before the first copy: it waits until the input is complete.
template <class Hook, class Ready>
__device__ __forceinline__ void gemm_produce_x(const Shared &S, const Plan &pl, const uint4 *X, const Cols &cols, Rings &r, uint64_t pol, Hook &&after_first,
                                               Ready &&ready) {
    Smem *sm = S.sm;
    const int lane = threadIdx.x & 31;
    const int nch = pl.nch, XC = cols.chunks();
    const unsigned char *src = reinterpret_cast<const unsigned char *>(X) + cols.cp0 * 4096;
    // as many rounds as the plan has groups; a CTA without any still passes `ready` and the hook
    Groups g(pl);
    bool first = true;
#pragma unroll 1
    do {
#pragma unroll 1
        for (int kc = 0; kc < nch; kc += XC) {
            const bool some = g.left > 0;
            if (some) mbar_wait(S, &sm->x_empty[r.xs], r.xp ^ 1);
            if (first) ready();
            if (some) {
                const int nc = min(XC, nch - kc);
#pragma unroll 1
                for (int t = 0; t < cols.tiles(); ++t) {
                    const uint32_t bytes = (uint32_t)min(cols.ncp - 4 * t, 4) * 4096u;
                    if (t > 0) mbar_wait(S, &sm->x_empty[r.xs], r.xp ^ 1);
                    if (lane == 0 && !aborted(S)) {
                        mbar_expect_tx(&sm->x_full[r.xs], bytes * nc);
                        for (int q = 0; q < nc; ++q)   // chunk kc+q: column pairs cp0 + 4 t .. at [q][pair] of the stage
                            bulk_g2s(sm->x[r.xs] + q * bytes, src + (size_t)(kc + q) * X_BLOCK + t * 16384, bytes, &sm->x_full[r.xs], pol);
                    }
                    r.next_x();
                }
            }
            if (first) { after_first(); first = false; }
            if (!some) break;
        }
        g.next();
    } while (g.left > 0);
}
struct NoHook {
    __device__ __forceinline__ void operator()() const {}
};

// The 32 k-steps of one weight stage: fragment loads run four steps ahead of the multiply-adds that use them.
// Even k-steps accumulate into acc[0] (high parts) and acc[2] (low parts), odd ones into acc[1] and acc[3].  (A stage of one warp
// is bound by the shared-memory reads of all eight, 200 cycles of the SM for 16 KB, not by the length of these chains.)
template <int T>
__device__ __forceinline__ void stage_full(float (&acc)[TILES][4][4], uint32_t ws, const uint32_t (&xs)[TILES], int a_hi, int a_sw) {
    constexpr int PF = T == 1 ? 4 : 2;
    uint32_t a[PF][4];
    uint4 b[PF][T];
#pragma unroll
    for (int j = 0; j < PF; ++j) {
        ldmatrix_x4_at(a[j], ws + (j >> 2) * 2048 + (((((j & 3) << 1) | a_hi) ^ a_sw) << 4));
#pragma unroll
        for (int t = 0; t < T; ++t) b[j][t] = lds128(xs[t] + j * 128);
    }
#pragma unroll
    for (int j = 0; j < KSTEPS; ++j) {
        const int cur = j % PF;
#pragma unroll
        for (int t = 0; t < T; ++t) {
            mma16816(acc[t][j & 1], a[cur], b[cur][t].x, b[cur][t].y);
            mma16816(acc[t][(j & 1) + 2], a[cur], b[cur][t].z, b[cur][t].w);
        }
        if (j + PF < KSTEPS) {
            const int ks = j + PF;
            ldmatrix_x4_at(a[cur], ws + (ks >> 2) * 2048 + (((((ks & 3) << 1) | a_hi) ^ a_sw) << 4));
#pragma unroll
            for (int t = 0; t < T; ++t) b[cur][t] = lds128(xs[t] + ks * 128);
        }
    }
}
// The gate and up stages of a chunk together: a k-step's activations are read once for both.  Three column tiles: 20 instead of 32
// shared-memory cycles a k-step and warp.
template <int T>
__device__ __forceinline__ void stage_full2(float (&acc0)[TILES][4][4], float (&acc1)[TILES][4][4], uint32_t ws0, uint32_t ws1, const uint32_t (&xs)[TILES], int a_hi,
                                            int a_sw) {
    constexpr int PF = 2;
    uint32_t a0[PF][4], a1[PF][4];
    uint4 b[PF][T];
    auto load = [&](int cur, int ks) {
        const uint32_t at = (ks >> 2) * 2048 + (((((ks & 3) << 1) | a_hi) ^ a_sw) << 4);
        ldmatrix_x4_at(a0[cur], ws0 + at);
        ldmatrix_x4_at(a1[cur], ws1 + at);
#pragma unroll
        for (int t = 0; t < T; ++t) b[cur][t] = lds128(xs[t] + ks * 128);
    };
#pragma unroll
    for (int j = 0; j < PF; ++j) load(j, j);
#pragma unroll
    for (int j = 0; j < KSTEPS; ++j) {
        const int cur = j % PF;
#pragma unroll
        for (int t = 0; t < T; ++t) {
            mma16816(acc0[t][j & 1], a0[cur], b[cur][t].x, b[cur][t].y);
            mma16816(acc1[t][j & 1], a1[cur], b[cur][t].x, b[cur][t].y);
            mma16816(acc0[t][(j & 1) + 2], a0[cur], b[cur][t].z, b[cur][t].w);
            mma16816(acc1[t][(j & 1) + 2], a1[cur], b[cur][t].z, b[cur][t].w);
        }
        if (j + PF < KSTEPS) load(cur, j + PF);
    }
}
// The same for up to four columns: their high parts are token columns 0..3 of one multiply-add, their low parts 4..7.
// Half the multiply-adds and half the shared-memory reads; every sum has the order it has above.
__device__ __forceinline__ void stage_packed(float (&acc)[4][4], uint32_t ws, uint32_t xs, int a_hi, int a_sw) {
    constexpr int PF = 4;
    uint32_t a[PF][4];
    uint2 b[PF];
#pragma unroll
    for (int j = 0; j < PF; ++j) {
        ldmatrix_x4_at(a[j], ws + (j >> 2) * 2048 + (((((j & 3) << 1) | a_hi) ^ a_sw) << 4));
        b[j] = lds64(xs + j * 128);
    }
#pragma unroll
    for (int j = 0; j < KSTEPS; ++j) {
        const int cur = j % PF;
        mma16816(acc[j & 1], a[cur], b[cur].x, b[cur].y);
        if (j + PF < KSTEPS) {
            const int ks = j + PF;
            ldmatrix_x4_at(a[cur], ws + (ks >> 2) * 2048 + (((((ks & 3) << 1) | a_hi) ^ a_sw) << 4));
            b[cur] = lds64(xs + ks * 128);
        }
    }
}

// A parked stage (see park_stage): the fragments come back from tensor memory, eight k-steps at a time, the next eight on their way
// while these are multiplied.  The same multiply-adds in the same order as above.
template <bool PACKED>
__device__ __forceinline__ void stage_parked(float (&acc)[4][4], uint32_t tm, uint32_t xs) {
    uint32_t a[2][32];
    tmem_ld32_start(a[0], tm);
#pragma unroll
    for (int h = 0; h < 4; ++h) {
        uint4 b[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const uint32_t p = xs + (8 * h + j) * 128;
            if (PACKED) {
                const uint2 v = lds64(p);
                b[j] = make_uint4(v.x, v.y, 0, 0);
            } else {
                b[j] = lds128(p);
            }
        }
        uint32_t(&cur)[32] = a[h & 1];
        tmem_ld_wait(cur);
        if (h < 3) tmem_ld32_start(a[(h + 1) & 1], tm + 32 * (h + 1));
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const uint32_t f[4] = {cur[4 * j], cur[4 * j + 1], cur[4 * j + 2], cur[4 * j + 3]};
            mma16816(acc[j & 1], f, b[j].x, b[j].y);
            if (!PACKED) mma16816(acc[(j & 1) + 2], f, b[j].z, b[j].w);
        }
    }
}

// Weight stages parked in tensor memory.  Between a phase's end and the arrival of the next one's activations (3 to 4 us: report,
// last CTA's report seen, copy) the consumers have nothing to multiply, and the nine stages of the ring cover 3 us of the
// stream only: HBM idled for the rest.  So the warps use the wait to move the stages they own from the ring to tensor memory, up to
// two each, as the fragments that the multiply-add wants; the ring's slots go back to the producer at once.  That makes 25
// stages (400 KB) per CTA, and the parked ones do not pass through shared memory again when the activations are there.
// Warp w can address the lanes of quadrant w % 4 only; it holds its stages there in columns 256 (w / 4) on, 128 a stage.
// A layer of the 8B shape (1B), us, with no, one and two stages a warp: QKV 12.3, 11.2, 10.9 (6.4, 5.8, 5.7), O 9.3, 7.5, 7.5 (5.4,
// 4.8, 4.9), gate-up 39.0, 39.2, 36.7 (13.5, 13.2, 10.7), down 20.9, 19.2, 18.6 (9.3, 7.7, 8.0); attention, whose K and V blocks have
// less time to arrive, 10.0, 10.2, 10.2 (6.6 each).  (The kernel of one column tile only.  With more than four columns in use the
// products of the other one are bound by their activations; its steps of up to four would gain too, but three tiles' sums leave no
// registers for it: some 200 bytes are spilled as it is.)
constexpr int PARK_MAX = 2, PARK_COLS = 512;
// The CTA's tensor memory, all of it (there is one CTA per SM); both by the same whole warp.
__device__ __forceinline__ void park_alloc(Smem *sm) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s32(&sm->tmem)), "r"(PARK_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void park_free(Smem *sm) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(sm->tmem), "r"(PARK_COLS) : "memory");
}
__device__ __forceinline__ void park_stage(uint32_t ws, int a_hi, int a_sw, uint32_t tm) {
#pragma unroll
    for (int h = 0; h < 4; ++h) {
        uint32_t v[32];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int ks = 8 * h + j;
            uint32_t a[4];
            ldmatrix_x4_at(a, ws + (ks >> 2) * 2048 + (((((ks & 3) << 1) | a_hi) ^ a_sw) << 4));
#pragma unroll
            for (int i = 0; i < 4; ++i) v[4 * j + i] = a[i];
        }
        tmem_st32(tm + 32 * h, v);
    }
    tmem_st_wait();
}

// Consumer warps.  Within a group of up to eight tiles the warps are arranged as TS tile slots x
// KS k-splits (TS * KS = 8, TS the smallest power of two holding the group); a warp multiplies
// the stages of its slot whose k chunk is ks_id (mod KS).  The arrangement depends only on the tile partition, never on which
// token columns are in use.
//
// All warps' sums then meet in shared memory and every thread finishes elements of its own: half-warp u takes (tile slot
// u mod E, the (u / E)-th column in use; E: element_shift), lane % 16 the row, in passes of sixteen half-warps; it adds the k-splits in index
// order and calls `epi(pass, active, tile, row, column, d0, d1)` (the whole warp calls it together).  One warp per tile finishing
// four elements a thread, the k-splits one after the other, was a chain of 1.6 us at the end of every phase.
// `epi.pre(pass, tile, row, column)` runs in the same thread before the group's first stage: a place to start loads the epilogue will
// need.
//
// One body for every product of a program (the caller loops over its phases and branches on the phase in `pre` and `epi`): with
// a copy of it per product and role the persistent kernel was 790 KB of code, more than the instruction caches hold, and every
// phase began and ended with instruction fetches from L2 on its critical path.
// PARK: the kernel has tensor memory for parked stages (sm->tmem), of which a warp parks at most `park` (up to PARK_MAX).  (As a
// member of `S`, which lives in local memory, the limit cost 0.4 % of a short request.)
// k steps past K multiply zeros (the tensor map fills weights with them, the activation blocks are padded with them).
template <bool PARK, class Epi>
__device__ __forceinline__ void gemm_consume(const Shared &S, const Plan &pl, const Cols &cols, unsigned mask, unsigned long long *part, unsigned phase_id, int cta,
                                             Rings &r, const Epi &epi, int park) {
    Smem *sm = S.sm;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nch = pl.nch, pair = pl.pair, XC = cols.chunks();
    const bool packed = cols.packed();
    const int s0_own_k0 = pl.s0_own_k0, s0_pub_k1 = pl.s0_pub_k1, sl_k1 = pl.sl_k1;
    // ldmatrix source of this lane inside a stage: row (lane%8) + 8 ((lane/8)%2), 16-byte chunk lane/16 of the k-step
    const int a_row = (lane & 7) + ((lane >> 3) & 1) * 8;
    const int a_off = a_row * 128, a_hi = lane >> 4, a_sw = a_row & 7;
    const int nt = cols.tiles();
    // this lane's column pair of every tile, counted from the first fetched (past the last: any, its columns are not in use), and
    // its 16 (8) bytes
    int x_off[TILES];
#pragma unroll
    for (int t = 0; t < TILES; ++t) {
        const int xpair = min(packed ? (lane >> 3) & 1 : lane >> 3, max(cols.ncp - 1 - 4 * t, 0));
        x_off[t] = xpair * 4096 + (lane & 7) * 16 + (packed ? (lane >> 4) * 8 : 0);
    }
    const int nact = __popc(mask), row = lane & 15;
    uint32_t known = r.w;
    bool first = true;
    const int esh = element_shift(Groups(pl).left), eslots = 1 << esh;
    const int n_pass = ((nact << esh) + 15) >> 4;
#pragma unroll 1
    for (Groups g(pl); g.left > 0; g.next()) {
        const int ng = g.slots(), lts = 32 - __clz(ng - 1);   // (clz(0) = 32)
        const int TS = 1 << lts, KS = CONS_WARPS >> lts;
        const int slot_id = warp & (TS - 1), ks_id = warp >> lts;
        const bool mine = slot_id < ng;
        const bool pub_only = slot_id > 0 && slot_id == ng - 1 && sl_k1 < nch;
        // this warp's slot: chunks below my_pub_k1 go to the published part, chunks from my_own_k0 to its own tile
        const int my_pub_k1 = !mine ? 0 : slot_id == 0 ? s0_pub_k1 : pub_only ? sl_k1 : 0;
        const int my_own_k0 = (!mine || pub_only) ? nch : slot_id == 0 ? s0_own_k0 : 0;
        const int own_tile = (mine && !pub_only) ? g.g0 + slot_id : -1;
        const bool tail = own_tile >= 0 && my_own_k0 > 0;   // the head part of this tile comes from CTA cta - 1
        // this thread's elements: columns by pass, five bits each
        unsigned long long my_cols = 0;
#pragma unroll 1
        for (int ps = 0; ps < n_pass; ++ps) {
            const int u = 16 * ps + 2 * warp + (lane >> 4), slot = u & (eslots - 1);
            int ci = u >> esh;
            unsigned m = mask;
            for (; ci > 0 && m; --ci) m &= m - 1;
            const bool act = m != 0 && slot < ng && !(slot > 0 && slot == ng - 1 && sl_k1 < nch);
            my_cols |= (unsigned long long)(act ? __ffs(m) - 1 : 31) << (5 * ps);
            if (act && ps < STASH_PASSES) epi.pre(ps, g.g0 + slot, row, __ffs(m) - 1);
        }
        // This warp's chunks in order: n_pub of the part it publishes, then those of its own tile; every KS-th one from the first of
        // the part.  (A warp then multiplies all 32 k-steps of a stage, which amortises the per-stage waiting and set-up: splitting
        // every stage among the warps streamed 20-30 % slower.)
        const int lks = 3 - lts, n_pub = max(0, my_pub_k1 - ks_id + KS - 1) >> lks, n_all = n_pub + (max(0, nch - my_own_k0 - ks_id + KS - 1) >> lks);
        auto chunk_of = [&](int j) { return j < n_pub ? ks_id + (j << lks) : my_own_k0 + ks_id + ((j - n_pub) << lks); };
        auto stage_of = [&](int kc) {   // number of its (first) weight stage at chunk kc
            const bool gap0 = slot_id > 0 && kc >= s0_pub_k1 && kc < s0_own_k0;   // slot 0 has none here
            return r.w + (uint32_t)((stages_before(pl, ng, kc) + slot_id - gap0) * pair);
        };
        // stages parked while the activations are on their way: those that land before they do, at most PARK_MAX
        int n_parked = 0, n_used = 0;
        const uint32_t tm = PARK ? sm->tmem + ((uint32_t)(warp & 3) << 21) + (uint32_t)(warp >> 2) * (128 * PARK_MAX) : 0u;
        if (PARK && first) {
            unsigned long long t0 = 0;
            const int most = min(n_all * pair, park);
#pragma unroll 1
            while (n_parked < most) {
                const uint32_t i = stage_of(chunk_of(pair == 2 ? n_parked >> 1 : n_parked)) + (pair == 2 ? n_parked & 1 : 0), wslot = i % NW;
                bool go = true;
#pragma unroll 1
                for (uint32_t it = 0;; ++it) {
                    if (__any_sync(0xffffffffu, mbar_test(&sm->x_full[r.xs], r.xp))) { go = false; break; }
                    if ((int)(known - i) <= 0) known = w_issued_get(sm);
                    if (__all_sync(0xffffffffu, (int)(known - i) > 0 && mbar_test(&sm->w_full[wslot], (i / NW) & 1))) break;
                    if ((it & 127u) == 127u || S.wait_ns < SHORT_LIMIT_NS) {   // the wait for the activations below reports what is wrong
                        bool stop = aborted(S) || *(volatile int *)S.err != 0;
                        const unsigned long long t = gtime();
                        if (t0 == 0) t0 = t;
                        else if (t - t0 > S.wait_ns) stop = true;
                        if (__any_sync(0xffffffffu, stop)) { go = false; break; }
                    }
                }
                if (!go) break;
                park_stage(s32(sm->w[wslot]) + a_off, a_hi, a_sw, tm + 128 * n_parked);
                ++n_parked;
                __syncwarp();
                if (lane == 0) mbar_arrive(&sm->w_empty[wslot]);
            }
            r.parked += n_parked;
        }
        float acc0[TILES][4][4], acc1[TILES][4][4];   // [column tile][even/odd step x hi/lo][fragment] of the one or two matrices
        auto clear = [&]() {
#pragma unroll
            for (int t = 0; t < TILES; ++t)
#pragma unroll
                for (int q = 0; q < 4; ++q)
#pragma unroll
                    for (int i = 0; i < 4; ++i) acc0[t][q][i] = acc1[t][q][i] = 0.f;
        };
        clear();
        // fold the partial accumulators in a fixed order: the chains of the high parts, those of the low parts, both.
        // The result of column pair cp0 + 4 t + j stands in tile t, lanes with lane % 4 = j.
        float d0[TILES][4], d1[TILES][4];
        auto fold = [&](float (&d)[TILES][4], float (&acc)[TILES][4][4]) {
#pragma unroll
            for (int t = 0; t < TILES; ++t)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float hi = acc[t][0][i] + acc[t][1][i];
                    d[t][i] = hi + (packed ? __shfl_xor_sync(0xffffffffu, hi, 2) : acc[t][2][i] + acc[t][3][i]);
                }
        };
        // Activation stages are shared: every warp waits for and releases each of them.  A warp goes from one of its own chunks to the
        // next; looking at every chunk cost 400 cycles for each that is not its own, which parked stages would not have hidden.
        int x0 = 0;                       // first chunk of the activation stage(s) at hand
        uint32_t xt[TILES];               // this lane's bytes of them, by column tile
        auto x_wait = [&]() {
            uint32_t xs = r.xs, xp = r.xp;
#pragma unroll
            for (int t = 0; t < TILES; ++t) {
                xt[t] = s32(sm->x[xs]) + x_off[t];
                if (t < nt) {
                    mbar_wait(S, &sm->x_full[xs], xp);
                    if (TILES > 1 && ++xs == NX) { xs = 0; xp ^= 1; }
                }
            }
        };
        auto x_release = [&]() {
            __syncwarp();
#pragma unroll 1
            for (int t = 0; t < nt; ++t) {
                if (lane == 0) mbar_arrive(&sm->x_empty[r.xs]);
                r.next_x();
            }
            x0 += XC;
        };
        x_wait();
        if (threadIdx.x == 0 && first) trace(S, EV_X0, 0);
        first = false;
#pragma unroll 1
        for (int j = 0;; ++j) {
            if (j == n_pub && my_pub_k1 > 0) {
                // The head part of a split tile is complete: every k-split warp publishes its own sums
                // (no meeting inside the CTA in the middle of the stream) and starts over for the tail
                // part that may follow in this slot.
                fold(d0, acc0);
                if (pair == 2) fold(d1, acc1);
#pragma unroll
                for (int t = 0; t < TILES; ++t) {
                    if (t >= nt) break;
                    unsigned long long *pb = part + (size_t)((cta * CONS_WARPS + ks_id) * TILES + t) * 256;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        st_relaxed_u64(pb + i * 32 + lane, ((unsigned long long)phase_id << 32) | __float_as_uint(d0[t][i]));
                        if (pair == 2) st_relaxed_u64(pb + (4 + i) * 32 + lane, ((unsigned long long)phase_id << 32) | __float_as_uint(d1[t][i]));
                    }
                }
                clear();
            }
            if (j >= n_all) break;
            const int kc = chunk_of(j);
            while (kc >= x0 + XC) { x_release(); x_wait(); }
            uint32_t xc[TILES];
#pragma unroll
            for (int t = 0; t < TILES; ++t) xc[t] = xt[t] + (t == 0 ? (kc - x0) * cols.ncp * 4096 : 0);
            uint32_t i = stage_of(kc);
            if (TILES > 1 && pair == 2 && !packed) {
                w_wait(S, i, known);
                w_wait(S, i + 1, known);
                const uint32_t ws0 = s32(sm->w[i % NW]) + a_off, ws1 = s32(sm->w[(i + 1) % NW]) + a_off;
                if (nt == 1) stage_full2<1>(acc0, acc1, ws0, ws1, xc, a_hi, a_sw);
                else if (nt == 2) stage_full2<TILES < 2 ? 1 : 2>(acc0, acc1, ws0, ws1, xc, a_hi, a_sw);
                else stage_full2<TILES>(acc0, acc1, ws0, ws1, xc, a_hi, a_sw);
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(&sm->w_empty[i % NW]);
                    mbar_arrive(&sm->w_empty[(i + 1) % NW]);
                }
                continue;
            }
#pragma unroll 1
            for (int p = 0; p < pair; ++p, ++i) {
                if (PARK && n_used < n_parked) {
                    const uint32_t at = tm + 128 * n_used++;
                    if (packed) {
                        if (p == 0) stage_parked<true>(acc0[0], at, xc[0]);
                        else stage_parked<true>(acc1[0], at, xc[0]);
                    } else {
                        if (p == 0) stage_parked<false>(acc0[0], at, xc[0]);
                        else stage_parked<false>(acc1[0], at, xc[0]);
                    }
                    continue;
                }
                w_wait(S, i, known);
                const uint32_t wslot = i % NW;
                const uint32_t ws = s32(sm->w[wslot]) + a_off;
                if (packed) {
                    if (p == 0) stage_packed(acc0[0], ws, xc[0], a_hi, a_sw);
                    else stage_packed(acc1[0], ws, xc[0], a_hi, a_sw);
                } else if (TILES == 1) {
                    if (p == 0) stage_full<1>(acc0, ws, xc, a_hi, a_sw);
                    else stage_full<1>(acc1, ws, xc, a_hi, a_sw);
                } else if (nt == 1) {   // (several tiles: the two matrices of a pair were multiplied together above, this is a single one)
                    stage_full<1>(acc0, ws, xc, a_hi, a_sw);
                } else if (nt == 2) {
                    stage_full<TILES < 2 ? TILES : 2>(acc0, ws, xc, a_hi, a_sw);
                } else {
                    stage_full<TILES>(acc0, ws, xc, a_hi, a_sw);
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&sm->w_empty[wslot]);
            }
        }
        for (x_release(); x0 < nch; x_release()) x_wait();
        r.w += (uint32_t)(stages_before(pl, ng, nch) * pair);
        if (threadIdx.x == 0 && g.left <= CONS_WARPS) trace(S, EV_MAIN_END, 0);
        fold(d0, acc0);
        if (pair == 2) fold(d1, acc1);
        // The head part published by CTA cta - 1, in ksp k-splits: this slot's k-split warp j fetches
        // the published splits j, j + KS, ... (all at once: one round trip) and adds them to its own
        // sums in index order; the fixed-order reduction below then covers both parts.
        if (tail) {
            unsigned long long t0 = 0;
            for (uint32_t it = 0;; ++it) {
                bool ok = true;
                float add[2][TILES][4];
#pragma unroll
                for (int p = 0; p < 2; ++p)
#pragma unroll
                    for (int t = 0; t < TILES; ++t)
#pragma unroll
                        for (int i = 0; i < 4; ++i) add[p][t][i] = 0.f;
                for (int q = ks_id; q < pl.ksp; q += KS) {
#pragma unroll
                    for (int t = 0; t < TILES; ++t) {
                        if (t >= nt) break;
                        const unsigned long long *pb = part + (size_t)(((cta - 1) * CONS_WARPS + q) * TILES + t) * 256;
#pragma unroll
                        for (int p = 0; p < 2; ++p) {
                            if (p >= pair) break;
#pragma unroll
                            for (int i = 0; i < 4; ++i) {
                                const unsigned long long v = ld_relaxed_u64(pb + (p * 4 + i) * 32 + lane);
                                ok = ok && (unsigned)(v >> 32) == phase_id;
                                add[p][t][i] += __uint_as_float((unsigned)v);
                            }
                        }
                    }
                }
                if (__all_sync(0xffffffffu, ok)) {
#pragma unroll
                    for (int t = 0; t < TILES; ++t)
#pragma unroll
                        for (int i = 0; i < 4; ++i) { d0[t][i] += add[0][t][i]; d1[t][i] += add[1][t][i]; }
                    break;
                }
                if ((it & 15u) == 15u || S.wait_ns < SHORT_LIMIT_NS) {   // bounded like every other wait on another CTA
                    bool stop = aborted(S) || *(volatile int *)S.err != 0;
                    const unsigned long long t = gtime();
                    if (t0 == 0) t0 = t;
                    else if (t - t0 > S.wait_ns) { if (lane == 0) raise_error(S, ERR_TIMEOUT_GRID); stop = true; }
                    if (__any_sync(0xffffffffu, stop)) { *(volatile int *)&S.sm->abort = 1; break; }
                }
                __nanosleep(64);
            }
        }
        float *red = reinterpret_cast<float *>(sm->scratch);   // [matrix][warp][column tile][fragment element][lane]
#pragma unroll
        for (int t = 0; t < TILES; ++t) {
            if (t >= nt) break;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                red[((warp * TILES + t) * 4 + i) * 32 + lane] = d0[t][i];
                if (pair == 2) red[(((CONS_WARPS + warp) * TILES + t) * 4 + i) * 32 + lane] = d1[t][i];
            }
        }
        bar_consumers();
#pragma unroll 1
        for (int ps = 0; ps < n_pass; ++ps) {
            const int slot = (16 * ps + 2 * warp + (lane >> 4)) & (eslots - 1), cn = (int)(my_cols >> (5 * ps)) & 31;
            const bool act = cn < MAX_COLS;
            const int col = act ? cn : 0;
            // element (row, column) of a warp's sums: fragment element 2 (row / 8) + column % 2 of lane 4 (row % 8) + column pair % 4, tile pair / 4
            const int pr = act ? (col >> 1) - cols.cp0 : 0;
            const float *o = red + ((((slot & (TS - 1)) * TILES + (pr >> 2)) * 4 + 2 * (row >> 3) + (col & 1)) * 32 + ((row & 7) << 2) + (pr & 3));
            float v0[CONS_WARPS], v1[CONS_WARPS];
            const int step = (TILES * 128) << lts;   // floats from one k-split to the next
#pragma unroll
            for (int q = 0; q < CONS_WARPS; ++q) {
                v0[q] = q < KS ? o[q * step] : 0.f;
                v1[q] = q < KS && pair == 2 ? o[CONS_WARPS * (TILES * 128) + q * step] : 0.f;
            }
            float e0 = v0[0], e1 = v1[0];
#pragma unroll
            for (int q = 1; q < CONS_WARPS; ++q)
                if (q < KS) { e0 += v0[q]; e1 += v1[q]; }
            epi(ps, act, g.g0 + slot, row, col, e0, e1);
        }
        if (g.left > CONS_WARPS) bar_consumers();   // the next group writes the exchange area again (after the last one the caller meets)
    }
}

// The dynamic shared memory is requested SMEM_BYTES long; the structure starts at its first
// 1024-byte boundary.
constexpr size_t SMEM_BYTES = sizeof(Smem) + 1024;
static_assert(SMEM_BYTES <= 232448, "exceeds the 227 KB of shared memory a block may use");
__device__ __forceinline__ Smem *smem_base(unsigned char *raw) {
    const uint32_t a = s32(raw);
    return reinterpret_cast<Smem *>(raw + ((1024u - (a & 1023u)) & 1023u));
}

// Shared-memory set-up by the whole block (call once, followed by __syncthreads()).
__device__ __forceinline__ void smem_init(Smem *sm) {
    if (threadIdx.x == 0) {
        for (int i = 0; i < NW; ++i) { mbar_init(&sm->w_full[i], 1); mbar_init(&sm->w_empty[i], 1); }
        for (int i = 0; i < NX; ++i) { mbar_init(&sm->x_full[i], 1); mbar_init(&sm->x_empty[i], CONS_WARPS); }
        sm->abort = 0;
        sm->trace_n = 0;
        sm->vec_seq = 0;
        sm->w_issued = 0;
        fence_mbar_init();
        fence_proxy_async();
    }
}

// After an error the producers stop issuing copies; give the ones already in flight time to land
// before the block's shared memory is released.
__device__ __forceinline__ void settle_on_abort(const Shared &S) {
    __syncthreads();
    if (!aborted(S)) return;
    const unsigned long long t0 = gtime();
    while (gtime() - t0 < 200000ull) __nanosleep(1000);
}

}  // namespace ADA_ST
}  // namespace ada

#endif
