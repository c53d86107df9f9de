// Dense products of the prompt pass ("KV cache <- LM(x)", first line of Algorithm 1) on the fifth-generation
// tensor cores of sm_100a: tcgen05.mma over pairs of CTAs (cta_group::2) with the accumulators in tensor memory,
// operands staged in shared memory by TMA, and the operation that follows a product fused into its epilogue.
//
// A block of prompt positions (up to PF_ROWS) goes through a weight matrix in one product
//     Y[m][n] = sum_k X[m][k] W[n][k],   m < rows positions, n < N weight rows.
// X arrives as two bf16 matrices, a high part and a low part (x = hi + lo, as everywhere in this library: fp32
// activations lose nothing), both multiplied into the same fp32 accumulator: 4 m n k floating-point operations.
//
// What bounds it.  Below about 128 positions the weights' way from HBM, above it the tensor cores and the L2 cache
// together: the gate / up product of a 1024-position block of the 8B shape keeps the tensor pipe 79 % busy while 8.7 TB/s
// move from L2 to the SMs (profiles/k_dense_gemm_8b_1024_ncu.md).  The weights are the 256-row operand of a pair of CTAs, the positions the other one, 32 to 256 wide in
// steps of 32: a block is cut into equal position tiles, so that little is multiplied for padding (777 positions: 4 tiles
// of 224; with positions as the 256-row operand a prompt of 45 positions cost as much as one of 256).  At full width a
// k block of 64 costs a CTA 48 KB of shared-memory fill per 1024 tensor-core cycles; one CTA per tile of 128 x 128 needed
// 48 KB per 512 cycles and 2.7 times the L2 traffic per weight byte.
//
// Accumulation.  The tensor core adds into its fp32 accumulator with truncation, so an accumulator falls short by
// 1.5e-8 of the sum per addition (1e-3 absolute at K = 14336 with sums of size 10).  A product is therefore cut into chunks
// of 512 k, shallow ones of 256 (chunk_blocks); a chunk accumulates in one of two 256-column tensor-memory buffers while the
// epilogue warps add the other one, already complete, to fp32 registers (round to nearest).  Error of the sums alone, 2-norm:
// 1.10e-6 with chunks of 512, 0.56e-6 of 256, 0.30e-6 of 128; the split of the activations is 2.45e-6.  Chunks of 256 (128)
// everywhere cost a 777-token prompt of the 8B shape 4 % (22 %): the epilogue then holds up the tensor core.
//
// Order of the sums.  It is a function of N, K and the device alone, so that the cache rows of a prompt's prefix have the
// same bits whatever follows the prefix.  The chunks of a tile form 1 to 4 groups (as many as one position
// tile has pairs to spare for, so that short prompts can use them side by side).  A group is summed from zero in the order
// of its chunks, the groups are then added in their order: ((g0 + g1) + g2) + g3.  A pair that holds several groups of a
// tile keeps the running total in scratch while it sums the next group (there are registers for one set of sums); that
// traffic runs under the tensor core's next chunk.
//
// Work division.  A tile may be cut between pairs (GemmPlan, plan_dense):
//   * with more tiles than pairs, tiles in excess of whole waves are divided by chunks ("stream-K"), every pair getting the
//     same number (+- 1), at least a tile's worth.  A tile then has at most two pieces, and the pair with the second one
//     goes on from the total and the unfinished group of the first;
//   * with fewer, between groups only.  Every piece starts its group from zero; the pair that holds the last group adds
//     the other pairs' sums before its own.
// What another pair waits for is computed first thing in the kernel, and a pair only ever waits for pairs with a lower
// number, so no assumption about co-residency is made.  With whole tiles a 1024-position block of the 8B shape would fill
// 83 % of its waves, a 500-position one 60 %.
//
// Roles of a CTA: warp 0 issues the TMA loads, warp 1 allocates the tensor memory and (in the first CTA of the pair)
// issues the MMAs, warps 4..11 read the accumulators and run the epilogue.  Every wait is bounded; on expiry an
// error word is set, the roles leave their loops, the tensor memory is released and the kernel ends.
#pragma once

#include "kernels.cuh"
#include "stream.cuh"
#include "tmem.cuh"

namespace ada {
namespace dg {

using namespace st;

constexpr int PF_ROWS = 2048;  // prompt positions of one block: 32 layers of launches and ragged waves are paid once per
                               // block; activations of a block stay below the size of the L2 cache per product
constexpr int BW = 128;        // weight rows one CTA of a pair holds (UMMA M = 256 over the pair)
constexpr int TW = 2 * BW;
constexpr int NT_MAX = 256;    // positions per tile, at most
constexpr int BK = 64;         // k elements per stage: one 128-byte swizzle row
constexpr int MAX_STAGES = 12;
constexpr int GEPI_WARPS = 8;  // epilogue warps: lane quadrant (warp % 4) x half of the tile's positions
constexpr int GTHREADS = 128 + 32 * GEPI_WARPS;
// The register file is divided per warpgroup at launch (168 a thread); the epilogue warps hold 128 sums each and take
// what the first warpgroup (TMA, MMA, two idle warps) gives back: (40 + 232 + 232) x 128 = 168 x 384.
constexpr int GREGS_ISSUE = 40, GREGS_EPI = 232;
constexpr int W_BYTES = BW * BK * 2;
constexpr int RING_BYTES = 196608;
constexpr int TMEM_COLS = 512; // two accumulator buffers of 256 fp32 columns
constexpr int MAX_GROUPS = 4;
constexpr size_t GPART_WARP = 128 * 32 * sizeof(float);           // sums of one epilogue warp
constexpr size_t GPART_SLOT = GEPI_WARPS * GPART_WARP;
// per CTA: what it publishes (the total of whole groups; the unfinished group), and the running total of a tile it keeps
constexpr int SLOT_TOTAL = 0, SLOT_GROUP = 1, SLOT_OWN = 2;
constexpr size_t GPART_CTA = 3 * GPART_SLOT;

struct DSmem {   // must start on a 1024-byte boundary (swizzle pattern)
    // stages of [W 128 x 64 (SwiGLU: 16 rows of gate, 16 of up, ...) | X.hi NT / 2 x 64 | X.lo NT / 2 x 64], rows of 128 B: as many as fit
    alignas(1024) unsigned char ring[RING_BYTES];
    alignas(8) unsigned long long full[MAX_STAGES], empty[MAX_STAGES], acc_full[2], acc_empty[2];
    alignas(16) float stash[GEPI_WARPS][32][32];   // per epilogue warp: 32 positions x its 32 weight rows
    unsigned long long wait_ns;
    uint32_t tmem_base;
    int abort;
};
constexpr size_t DSMEM_BYTES = sizeof(DSmem) + 1024;
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

__device__ __forceinline__ void umma_pair(uint32_t d_tmem, unsigned long long adesc, unsigned long long bdesc, uint32_t id, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(id), "r"(accumulate)
        : "memory");
}
// The barrier at this offset of both CTAs is arrived on once every MMA issued so far by this thread has completed.
__device__ __forceinline__ void umma_commit_pair(unsigned long long *bar) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(s32(bar)), "h"((uint16_t)3)
                 : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t (&v)[16], uint32_t addr) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];\n\t"
                 "tcgen05.wait::ld.sync.aligned;"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                   "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
                 : "r"(addr)
                 : "memory");
}
__device__ __forceinline__ void tmem_ld128(uint32_t (&v)[128], uint32_t addr) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x128.b32 {"
                 "%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
                 "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, "
                 "%32, %33, %34, %35, %36, %37, %38, %39, %40, %41, %42, %43, %44, %45, %46, %47, "
                 "%48, %49, %50, %51, %52, %53, %54, %55, %56, %57, %58, %59, %60, %61, %62, %63, "
                 "%64, %65, %66, %67, %68, %69, %70, %71, %72, %73, %74, %75, %76, %77, %78, %79, "
                 "%80, %81, %82, %83, %84, %85, %86, %87, %88, %89, %90, %91, %92, %93, %94, %95, "
                 "%96, %97, %98, %99, %100, %101, %102, %103, %104, %105, %106, %107, %108, %109, %110, %111, "
                 "%112, %113, %114, %115, %116, %117, %118, %119, %120, %121, %122, %123, %124, %125, %126, %127"
                 "}, [%128];\n\t"
                 "tcgen05.wait::ld.sync.aligned;"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                   "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
                   "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
                   "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31]),
                   "=r"(v[32]), "=r"(v[33]), "=r"(v[34]), "=r"(v[35]), "=r"(v[36]), "=r"(v[37]), "=r"(v[38]), "=r"(v[39]),
                   "=r"(v[40]), "=r"(v[41]), "=r"(v[42]), "=r"(v[43]), "=r"(v[44]), "=r"(v[45]), "=r"(v[46]), "=r"(v[47]),
                   "=r"(v[48]), "=r"(v[49]), "=r"(v[50]), "=r"(v[51]), "=r"(v[52]), "=r"(v[53]), "=r"(v[54]), "=r"(v[55]),
                   "=r"(v[56]), "=r"(v[57]), "=r"(v[58]), "=r"(v[59]), "=r"(v[60]), "=r"(v[61]), "=r"(v[62]), "=r"(v[63]),
                   "=r"(v[64]), "=r"(v[65]), "=r"(v[66]), "=r"(v[67]), "=r"(v[68]), "=r"(v[69]), "=r"(v[70]), "=r"(v[71]),
                   "=r"(v[72]), "=r"(v[73]), "=r"(v[74]), "=r"(v[75]), "=r"(v[76]), "=r"(v[77]), "=r"(v[78]), "=r"(v[79]),
                   "=r"(v[80]), "=r"(v[81]), "=r"(v[82]), "=r"(v[83]), "=r"(v[84]), "=r"(v[85]), "=r"(v[86]), "=r"(v[87]),
                   "=r"(v[88]), "=r"(v[89]), "=r"(v[90]), "=r"(v[91]), "=r"(v[92]), "=r"(v[93]), "=r"(v[94]), "=r"(v[95]),
                   "=r"(v[96]), "=r"(v[97]), "=r"(v[98]), "=r"(v[99]), "=r"(v[100]), "=r"(v[101]), "=r"(v[102]), "=r"(v[103]),
                   "=r"(v[104]), "=r"(v[105]), "=r"(v[106]), "=r"(v[107]), "=r"(v[108]), "=r"(v[109]), "=r"(v[110]), "=r"(v[111]),
                   "=r"(v[112]), "=r"(v[113]), "=r"(v[114]), "=r"(v[115]), "=r"(v[116]), "=r"(v[117]), "=r"(v[118]), "=r"(v[119]),
                   "=r"(v[120]), "=r"(v[121]), "=r"(v[122]), "=r"(v[123]), "=r"(v[124]), "=r"(v[125]), "=r"(v[126]), "=r"(v[127])
                 : "r"(addr)
                 : "memory");
}

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
        if ((it & 255u) == 0 || sm->wait_ns < SHORT_LIMIT_NS) {
            if (*(volatile int *)&sm->abort) return false;
            const unsigned long long t = gtime();
            if (t0 == 0) t0 = t;
            else if (t - t0 > sm->wait_ns) {
                atomicCAS(err, 0, ERR_TIMEOUT_MBAR);
                *(volatile int *)&sm->abort = 1;
                return false;
            }
        }
    }
}

// Division of one product's tiles over the CTA pairs (worked out on the host, plan_dense, down to every pair's share: a
// division on the device is cold code in front of a kernel's first load).  Tiles are numbered with the position tile fastest,
// so that the pairs at work at one time share weight rows.  The tiles from `whole` on are divided over the pairs, by chunks or
// by groups: pair p holds (tile - whole) << 16 | chunk from start[p] to start[p + 1]; the tiles before are dealt out whole.
constexpr int MAX_PAIRS = 76;
struct GemmPlan {
    int nt, mt, ck, chunks, groups, pairs;   // positions per tile, position tiles; k blocks of a chunk, chunks and groups of a tile
    int tiles, whole;
    int group[MAX_GROUPS + 2];               // first chunk of each group; `chunks` for the last group's end and behind
    int start[MAX_PAIRS + 1];
};

struct Seg { int tile, c0, c1; };   // chunks [c0, c1) of a tile
struct Sched {
    const GemmPlan &g;
    int pair, t_first, c_first, t_last, c_last, i, phase;   // phase 0: last shared tile, 1: the whole ones between, 2: whole tiles, 3: first shared tile, 4: end
    __host__ __device__ __forceinline__ Sched(const GemmPlan &g_, int pair_) : g(g_), pair(pair_), t_first(0), c_first(0), t_last(0), c_last(0), i(pair_), phase(2) {
        const int beg = g.start[pair], end = g.start[pair + 1];
        if (end > beg) {
            t_first = beg >> 16;
            c_first = beg & 0xffff;
            c_last = end & 0xffff;
            t_last = (end >> 16) - (c_last == 0);
            if (c_last == 0) c_last = g.chunks;
            phase = 0;
        }
    }
    // Pieces another pair waits for come first, the piece that waits for others comes last.
    __host__ __device__ __forceinline__ bool next(Seg &s) {
        if (phase == 0) {
            phase = 1;
            i = t_last - 1;
            if (t_last != t_first || c_last < g.chunks) {
                s.tile = g.whole + t_last;
                s.c0 = t_last == t_first ? c_first : 0;
                s.c1 = c_last;
                return true;
            }
        }
        if (phase == 1) {
            if (i > t_first) {
                s.tile = g.whole + i--;
                s.c0 = 0;
                s.c1 = g.chunks;
                return true;
            }
            phase = 2;
            i = pair;
        }
        if (phase == 2) {
            if (i < g.whole) {
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
            if (g.start[pair + 1] > g.start[pair] && (t_first != t_last || c_last == g.chunks)) {
                s.tile = g.whole + t_first;
                s.c0 = c_first;
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
    int rows, N, K;               // positions, weight rows (SwiGLU: of one of the two matrices), depth
    float *Y; int ldy;            // STORE, ADD
    __nv_bfloat16 *hi, *lo;       // QKV: scaled queries [rows][q features]; SwiGLU: activations [rows][N]
    const float *cs;              // QKV: cos, sin [rows][hd / 2][2]
    const float *rstd;            // QKV, SwiGLU: 1 / rms of the rows, applied to the products
    int layer, seq, pos0;         // QKV: rows are positions pos0 .. of sequence seq
    float *part;                  // [CTA][slot]: sums of tiles cut between pairs, running totals (null: one group, nothing cut)
    unsigned *flag;               // [CTA][epilogue warp]: launch number of the sums published last
    unsigned epoch;
    int *err;
    unsigned long long wait_ns;   // limit of every wait
};

// a pair of fp32 values as bf16 high parts and low parts
__device__ __forceinline__ void split2(float a, float b, uint32_t &hi, uint32_t &lo) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    const __nv_bfloat162 l = __floats2bfloat162_rn(a - __low2float(h), b - __high2float(h));
    hi = *reinterpret_cast<const uint32_t *>(&h);
    lo = *reinterpret_cast<const uint32_t *>(&l);
}

// Epilogues.  A lane holds one weight row and acc[j] its value for position m0 + j.  Thirty-two positions at a time go through
// shared memory (x[position][weight row of the warp]), from where they are written in whole sectors.  What a round needs
// from memory is loaded before anything is stored: the compiler cannot move a load over a store that might alias, and one
// round trip to L2 per position made the QKV epilogue 40 us long.
template <class Body> __device__ __forceinline__ void epi_rounds(const float (&acc)[128], float (*x)[32], int lane, int left, Body &&body) {
#pragma unroll 1
    for (int g = 0; 32 * g < left; ++g) {
        __syncwarp();
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (g == k) {
#pragma unroll
                for (int j = 0; j < 32; ++j) x[j][lane] = acc[32 * k + j];
            }
        __syncwarp();
        body(32 * g, min(32, left - 32 * g));
    }
}

// One set of sums of an epilogue warp in scratch: 16 bytes of every lane side by side.
__device__ __forceinline__ void sums_store(const float (&acc)[128], float4 *o, int nh) {
#pragma unroll
    for (int j = 0; j < 32; ++j)
        if (4 * j < nh) __stcg(o + 32 * j, make_float4(acc[4 * j], acc[4 * j + 1], acc[4 * j + 2], acc[4 * j + 3]));
}
// acc += what sums_store left: sixteen loads in flight, more would not fit beside the sums.
__device__ __forceinline__ void sums_add(float (&acc)[128], const float4 *src, int nh) {
#pragma unroll
    for (int j0 = 0; j0 < 32; j0 += 16) {
        if (4 * j0 >= nh) break;
        float4 r[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) r[j] = 4 * (j0 + j) < nh ? ld_cg_inorder(src + 32 * (j0 + j)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const int e = 4 * (j0 + j);
            acc[e] += r[j].x; acc[e + 1] += r[j].y; acc[e + 2] += r[j].z; acc[e + 3] += r[j].w;
        }
    }
}

// Y[m][n] = or += x: four neighbouring n per lane, four positions per access.  N arbitrary, ldy a multiple of 4.
template <bool ADD> __device__ __forceinline__ void epi_rows(const float (*x)[32], float *y, int ldy, int n_left, int lane, int left) {
    const int n = 4 * (lane & 7);
    y += n;
    if (n + 4 <= n_left) {
        float4 r[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int j = 4 * i + (lane >> 3);
            r[i] = *reinterpret_cast<const float4 *>(&x[j][n]);
            if (ADD && j < left) {
                const float4 o = *reinterpret_cast<const float4 *>(y + (size_t)j * ldy);
                r[i].x += o.x; r[i].y += o.y; r[i].z += o.z; r[i].w += o.w;
            }
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int j = 4 * i + (lane >> 3);
            if (j < left) *reinterpret_cast<float4 *>(y + (size_t)j * ldy) = r[i];
        }
    } else {
        for (int j = lane >> 3; j < left; j += 4)
            for (int e = 0; n + e < n_left; ++e) y[(size_t)j * ldy + e] = x[j][n + e] + (ADD ? y[(size_t)j * ldy + e] : 0.f);
    }
}

// q, k and v: the products are those of the rows before normalisation (k_norm_split_rows) and take its factor here.
// The weight rows come reordered (see k_repack_qkv), so that rows r and r + 8 of 16 are the partners of a rotation.
// q and k are rotated, q is scaled and split into bf16 high and low parts, k and v go to the cache rows of the positions
// (16-byte chunks xor-swizzled, see kv_swz).  n_w: first weight row of the warp; all 32 belong to one head.  A lane
// computes one pair of partners for every second position and, with its neighbour, writes two neighbouring features.
template <int HD> __device__ __forceinline__ void epi_qkv(const Ctx &c, const GemmArgs &a, const float (*x)[32], int n_w, int lane, int m0, int left) {
    const int qd = c.nq * HD, kvd = c.nkv * HD;
    const int which = n_w < qd ? 0 : n_w < qd + kvd ? 1 : 2;
    const int nr = n_w - (which == 0 ? 0 : which == 1 ? qd : qd + kvd), head = nr / HD, r0 = nr % HD;   // first row within the head
    const int l = lane & 15, row = (l >> 3) * 16 + (l & 7);          // the pair is rows `row` and `row` + 8 of the warp's 32
    const bool odd = lane & 1;
    const int jj = r0 / 2 + l;                                        // frequency of the pair
    // features this lane writes: of the rotation's lower half (even lanes) or upper half (odd lanes); v rows are in order
    const int fe = which < 2 ? (jj & ~1) + (odd ? HD / 2 : 0) : r0 + (row & ~1) + (odd ? 8 : 0);
    const float scale = which == 0 ? rsqrtf((float)HD) : 1.f;
    const int32_t *table = c.page_table + (size_t)a.seq * c.max_pages;
    __nv_bfloat16 *pool = reinterpret_cast<__nv_bfloat16 *>(c.kv_pool);
    float2 cs[16];
    float rstd[16];
    int page[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const int m = m0 + min(2 * i + (lane >> 4), left - 1);
        rstd[i] = a.rstd[m];
        if (which < 2) cs[i] = *reinterpret_cast<const float2 *>(a.cs + ((size_t)m * (HD / 2) + jj) * 2);
        if (which > 0) page[i] = table[(a.pos0 + m) >> c.page_shift];
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const int jm = 2 * i + (lane >> 4), m = m0 + jm;
        float y0 = x[jm][row] * rstd[i], y1 = x[jm][row + 8] * rstd[i];
        if (which < 2) {   // the same in every lane
            const float z0 = y0 * cs[i].x - y1 * cs[i].y, z1 = y1 * cs[i].x + y0 * cs[i].y;
            y0 = z0 * scale; y1 = z1 * scale;
        }
        const float got = __shfl_xor_sync(0xffffffffu, odd ? y0 : y1, 1);
        const float v0 = odd ? got : y0, v1 = odd ? y1 : got;
        if (jm < left) {
            if (which == 0) {
                uint32_t h, w;
                split2(v0, v1, h, w);
                const size_t o = (size_t)m * qd + head * HD + fe;
                *reinterpret_cast<uint32_t *>(a.hi + o) = h;
                *reinterpret_cast<uint32_t *>(a.lo + o) = w;
            } else {
                const int pos = a.pos0 + m, t = pos & (c.page_tokens - 1);
                const size_t base = ((((size_t)page[i] * c.L + a.layer) * 2 + (which - 1)) * c.nkv + head) * ((size_t)c.page_tokens * HD) + (size_t)t * HD;
                *reinterpret_cast<__nv_bfloat162 *>(pool + base + ((((fe >> 3) ^ (pos & c.kv_swz)) << 3) | (fe & 7))) = __floats2bfloat162_rn(v0, v1);
            }
        }
    }
}

// SwiGLU: rows 0 .. 15 are the gate values of sixteen features, rows 16 .. 31 their up values; a lane takes two neighbouring
// features of every fourth position.  The activations are split into bf16 high and low parts.
__device__ __forceinline__ void epi_swiglu(const float (*x)[32], const float *rstd, __nv_bfloat16 *hi, __nv_bfloat16 *lo, int ld, int lane, int left) {
    const int n = 2 * (lane & 7);
    uint32_t h[8], l[8];
    float rs[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) rs[i] = rstd[min(4 * i + (lane >> 3), left - 1)];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int j = 4 * i + (lane >> 3);
        float2 g = *reinterpret_cast<const float2 *>(&x[j][n]), u = *reinterpret_cast<const float2 *>(&x[j][16 + n]);
        g.x *= rs[i]; g.y *= rs[i]; u.x *= rs[i]; u.y *= rs[i];
        split2(g.x / (1.0f + expf(-g.x)) * u.x, g.y / (1.0f + expf(-g.y)) * u.y, h[i], l[i]);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int j = 4 * i + (lane >> 3);
        if (j < left) {
            *reinterpret_cast<uint32_t *>(hi + (size_t)j * ld + n) = h[i];
            *reinterpret_cast<uint32_t *>(lo + (size_t)j * ld + n) = l[i];
        }
    }
}

// Waits until the epilogue warp ew of a CTA has published its sums of this launch (whole warp).
template <typename SM> __device__ __forceinline__ bool flag_wait(SM *sm, const GemmArgs &a, int cta, int ew) {
    const unsigned *f = a.flag + cta * GEPI_WARPS + ew;
    const unsigned long long t0 = gtime();
    bool ok = true;
    for (;;) {
        unsigned v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(f) : "memory");
        if (v == a.epoch) break;
        if (*(volatile int *)&sm->abort) { ok = false; break; }
        if (gtime() - t0 > a.wait_ns) {
            atomicCAS(a.err, 0, ERR_TIMEOUT_MBAR);
            *(volatile int *)&sm->abort = 1;
            ok = false;
            break;
        }
    }
    return __all_sync(0xffffffffu, ok);
}

// mapXhi / mapXlo: 2-D maps over the bf16 matrices [rows][K] (box 64 x plan.nt / 2); mapW0, mapW1: over the weight matrices
// [N][K] (box 64 x 128; SwiGLU: gate and up, box 64 x 16); all 128-byte swizzled, zero fill outside.  K a multiple of 64.
// Grid: 2 x plan.pairs CTAs.
template <int EPI, int HD>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(GTHREADS, 1)
k_dense_gemm(const __grid_constant__ CUtensorMap mapXhi, const __grid_constant__ CUtensorMap mapXlo, const __grid_constant__ CUtensorMap mapW0,
             const __grid_constant__ CUtensorMap mapW1, const __grid_constant__ Ctx c, const __grid_constant__ GemmArgs a) {
    extern __shared__ unsigned char dsm_raw[];
    DSmem *sm = reinterpret_cast<DSmem *>(dsm_raw + ((1024u - (s32(dsm_raw) & 1023u)) & 1023u));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    const int pair = blockIdx.x >> 1, nkb = a.K / BK, nt = a.plan.nt, ck = a.plan.ck;
    const int x_bytes = nt / 2 * BK * 2, stage_bytes = W_BYTES + 2 * x_bytes, stages = min(MAX_STAGES, RING_BYTES / stage_bytes);
    pdl_trigger();
    if (threadIdx.x == 0) {
        for (int i = 0; i < MAX_STAGES; ++i) { mbar_init(&sm->full[i], 1); mbar_init(&sm->empty[i], 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(&sm->acc_full[i], 1); mbar_init(&sm->acc_empty[i], 2 * GEPI_WARPS); }
        sm->abort = 0;
        sm->wait_ns = a.wait_ns;
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
            auto load_w = [&](int st, int kb, int tn) {
                if (rank == 0) mbar_expect_tx(&sm->full[st], 2u * (uint32_t)stage_bytes);   // both CTAs' tiles complete on the first CTA's barrier
                const uint32_t bar = map_to_cta(&sm->full[st], 0);
                unsigned char *dst = sm->ring + st * stage_bytes;
                if (EPI == EPI_SWIGLU) {   // sixteen gate rows, the same rows of up, ...: one warp's lanes hold both
                    for (int i = 0; i < 4; ++i) {
                        const int f = tn * BW + (int)rank * 64 + 16 * i;
                        tma_load_2d_pair(dst + i * 4096, &mapW0, kb * BK, f, bar);
                        tma_load_2d_pair(dst + i * 4096 + 2048, &mapW1, kb * BK, f, bar);
                    }
                } else tma_load_2d_pair(dst, &mapW0, kb * BK, tn * TW + (int)rank * BW, bar);
            };
            // the weights of the first stages do not depend on earlier kernels
            int ahead = 0;
            {
                Sched sch(a.plan, pair);
                Seg s;
                if (sch.next(s)) {
                    const int kb0 = s.c0 * ck, kb1 = min(s.c1 * ck, nkb);
                    for (; ahead < stages && kb0 + ahead < kb1; ++ahead) load_w(ahead, kb0 + ahead, s.tile / a.plan.mt);
                }
            }
            pdl_wait();
            Sched sch(a.plan, pair);
            Seg s;
            int it = 0, st = 0;
            uint32_t ph = 1;
            bool ok = true;
            while (ok && sch.next(s)) {
                const int tm = s.tile % a.plan.mt, tn = s.tile / a.plan.mt, x0 = tm * nt + (int)rank * (nt / 2), kb1 = min(s.c1 * ck, nkb);
                for (int kb = s.c0 * ck; kb < kb1; ++kb, ++it) {
                    if (it >= ahead) {
                        ok = dwait(sm, a.err, &sm->empty[st], ph);
                        if (!ok) break;
                        load_w(st, kb, tn);
                    }
                    const uint32_t bar = map_to_cta(&sm->full[st], 0);
                    unsigned char *dst = sm->ring + st * stage_bytes + W_BYTES;
                    tma_load_2d_pair(dst, &mapXhi, kb * BK, x0, bar);
                    tma_load_2d_pair(dst + x_bytes, &mapXlo, kb * BK, x0, bar);
                    if (++st == stages) { st = 0; ph ^= 1; }
                }
            }
        }
        if (warp == 1 && lane == 0 && rank == 0) {
            const uint32_t id = Idesc<TW, 0>::v | ((uint32_t)(nt >> 3) << 17);
            Sched sch(a.plan, pair);
            Seg s;
            int ch = 0, st = 0;
            uint32_t ph = 0;
            bool ok = true;
            while (ok && sch.next(s)) {
                for (int cc = s.c0; ok && cc < s.c1; ++cc, ++ch) {
                    const int b = ch & 1, kb1 = min((cc + 1) * ck, nkb);
                    ok = dwait(sm, a.err, &sm->acc_empty[b], ((ch >> 1) & 1) ^ 1);
                    if (!ok) break;
                    tc_fence_after();
                    uint32_t add = 0;
                    for (int kb = cc * ck; kb < kb1; ++kb) {
                        ok = dwait(sm, a.err, &sm->full[st], ph);
                        if (!ok) break;
                        tc_fence_after();
                        const uint32_t base = s32(sm->ring + st * stage_bytes);
                        const unsigned long long w = smem_desc(base), xh = smem_desc(base + W_BYTES), xl = smem_desc(base + W_BYTES + x_bytes);
                        const uint32_t acc = tmem + (uint32_t)(b * 256);
#pragma unroll
                        for (int k = 0; k < BK / 16; ++k) {   // 32 bytes further along the swizzled row per K = 16 step
                            umma_pair(acc, w + 2 * k, xh + 2 * k, id, k == 0 ? add : 1u);
                            umma_pair(acc, w + 2 * k, xl + 2 * k, id, 1u);
                        }
                        add = 1u;
                        umma_commit_pair(&sm->empty[st]);   // the stage is free in both CTAs once these MMAs have read it
                        if (++st == stages) { st = 0; ph ^= 1; }
                    }
                    umma_commit_pair(&sm->acc_full[b]);
                }
            }
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(GREGS_EPI));
        // epilogue: warp w may read the 32 lanes 32 (w % 4) .. of the tensor memory; lane = weight row within the CTA's 128
        const int q = warp & 3, h = (warp - 4) >> 2, ew = warp - 4, nh = nt / 2;
        const uint32_t t_lane = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(h * nh);
        pdl_wait();
        Sched sch(a.plan, pair);
        Seg s;
        int ch = 0;
        bool ok = true;
        while (ok && sch.next(s)) {
            const int tm = s.tile % a.plan.mt, tn = s.tile / a.plan.mt;
            // first position; first weight row (SwiGLU: feature) of the warp
            const int m0 = tm * nt + h * nh, n_w = EPI == EPI_SWIGLU ? tn * BW + (int)rank * 64 + q * 16 : tn * TW + (int)rank * BW + q * 32;
            const int left = min(nh, a.rows - m0);
            const bool live = left > 0 && n_w < a.N;   // the same in every lane, and in the same warp of every pair
            float acc[128];
#pragma unroll
            for (int j = 0; j < 128; ++j) acc[j] = 0.f;
            const int chunks = a.plan.chunks, end = s.c1;
            const bool last = end == chunks;                 // this pair finishes the tile
            const bool middle = s.c0 > 0 && !last;           // one group, published by itself
            const int cta = 2 * pair + (int)rank;
            auto slot = [&](int at, int which) {
                return reinterpret_cast<float4 *>(reinterpret_cast<unsigned char *>(a.part) + (size_t)at * GPART_CTA + which * GPART_SLOT + ew * GPART_WARP) + lane;
            };
            int cc = s.c0, grp = 0;
            while (a.plan.group[grp + 1] <= cc) ++grp;
            // Steps of a segment, each in one place of the code (the instruction cache is what a second copy of 128 additions
            // costs: 6 us per launch): add sums from scratch, store the sums and go on from zero, multiply to the end of the
            // group or of the segment.
            const int own_slot = last ? SLOT_OWN : SLOT_TOTAL;
            int add_from = 0, add_n = 0, add_slot = SLOT_TOTAL;   // sums to add: add_slot of add_n CTAs from add_from on, every second one
            float4 *store_to = nullptr;
            bool own_total = false;                          // the total of the groups before this one is in this CTA's scratch
            bool group_done = false, publish = false;
            if (live && cc > a.plan.group[grp]) {     // the pair before this one began the group
                add_from = cta - 2;
                add_n = 1;
                add_slot = SLOT_GROUP;
            }
            while (ok) {
                for (; add_n > 0; --add_n, add_from += 2) {
                    if (add_from != cta && !(ok = flag_wait(sm, a, add_from, ew))) break;
                    sums_add(acc, slot(add_from, add_from == cta ? own_slot : add_slot), nh);
                }
                if (!ok) break;
                if (store_to) {
                    sums_store(acc, store_to, nh);
                    if (publish) break;
                    store_to = nullptr;
#pragma unroll
                    for (int j = 0; j < 128; ++j) acc[j] = 0.f;
                    if (group_done) {   // these were set aside: first the other pairs' in their order, then they themselves
                        add_n = (cta - add_from) / 2 + 1;
                        continue;
                    }
                }
                if (group_done) {
                    group_done = false;
                    ++grp;
                    if (cc == end && last) break;
                    if (live) {
                        store_to = slot(cta, own_slot);
                        publish = cc == end;
                        own_total = true;
                        continue;
                    }
                    if (cc == end) break;
                }
                const int grp_end = a.plan.group[grp + 1], stop = min(end, grp_end);
                for (; cc < stop; ++cc, ++ch) {
                    const int b = ch & 1;
                    ok = dwait(sm, a.err, &sm->acc_full[b], (ch >> 1) & 1);
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                    tc_fence_after();
                    if (live) {
#pragma unroll
                        for (int g = 0; g < 8; ++g)
                            if (16 * g < nh) {
                                uint32_t v[16];
                                tmem_ld16(v, t_lane + (uint32_t)(b * 256 + 16 * g));
#pragma unroll
                                for (int e = 0; e < 16; ++e) acc[16 * g + e] += __uint_as_float(v[e]);
#pragma unroll
                                for (int e = 0; e < 16; ++e) asm volatile("" : "+f"(acc[16 * g + e]));
                            }
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_at(map_to_cta(&sm->acc_empty[b], 0));
                }
                if (!ok) break;
                if (stop < grp_end) {             // the next pair goes on with this group
                    if (!live) break;
                    store_to = slot(cta, SLOT_GROUP);
                    publish = true;
                    continue;
                }
                group_done = true;
                if (!live || grp == 0 || middle) continue;
                if (own_total) { add_from = cta; add_n = 1; }
                else {                            // other pairs hold the groups before this one
                    int p0 = pair - 1;
                    while (p0 > 0 && a.plan.start[p0] > (s.tile - a.plan.whole) << 16) --p0;
                    add_from = 2 * p0 + (int)rank;
                    add_slot = SLOT_TOTAL;
                    if (p0 == pair - 1) add_n = 1;
                    else store_to = slot(cta, own_slot);
                }
            }
            if (!ok || !live) continue;
            if (!last) {   // another pair finishes this tile
                __threadfence();
                __syncwarp();
                if (lane == 0) asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(a.flag + cta * GEPI_WARPS + ew), "r"(a.epoch) : "memory");
                continue;
            }
            float(*x)[32] = sm->stash[ew];
            epi_rounds(acc, x, lane, left, [&](int j0, int cnt) {
                const int m = m0 + j0;
                if constexpr (EPI == EPI_STORE || EPI == EPI_ADD) epi_rows<EPI == EPI_ADD>(x, a.Y + (size_t)m * a.ldy + n_w, a.ldy, a.N - n_w, lane, cnt);
                else if constexpr (EPI == EPI_QKV) epi_qkv<HD>(c, a, x, n_w, lane, m, cnt);
                else epi_swiglu(x, a.rstd + m, a.hi + (size_t)m * a.N + n_w, a.lo + (size_t)m * a.N + n_w, a.N, lane, cnt);   // N is a multiple of 64: the warp's features are all there
            });
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

// RMSNorm and split in one pass: x = resid[r] * g -> high and low parts, rstd[r] = 1 / sqrt(mean(resid[r]^2) + eps), which the
// epilogue of the product applies.  (The factor before the split would cost the first layer the exactness of its split: bf16
// embeddings have no low part, their products with the factor have one, and five times as many rounded K and V differed.)
// One CTA (256 threads) per row, four elements per access; K a multiple of 64.
__global__ void __launch_bounds__(256) k_norm_split_rows(const float *X, int K, const __nv_bfloat16 *__restrict__ gain,
                                                         float eps, __nv_bfloat16 *hi, __nv_bfloat16 *lo, float *rstd) {
    const int r = blockIdx.x;
    __shared__ float red[8];
    pdl_begin();
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
    if (threadIdx.x == 0) rstd[r] = 1.0f / sqrtf(tot / K + eps);
    for (int i = threadIdx.x; i < K / 4; i += 256) {
        const float4 v = x[i];
        const uint2 gq = reinterpret_cast<const uint2 *>(gain)[i];
        uint2 h, l;
        split2(v.x * __uint_as_float(gq.x << 16), v.y * __uint_as_float(gq.x & 0xffff0000u), h.x, l.x);
        split2(v.z * __uint_as_float(gq.y << 16), v.w * __uint_as_float(gq.y & 0xffff0000u), h.y, l.y);
        reinterpret_cast<uint2 *>(hi + (size_t)r * K)[i] = h;
        reinterpret_cast<uint2 *>(lo + (size_t)r * K)[i] = l;
    }
}

// fp32 rows X[r][ldx] -> the two bf16 matrices [rows][K] the dense GEMM reads: high part and low part (x = hi + lo).  One
// block per row.
__global__ void k_split_rows(const float *__restrict__ X, int ldx, int K, __nv_bfloat16 *__restrict__ hi, __nv_bfloat16 *__restrict__ lo) {
    const int r = blockIdx.x;
    for (int k = threadIdx.x; k < K; k += blockDim.x) {
        const float v = X[(size_t)r * ldx + k];
        const __nv_bfloat16 h = __float2bfloat16_rn(v);
        hi[(size_t)r * K + k] = h;
        lo[(size_t)r * K + k] = __float2bfloat16_rn(v - __bfloat162float(h));
    }
}

// ---------------------------------------------------------------- causal attention of a block of prompt positions
//
// Work item = one kv head x 256 query rows: two tiles of 128 rows, a row being one (position, q head of the kv head's
// group) pair, so that the q heads of a group share every K and V tile.  K and V tiles of 128 positions come from the
// cache pages by TMA exactly as they are stored: the cache's own 16-byte-chunk swizzle is the 128-byte swizzle of the
// tensor core's operand layouts (K: K-major; V: MN-major), so nothing is rearranged.  Per tile and key tile
//     S = Q.lo K^T + Q.hi K^T  (tensor memory, 128 columns)  ->  softmax, one thread per row  ->
//     P as bf16 high and low parts over the columns of S  ->  O += P V  (A operand from tensor memory).
// The two tiles take turns: the tensor core works on one while the 128 threads of the other compute its softmax.
// Online softmax with a lazy reference: O is rescaled only when a row's maximum has grown by more than 2^8 since its
// reference was set (the reference cancels in the end), so most key tiles touch O in the tensor core only.
//
// What bounds it: the tensor core, 4 x 128 x 128 x HD multiply-adds per tile and key tile (high and low parts of Q and
// of P), 2048 cycles at HD = 128; the softmax of a tile takes about 1500 cycles of its warps and hides behind the other
// tile.  Key tiles of 128 because an S of 64 columns would read Q from shared memory twice as often as its bandwidth
// (128 B per cycle) allows.  Rows are independent of each other, so positions past the prompt only waste work.
//
// A masked position has probability zero, which hides everything but a V that is not finite.  So the V tiles that some row
// of the item must not see whole are gone over before the tensor core reads them: rows behind the item's last position
// are cleared (they hold another sequence's rows, or none), and a value that is not finite becomes zero, its feature
// remembered with the position: the rows that do see it get NaN in the end, which is what p * V would have left of them.
// One warp, 0.3 us per tile, for the one to three key tiles at the diagonal.
constexpr int AT_Q = 128, AT_K = 128, AT_THREADS = 384;
constexpr int AT_REGS_ISSUE = 56, AT_REGS_SOFT = 224;   // (56 + 224 + 224) x 128 = 168 x 384
template <int HD> struct AtSmem {   // must start on a 1024-byte boundary
    static constexpr int HALF = AT_Q * 128;             // 128 rows x 64 features
    static constexpr int KV = HD / 64 * AT_K * 128;     // one K or V tile
    static constexpr int SLOTS = HD == 128 ? 3 : 6;
    alignas(1024) unsigned char q[2][2][HD / 64][HALF];  // [tile][high | low][64-feature group]
    alignas(1024) unsigned char kv[SLOTS][KV];           // ring of K and V tiles in turn
    alignas(8) unsigned long long q_full[2], kv_full[SLOTS], kv_empty[SLOTS], s_full[2], p_full[2], o_full[2], diag;
    int bad[HD];                                         // per feature: first position of a causally cut key tile whose V is not finite
    int any_bad;
    unsigned long long wait_ns;
    uint32_t tmem_base;
    int abort;
};
template <int HD> constexpr size_t at_smem_bytes() { return sizeof(AtSmem<HD>) + 1024; }
static_assert(at_smem_bytes<128>() <= 232448, "exceeds the 227 KB of shared memory a block may use");

// Descriptor of V [128 positions][64 features] x groups as the MN-major B operand: 64-feature groups AT_K x 128 bytes
// apart (leading byte offset), groups of eight positions 1024 bytes apart (stride byte offset), 128-byte swizzle.
__device__ __forceinline__ unsigned long long smem_desc_mn(uint32_t saddr) {
    return (unsigned long long)((saddr >> 4) & 0x3fffu) | ((unsigned long long)(AT_K * 128 / 16) << 16) | (64ull << 32) | (1ull << 46) | (2ull << 61);
}
__device__ __forceinline__ void umma_ss(uint32_t d, unsigned long long a, unsigned long long b, uint32_t id, uint32_t accumulate) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d), "l"(a), "l"(b),
                 "r"(id), "r"(accumulate)
                 : "memory");
}
__device__ __forceinline__ void umma_ts(uint32_t d, uint32_t a, unsigned long long b, uint32_t id, uint32_t accumulate) {   // A from tensor memory
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d), "r"(a), "l"(b),
                 "r"(id), "r"(accumulate)
                 : "memory");
}
__device__ __forceinline__ void umma_commit(unsigned long long *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(s32(bar)) : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t addr, const uint32_t *v) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};" ::"r"(addr),
                 "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
                   "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
                 : "memory");
}
__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ void tma_tile_2d(void *dst, const CUtensorMap *map, int c0, int c1, unsigned long long *bar) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(s32(dst)), "l"(map),
                 "r"(c0), "r"(c1), "r"(s32(bar))
                 : "memory");
}
__device__ __forceinline__ void tma_tile_3d(void *dst, const CUtensorMap *map, int c0, int c1, int c2, unsigned long long *bar) {
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(s32(dst)),
                 "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(s32(bar))
                 : "memory");
}

// Takes the values that are not finite out of the first `seen` rows of a V tile (positions from p0 on); see above.  Rare, and out
// of line for that reason.  Chunk c of row r is stored at c ^ (r % 8).
template <int HD> __device__ __noinline__ void pf_attn_take_out(AtSmem<HD> *sm, unsigned char *tile, int p0, int seen, int lane) {
    if (*(volatile int *)&sm->any_bad == 0)
        for (int f = lane; f < HD; f += 32) sm->bad[f] = INT_MAX;
    __syncwarp();
    for (int g = 0; g < HD / 64; ++g)
        for (int i = lane; i < seen * 8; i += 32) {
            __nv_bfloat16 *x = reinterpret_cast<__nv_bfloat16 *>(tile + g * (AT_K * 128) + i * 16);
            const int row = i >> 3, f = g * 64 + ((i ^ row) & 7) * 8;
            for (int e = 0; e < 8; ++e)
                if (!isfinite(__bfloat162float(x[e]))) {
                    atomicMin(&sm->bad[f + e], p0 + row);
                    x[e] = __float2bfloat16_rn(0.f);
                }
        }
    __syncwarp();
    if (lane == 0) *(volatile int *)&sm->any_bad = 1;
    __syncwarp();
}

// mapQhi / mapQlo: 3-D maps over the queries [rows][q heads][HD] (box 64 x GROUP x 128 / GROUP, 128-byte swizzle, rows past
// the block read as zero).  mapKV: 2-D map over the page pool as rows of HD elements (box 64 x kv_box rows, no swizzle).
// Grid: (256-row items of the block) x kv heads, the items with the longest context first.
template <int HD, int GROUP>
__global__ void __launch_bounds__(AT_THREADS, 1)
k_pf_attn(const __grid_constant__ CUtensorMap mapQhi, const __grid_constant__ CUtensorMap mapQlo, const __grid_constant__ CUtensorMap mapKV,
          const __grid_constant__ Ctx c, int layer, int rows, int seq, int pos0, int kv_box, __nv_bfloat16 *ohi,
          __nv_bfloat16 *olo, int *err, unsigned long long wait_ns) {
    typedef AtSmem<HD> Sm;
    constexpr int PT = AT_Q / GROUP, SLOTS = Sm::SLOTS, HG = HD / 64;
    extern __shared__ unsigned char dsm_raw[];
    Sm *sm = reinterpret_cast<Sm *>(dsm_raw + ((1024u - (s32(dsm_raw) & 1023u)) & 1023u));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int kvh = blockIdx.x % c.nkv, item = gridDim.x / c.nkv - 1 - blockIdx.x / c.nkv;
    const int r0 = item * 2 * PT;                                  // first row (position within the block) of the item
    const int last = pos0 + min(r0 + 2 * PT, rows) - 1;            // last position any row of the item sees
    int n_kt[2];                                                   // key tiles of the two query tiles (0: the tile has no rows)
#pragma unroll
    for (int t = 0; t < 2; ++t) n_kt[t] = r0 + t * PT < rows ? (pos0 + min(r0 + (t + 1) * PT, rows) - 1) / AT_K + 1 : 0;
    const int n = max(n_kt[0], n_kt[1]);
    pdl_trigger();
    if (threadIdx.x == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(&sm->q_full[i], 1); mbar_init(&sm->s_full[i], 1); mbar_init(&sm->p_full[i], 4); mbar_init(&sm->o_full[i], 1);
        }
        for (int i = 0; i < SLOTS; ++i) { mbar_init(&sm->kv_full[i], 1); mbar_init(&sm->kv_empty[i], 1); }
        mbar_init(&sm->diag, 1);
        sm->any_bad = 0;
        sm->abort = 0;
        sm->wait_ns = wait_ns;
        fence_mbar_init();
        fence_proxy_async();
    }
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s32(&sm->tmem_base)), "r"(TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *(volatile uint32_t *)&sm->tmem_base;   // columns: S of the tiles at 0 and 128, O at 256 and 384

    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(AT_REGS_ISSUE));
        if (warp == 0) {
            pdl_wait();
            const int32_t *table = c.page_table + (size_t)seq * c.max_pages;
            const int last_page = last >> c.page_shift;
            if (lane == 0)
                for (int t = 0; t < 2; ++t) {
                    if (n_kt[t] == 0) continue;
                    mbar_expect_tx(&sm->q_full[t], 2u * HG * Sm::HALF);
                    for (int g = 0; g < HG; ++g) {
                        tma_tile_3d(sm->q[t][0][g], &mapQhi, g * 64, kvh * GROUP, r0 + t * PT, &sm->q_full[t]);
                        tma_tile_3d(sm->q[t][1][g], &mapQlo, g * 64, kvh * GROUP, r0 + t * PT, &sm->q_full[t]);
                    }
                }
            bool ok = true;
            int n_cut = 0;
            for (int it = 0; ok && it < 2 * n; ++it) {   // K of key tile 0, V of key tile 0, K of key tile 1, ...
                const int st = it % SLOTS, j = it >> 1, which = it & 1;
                ok = dwait(sm, err, &sm->kv_empty[st], ((it / SLOTS) & 1) ^ 1);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                const bool cut = which == 1 && (j + 1) * AT_K - 1 > pos0 + r0;   // some row of the item does not see the whole tile
                unsigned long long *bar = cut ? &sm->diag : &sm->kv_full[st];
                if (lane == 0) {
                    mbar_expect_tx(bar, (uint32_t)Sm::KV);
                    for (int r = 0; r < AT_K; r += kv_box) {
                        const int p = j * AT_K + r, page = table[min(p >> c.page_shift, last_page)];
                        const int row = (int)(((((long long)page * c.L + layer) * 2 + which) * c.nkv + kvh) * c.page_tokens) + (p & (c.page_tokens - 1));
                        for (int g = 0; g < HG; ++g) tma_tile_2d(sm->kv[st] + g * (AT_K * 128) + r * 128, &mapKV, g * 64, row, bar);
                    }
                }
                __syncwarp();
                if (cut) {
                    ok = dwait(sm, err, &sm->diag, n_cut & 1);
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                    ++n_cut;
                    const int seen = min(AT_K, last + 1 - j * AT_K);   // rows of the tile that the item sees
                    uint32_t found = 0;
                    for (int g = 0; g < HG; ++g) {
                        uint4 *v = reinterpret_cast<uint4 *>(sm->kv[st] + g * (AT_K * 128));
                        int i = lane;
#pragma unroll 8
                        for (; i < seen * 8; i += 32) {   // exponent bits all set: adding one to them carries into the sign bit
                            const uint4 x = v[i];
                            found |= ((x.x & 0x7f807f80u) + 0x00800080u) | ((x.y & 0x7f807f80u) + 0x00800080u) |
                                     ((x.z & 0x7f807f80u) + 0x00800080u) | ((x.w & 0x7f807f80u) + 0x00800080u);
                        }
                        for (; i < AT_K * 8; i += 32) v[i] = make_uint4(0, 0, 0, 0);
                    }
                    if (__any_sync(0xffffffffu, (found & 0x80008000u) != 0)) pf_attn_take_out<HD>(sm, sm->kv[st], j * AT_K, seen, lane);
                    fence_proxy_async();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&sm->kv_full[st]);
                }
            }
        } else if (warp == 1 && lane == 0) {
            constexpr uint32_t ID_S = Idesc<AT_Q, AT_K>::v, ID_O = Idesc<AT_Q, HD>::v | (1u << 16);   // bit 16: B is MN-major
            bool ok = true;
            auto issue_s = [&](int t, int st) {
                const uint32_t d = tmem + (uint32_t)(t * AT_K);
                uint32_t add = 0;
#pragma unroll 1
                for (int i = 2 * HG - 1; i >= 0; --i) {   // low parts first: the small products are added up before the large ones
                    const int part = i / HG, g = i % HG;
                    const unsigned long long qd = smem_desc(s32(sm->q[t][part][g])), kd = smem_desc(s32(sm->kv[st] + g * (AT_K * 128)));
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        umma_ss(d, qd + 2 * k, kd + 2 * k, ID_S, add);
                        add = 1u;
                    }
                }
                umma_commit(&sm->s_full[t]);
            };
            if (n > 0) ok = dwait(sm, err, &sm->kv_full[0], 0);
            tc_fence_after();
            for (int t = 0; ok && t < 2; ++t) {
                if (n_kt[t] == 0) continue;
                ok = dwait(sm, err, &sm->q_full[t], 0);
                if (!ok) break;
                tc_fence_after();
                issue_s(t, 0);
            }
            if (ok) umma_commit(&sm->kv_empty[0]);
            for (int j = 0; ok && j < n; ++j) {
                const int iv = 2 * j + 1, ik = 2 * j + 2, sv = iv % SLOTS, sk = ik % SLOTS;
                ok = dwait(sm, err, &sm->kv_full[sv], (iv / SLOTS) & 1);
                if (!ok) break;
                tc_fence_after();
                bool have_k = false;
                for (int t = 0; ok && t < 2; ++t) {
                    if (j >= n_kt[t]) continue;
                    ok = dwait(sm, err, &sm->p_full[t], j & 1);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t d = tmem + 256u + (uint32_t)(t * 128), pa = tmem + (uint32_t)(t * AT_K);
                    uint32_t add = j > 0 ? 1u : 0u;
#pragma unroll 1
                    for (int i = 3; i >= 0; --i) {   // P.lo, then P.hi, half of the positions at a time
                        const unsigned long long vd = smem_desc_mn(s32(sm->kv[sv])) + 512 * (i & 1);
                        const uint32_t pi = pa + (uint32_t)(32 * i);
#pragma unroll
                        for (int k = 0; k < 4; ++k) {   // sixteen positions: two groups of eight rows of V, eight columns of P
                            umma_ts(d, pi + (uint32_t)(8 * k), vd + 128 * k, ID_O, add);
                            add = 1u;
                        }
                    }
                    if (t == 1 || n_kt[1] <= j) umma_commit(&sm->kv_empty[sv]);
                    if (j + 1 < n_kt[t]) {
                        if (!have_k) {
                            ok = dwait(sm, err, &sm->kv_full[sk], (ik / SLOTS) & 1);
                            if (!ok) break;
                            tc_fence_after();
                            have_k = true;
                        }
                        issue_s(t, sk);
                    } else umma_commit(&sm->o_full[t]);
                }
                if (ok && j + 1 < n) umma_commit(&sm->kv_empty[sk]);
            }
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(AT_REGS_SOFT));
        const int t = (warp - 4) >> 2, q = warp & 3, row = q * 32 + lane;
        const int r = r0 + t * PT + row / GROUP, pos = pos0 + r;             // row of the block, its position
        const int pos_min = pos0 + r0 + t * PT;                              // smallest position of the tile
        const uint32_t t_s = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(t * AT_K), t_o = tmem + ((uint32_t)(q * 32) << 16) + 256u + (uint32_t)(t * 128);
        constexpr float LOG2E = 1.4426950408889634f;
        pdl_wait();
        float ref = 0.f, l = 0.f;   // ref: reference exponent (log2 units) the row's P, O and l are relative to
        bool ok = true;
        for (int j = 0; ok && j < n_kt[t]; ++j) {
            ok = dwait(sm, err, &sm->s_full[t], j & 1);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after();
            uint32_t s[128];
            tmem_ld128(s, t_s);
            if ((j + 1) * AT_K - 1 > pos_min) {   // some row of the tile does not see all of these positions
                const int lim = pos - j * AT_K;
#pragma unroll
                for (int e = 0; e < 128; ++e) s[e] = e <= lim ? s[e] : 0xff800000u;
            }
            float mx[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) mx[e] = __uint_as_float(s[e]);
#pragma unroll
            for (int e = 4; e < 128; ++e) mx[e & 3] = fmaxf(mx[e & 3], __uint_as_float(s[e]));
            const float m2 = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * LOG2E;
            if (j == 0) ref = m2;
            else if (__any_sync(0xffffffffu, m2 > ref + 8.f)) {
                // the previous key tile's O is complete (its products were issued before those of this S)
                const float nr = m2 > ref + 8.f ? m2 : ref, f = ex2(ref - nr);
                ref = nr;
                l *= f;
#pragma unroll 1
                for (int b = 0; b < HD / 32; ++b) {
                    uint32_t v[32];
                    tmem_ld32(v, t_o + 32 * b);
#pragma unroll
                    for (int e = 0; e < 32; ++e) v[e] = __float_as_uint(__uint_as_float(v[e]) * f);
                    tmem_st32(t_o + 32 * b, v);
                }
            }
            float sum[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int b = 0; b < 4; ++b) {   // 32 probabilities -> 16 words of high parts and 16 of low parts
                uint32_t h[16], lo[16];
#pragma unroll
                for (int e = 0; e < 16; ++e) {
                    const float p0 = ex2(fmaf(__uint_as_float(s[32 * b + 2 * e]), LOG2E, -ref)), p1 = ex2(fmaf(__uint_as_float(s[32 * b + 2 * e + 1]), LOG2E, -ref));
                    sum[2 * (e & 1)] += p0;
                    sum[2 * (e & 1) + 1] += p1;
                    split2(p0, p1, h[e], lo[e]);
                }
                tmem_st16(t_s + 16 * b, h);
                tmem_st16(t_s + 64 + 16 * b, lo);
            }
            l += (sum[0] + sum[1]) + (sum[2] + sum[3]);
            tmem_st_wait();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm->p_full[t]);
        }
        if (ok && n_kt[t] > 0) {
            ok = dwait(sm, err, &sm->o_full[t], 0);
            ok = __all_sync(0xffffffffu, ok);
            tc_fence_after();
            if (ok) {
                const float inv = 1.0f / l;
                const bool any_bad = *(volatile int *)&sm->any_bad != 0;
                const size_t o = ((size_t)r * c.nq + kvh * GROUP + row % GROUP) * HD;
#pragma unroll 1
                for (int b = 0; b < HD / 32; ++b) {
                    uint32_t v[32];
                    tmem_ld32(v, t_o + 32 * b);
                    if (any_bad)
#pragma unroll
                        for (int e = 0; e < 32; ++e) v[e] = pos >= *(volatile int *)&sm->bad[32 * b + e] ? 0x7fc00000u : v[e];
                    if (r < rows)
#pragma unroll
                        for (int e = 0; e < 32; e += 8) {
                            uint4 h, w;
                            split2(__uint_as_float(v[e]) * inv, __uint_as_float(v[e + 1]) * inv, h.x, w.x);
                            split2(__uint_as_float(v[e + 2]) * inv, __uint_as_float(v[e + 3]) * inv, h.y, w.y);
                            split2(__uint_as_float(v[e + 4]) * inv, __uint_as_float(v[e + 5]) * inv, h.z, w.z);
                            split2(__uint_as_float(v[e + 6]) * inv, __uint_as_float(v[e + 7]) * inv, h.w, w.w);
                            *reinterpret_cast<uint4 *>(ohi + o + 32 * b + e) = h;
                            *reinterpret_cast<uint4 *>(olo + o + 32 * b + e) = w;
                        }
                }
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
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    }
}

}  // namespace dg
}  // namespace ada
