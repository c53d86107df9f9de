// fp32 models: whole calls of Algorithm 1, and prompt passes, in one cooperative launch.
//
// A small fp32 model stays in the L2 cache and a step of it is a chain of short products: 22 launches of about 5 us each per
// early exit, and a read-back to decide what to launch next.  Here one CTA per SM walks the layers on the device, and nothing
// but data passes between the CTAs:
//   * every value that another CTA needs travels as an 8-byte word (phase number, fp32 value), written and read by single
//     accesses: whoever sees the expected phase number has the value, so no barrier, fence or counter stands between a
//     product and the next one.  A phase costs one store, one load and its arithmetic;
//   * each CTA keeps the whole decoding state and takes every decision (Eq. 1, verification, rollback) itself, from the same
//     numbers in the same order; CTA 0 also writes them back.  Nobody waits for a decision to be published;
//   * the weights of a warp's first outputs are in registers before the input they multiply has arrived.
// Phases of a layer: RMSNorm + q, k, v with rotation | attention partials (row, head, 128-position chunk) | their merge + O +
// residual | RMSNorm + gate, up, SwiGLU | down + residual.  A buffer is written again a layer later, and a reader that comes late
// would not find its phase number any more.  What holds the writers back is the reader's own next output, which they wait for: so
// every CTA must own an output between each of its reads and the next writing of what it read.  The grid has no more CTAs than the
// model has features (grid_for): each then owns one of O and one of down in every layer, and one of the two lies in every such
// interval (XA: read by q, k, v, written by down; XB: gate / up, O; HT: down, gate / up; PT: O, attention; head partials and
// staged logits: a head, the next one).  What has to last longer than a phase (cache rows, the residual of rows that wait at an
// exit layer, staged logits) is stored plainly and ordered by the exchange of head partials that ends every step: a fence
// before, a fence after.
//
// Invariance rule as in kernels.cuh: a row's numbers depend on that row's inputs and the launch geometry only.
//
// Measured, four layers of width 256 (16 + 128 tokens, up to five early ones): 10.1 ms, 20.2 with a launch per operation.  Plain
// decoding takes 102 us a token: some 3 to 7 us a phase, an exchange through L2 with the latency of its loads before and after.
#pragma once

#include "kernels.cuh"

namespace ada {
namespace rs {

constexpr int THREADS = 256, WARPS = 8;
constexpr int MAX_L = 128;             // layers (their weight pointers are kernel arguments)
constexpr int MAX_SLOTS = 16;          // rows per sequence
constexpr int MAX_R = 64;              // rows of a pass
constexpr int TOK_RING = 32;           // tokens kept per sequence, by position
constexpr int U = 6;                   // 16-byte pieces of a weight row per lane in registers at a time
constexpr int ERR_TIMEOUT = 1, ERR_STEPS = 2;
typedef unsigned long long u64;

struct LayerPtrs { const float *attn_norm, *ffn_norm, *wq, *wk, *wv, *wo, *wg, *wu, *wd; };

struct Args {
    Ctx c;
    const float *tok_embed, *lm_head, *final_norm;
    LayerPtrs layer[MAX_L];
    const float *head_T[MAX_L];          // by 1-based layer (null: identity)
    float head_scale[MAX_L];
    unsigned char exit_at[MAX_L];        // the call consults the head after 1-based layer e
    float rope_base, gamma;
    int batch, max_early, eos_id, tape_n, capture_cap;
    long long max_steps;                 // more steps than any call takes
    u64 *XA, *XB, *QT, *PT, *HT, *TT, *HP;   // exchanged words: layer input, FFN input, q | k | v, attention partials [row][q head][c.n_chunks: as
                                         // many as the call can reach][hd + 2], FFN activations, T output, head partials
    int R;                               // rows of the buffers
    int ku;                              // widest product input: max(d_model, q width, d_ff)
    int cs_ring;                         // rotary factors kept per sequence (a power of two above the rows in flight)
    int page_words;                      // entries of the page table that are kept in shared memory: all, or none
    int store_logits, prof;
    int pf_seq, pf_n;                    // prompt passes of this sequence (pf_n tokens), or pf_n = 0: decode
    int pf_rows;                         // prompt positions per pass
    int *err;
    u64 wait_ns;
};

// decoding state, one copy per CTA
struct State {
    int len[ADA_MAX_BATCH], base[ADA_MAX_BATCH], target[ADA_MAX_BATCH], done[ADA_MAX_BATCH], climbing[ADA_MAX_BATCH], eos_hit[ADA_MAX_BATCH];
    int tok[ADA_MAX_BATCH][TOK_RING];
    int fl[MAX_R], pos[MAX_R];           // rows of the pass: layer at which a row resumes (INT_MAX: idle), its position
    HeadResult hr[MAX_R];
    int n_climbing, n_done, tape_i, log_n, cap_n, keep, keep_row, abort;
};
struct Shm {   // carved from dynamic shared memory
    float *xs, *us, *cs, *ao;            // residual rows [R][d]; product input [R][ku]; rotary factors; attention merge [WARPS][hd + 2]
    Msa *red;                            // [WARPS][R]
    int *fill;                           // [batch][L]
    State *st;
    double *freq;                        // rotary frequencies [hd / 2]
};
__host__ __device__ constexpr size_t walker_bytes(size_t n) { return (n + 15) / 16 * 16; }
__host__ __device__ inline size_t shm_bytes(int R, int d, int ku, int hd, int n_cs, int batch, int L) {
    return sizeof(float) * ((size_t)R * d + (size_t)R * ku + (size_t)n_cs * hd + (size_t)WARPS * (hd + 2)) + sizeof(Msa) * WARPS * (size_t)R +
           sizeof(int) * (size_t)batch * L + sizeof(State) + sizeof(double) * (hd / 2) + walker_bytes(sizeof(Args) + sizeof(Shm) + sizeof(u64)) + 64;
}

// CTAs of a launch on a device of `sms` SMs (see above why no more than d), and the units of a product of `units` that CTA `cta` of
// them works on: unit u is warp u / grid's of CTA u mod grid (Product).
constexpr int MAX_GRID = 256;
__host__ __device__ constexpr int grid_for(int sms, int d) { return sms < MAX_GRID ? (sms < d ? sms : d) : (MAX_GRID < d ? MAX_GRID : d); }
__host__ __device__ constexpr int units_of(int units, int cta, int grid) { return units > cta ? (units - cta + grid - 1) / grid : 0; }

__device__ __forceinline__ int popc64(u64 m) { return __popcll(m); }
__device__ __forceinline__ u64 now() { u64 t; asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t)); return t; }
__device__ __forceinline__ void put(u64 *p, float v, unsigned tag) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(((u64)tag << 32) | __float_as_uint(v)) : "memory");
}
__device__ __forceinline__ bool get(const u64 *p, float &v, unsigned tag) {
    u64 x;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(x) : "l"(p) : "memory");
    v = __uint_as_float((unsigned)x);
    return (unsigned)(x >> 32) == tag;
}
__device__ __forceinline__ bool get2(const u64 *p, float &a, float &b, unsigned tag) {   // two words; 16-byte aligned
    u64 x, y;
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(x), "=l"(y) : "l"(p) : "memory");
    a = __uint_as_float((unsigned)x);
    b = __uint_as_float((unsigned)y);
    return (unsigned)(x >> 32) == tag && (unsigned)(y >> 32) == tag;
}

// Bounded repetition of `load` until it reports success.  Once a wait has run out, here or anywhere in the grid, all waits fall
// through and the CTAs run to the end of the step on whatever is there.
template <class F> __device__ __forceinline__ void until(const Args &A, State *st, F &&load) {
    u64 t0 = 0;
    for (unsigned it = 0;; ++it) {
        if (load()) return;
        if ((it & 31u) == 31u || A.wait_ns < 1000000ull) {
            if (*(volatile int *)&st->abort) return;
            if (*(volatile int *)A.err != 0) { *(volatile int *)&st->abort = 1; return; }
            const u64 t = now();
            if (t0 == 0) t0 = t;
            else if (t - t0 > A.wait_ns) { atomicCAS(A.err, 0, ERR_TIMEOUT); *(volatile int *)&st->abort = 1; return; }
        }
    }
}

__device__ __forceinline__ u64 active_rows(const State *st, int R, int layer) {   // every warp for itself
    const int lane = threadIdx.x & 31;
    const unsigned lo = __ballot_sync(0xffffffffu, lane < R && st->fl[lane] <= layer);
    const unsigned hi = R > 32 ? __ballot_sync(0xffffffffu, lane + 32 < R && st->fl[lane + 32 < MAX_R ? lane + 32 : 0] <= layer) : 0u;
    return ((u64)hi << 32) | lo;
}

// ---------------------------------------------------------------- products

// NW weight rows of a unit, the first U 16-byte pieces per lane.
template <int NW> struct Wreg { float4 w[NW][U]; };
template <int NW, class Ptr> __device__ __forceinline__ void load_w(Wreg<NW> &r, const Ptr &wptr, int unit, int K, int c0) {
    const int lane = threadIdx.x & 31, nch = K / 4;
#pragma unroll
    for (int i = 0; i < NW; ++i) {
        const float *w = wptr(unit, i);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int cc = c0 + lane + 32 * u;
            r.w[i][u] = w != nullptr && cc < nch ? __ldg(reinterpret_cast<const float4 *>(w) + cc) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
}
// A product of `units` units (NW weight rows each) over the rows in `mask`: units are dealt to the warps of the grid, groups of
// eight rows apart where there are more.  `same_warp`: a unit belongs to the same warp in every group.  (The head needs it: a warp
// folds its units' exponentials before they meet the others', and a row's group depends on how many rows are in front of it.)
// Before the input has arrived: the constructor loads the first unit's weights.  Then run(): out(unit, row, sums) by the whole warp.
template <int NW, class Ptr> struct Product {
    const Ptr &wptr;
    int K, units, groups, first, stride, pitch;   // item unit + pitch * group is item / stride's of warp item % stride
    Wreg<NW> r;
    __device__ __forceinline__ Product(const Ptr &p, int K_, int units_, u64 mask, bool same_warp = false)
        : wptr(p), K(K_), units(units_), groups((popc64(mask) + 7) >> 3), first((int)(threadIdx.x >> 5) * (int)gridDim.x + (int)blockIdx.x), stride(WARPS * (int)gridDim.x) {
        pitch = same_warp ? (units + stride - 1) / stride * stride : units;
        const int unit = groups == 1 ? first : first % pitch;   // (up to eight rows: no division in front of the first load)
        if (first < pitch * groups && unit < units) load_w<NW>(r, wptr, unit, K, 0);
    }
    // Two rows at a time; a weight row of up to 128 U elements is loaded once for all rows of the group.
    template <class Out> __device__ __forceinline__ void run(const float *us, int ldu, u64 mask, Out &&out) {
        const int lane = threadIdx.x & 31, nch = K / 4;
        int at = 0;   // piece of the unit's weights in registers
#pragma unroll 1
        for (int wk = first; wk < pitch * groups; wk += stride) {
            const int grp = groups == 1 ? 0 : wk / pitch, unit = wk - grp * pitch;
            if (unit >= units) continue;
            u64 m = mask;
            for (int i = 0; i < 8 * grp; ++i) m &= m - 1;
            if (wk != first) at = -1;
#pragma unroll 1
            for (int j = 0; j < 8 && m; j += 2) {
                const int r0 = __ffsll((long long)m) - 1;
                m &= m - 1;
                const bool two = m != 0;
                const int r1 = two ? __ffsll((long long)m) - 1 : r0;
                m &= m - 1;
                float acc[2][NW];
#pragma unroll
                for (int i = 0; i < NW; ++i) acc[0][i] = acc[1][i] = 0.f;
                const float4 *x0 = reinterpret_cast<const float4 *>(us + (size_t)r0 * ldu) + lane, *x1 = reinterpret_cast<const float4 *>(us + (size_t)r1 * ldu) + lane;
#pragma unroll 1
                for (int c0 = 0; c0 < nch; c0 += 32 * U) {
                    if (at != c0) load_w<NW>(r, wptr, unit, K, c0);
                    at = c0;
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        if (c0 + 32 * u + lane >= nch) break;
                        const float4 v0 = x0[c0 + 32 * u], v1 = x1[c0 + 32 * u];
#pragma unroll
                        for (int i = 0; i < NW; ++i) {
                            acc[0][i] = fmaf(r.w[i][u].x, v0.x, acc[0][i]); acc[1][i] = fmaf(r.w[i][u].x, v1.x, acc[1][i]);
                            acc[0][i] = fmaf(r.w[i][u].y, v0.y, acc[0][i]); acc[1][i] = fmaf(r.w[i][u].y, v1.y, acc[1][i]);
                            acc[0][i] = fmaf(r.w[i][u].z, v0.z, acc[0][i]); acc[1][i] = fmaf(r.w[i][u].z, v1.z, acc[1][i]);
                            acc[0][i] = fmaf(r.w[i][u].w, v0.w, acc[0][i]); acc[1][i] = fmaf(r.w[i][u].w, v1.w, acc[1][i]);
                        }
                    }
                }
#pragma unroll
                for (int i = 0; i < NW; ++i) { acc[0][i] = warp_sum(acc[0][i]); acc[1][i] = warp_sum(acc[1][i]); }
                out(unit, r0, acc[0]);
                if (two) out(unit, r1, acc[1]);
            }
        }
    }
};

// ---------------------------------------------------------------- the walker

// The phases are functions of their own: inlined into one body, their addresses and prefetched weights together spilled
// thousands of bytes; a call costs little beside a phase.  The object they work on, the arguments with it, lives in shared
// memory (a copy per thread in local memory, and arguments read through a pointer to the parameters, were loads from L2 in front
// of every phase: their L1 lines do not survive the fences of a step).
// `tag`: number of the phase whose output is being written; `tag_x`: of the last layer output.
template <int EPL> struct Walker {   // EPL = head_dim / 32
    static constexpr int HD = 32 * EPL, HALF = HD / 2;
    Args A;
    Shm s;
    u64 t_last;   // thread 0 of CTA 0

    __device__ __forceinline__ int lane() const { return threadIdx.x & 31; }
    __device__ __forceinline__ int warp() const { return threadIdx.x >> 5; }
    __device__ __forceinline__ int seq_of(int r) const { return A.pf_n > 0 ? A.pf_seq : r / A.c.slots; }
    __device__ __forceinline__ void book(int cls) {
        if (!A.prof || blockIdx.x != 0 || threadIdx.x != 0) return;
        const u64 t = now();
        atomicAdd(reinterpret_cast<u64 *>(&A.c.st->st.phase_ns[cls]), t - t_last);
        atomicAdd(reinterpret_cast<u64 *>(&A.c.st->st.phase_count[cls]), 1ull);
        t_last = t;
    }
    __device__ __forceinline__ void bump(long long *p, long long v) const {
        if (blockIdx.x == 0) atomicAdd(reinterpret_cast<u64 *>(p), (u64)v);
    }

    // rotary factors of position pos, into entry `at`, by one warp
    __device__ __forceinline__ void rotary(int at, int pos) const {
        for (int j = lane(); j < HALF; j += 32) {
            double sn, cs;
            sincos((double)pos * s.freq[j], &sn, &cs);
            s.cs[(size_t)at * HD + 2 * j] = (float)cs;
            s.cs[(size_t)at * HD + 2 * j + 1] = (float)sn;
        }
    }
    __device__ __forceinline__ int cs_at(int r) const { return A.pf_n > 0 ? r : seq_of(r) * A.cs_ring + (s.st->pos[r] & (A.cs_ring - 1)); }

    // Rows of `mask` of the residual stream into xs, and normalised with `gain` into us; one warp per row.  Where a row comes from:
    // its embedding (fresh: layer 0), the residual it was parked with (it resumes at this layer), or the exchanged words of
    // phase `want` in `X`.
    __device__ __forceinline__ void load_norm(u64 mask, const u64 *X, unsigned want, int layer, const float *gain) const {
        const int d = A.c.d;
        int i = 0;
        for (u64 m = mask; m; m &= m - 1, ++i) {
            if (i % WARPS != warp()) continue;
            const int r = __ffsll((long long)m) - 1;
            const float *plain = nullptr;
            if (layer == 0) plain = A.tok_embed + (size_t)s.st->tok[seq_of(r)][s.st->pos[r] & (TOK_RING - 1)] * d;
            else if (layer > 0 && s.st->fl[r] == layer) plain = A.c.resid + (size_t)r * d;
            float ss = 0.f;
            float *xr = s.xs + (size_t)r * d, *ur = s.us + (size_t)r * A.ku;
            float2 v[8], g[8];   // up to 512 elements of the row and of the gain stay in registers
#pragma unroll 1
            for (int k0 = 0; k0 < d; k0 += 64 * 8) {
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const int k = k0 + 64 * q + 2 * lane();
                    g[q] = k < d ? __ldg(reinterpret_cast<const float2 *>(gain + k)) : make_float2(0.f, 0.f);
                }
                until(A, s.st, [&]() {
                    bool ok = true;
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const int k = k0 + 64 * q + 2 * lane();
                        v[q] = make_float2(0.f, 0.f);
                        if (k >= d) continue;
                        if (plain) v[q] = __ldcg(reinterpret_cast<const float2 *>(plain + k));
                        else ok = get2(X + (size_t)r * d + k, v[q].x, v[q].y, want) && ok;
                    }
                    return ok;
                });
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const int k = k0 + 64 * q + 2 * lane();
                    if (k < d) *reinterpret_cast<float2 *>(xr + k) = v[q];
                    ss = fmaf(v[q].x, v[q].x, ss);
                    ss = fmaf(v[q].y, v[q].y, ss);
                }
            }
            const float rstd = 1.0f / sqrtf(warp_sum(ss) / d + A.c.eps);
            if (d <= 64 * 8) {
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const int k = 64 * q + 2 * lane();
                    if (k < d) *reinterpret_cast<float2 *>(ur + k) = make_float2(v[q].x * rstd * g[q].x, v[q].y * rstd * g[q].y);
                }
            } else {
                for (int k = 2 * lane(); k < d; k += 64) {   // each lane its own elements
                    const float2 x = *reinterpret_cast<const float2 *>(xr + k), gn = __ldg(reinterpret_cast<const float2 *>(gain + k));
                    *reinterpret_cast<float2 *>(ur + k) = make_float2(x.x * rstd * gn.x, x.y * rstd * gn.y);
                }
            }
        }
    }
    // rows of exchanged words as they are, 256 elements of a row per warp at a time
    __device__ __forceinline__ void load_words(u64 mask, const u64 *X, unsigned want, int K) const {
        const int parts = (K + 255) >> 8;
        int i = 0;
        for (u64 m = mask; m; m &= m - 1) {
            const int r = __ffsll((long long)m) - 1;
            for (int pt = 0; pt < parts; ++pt, ++i) {
                if (i % WARPS != warp()) continue;
                float a[4], b[4];
                until(A, s.st, [&]() {
                    bool ok = true;
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int k = 256 * pt + 64 * q + 2 * lane();
                        if (k < K) ok = get2(X + (size_t)r * K + k, a[q], b[q], want) && ok;
                    }
                    return ok;
                });
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int k = 256 * pt + 64 * q + 2 * lane();
                    if (k < K) *reinterpret_cast<float2 *>(s.us + (size_t)r * A.ku + k) = make_float2(a[q], b[q]);
                }
            }
        }
    }

    // ---- q, k, v: rotated (q, k), exchanged, and k, v to their cache rows.  A unit is a rotation's pair of features (i, i + hd/2) of a
    // q or k head, or two neighbouring features of v.
    __device__ __noinline__ void qkv(int l, u64 mask, unsigned tag_x, unsigned tag) {
        const Ctx &c = A.c;
        const LayerPtrs &w = A.layer[l];
        const int nqk = (c.nq + c.nkv) * HALF, units = nqk + c.nkv * HALF;
        auto wptr = [&](int u, int i) -> const float * {
            if (u < nqk) {
                const int h = u / HALF, j = u - h * HALF + i * HALF;
                return h < c.nq ? w.wq + (size_t)(h * HD + j) * c.d : w.wk + (size_t)((h - c.nq) * HD + j) * c.d;
            }
            return w.wv + (size_t)(2 * (u - nqk) + i) * c.d;
        };
        Product<2, decltype(wptr)> p(wptr, c.d, units, mask);
        load_norm(mask, A.XA, tag_x, l, w.attn_norm);
        __syncthreads();
        float *pool = reinterpret_cast<float *>(c.kv_pool);
        p.run(s.us, A.ku, mask, [&](int u, int r, float (&a)[2]) {
            if (lane() != 0) return;
            const int pos = s.st->pos[r], sq = seq_of(r);
            u64 *q = A.QT + (size_t)r * c.qkv_rows;
            if (u < nqk) {
                const int h = u / HALF, j = u - h * HALF;
                const float co = s.cs[(size_t)cs_at(r) * HD + 2 * j], si = s.cs[(size_t)cs_at(r) * HD + 2 * j + 1];
                const float y0 = a[0] * co - a[1] * si, y1 = a[1] * co + a[0] * si;
                put(q + h * HD + j, y0, tag);
                put(q + h * HD + j + HALF, y1, tag);
                if (h >= c.nq) {
                    float *o = pool + kv_index(c, sq, l, 0, h - c.nq, pos);
                    o[j] = y0;
                    o[j + HALF] = y1;
                }
            } else {
                const int v = 2 * (u - nqk), h = v / HD, j = v - h * HD;
                put(q + (c.nq + c.nkv) * HD + v, a[0], tag);
                put(q + (c.nq + c.nkv) * HD + v + 1, a[1], tag);
                float *o = pool + kv_index(c, sq, l, 1, h, pos);
                o[j] = a[0];
                o[j + 1] = a[1];
            }
        });
        __syncthreads();
        book(2);
    }

    __device__ __forceinline__ bool words(const u64 *p, float (&v)[EPL], unsigned want) const {
        bool ok = true;
        if constexpr (EPL == 1) ok = get(p, v[0], want);
        else {
#pragma unroll
            for (int e = 0; e < EPL; e += 2) ok = get2(p + e, v[e], v[e + 1], want) && ok;
        }
        return ok;
    }

    // EPL elements of a cache row, or zeros
    __device__ __forceinline__ static void cached(float (&v)[EPL], const float *p, bool there) {
        if constexpr (EPL == 1) v[0] = there ? __ldcg(p) : 0.f;
        else {
#pragma unroll
            for (int e = 0; e < EPL; e += 2) {
                const float2 x = there ? __ldcg(reinterpret_cast<const float2 *>(p + e)) : make_float2(0.f, 0.f);
                v[e] = x.x;
                v[e + 1] = x.y;
            }
        }
    }
    // ---- attention: one (row, q head, 128-position chunk) per CTA at a time, sixteen positions per warp.  Positions of this pass
    // come from the exchanged words, earlier ones from the cache (requested before the queries have arrived).
    __device__ __noinline__ void attention(int l, u64 mask, unsigned tag) {
        const Ctx &c = A.c;
        const unsigned want = tag - 1;
        const float *pool = reinterpret_cast<const float *>(c.kv_pool);
        const float scale = rsqrtf((float)HD);
        int total = 0;
        for (u64 m = mask; m; m &= m - 1) total += c.nq * (s.st->pos[__ffsll((long long)m) - 1] / kAttnChunk + 1);
        for (int it = blockIdx.x; it < total; it += gridDim.x) {
            int k = it, r = 0, nch = 1;
            for (u64 m = mask; m; m &= m - 1) {
                r = __ffsll((long long)m) - 1;
                nch = s.st->pos[r] / kAttnChunk + 1;
                if (k < c.nq * nch) break;
                k -= c.nq * nch;
            }
            const int h = k / nch, chunk = k - h * nch, kvh = h / c.group, sq = seq_of(r), pos = s.st->pos[r];
            const int row0 = A.pf_n > 0 ? 0 : sq * c.slots, pos0 = s.st->pos[row0];                       // the sequence's first row and its position
            const int lo = A.pf_n > 0 ? pos0 : s.fill[sq * c.L + l];                                       // positions from here on belong to this pass
            const int t0 = chunk * kAttnChunk + 16 * warp();
            float kk[16][EPL], vv[16][EPL], q[EPL];
            const int tc = min(t0, pos);   // (a warp past the row's position multiplies nothing)
            const float *kp = pool + kv_index(c, sq, l, 0, kvh, tc) + lane() * EPL, *vp = pool + kv_index(c, sq, l, 1, kvh, tc) + lane() * EPL;
            // sixteen positions lie in one cache page (pages hold a multiple of sixteen, warps start at multiples of sixteen)
#pragma unroll
            for (int u = 0; u < 16; ++u) {
                const bool old = t0 + u <= pos && t0 + u < lo;
                cached(kk[u], kp + u * HD, old);
                cached(vv[u], vp + u * HD, old);
            }
            until(A, s.st, [&]() {
                bool ok = words(A.QT + (size_t)r * c.qkv_rows + h * HD + lane() * EPL, q, want);
#pragma unroll
                for (int u = 0; u < 16; ++u) {
                    const int t = t0 + u;
                    if (t <= pos && t >= lo) {
                        const u64 *x = A.QT + (size_t)(row0 + t - pos0) * c.qkv_rows + (c.nq + kvh) * HD + lane() * EPL;
                        ok = words(x, kk[u], want) && ok;
                        ok = words(x + c.nkv * HD, vv[u], want) && ok;
                    }
                }
                return ok;
            });
            // scores: sixteen sums over the lanes at once, halving the number of values a lane holds with every exchange;
            // lanes 2 u and 2 u + 1 end with position u
            float x[16];
#pragma unroll
            for (int u = 0; u < 16; ++u) {
                x[u] = 0.f;
#pragma unroll
                for (int e = 0; e < EPL; ++e) x[u] = fmaf(q[e], kk[u][e], x[u]);
            }
#pragma unroll
            for (int n = 8; n >= 1; n >>= 1) {
                const bool up = (lane() & (2 * n)) != 0;
#pragma unroll
                for (int u = 0; u < n; ++u) {
                    const float give = up ? x[u] : x[u + n], keep = up ? x[u + n] : x[u];
                    x[u] = keep + __shfl_xor_sync(0xffffffffu, give, 2 * n);
                }
            }
            x[0] += __shfl_xor_sync(0xffffffffu, x[0], 1);
            const float sc = t0 + (lane() >> 1) <= pos ? x[0] * scale : -INFINITY;
            float mx = sc;
#pragma unroll
            for (int o = 2; o < 32; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            const float pr = mx == -INFINITY ? 0.f : expf(sc - mx);
            float ls = pr;
#pragma unroll
            for (int o = 2; o < 32; o <<= 1) ls += __shfl_xor_sync(0xffffffffu, ls, o);
            float acc[EPL];
#pragma unroll
            for (int e = 0; e < EPL; ++e) acc[e] = 0.f;
#pragma unroll
            for (int u = 0; u < 16; ++u) {
                const float pu = __shfl_sync(0xffffffffu, pr, 2 * u);
#pragma unroll
                for (int e = 0; e < EPL; ++e) acc[e] = fmaf(pu, vv[u][e], acc[e]);
            }
            float *ao = s.ao + (size_t)warp() * (HD + 2);
#pragma unroll
            for (int e = 0; e < EPL; ++e) ao[lane() * EPL + e] = acc[e];
            if (lane() == 0) { ao[HD] = mx; ao[HD + 1] = ls; }
            __syncthreads();
            if (threadIdx.x < HD) {
                float M = -INFINITY, den = 0.f, o = 0.f;
#pragma unroll
                for (int w = 0; w < WARPS; ++w) M = fmaxf(M, s.ao[w * (HD + 2) + HD]);
#pragma unroll
                for (int w = 0; w < WARPS; ++w) {
                    const float f = expf(s.ao[w * (HD + 2) + HD] - M);
                    den = fmaf(s.ao[w * (HD + 2) + HD + 1], f, den);
                    o = fmaf(s.ao[w * (HD + 2) + threadIdx.x], f, o);
                }
                u64 *out = A.PT + (((size_t)r * c.nq + h) * c.n_chunks + chunk) * (HD + 2);
                put(out + threadIdx.x, o, tag);
                if (threadIdx.x == 0) { put(out + HD, M, tag); put(out + HD + 1, den, tag); }
            }
            __syncthreads();
        }
        book(4);
    }

    // chunk partials of every head, merged in ascending order, as the O product's input
    __device__ __forceinline__ void load_attention(u64 mask, unsigned want) const {
        const Ctx &c = A.c;
        int i = 0;   // 64 features of a row per warp at a time
        for (u64 m = mask; m; m &= m - 1) {
            const int r = __ffsll((long long)m) - 1, nch = s.st->pos[r] / kAttnChunk + 1;
            for (int k0 = 0; k0 < c.nq * HD; k0 += 64, ++i) {
                const int k = k0 + 2 * lane();
                if (i % WARPS != warp() || k >= c.nq * HD) continue;
                const int h = k / HD, dim = k - h * HD;
                const u64 *part = A.PT + ((size_t)r * c.nq + h) * c.n_chunks * (HD + 2);
                float M = -INFINITY, den = 0.f, ox = 0.f, oy = 0.f;
                for (int c0 = 0; c0 < nch; c0 += 4) {
                    float pm[4], pl[4], px[4], py[4];
                    until(A, s.st, [&]() {
                        bool ok = true;
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            pm[q] = -INFINITY; pl[q] = px[q] = py[q] = 0.f;
                            if (c0 + q >= nch) continue;
                            ok = get2(part + (size_t)(c0 + q) * (HD + 2) + HD, pm[q], pl[q], want) && ok;
                            ok = get2(part + (size_t)(c0 + q) * (HD + 2) + dim, px[q], py[q], want) && ok;
                        }
                        return ok;
                    });
                    float Mn = M;
#pragma unroll
                    for (int q = 0; q < 4; ++q) Mn = fmaxf(Mn, pm[q]);
                    const float f = M == -INFINITY ? 0.f : expf(M - Mn);
                    den *= f; ox *= f; oy *= f;
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float g = pm[q] == -INFINITY ? 0.f : expf(pm[q] - Mn);
                        den = fmaf(pl[q], g, den); ox = fmaf(px[q], g, ox); oy = fmaf(py[q], g, oy);
                    }
                    M = Mn;
                }
                *reinterpret_cast<float2 *>(s.us + (size_t)r * A.ku + k) = make_float2(ox / den, oy / den);
            }
        }
    }

    // O and down: residual + product, exchanged; the layer's output is also kept (a row may wait at an exit layer)
    __device__ __noinline__ void o_product(int l, u64 mask, unsigned tag) {
        const Ctx &c = A.c;
        const float *W = A.layer[l].wo;
        const int K = c.nq * HD;
        auto wptr = [&](int u, int) { return W + (size_t)u * K; };
        const unsigned want = tag - 1;
        Product<1, decltype(wptr)> p(wptr, K, c.d, mask);
        load_attention(mask, want);
        __syncthreads();
        p.run(s.us, A.ku, mask, [&](int n, int r, float (&a)[1]) {
            if (lane() == 0) put(A.XB + (size_t)r * c.d + n, s.xs[(size_t)r * c.d + n] + a[0], tag);
        });
        __syncthreads();
        book(5);
    }
    __device__ __noinline__ void gate_up(int l, u64 mask, unsigned tag) {
        const Ctx &c = A.c;
        const LayerPtrs &w = A.layer[l];
        auto wptr = [&](int u, int i) { return (i ? w.wu : w.wg) + (size_t)u * c.d; };
        const unsigned want = tag - 1;
        Product<2, decltype(wptr)> p(wptr, c.d, c.dff, mask);
        // the rotary factors of the token that this step may emit, by warps that are waiting (their entry's position is complete)
        if (l == 0 && A.pf_n == 0)
            for (int q = WARPS - 1 - warp(); q < A.batch; q += WARPS)
                if (!s.st->done[q]) rotary(q * A.cs_ring + (s.st->len[q] & (A.cs_ring - 1)), s.st->len[q]);
        load_norm(mask, A.XB, want, -1, w.ffn_norm);
        __syncthreads();
        p.run(s.us, A.ku, mask, [&](int n, int r, float (&a)[2]) {
            if (lane() == 0) put(A.HT + (size_t)r * c.dff + n, a[0] / (1.0f + expf(-a[0])) * a[1], tag);
        });
        __syncthreads();
        book(6);
    }
    __device__ __noinline__ void down(int l, u64 mask, unsigned tag) {
        const Ctx &c = A.c;
        const float *W = A.layer[l].wd;
        auto wptr = [&](int u, int) { return W + (size_t)u * c.dff; };
        const unsigned want = tag - 1;
        Product<1, decltype(wptr)> p(wptr, c.dff, c.d, mask);
        load_words(mask, A.HT, want, c.dff);
        __syncthreads();
        p.run(s.us, A.ku, mask, [&](int n, int r, float (&a)[1]) {
            if (lane() != 0) return;
            const float v = s.xs[(size_t)r * c.d + n] + a[0];
            put(A.XA + (size_t)r * c.d + n, v, tag);
            c.resid[(size_t)r * c.d + n] = v;
        });
        __syncthreads();
        book(8);
    }

    // ---- head over the rows of `mask` (layer1: 1-based layer, 0 = final): every CTA's (max, sum exp, argmax) of its vocabulary
    // entries, exchanged, and merged by every CTA alike into st->hr.
    __device__ __noinline__ void head(int layer1, u64 mask, unsigned tag_x, unsigned tag) {
        const Ctx &c = A.c;
        const float *T = layer1 > 0 ? A.head_T[layer1] : nullptr;
        const float scale = layer1 > 0 ? A.head_scale[layer1] : 1.0f;
        const int n_units = (c.vocab + 1) / 2;
        auto wptr = [&](int u, int i) -> const float * { return 2 * u + i < c.vocab ? A.lm_head + (size_t)(2 * u + i) * c.d : nullptr; };
        // What this thread stored plainly in the step (cache rows, residuals) is ordered before the partials below; here, where it waits
        // for the layer's output anyway.
        __threadfence();
        if (T) {
            auto tptr = [&](int u, int) { return T + (size_t)u * c.d; };
            Product<1, decltype(tptr)> p(tptr, c.d, c.d, mask);
            load_norm(mask, A.XA, tag_x, -1, A.final_norm);
            __syncthreads();
            p.run(s.us, A.ku, mask, [&](int n, int r, float (&a)[1]) {
                if (lane() == 0) put(A.TT + (size_t)r * c.d + n, a[0], tag - 1);
            });
            __syncthreads();
            book(10);
        }
        for (int r = lane(); r < A.R; r += 32) { Msa &m = s.red[warp() * A.R + r]; m.m = -INFINITY; m.s = 0.f; m.i = INT_MAX; }
        Product<2, decltype(wptr)> p(wptr, c.d, n_units, mask, true);
        if (T) load_words(mask, A.TT, tag - 1, c.d);
        else load_norm(mask, A.XA, tag_x, -1, A.final_norm);
        __syncthreads();
        p.run(s.us, A.ku, mask, [&](int u, int r, float (&a)[2]) {
            if (lane() != 0) return;
            Msa run = s.red[warp() * A.R + r];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int n = 2 * u + i;
                if (n >= c.vocab) break;
                Msa one;
                one.m = a[i] * scale; one.s = 1.f; one.i = n;
                if (A.store_logits && layer1 == 0) c.logit_stage[(size_t)r * c.vocab + n] = one.m;
                run = msa_merge(run, one);
            }
            s.red[warp() * A.R + r] = run;
        });
        if (A.store_logits && layer1 == 0) __threadfence();   // the staged logits too
        __syncthreads();
        if (threadIdx.x < A.R && ((mask >> threadIdx.x) & 1ull)) {
            const int r = threadIdx.x;
            Msa a = s.red[r];
#pragma unroll
            for (int w = 1; w < WARPS; ++w) a = msa_merge(a, s.red[w * A.R + r]);
            u64 *o = A.HP + ((size_t)blockIdx.x * A.R + r) * 4;
            put(o, a.m, tag);
            put(o + 1, a.s, tag);
            put(o + 2, __int_as_float(a.i), tag);
        }
        meet(mask, tag);
        book(9);
    }
    // the partials of all CTAs: one warp per row, lane l merges CTAs l, l + 32, ..., then the lanes by a butterfly
    __device__ __forceinline__ void meet(u64 mask, unsigned tag) {
        int i = 0;
        for (u64 m = mask; m; m &= m - 1, ++i) {
            if (i % WARPS != warp()) continue;
            const int r = __ffsll((long long)m) - 1, G = gridDim.x;
            Msa a;
            a.m = -INFINITY; a.s = 0.f; a.i = INT_MAX;
            for (int b0 = 0; b0 < G; b0 += 32 * 5) {
                float pm[5], ps[5], pi[5];
                until(A, s.st, [&]() {
                    bool ok = true;
#pragma unroll
                    for (int q = 0; q < 5; ++q) {
                        const int b = b0 + 32 * q + lane();
                        if (b >= G) continue;
                        const u64 *o = A.HP + ((size_t)b * A.R + r) * 4;
                        ok = get2(o, pm[q], ps[q], tag) && ok;
                        ok = get(o + 2, pi[q], tag) && ok;
                    }
                    return ok;
                });
#pragma unroll
                for (int q = 0; q < 5; ++q) {
                    const int b = b0 + 32 * q + lane();
                    if (b >= G) continue;
                    Msa x;
                    x.m = pm[q]; x.s = ps[q]; x.i = __float_as_int(pi[q]);
                    if (x.m != -INFINITY) a = msa_merge(a, x);
                }
            }
            __syncwarp();
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                Msa x;
                x.m = __shfl_xor_sync(0xffffffffu, a.m, o);
                x.s = __shfl_xor_sync(0xffffffffu, a.s, o);
                x.i = __shfl_xor_sync(0xffffffffu, a.i, o);
                a = msa_merge(a, x);
            }
            if (lane() == 0) {
                HeadResult hr;
                hr.token = min(a.i, A.c.vocab - 1);   // (no logit is a number: no argmax)
                hr.zmax = a.m; hr.sumexp = a.s; hr.p = 1.0f / a.s;
                s.st->hr[r] = hr;
                if (blockIdx.x == 0) A.c.head_res[r] = hr;
            }
        }
        __threadfence();   // and what the other CTAs stored before their partials is seen from here on
        __syncthreads();
    }

    // the kept rows' staged logits of sequence 0 into the capture buffer
    __device__ __forceinline__ void capture() const {
        const Ctx &c = A.c;
        if (!c.capture) return;
        const int keep = s.st->keep, at = s.st->cap_n - keep, V = c.vocab;
        for (int j = 0; j < keep; ++j) {
            const float *src = c.logit_stage + (size_t)(s.st->keep_row + j) * V;
            float *dst = c.capture + (size_t)(at + j) * V;
            for (int i = blockIdx.x * THREADS + threadIdx.x; i < V; i += gridDim.x * THREADS) dst[i] = __ldcg(src + i);
        }
    }
    // (thread 0) `keep` rows from row `row` on go to the capture buffer, as many as it still holds
    __device__ __forceinline__ void note_capture(int keep, int row) const {
        s.st->keep = s.st->keep_row = 0;
        if (!A.c.capture) return;
        const int n = max(0, min(keep, A.capture_cap - s.st->cap_n));
        s.st->keep = n;
        s.st->keep_row = row;
        s.st->cap_n += n;
    }
    __device__ __forceinline__ void set_token(int sq, int pos, int t) const {
        t = min(max(t, 0), A.c.vocab - 1);
        s.st->tok[sq][pos & (TOK_RING - 1)] = t;
        if (blockIdx.x == 0) A.c.tokens[(size_t)sq * A.c.max_seq + pos] = t;
    }
    __device__ __forceinline__ void set_fill(int sq, int l, int v) const {
        s.fill[sq * A.c.L + l] = v;
        if (blockIdx.x == 0) A.c.fill[sq * A.c.L + l] = v;
    }

    // Eq. 1 after the head at 1-based layer e (thread 0 of every CTA; the same rules as k_exit_control)
    __device__ __forceinline__ void exit_control(int e) const {
        const Ctx &c = A.c;
        State *st = s.st;
        DevState *g = c.st;
        int nclimb = 0;
        for (int q = 0; q < A.batch; ++q) {
            if (!st->climbing[q]) continue;
            const int len = st->len[q], slot = len - 1 - st->base[q];
            if (slot < A.max_early && len < st->target[q]) {
                const HeadResult hr = st->hr[q * c.slots + slot];
                bool decide = hr.p > A.gamma;
                if (q == 0 && st->tape_i < A.tape_n) {
                    const uint8_t t = g->tape[st->tape_i++];
                    if (t == 0) decide = false;
                    if (t == 1) decide = true;
                }
                bump(&g->st.head_evals, 1);
                if (c.head_log && st->log_n < kHeadLogCap) {
                    if (blockIdx.x == 0) {
                        float *hl = c.head_log + 4 * (size_t)st->log_n;
                        hl[0] = (float)__ldcg(&g->st.steps); hl[1] = (float)e; hl[2] = (float)hr.token; hl[3] = hr.p;
                    }
                    st->log_n++;
                }
                if (decide) {
                    long long rl = 0;
                    for (int l = 0; l < e; ++l) {
                        rl += len - s.fill[q * c.L + l];
                        set_fill(q, l, len);
                    }
                    bump(&g->st.row_layers, rl);
                    set_token(q, len, hr.token);
                    st->len[q] = len + 1;
                    bump(&g->st.early_exits, 1);
                    bump(&g->st.exits_at_layer[e], 1);
                    bump(&g->st.steps, 1);
                    st->climbing[q] = 0;
                    for (int j = 0; j < c.slots; ++j) st->fl[q * c.slots + j] = INT_MAX;
                }
            }
            nclimb += st->climbing[q];
        }
        st->n_climbing = nclimb;
        if (nclimb == 0) bump(&g->st.layer_passes, e);
    }
    // Verification at the last layer (thread 0 of every CTA; the same rules as k_verify)
    __device__ __forceinline__ void verify() const {
        const Ctx &c = A.c;
        State *st = s.st;
        DevState *g = c.st;
        int ndone = 0, keep0 = 0;
        for (int q = 0; q < A.batch; ++q) {
            if (st->climbing[q]) {
                const int len = st->len[q], base = st->base[q], nrow = len - base;
                const HeadResult *hr = st->hr + q * c.slots;
                long long rl = 0;
                for (int l = 0; l < c.L; ++l) rl += len - s.fill[q * c.L + l];
                bump(&g->st.row_layers, rl);
                int bad = -1;
                for (int j = 0; j + 1 < nrow; ++j)
                    if (hr[j].token != st->tok[q][(base + j + 1) & (TOK_RING - 1)]) { bad = j; break; }
                int new_base, keep;
                if (bad < 0) {
                    bump(&g->st.accepted, nrow - 1);
                    set_token(q, len, hr[nrow - 1].token);
                    new_base = len;
                    keep = nrow;
                } else {
                    bump(&g->st.accepted, bad);
                    bump(&g->st.rejected, 1);
                    bump(&g->st.discarded, nrow - 2 - bad);
                    new_base = base + bad + 1;
                    set_token(q, new_base, hr[bad].token);
                    keep = bad + 1;
                }
                // "while t_i != [EOS]" (Algorithm 1): the first verified end-of-sequence token ends the sequence
                int target = st->target[q];
                if (A.eos_id >= 0) {
                    for (int j = 0; j < keep; ++j)
                        if (hr[j].token == A.eos_id) {
                            if (base + j + 2 <= target) { target = base + j + 2; st->eos_hit[q] = 1; }
                            break;
                        }
                }
                int new_len = new_base + 1;
                if (new_len > target) {
                    bump(&g->st.truncated, new_len - target);
                    new_len = target;
                    new_base = new_len - 1;
                }
                keep = new_len - 1 - base;   // verified tokens that stay
                for (int l = 0; l < c.L; ++l) set_fill(q, l, new_base);
                st->len[q] = new_len;
                st->base[q] = new_base;
                bump(&g->st.verify_steps, 1);
                bump(&g->st.steps, 1);
                st->climbing[q] = 0;
                if (new_len >= target) st->done[q] = 1;
                if (q == 0) keep0 = keep;
            }
            ndone += st->done[q];
        }
        note_capture(keep0, 0);
        bump(&g->st.layer_passes, c.L);
        st->n_climbing = 0;
        st->n_done = ndone;
    }

    // the phases tag + 1 .. tag + 5; `tag` becomes the last of them, the layer's output
    __device__ __forceinline__ void layers(int l, u64 mask, unsigned tag_x, unsigned &tag) {
        qkv(l, mask, tag_x, tag + 1);
        attention(l, mask, tag + 2);
        o_product(l, mask, tag + 3);
        gate_up(l, mask, tag + 4);
        down(l, mask, tag + 5);
        tag += 5;
    }
    __device__ __forceinline__ bool aborted() const { return *(volatile int *)&s.st->abort != 0; }

    __device__ __forceinline__ void decode() {
        const Ctx &c = A.c;
        State *st = s.st;
        DevState *g = c.st;
        const int batch = A.batch, rows = batch * c.slots, tid = threadIdx.x;
        for (int q = tid; q < batch; q += THREADS) {
            st->len[q] = g->len[q]; st->base[q] = g->base[q]; st->target[q] = g->target_len[q]; st->done[q] = g->done[q]; st->eos_hit[q] = g->eos_hit[q];
        }
        for (int i = tid; i < batch * c.L; i += THREADS) s.fill[i] = c.fill[i];
        for (int i = tid; i < batch * TOK_RING; i += THREADS) {   // the last TOK_RING positions up to the newest
            const int q = i / TOK_RING, pos = g->len[q] - 1 - (i % TOK_RING);
            if (pos >= 0) st->tok[q][pos & (TOK_RING - 1)] = c.tokens[(size_t)q * c.max_seq + pos];
        }
        if (tid == 0) { st->tape_i = 0; st->log_n = 0; st->cap_n = g->capture_n; st->n_done = g->n_done; st->n_climbing = 0; }
        __syncthreads();
        // rotary factors of the positions in flight
        for (int i = warp(); i < batch * A.cs_ring; i += WARPS) {
            const int q = i / A.cs_ring, pos = st->base[q] + i % A.cs_ring;
            if (pos < st->len[q]) rotary(q * A.cs_ring + (pos & (A.cs_ring - 1)), pos);
        }
        __syncthreads();
        unsigned tag = 0, tag_x = 0;
        for (long long step = 0; st->n_done < batch; ++step) {
            if (step >= A.max_steps) {   // every step emits or verifies a token
                if (tid == 0 && blockIdx.x == 0) atomicCAS(A.err, 0, ERR_STEPS);
                break;
            }
            // the step's rows: per sequence the early tokens in flight and the newest one, each with the layer at which it resumes
            for (int r = tid; r < MAX_R; r += THREADS) {
                const int q = min(r / c.slots, batch - 1), pos = st->base[q] + (r - q * c.slots);
                int fl = INT_MAX;
                if (r < rows && !st->done[q] && pos < st->len[q]) {
                    fl = 0;
                    for (int l = 0; l < c.L; ++l) fl += s.fill[q * c.L + l] > pos;
                }
                st->fl[r] = fl;
                st->pos[r] = pos;
            }
            if (tid < batch) st->climbing[tid] = !st->done[tid];
            __syncthreads();
            book(0);
            bool up = true;
            for (int l = 0; l < c.L && up; ++l) {
                layers(l, active_rows(st, rows, l), tag_x, tag);
                tag_x = tag;
                if (l + 1 < c.L && A.exit_at[l + 1]) {
                    u64 sel = 0;   // newest rows that may leave early
                    for (int q = 0; q < batch; ++q) {
                        const int slot = st->len[q] - 1 - st->base[q];
                        if (st->climbing[q] && slot < A.max_early && st->len[q] < st->target[q]) sel |= 1ull << (q * c.slots + slot);
                    }
                    if (sel) {
                        tag += 2;   // (the first: T's output)
                        head(l + 1, sel, tag_x, tag);
                        if (tid == 0) exit_control(l + 1);
                        __syncthreads();
                        book(0);
                        up = st->n_climbing > 0;
                    }
                }
            }
            if (up) {
                tag += 2;
                head(0, active_rows(st, rows, c.L - 1), tag_x, tag);
                if (tid == 0) verify();
                __syncthreads();
                capture();
                book(0);
            }
            if (aborted()) break;
            __syncthreads();   // everybody has read the state that the next step's set-up rewrites
        }
        __syncthreads();
        if (blockIdx.x == 0) {
            for (int q = tid; q < batch; q += THREADS) { g->len[q] = st->len[q]; g->base[q] = st->base[q]; g->done[q] = st->done[q]; g->eos_hit[q] = st->eos_hit[q]; }
            if (tid == 0) { g->tape_i = st->tape_i; g->head_log_n = st->log_n; g->capture_n = st->cap_n; g->n_done = st->n_done; g->n_climbing = 0; }
        }
    }

    // prompt passes of one sequence (KV cache <- LM(x)): up to pf_rows positions at a time, then the head on the last one
    __device__ __forceinline__ void prefill() {
        const Ctx &c = A.c;
        State *st = s.st;
        DevState *g = c.st;
        const int tid = threadIdx.x, sq = A.pf_seq;
        if (tid == 0) st->cap_n = g->capture_n;
        unsigned tag = 0, tag_x = 0;
        for (int p0 = 0; p0 < A.pf_n; p0 += A.pf_rows) {
            const int n = min(A.pf_rows, A.pf_n - p0);
            const bool last = p0 + n == A.pf_n;
            for (int r = tid; r < MAX_R; r += THREADS) { st->fl[r] = r < n ? 0 : INT_MAX; st->pos[r] = p0 + min(r, n - 1); }
            // (tokens are kept by position modulo TOK_RING: a pass takes at most as many)
            for (int r = tid; r < n; r += THREADS) st->tok[sq][(p0 + r) & (TOK_RING - 1)] = c.tokens[(size_t)sq * c.max_seq + p0 + r];
            for (int r = warp(); r < n; r += WARPS) rotary(r, p0 + r);
            __syncthreads();
            for (int l = 0; l < c.L; ++l) {
                layers(l, active_rows(st, n, l), tag_x, tag);
                tag_x = tag;
            }
            if (last) {
                tag += 2;
                head(0, 1ull << (n - 1), tag_x, tag);
            } else {   // the next pass reads this one's cache rows
                __threadfence();
                __syncthreads();
                ++tag;
                if (tid == 0) { u64 *o = A.HP + (size_t)blockIdx.x * A.R * 4; put(o, -INFINITY, tag); put(o + 1, 0.f, tag); put(o + 2, 0.f, tag); }
                meet(1ull, tag);
            }
            if (aborted()) break;
        }
        if (tid == 0) {
            const int n_last = (A.pf_n - 1) % A.pf_rows;
            set_token(sq, A.pf_n, st->hr[n_last].token);
            if (blockIdx.x == 0) {
                for (int l = 0; l < c.L; ++l) c.fill[sq * c.L + l] = A.pf_n;
                g->base[sq] = A.pf_n;
                g->len[sq] = A.pf_n + 1;
                g->n_prompt[sq] = A.pf_n;
                g->done[sq] = 1;
            }
            note_capture(sq == 0 ? 1 : 0, n_last);
        }
        __syncthreads();
        capture();
        if (tid == 0 && blockIdx.x == 0 && sq == 0 && c.capture) g->capture_n = st->cap_n;
    }
};

template <int EPL> __global__ void __launch_bounds__(THREADS, 1) k_decode_resident(const __grid_constant__ Args args) {
    extern __shared__ __align__(16) unsigned char raw[];
    Walker<EPL> &w = *reinterpret_cast<Walker<EPL> *>(raw);
    static_assert(sizeof(Args) % 4 == 0, "the arguments are copied by words");
    for (int i = threadIdx.x; i < (int)(sizeof(Args) / 4); i += THREADS) reinterpret_cast<int *>(&w.A)[i] = reinterpret_cast<const int *>(&args)[i];
    const Ctx &c = args.c;
    if (threadIdx.x == 0) {
        unsigned char *at = raw + walker_bytes(sizeof(Walker<EPL>));
        w.s.freq = reinterpret_cast<double *>(at);
        float *f = reinterpret_cast<float *>(at + sizeof(double) * (c.hd / 2));
        const int batch = args.batch, n_cs = max(args.R, batch * args.cs_ring);
        w.s.xs = f; f += (size_t)args.R * c.d;
        w.s.us = f; f += (size_t)args.R * args.ku;
        w.s.cs = f; f += (size_t)n_cs * c.hd;
        w.s.ao = f; f += (size_t)WARPS * (c.hd + 2);
        w.s.red = reinterpret_cast<Msa *>(f); f += 3 * (size_t)WARPS * args.R;
        w.s.fill = reinterpret_cast<int *>(f); f += (size_t)batch * c.L;
        w.s.st = reinterpret_cast<State *>(f);
        w.s.st->abort = 0;
        w.s.st->keep = w.s.st->keep_row = 0;
        w.t_last = now();
    }
    __syncthreads();
    if (args.page_words > 0) {   // the page table, behind the rest: an entry is looked up for every cache row that is written or read, each a load from L2
        int32_t *table = reinterpret_cast<int32_t *>(w.s.st + 1);
        for (int i = threadIdx.x; i < args.page_words; i += THREADS) table[i] = c.page_table[i];
        if (threadIdx.x == 0) w.A.c.page_table = table;
    }
    for (int j = threadIdx.x; j < c.hd / 2; j += THREADS) w.s.freq[j] = pow((double)args.rope_base, -2.0 * j / c.hd);
    __syncthreads();
    if (args.pf_n > 0) w.prefill();
    else w.decode();
}

}  // namespace rs
}  // namespace ada
