// The persistent decode kernel: Algorithm 1 of the paper, one cooperative launch for many steps.
//
// One CTA per SM: a warp that produces weights and K / V blocks, one that produces activations and queries, eight consumers.
// Every CTA walks the same program
//     control | for each layer: QKV | attention | O | gate-up | down | [head, control] ... | final head | control
// with a grid barrier between phases.  The weight producer is not held by those barriers (but for cache rows
// of the pass itself): it keeps the TMA ring full with the tiles of the coming phases, so HBM keeps streaming while the
// grid meets, and the consumers move what has landed on to tensor memory (park_stage in stream.cuh).  Measured, one layer in a plain
// step (1B / 8B shape): QKV 5.7 / 10.9 us, attention 6.6 / 10.2 (60 / 1040 positions), O 4.9 / 7.5, gate-up 10.7 / 36.7, down 8.0 / 18.6,
// of which a phase's own bytes take 1.9 / 7.8, - / 0.7, 1.3 / 5.2, 10.3 / 36, 5.1 / 18.  (Not a floor of the phase: up to 25 stages a
// CTA, 9 us of the stream, have been fetched in earlier phases, and as many of the next ones' are fetched in it.  Boxes differ by up to
// 0.6 us a phase.)  All decoding state (sequence, per-layer fill levels, in-flight tokens, row
// residuals, counters) lives in device memory; the control points run in CTA 0, which publishes
// each decision (continue the climb, start the next token, stop) to the other CTAs through a
// sequence-numbered record.  The host launches, waits, and launches again until the call is done.
//
// Token columns: the tokens of a pass (per sequence the newest token and the early-predicted
// tokens still in flight, Algorithm 1's P[l] (+) t_i) are the columns of one or three tensor-core
// tiles; column = (position - base) x sequences of the launch + sequence, fixed for the life of a token.  Per-column buffers therefore
// persist across steps: a token that left the climb at layer e finds its residual, its
// normalisation partial sums and its layer-(e+1) GEMM input where its last pass left them.
// Each column's numbers depend only on that column's own inputs (never on which other columns
// ride along), which is what makes the adaptive output bit-identical to plain greedy decoding.
#include "kernels.cuh"
#include "stream.cuh"   // (compiled once per number of column tiles, like this file: see there)

namespace ada {
namespace ADA_MG {

using namespace ADA_ST;

constexpr int ACT_CONTINUE = 1, ACT_NEWSTEP = 2, ACT_STOP = 3;
constexpr int CTRL_START = 0, CTRL_HEAD = 1, CTRL_TOP = 2;
constexpr int ATT_CHUNK = kAttnChunk; // positions per attention work item (fixed: anchored at position 0)

constexpr int NO_LAYER = 255;   // above every layer index (ADA_MAX_LAYERS - 1 layers at most)
static_assert(ADA_MAX_LAYERS <= 256, "layer indexes are kept in a byte");

struct StepDesc {
    int n_cols;                // columns with a token (in flight + newest, over all sequences of the launch)
    int newest_mask;           // columns holding the newest token of their sequence
    int head_mask;             // newest columns that may consult intermediate heads in this step
    int pmax;                  // highest position of the step
    int fresh;                 // columns whose token enters at layer 1 in this step (their embedding is set up by the control point)
    int run_final;             // the step ends with the final head (0: a prompt pass that is not the last)
    unsigned char first_layer[MAX_COLS];   // 0-based layer at which the column resumes (NO_LAYER: no token, or its sequence has left the step)
    int pos[MAX_COLS];
    int seq_pmax[MAX_SEQS];    // per sequence of the launch: position of its newest token (-1: the sequence is not in this step)
};
static_assert(sizeof(StepDesc) <= sizeof(Smem::desc[0]), "the step descriptor must fit its shared-memory slot");

struct Pub {                   // what CTA 0 publishes at a control point
    unsigned seq;
    int action;
    StepDesc d;
    int cap_keep, cap_at, cap_row0;   // logit capture (test hook): rows to copy, where to, first row of the staging buffer
    int pad[5];
};

// ---------------------------------------------------------------- small helpers

__device__ __forceinline__ float ldcg(const float *p) { return __ldcg(p); }

__device__ __forceinline__ unsigned active_mask(const StepDesc &d, int layer) {
    unsigned m = 0;
#pragma unroll
    for (int c = 0; c < MAX_COLS; ++c) m |= (d.first_layer[c] <= layer ? 1u : 0u) << c;
    return m;
}

// RMSNorm factors 1/sqrt(mean square + eps) of all columns from the per-tile sums of squares
// ssq[tile][column], by the activation producer warp, eight columns at a time: lane l sums column l%8 over the tiles
// l/8 + 4u in ascending order (32 loads in flight), the four lanes of a column are folded by a
// butterfly.  The order is fixed, so the factor of a column does not depend on the other columns.
__device__ __forceinline__ void rstd_produce(Smem *sm, const float *ssq, int ntiles, int d, float eps, unsigned seq) {
    const int lane = threadIdx.x & 31, sub = lane >> 3;
#pragma unroll 1
    for (int ct = 0; ct < TILES; ++ct) {
        const int col = 8 * ct + (lane & 7);
        float s = 0.f;
        for (int t0 = 0; t0 < ntiles; t0 += 128) {
            float v[32];
#pragma unroll
            for (int u = 0; u < 32; ++u) {
                const int t = t0 + sub + 4 * u;
                v[u] = t < ntiles ? ldcg(ssq + (size_t)t * MAX_COLS + col) : 0.f;
            }
#pragma unroll
            for (int u = 0; u < 32; ++u) s += v[u];
        }
        s += __shfl_xor_sync(0xffffffffu, s, 8);
        s += __shfl_xor_sync(0xffffffffu, s, 16);
        if (lane < 8) sm->vec[col] = 1.0f / sqrtf(s / (float)d + eps);
    }
    __threadfence_block();
    __syncwarp();
    if (lane == 0) *(volatile unsigned *)&sm->vec_seq = seq;
}

// The end of a phase as seen by the consumers of a CTA: they report it to the grid and go on.  Whoever needs what the other
// CTAs wrote waits for the counter: the activation producer before it fetches a product's input, the consumers themselves
// (consumers_meet) where they read other CTAs' results directly.  Consumers of a product wait for its first input stage only,
// and set up its epilogue's operands while the grid is still meeting.
__device__ __forceinline__ void consumers_arrive(const Shared &S, unsigned *ctr, int cls) {
    if (threadIdx.x == 0) trace(S, EV_EPI_END, cls);
    bar_consumers();
    if (threadIdx.x == 0) {
        grid_arrive(ctr);
        trace(S, EV_ARRIVE, cls);
    }
}
__device__ __forceinline__ void consumers_meet(const Shared &S, const unsigned *ctr, unsigned target) {
    if (threadIdx.x == 0) grid_wait(S, ctr, target);
    bar_consumers();
}

// Merge the per-CTA (max, sum exp, argmax) partials of one column, by one whole warp: lane i folds
// CTAs i, i+32, ... in ascending order, then the lanes are folded by a butterfly (the merge is
// symmetric, so every lane ends with the same value).
__device__ __forceinline__ HeadResult merge_head(const float *head_part, int G, int col) {
    const int lane = threadIdx.x & 31;
    Msa a; a.m = -INFINITY; a.s = 0.f; a.i = INT_MAX;
    for (int b0 = lane; b0 < G; b0 += 32 * 8) {   // eight CTAs' partials in flight per lane, merged in ascending order
        float4 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int b = b0 + 32 * u;
            v[u] = b < G ? __ldcg(reinterpret_cast<const float4 *>(head_part + ((size_t)b * MAX_COLS + col) * 4)) : make_float4(-INFINITY, 0.f, __int_as_float(INT_MAX), 0.f);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            if (b0 + 32 * u < G) {
                Msa x; x.m = v[u].x; x.s = v[u].y; x.i = __float_as_int(v[u].z);
                a = msa_merge(a, x);
            }
        }
    }
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        Msa o;
        o.m = __shfl_xor_sync(0xffffffffu, a.m, off);
        o.s = __shfl_xor_sync(0xffffffffu, a.s, off);
        o.i = __shfl_xor_sync(0xffffffffu, a.i, off);
        a = msa_merge(a, o);
    }
    HeadResult hr; hr.token = a.i; hr.zmax = a.m; hr.sumexp = a.s; hr.p = 1.0f / a.s;
    return hr;
}

// ---------------------------------------------------------------- sampling (CTA 0, consumer warps)

constexpr int DRAW_CHUNK = 128;                 // vocabulary entries per partial sum
constexpr int DRAW_OFFSET = 12288;              // the draw's buffers sit in the consumers' scratch behind the control point's copies
constexpr int DRAW_MAX_CHUNKS = (SCRATCH_BYTES - DRAW_OFFSET - 4 * (CONS_THREADS + DRAW_CHUNK + 8)) / 4;
constexpr int DRAW_MAX_VOCAB = DRAW_MAX_CHUNKS * DRAW_CHUNK;

// Weights the draw is made from, in vocabulary order: exp(z - m) (a head's distribution up to its normaliser), or, with
// zq set, the positive part of exp(z - m) / s - exp(zq - mq) / sq (the distribution Eq. 2 resamples from, up to its normaliser).
struct DrawSrc {
    const float *z; float m, inv_s;
    const float *zq; float mq, inv_sq;
    __device__ __forceinline__ float weight_of(float zv, float qv) const {   // from the loaded logits (-inf: outside the vocabulary)
        const float a = __expf(zv - m);
        if (!zq) return a;
        return fmaxf(0.f, a * inv_s - __expf(qv - mq) * inv_sq);
    }
    __device__ __forceinline__ float weight(int v) const { return weight_of(__ldcg(z + v), zq ? __ldcg(zq + v) : 0.f); }
};

// Inverse-CDF draw by the consumer warps of one CTA: the first token, in vocabulary order, whose running sum of weights
// exceeds u x (sum of all weights); the last token of non-zero weight if rounding leaves none.  Returns the token to every
// thread (-1 if all weights are zero), with the sum of all weights and the drawn token's weight.  Partial sums per 128
// entries in a fixed order, so the result does not depend on timing.
__device__ __noinline__ int block_draw(Smem *sm, const DrawSrc &src, int V, float u, float &total, float &w_tok) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    float *psum = reinterpret_cast<float *>(sm->scratch + DRAW_OFFSET);   // [CONS_THREADS]
    float *wbuf = psum + CONS_THREADS;                                     // [DRAW_CHUNK]
    float *res = wbuf + DRAW_CHUNK;                                        // token, its weight
    float *csum = res + 8;                                                 // [chunks]
    const int n_chunks = (V + DRAW_CHUNK - 1) / DRAW_CHUNK;
    // pass 1: the sum of every chunk (warp w takes chunks w, w + 8, ...; eight chunks' loads in flight)
    const bool vec = (V & 3) == 0;   // rows start on 16-byte boundaries: one 16-byte load per lane and chunk
    for (int c0 = warp; vec && c0 < n_chunks; c0 += CONS_WARPS * 8) {
        float4 zv[8], qv[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int v = (c0 + j * CONS_WARPS) * DRAW_CHUNK + 4 * lane;
            const bool in = v < V;   // V is a multiple of 4: the four entries are inside together
            zv[j] = in ? __ldcg(reinterpret_cast<const float4 *>(src.z + v)) : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
            qv[j] = (src.zq && in) ? __ldcg(reinterpret_cast<const float4 *>(src.zq + v)) : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            float a = (src.weight_of(zv[j].x, qv[j].x) + src.weight_of(zv[j].y, qv[j].y)) + (src.weight_of(zv[j].z, qv[j].z) + src.weight_of(zv[j].w, qv[j].w));
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
            const int ch = c0 + j * CONS_WARPS;
            if (lane == 0 && ch < n_chunks) csum[ch] = a;
        }
    }
    for (int c0 = warp; !vec && c0 < n_chunks; c0 += CONS_WARPS * 8) {
        // all 32 (or 64) loads of the lane first, then the arithmetic: one round trip to L2 per eight chunks, not one per entry
        float zv[8][DRAW_CHUNK / 32], qv[8][DRAW_CHUNK / 32];
#pragma unroll
        for (int j = 0; j < 8; ++j)
#pragma unroll
            for (int it = 0; it < DRAW_CHUNK / 32; ++it) {
                const int v = (c0 + j * CONS_WARPS) * DRAW_CHUNK + it * 32 + lane;
                zv[j][it] = v < V ? __ldcg(src.z + v) : -INFINITY;
                qv[j][it] = (src.zq && v < V) ? __ldcg(src.zq + v) : -INFINITY;
            }
        float acc[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            float a = 0.f;
#pragma unroll
            for (int it = 0; it < DRAW_CHUNK / 32; ++it) a += src.weight_of(zv[j][it], qv[j][it]);
            acc[j] = a;
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            float a = acc[j];
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
            const int ch = c0 + j * CONS_WARPS;
            if (lane == 0 && ch < n_chunks) csum[ch] = a;
        }
    }
    bar_consumers();
    const int cpt = (n_chunks + CONS_THREADS - 1) / CONS_THREADS;   // chunks per thread of the second level
    {
        float a = 0.f;
        for (int j = 0; j < cpt; ++j) {
            const int ch = tid * cpt + j;
            a += ch < n_chunks ? csum[ch] : 0.f;
        }
        psum[tid] = a;
    }
    bar_consumers();
    // every thread walks the same two levels to the chunk that holds the crossing
    total = 0.f;
    for (int i = 0; i < CONS_THREADS; ++i) total += psum[i];
    w_tok = 0.f;
    if (!(total > 0.f)) return -1;
    const float target = u * total;
    float base = 0.f;
    int t_at = -1;
    for (int i = 0; i < CONS_THREADS; ++i) {
        if (base + psum[i] > target) { t_at = i; break; }
        base += psum[i];
    }
    int ch_at = -1;
    bool take_last = false;
    if (t_at >= 0) {
        for (int j = 0; j < cpt; ++j) {
            const int ch = t_at * cpt + j;
            if (ch >= n_chunks) break;
            if (base + csum[ch] > target) { ch_at = ch; break; }
            base += csum[ch];
        }
    }
    if (ch_at < 0) {   // rounding left no crossing: the last chunk of non-zero weight, its last such token
        take_last = true;
        for (int ch = n_chunks - 1; ch >= 0; --ch)
            if (csum[ch] > 0.f) { ch_at = ch; break; }
        if (ch_at < 0) return -1;
    }
    // pass 2: locate the token inside the chunk
    if (warp == 0) {
#pragma unroll
        for (int it = 0; it < DRAW_CHUNK / 32; ++it) {
            const int v = ch_at * DRAW_CHUNK + it * 32 + lane;
            wbuf[it * 32 + lane] = v < V ? src.weight(v) : 0.f;
        }
        __syncwarp();
        if (lane == 0) {
            float run = base;
            int tok = -1, last = -1;
            for (int i = 0; i < DRAW_CHUNK; ++i) {
                const float w = wbuf[i];
                if (w > 0.f) last = i;
                run += w;
                if (!take_last && run > target) { tok = i; break; }
            }
            if (tok < 0) tok = last < 0 ? 0 : last;
            res[0] = __int_as_float(ch_at * DRAW_CHUNK + tok);
            res[1] = wbuf[tok];
        }
    }
    bar_consumers();
    const int tok = __float_as_int(res[0]);
    w_tok = res[1];
    bar_consumers();   // the buffers may be rewritten by the next draw
    return tok;
}

// The same draw from a head's distribution exp(z - m), using what the head product already left behind: CTA b of the
// grid has published (max, sum of exp, argmax) of its own rows of the vocabulary, [16 t0(b), 16 t1(b)), a contiguous range in
// CTA order.  The running sum over the CTAs finds the CTA whose range holds the crossing; only that range's logits
// (vocabulary / grid entries) are read again.  Two round trips to L2 instead of a pass over the whole vocabulary by one CTA.
__device__ __noinline__ int block_draw_head(Smem *sm, const float *z, float m, const float *head_part, int col, int G, int V, float u,
                                            float &total, float &w_tok) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    float *psum = reinterpret_cast<float *>(sm->scratch + DRAW_OFFSET);   // second-level sums, then the located range
    float *wbuf = psum + CONS_THREADS;
    float *res = wbuf + DRAW_CHUNK;
    float *csum = res + 8;
    const int T = (V + 15) / 16;
    // (1) running sum over the CTAs' sums, by warp 0: lane l holds CTAs [l per, (l + 1) per)
    if (warp == 0) {
        const int per = (G + 31) / 32;
        float loc = 0.f;
        for (int k = 0; k < per; ++k) {
            const int b = lane * per + k;
            if (b < G) {
                const float4 v = __ldcg(reinterpret_cast<const float4 *>(head_part + ((size_t)b * MAX_COLS + col) * 4));
                loc += (v.x == -INFINITY) ? 0.f : v.y * __expf(v.x - m);
            }
        }
        float inc = loc;   // inclusive scan over the lanes
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const float o = __shfl_up_sync(0xffffffffu, inc, off);
            if (lane >= off) inc += o;
        }
        const float tot = __shfl_sync(0xffffffffu, inc, 31);
        const float target = u * tot;
        const unsigned hit = __ballot_sync(0xffffffffu, inc > target);
        int l_at = hit ? __ffs(hit) - 1 : -1;
        bool take_last = false;
        if (l_at < 0) {   // rounding left no crossing: the last lane of non-zero sum
            const unsigned pos = __ballot_sync(0xffffffffu, loc > 0.f);
            l_at = pos ? 31 - __clz(pos) : -1;
            take_last = true;
        }
        if (lane == (l_at < 0 ? 0 : l_at)) {
            int b_at = -1;
            float base = inc - loc;
            if (l_at >= 0) {
                float run = base;
                int last_b = -1;
                for (int k = 0; k < per; ++k) {   // the lane walks its CTAs again (the same values, from L2)
                    const int b = lane * per + k;
                    if (b >= G) break;
                    const float4 v = __ldcg(reinterpret_cast<const float4 *>(head_part + ((size_t)b * MAX_COLS + col) * 4));
                    const float wv = (v.x == -INFINITY) ? 0.f : v.y * __expf(v.x - m);
                    if (wv > 0.f) last_b = b;
                    if (!take_last && run + wv > target) { b_at = b; base = run; break; }
                    run += wv;
                }
                if (b_at < 0) { b_at = last_b; take_last = true; base = 0.f; }
            }
            res[0] = __int_as_float(b_at);
            res[1] = base;
            res[2] = tot;
            res[3] = take_last ? 1.f : 0.f;
        }
    }
    bar_consumers();
    const int b_at = __float_as_int(res[0]);
    const float base = res[1];
    total = res[2];
    const bool take_last = res[3] != 0.f;
    w_tok = 0.f;
    if (b_at < 0 || !(total > 0.f)) { bar_consumers(); return -1; }
    const float target = u * total;
    int t0, t1;
    cta_tile_range(T, b_at, G, t0, t1);
    const int v0 = t0 * 16, v1 = min(V, t1 * 16), n_sub = (v1 - v0 + DRAW_CHUNK - 1) / DRAW_CHUNK;
    // (2) sums of the 128-entry pieces of that range (one per warp and turn)
    for (int sub = warp; sub < n_sub; sub += CONS_WARPS) {
        float a = 0.f;
#pragma unroll
        for (int it = 0; it < DRAW_CHUNK / 32; ++it) {
            const int v = v0 + sub * DRAW_CHUNK + it * 32 + lane;
            a += v < v1 ? __expf(__ldcg(z + v) - m) : 0.f;
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
        if (lane == 0) csum[sub] = a;
    }
    bar_consumers();
    // (3) the piece that holds the crossing, then the entry inside it (warp 0; entries in vocabulary order)
    if (warp == 0) {
        float run = base;
        int sub_at = -1;
        bool tl = take_last;
        for (int sub = 0; sub < n_sub; ++sub) {
            if (!tl && run + csum[sub] > target) { sub_at = sub; break; }
            run += csum[sub];
        }
        if (sub_at < 0) {
            tl = true;
            for (int sub = n_sub - 1; sub >= 0; --sub)
                if (csum[sub] > 0.f) { sub_at = sub; break; }
        }
        int tok = -1;
        float wt = 0.f;
        if (sub_at >= 0) {
            // lane l holds the entries [4 l, 4 l + 4) of the piece
            float wv[4], loc = 0.f;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int v = v0 + sub_at * DRAW_CHUNK + 4 * lane + i;
                wv[i] = v < v1 ? __expf(__ldcg(z + v) - m) : 0.f;
                loc += wv[i];
            }
            float inc = loc;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const float o = __shfl_up_sync(0xffffffffu, inc, off);
                if (lane >= off) inc += o;
            }
            const float before = run + inc - loc;
            int my = -1;
            float r2 = before;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                r2 += wv[i];
                if (my < 0 && !tl && r2 > target) my = i;
            }
            const unsigned hit = __ballot_sync(0xffffffffu, my >= 0);
            int l_at, i_at;
            if (hit) {
                l_at = __ffs(hit) - 1;
                i_at = __shfl_sync(0xffffffffu, my, l_at);
            } else {   // the last entry of non-zero weight
                int lastp = -1;
#pragma unroll
                for (int i = 0; i < 4; ++i) if (wv[i] > 0.f) lastp = i;
                const unsigned pos = __ballot_sync(0xffffffffu, lastp >= 0);
                l_at = pos ? 31 - __clz(pos) : 0;
                i_at = max(__shfl_sync(0xffffffffu, lastp, l_at), 0);
            }
            float wsel = wv[0];
#pragma unroll
            for (int i = 1; i < 4; ++i) if (i == i_at) wsel = wv[i];
            wt = __shfl_sync(0xffffffffu, wsel, l_at);
            tok = v0 + sub_at * DRAW_CHUNK + 4 * l_at + i_at;
        }
        if (lane == 0) { res[4] = __int_as_float(tok); res[5] = wt; }
    }
    bar_consumers();
    const int tok = __float_as_int(res[4]);
    w_tok = res[5];
    bar_consumers();   // the buffers may be rewritten by the next draw
    return tok;
}

struct SampleArgs {
    const float *uniforms; float *q_stage; float4 *qinfo; const float *logit_stage; HeadResult *head_res; DevState *st;
    int vocab, max_seq, cps, L, seq0, nseq, exit_idx;
    const float *head_part; int G;   // the grid's per-CTA (max, sum of exp, argmax) of the head just evaluated
};

// Sampled decoding at a control point (its own function: its registers must not weigh on the streaming loops).
// After an intermediate head (Eq. 1): the newest token's successor is drawn from the head's distribution q; its
// probability q(t) is what the threshold test sees.  After the final head (Eq. 2): every early-predicted token t, in
// sequence order, is accepted with probability min{1, p*(t) / q(t)} -- the result stands in the column's head result as
// the token itself, so that the comparison of the bookkeeping accepts it -- and the first one that is not is replaced by
// a draw from Normalize(max(0, p* - q)); if all are accepted the next token is drawn from p* of the newest column.
__device__ __noinline__ void sample_stage(SampleArgs a, Smem *sm, bool after_head, const StepDesc *dprev, unsigned head_cols) {
    const int tid = threadIdx.x, V = a.vocab, cps = a.cps;
    HeadResult *hr_s = reinterpret_cast<HeadResult *>(sm->scratch + 8192);
    const int *tok_s = reinterpret_cast<const int *>(sm->scratch + 8192 + sizeof(HeadResult) * MAX_COLS);
    auto unif = [&](int s, int pos, int which) { return a.uniforms[((size_t)s * a.max_seq + pos) * SAMPLE_NU + which]; };
    if (after_head) {
        for (int col = 0; col < MAX_COLS; ++col) {
            if (!((head_cols >> col) & 1u)) continue;
            const int s = a.seq0 + (a.nseq == 1 ? 0 : col % a.nseq), pos = dprev->pos[col], slot = s * DRAFT_SLOTS + (pos & 7);
            float total, wt;
            const int tok = block_draw_head(sm, a.q_stage + (size_t)slot * V, hr_s[col].zmax, a.head_part, col, a.G, V, unif(s, pos + 1, 3 + a.exit_idx), total, wt);
            if (tid == 0) {
                hr_s[col].token = max(tok, 0);
                hr_s[col].p = tok < 0 ? 0.f : wt / total;
                a.head_res[col] = hr_s[col];
                a.qinfo[slot] = make_float4(hr_s[col].zmax, total, hr_s[col].p, 0.f);
            }
        }
    } else {
        for (int k = 0; k < a.nseq; ++k) {
            const int s = a.seq0 + k, ln = a.st->len[s], bs = a.st->base[s], nrow = ln - bs;
            if (nrow < 1 || nrow > cps || dprev->first_layer[(nrow - 1) * a.nseq + k] > a.L - 1) continue;
            bool rejected = false;
            for (int r = 0; r + 1 < nrow && !rejected; ++r) {
                const int col = r * a.nseq + k, pos_t = bs + r + 1, t = min(max(tok_s[col], 0), V - 1), slot = s * DRAFT_SLOTS + ((bs + r) & 7);
                const float *zs = a.logit_stage + (size_t)col * V;
                const float4 qi = a.qinfo[slot];
                const float ps = __expf(__ldcg(zs + t) - hr_s[col].zmax) / hr_s[col].sumexp;
                if (unif(s, pos_t, 1) * qi.z < ps) {   // accepted; every thread evaluates the same numbers
                    if (tid == 0) hr_s[col].token = t;
                    continue;
                }
                rejected = true;
                DrawSrc src{zs, hr_s[col].zmax, 1.f / hr_s[col].sumexp, a.q_stage + (size_t)slot * V, qi.x, 1.f / qi.y};
                float total, wt;
                int tok = block_draw(sm, src, V, unif(s, pos_t, 2), total, wt);
                if (tok < 0) {   // p* nowhere above q (they are equal up to rounding): draw from p*
                    DrawSrc plain{zs, hr_s[col].zmax, 0.f, nullptr, 0.f, 0.f};
                    tok = block_draw(sm, plain, V, unif(s, pos_t, 2), total, wt);
                }
                if (tid == 0) hr_s[col].token = max(tok, 0);
            }
            if (!rejected) {
                const int col = (nrow - 1) * a.nseq + k;
                float total, wt;
                const int tok = block_draw_head(sm, a.logit_stage + (size_t)col * V, hr_s[col].zmax, a.head_part, col, a.G, V, unif(s, ln, 0), total, wt);
                if (tid == 0) hr_s[col].token = max(tok, 0);
            }
        }
    }
    __threadfence_block();
    bar_consumers();
}

// ---------------------------------------------------------------- control point (CTA 0, consumer warps)

// What the bookkeeping works on, in the consumers' scratch.  (The next step's descriptor and the sequences' lengths as arrays of the
// bookkeeping warp were local memory, a load from L2 for each first touch behind the barrier's acquire: 13 us with eight sequences.)
struct Ctl {
    StepDesc nd;
    int len[MAX_SEQS], base[MAX_SEQS], target[MAX_SEQS], done[MAX_SEQS];
    int newest[MAX_SEQS];      // the newest token
};
constexpr int CTL_OFFSET = 8192 + ((int)sizeof(HeadResult) + 4) * MAX_COLS;
static_assert(CTL_OFFSET % 16 == 0 && CTL_OFFSET + (int)sizeof(Ctl) <= DRAW_OFFSET, "the control point's copies overlap the draw's buffers");

// Applies the outcome of the step that just ended (Eq. 1 after a head; verification and rollback,
// Eq. 2 at temperature zero, after the final head), then sets up the next step: its columns, the
// embeddings of its newest tokens, their rotary factors; finally publishes the action.
__device__ __forceinline__ void control_cta0(const MegaArgs &A, Smem *sm, int kind, int e, unsigned pub_no, const StepDesc &dprev,
                                          int &steps_started) {
    const Ctx &c = A.c;
    DevState *st = c.st;
    const MegaModel &M = A.m;
    const int tid = threadIdx.x, G = gridDim.x;
    const int nseq = A.nseq, seq0 = A.seq0, cps = c.slots, L = c.L;   // cps: token columns per sequence (slots)
    Pub *pub = reinterpret_cast<Pub *>(A.pub) + (pub_no & 1);
    // Shared-memory copies for the bookkeeping warp (fetched by many threads at once: a single
    // thread reading them from global memory one after the other spent 30 us here on round trips to L2):
    // the fill levels, the head results, and the tokens the verification compares with.
    int *fill_s = reinterpret_cast<int *>(sm->scratch);                                          // [nseq][L]
    HeadResult *hr_s = reinterpret_cast<HeadResult *>(sm->scratch + 8192);                       // [MAX_COLS]
    int *tok_s = reinterpret_cast<int *>(sm->scratch + 8192 + sizeof(HeadResult) * MAX_COLS);    // [MAX_COLS]: the token after the column's own
    static_assert(ADA_MAX_LAYERS * MAX_SEQS * sizeof(int) <= 8192, "fill levels of a launch's sequences must fit the scratch corner");
    Ctl &ctl = *reinterpret_cast<Ctl *>(sm->scratch + CTL_OFFSET);
    StepDesc &nd = ctl.nd;
    for (int i = tid; i < nseq * L; i += CONS_THREADS) fill_s[i] = c.fill[(size_t)seq0 * L + i];
    if (tid < (int)(sizeof(StepDesc) / 4)) reinterpret_cast<int *>(&nd)[tid] = reinterpret_cast<const int *>(&dprev)[tid];
    if (tid >= 64 && tid < 64 + MAX_SEQS) {
        const int k = tid - 64, s = seq0 + k;
        const bool in = k < nseq;
        const int ln = in ? st->len[s] : 0;
        ctl.len[k] = ln;
        ctl.base[k] = in ? st->base[s] : 0;
        ctl.target[k] = in ? st->target_len[s] : 0;
        ctl.done[k] = in ? st->done[s] : 1;
        ctl.newest[k] = in && ln > 0 && ln <= c.max_seq ? c.tokens[(size_t)s * c.max_seq + ln - 1] : 0;
    }
    if (tid >= CONS_THREADS - MAX_COLS) {
        const int j = tid - (CONS_THREADS - MAX_COLS), k = j % nseq;
        int v = -1;
        if (j / nseq < cps) {
            const int at = st->base[seq0 + k] + j / nseq + 1;
            if (at < c.max_seq) v = c.tokens[(size_t)(seq0 + k) * c.max_seq + at];
        }
        tok_s[j] = v;
    }
    // (a) head results of the columns that matter: warp w merges column w
    const unsigned head_cols = kind == CTRL_HEAD ? ((unsigned)dprev.head_mask & active_mask(dprev, e - 1))
                                                 : (kind == CTRL_TOP ? active_mask(dprev, L - 1) : 0u);
    if (kind != CTRL_START) {
#pragma unroll 1
        for (int w = tid >> 5; w < MAX_COLS; w += CONS_WARPS)
            if ((head_cols >> w) & 1u) {
                const HeadResult hr = merge_head(A.head_part, G, w);
                if ((tid & 31) == 0) { c.head_res[w] = hr; hr_s[w] = hr; }
            }
    }
    __threadfence_block();
    bar_consumers();
    // (a') sampled decoding replaces the tokens and probabilities the bookkeeping below works with
    if (A.sampling && kind != CTRL_START && !(kind == CTRL_TOP && st->pf_end > 0)) {
        SampleArgs sa{A.uniforms, A.q_stage, A.qinfo, c.logit_stage, c.head_res, st, c.vocab, c.max_seq, cps, L, seq0, nseq,
                      kind == CTRL_HEAD ? (int)M.exit_at[e] - 1 : 0, A.head_part, G};
        sample_stage(sa, sm, kind == CTRL_HEAD, &dprev, head_cols);
    }
    // (b) bookkeeping, one warp: every lane follows the same decisions, lane 0 writes them down, loops over the layers are shared out.
    // Every scalar it may need is read up front (the loads overlap); counters are bumped by reductions, which do not wait for memory.
    // The lanes have to agree on all of it, or they would part ways at the sums over the warp: the error word, which any CTA may set at
    // any time, is settled by a vote, and lane 0 writes nothing before every lane has read.
    if (tid < 32) {
        const int lane = tid;
        const bool w0 = lane == 0;
        auto bump = [&](long long *p, long long v) { if (w0) atomicAdd(reinterpret_cast<unsigned long long *>(p), (unsigned long long)v); };
        // fill levels of sequence k at layers below n become `to`; the sum of (from - old level)
        auto refill = [&](int k, int n, int from, int to) {
            int rl = 0;
            for (int l = lane; l < n; l += 32) {
                rl += from - fill_s[k * L + l];
                fill_s[k * L + l] = to;
                c.fill[(size_t)(seq0 + k) * L + l] = to;
            }
            return (long long)__reduce_add_sync(0xffffffffu, rl);
        };
        const bool stop0 = __any_sync(0xffffffffu, *(volatile int *)A.err != 0);
        const int pf_end0 = st->pf_end, pf_pos0 = st->pf_pos, max_early0 = st->max_early;
        const int tape_n0 = st->tape_n, hl_n0 = st->head_log_n;
        const int tape_i0 = st->tape_i;
        int tape_i = tape_i0, hl_n = hl_n0;
        const float gamma0 = st->gamma;
        const int eos0 = st->eos_id;
        const long long steps0 = __ldcg(&st->st.steps);   // past the L1: the counters are bumped by reductions
        int action = ACT_NEWSTEP, verified = 0;
        int keep_rows = 0, keep_row0 = 0;
        int pf_end = pf_end0, pf_pos = pf_pos0;
        __syncwarp();
        if (stop0) action = ACT_STOP;
        // ---- Eq. 1 after an intermediate head: every sequence whose newest token consulted it decides for itself
        if (action != ACT_STOP && kind == CTRL_HEAD) {
            unsigned still = 0;   // sequences that go on climbing in this step
            int n_steps_seen = 0;
            for (int k = 0; k < nseq; ++k) {
                const int s = seq0 + k, len = ctl.len[k], col = (len - 1 - ctl.base[k]) * nseq + k;
                if (col < 0 || col >= MAX_COLS || dprev.first_layer[col] > e - 1) continue;   // not in this step any more
                if (!((head_cols >> col) & 1u)) { still |= 1u << k; continue; }                // climbing, but may not exit early
                const HeadResult hr = hr_s[col];
                bool decide = hr.p > gamma0;
                if (s == 0 && tape_i < tape_n0) {
                    const uint8_t t = st->tape[tape_i++];
                    if (t == 0) decide = false;
                    if (t == 1) decide = true;
                }
                bump(&st->st.head_evals, 1);
                if (s == 0 && c.head_log && hl_n < kHeadLogCap) {
                    float *hl = c.head_log + 4 * (size_t)hl_n;
                    if (w0) { hl[0] = (float)(steps0 + n_steps_seen); hl[1] = (float)e; hl[2] = (float)hr.token; hl[3] = hr.p; }
                    ++hl_n;
                }
                if (!decide) { still |= 1u << k; continue; }
                bump(&st->st.row_layers, refill(k, e, len, len));
                const int token = min(max(hr.token, 0), c.vocab - 1);
                if (w0) {
                    c.tokens[(size_t)s * c.max_seq + len] = token;
                    ctl.newest[k] = token;
                    ctl.len[k] = len + 1;
                    st->len[s] = len + 1;
                    for (int j = k; j < MAX_COLS; j += nseq) {   // the sequence sits out the rest of the step
                        nd.first_layer[j] = NO_LAYER;
                        nd.head_mask &= ~(1 << j);
                    }
                }
                bump(&st->st.early_exits, 1);
                bump(&st->st.exits_at_layer[e], 1);
                bump(&st->st.steps, 1);
                ++n_steps_seen;
            }
            if (w0 && tape_i != tape_i0) st->tape_i = tape_i;
            if (w0 && hl_n != hl_n0) st->head_log_n = hl_n;
            if (still) action = ACT_CONTINUE;
            else bump(&st->st.layer_passes, e);   // the weights of layers 1..e were streamed once, for all the sequences
        }
        const bool prefilling = pf_end > 0;
        if (action != ACT_STOP && kind == CTRL_TOP && prefilling) {
            // a pass over prompt positions [pf_pos, pf_pos + n) of the launch's one sequence is complete at every layer
            const int s = seq0, n = dprev.n_cols, end = pf_pos + n;
            refill(0, L, 0, end);
            pf_pos = end;
            if (w0) st->pf_pos = end;
            if (end >= pf_end) {   // KV cache <- LM(x) done: the full-depth argmax at the last prompt token is the first generated token
                const int np = pf_end, token = min(max(hr_s[n - 1].token, 0), c.vocab - 1);
                pf_end = 0;
                keep_rows = 1;
                keep_row0 = n - 1;
                verified = s == 0;
                if (w0) {
                    c.tokens[(size_t)s * c.max_seq + np] = token;
                    ctl.newest[0] = token;
                    ctl.len[0] = np + 1; ctl.base[0] = np; ctl.done[0] = 1;
                    st->len[s] = np + 1;
                    st->base[s] = np;
                    st->n_prompt[s] = np;
                    st->done[s] = 1;
                    st->pf_end = 0;
                    st->keep_rows = 1;
                    st->keep_row0 = n - 1;
                }
            }
        }
        // ---- verification (Eq. 2 at temperature zero) of every sequence whose newest token reached the last layer
        if (action != ACT_STOP && kind == CTRL_TOP && !prefilling) {
            for (int k = 0; k < nseq; ++k) {
                const int s = seq0 + k, len = ctl.len[k], base = ctl.base[k], nrow = len - base;
                if (nrow < 1 || nrow > cps || dprev.first_layer[(nrow - 1) * nseq + k] > L - 1) continue;   // left the step at an exit layer, or idle
                int32_t *tok = c.tokens + (size_t)s * c.max_seq;
                int bad = -1;
                for (int j = 0; j + 1 < nrow; ++j)
                    if (hr_s[j * nseq + k].token != tok_s[j * nseq + k]) { bad = j; break; }
                int new_base, keep;
                const int token = min(max(hr_s[(bad < 0 ? nrow - 1 : bad) * nseq + k].token, 0), c.vocab - 1);
                if (bad < 0) {
                    bump(&st->st.accepted, nrow - 1);
                    new_base = len;
                    keep = nrow;
                } else {
                    bump(&st->st.accepted, bad);
                    bump(&st->st.rejected, 1);
                    bump(&st->st.discarded, nrow - 2 - bad);
                    new_base = base + bad + 1;
                    keep = bad + 1;
                }
                if (w0) tok[new_base] = token;
                // Algorithm 1 runs "while t_i != [EOS]": the verified tokens of this step (positions base + 1 .. new_base,
                // each equal to the full-depth argmax of the row before it) end the sequence at the first end-of-sequence
                // token among them.  An early-predicted end-of-sequence token stops nothing until it is verified here.
                int tgt = ctl.target[k];
                if (eos0 >= 0) {
                    for (int j = 0; j < keep; ++j)
                        if (min(max(hr_s[j * nseq + k].token, 0), c.vocab - 1) == eos0) {
                            if (base + j + 2 <= tgt) { tgt = base + j + 2; if (w0) st->eos_hit[s] = 1; }
                            break;
                        }
                }
                int new_len = new_base + 1;
                if (new_len > tgt) {
                    bump(&st->st.truncated, new_len - tgt);
                    new_len = tgt;
                    new_base = new_len - 1;
                }
                keep = new_len - 1 - base;   // verified tokens that stay: their logit rows are the ones a capture keeps
                bump(&st->st.row_layers, refill(k, L, len, new_base));
                if (w0) {
                    ctl.newest[k] = token;   // (a sequence that was cut short is done, and embeds nothing)
                    ctl.len[k] = new_len; ctl.base[k] = new_base;
                    st->len[s] = new_len;
                    st->base[s] = new_base;
                    if (new_len >= tgt) { ctl.done[k] = 1; st->done[s] = 1; }
                }
                bump(&st->st.verify_steps, 1);
                bump(&st->st.steps, 1);
                if (s == 0) {
                    keep_rows = keep;
                    keep_row0 = 0;
                    if (w0) { st->keep_rows = keep; st->keep_row0 = 0; }
                    verified = 1;
                }
            }
        }
        __syncwarp();
        if (action != ACT_STOP && kind == CTRL_TOP && !prefilling) bump(&st->st.layer_passes, L);
        if (action == ACT_NEWSTEP) {
            bool all_done = true;
            for (int k = 0; k < nseq; ++k) all_done = all_done && ctl.done[k];
            if (all_done) { action = ACT_STOP; if (w0) st->n_done = 1; }
            else if (steps_started >= A.step_budget) action = ACT_STOP;
        }
        if (action == ACT_NEWSTEP) {
            ++steps_started;
            int n_cols = 0, newest_mask = 0, head_mask = 0, pmax = 0, fresh = 0, run_final = 1;
            if (lane < MAX_COLS) { nd.first_layer[lane] = NO_LAYER; nd.pos[lane] = 0; }
            if (lane < MAX_SEQS) nd.seq_pmax[lane] = -1;
            __syncwarp();
            if (pf_end > 0) {   // next pass over the prompt: up to eight positions, all from layer 1
                const int n = min(MAX_COLS, pf_end - pf_pos);
                n_cols = n;
                newest_mask = 1 << (n - 1);
                pmax = pf_pos + n - 1;
                fresh = (1 << n) - 1;
                run_final = pf_pos + n >= pf_end;
                if (n < 1 || pmax >= c.max_seq) {
                    if (w0) atomicCAS(A.err, 0, ERR_BAD_STATE);
                    action = ACT_STOP;
                }
                if (lane < n) { nd.first_layer[lane] = 0; nd.pos[lane] = pf_pos + lane; }
                if (w0) nd.seq_pmax[0] = pmax;
            } else {
                for (int k = 0; k < nseq; ++k) {
                    if (ctl.done[k]) continue;   // a sequence that has reached its target idles while the others go on
                    const int len = ctl.len[k], base = ctl.base[k], nrow = len - base;
                    if (nrow < 1 || nrow > cps || nrow * nseq > MAX_COLS || len > c.max_seq || base < 0) {
                        if (w0) atomicCAS(A.err, 0, ERR_BAD_STATE);
                        action = ACT_STOP;
                        break;
                    }
                    for (int j = 0; j < nrow; ++j) {
                        const int pos = base + j;
                        int fl = 0;
                        for (int l = lane; l < L; l += 32) fl += fill_s[k * L + l] > pos;
                        fl = __reduce_add_sync(0xffffffffu, fl);
                        if (w0) { nd.first_layer[j * nseq + k] = (unsigned char)fl; nd.pos[j * nseq + k] = pos; }
                    }
                    const int cn = (nrow - 1) * nseq + k;
                    n_cols += nrow;
                    newest_mask |= 1 << cn;
                    fresh |= 1 << cn;
                    if (nrow - 1 < max_early0 && len < ctl.target[k]) head_mask |= 1 << cn;
                    if (w0) nd.seq_pmax[k] = len - 1;
                    pmax = max(pmax, len - 1);
                }
            }
            if (w0) { nd.n_cols = n_cols; nd.newest_mask = newest_mask; nd.head_mask = head_mask; nd.pmax = pmax; nd.fresh = fresh; nd.run_final = run_final; }
        }
        __syncwarp();
        if (action == ACT_NEWSTEP || action == ACT_CONTINUE)
            for (int i = lane; i < (int)(sizeof(StepDesc) / 4); i += 32) reinterpret_cast<int *>(&pub->d)[i] = reinterpret_cast<const int *>(&nd)[i];
        if (w0) {
            pub->action = action;
            pub->cap_keep = 0;
            if (kind == CTRL_TOP && c.capture && verified) {
                const int at = st->capture_n, keep = min(keep_rows, st->capture_cap - at);
                pub->cap_keep = max(keep, 0);
                pub->cap_at = at;
                pub->cap_row0 = keep_row0;
                if (keep > 0) st->capture_n = at + keep;
            }
            sm->bcast[0] = action;
        }
    }
    bar_consumers();
    const int action = sm->bcast[0];
    // (c) the embeddings of the tokens that enter, and their rotary factors
    if (action == ACT_NEWSTEP) {
        const __nv_bfloat16 *g0 = M.attn_norm[0];
        const int half = c.hd / 2, nf = __popc(nd.fresh);
        for (int i = tid; i < nf * half; i += CONS_THREADS) {
            const int w = i % half;
            unsigned m = (unsigned)nd.fresh;
            for (int q = i / half; q > 0; --q) m &= m - 1;
            const int col = __ffs(m) - 1, pos = nd.pos[col];
            // angle = pos * freq in double, reduced to [-pi, pi] in double, then single-precision sin / cos
            // (double-precision transcendentals with large arguments are slow on this GPU)
            const double a = (double)pos * A.rope_freq[w];
            const double r = a - 6.283185307179586476925 * rint(a * 0.15915494309189533577);
            float sn, cs;
            sincosf((float)r, &sn, &cs);
            c.rope_cs[((size_t)col * half + w) * 2 + 0] = cs;
            c.rope_cs[((size_t)col * half + w) * 2 + 1] = sn;
        }
        // 8 / 4 / 2 / 1 warps a column, eight elements a lane and turn, the next turn's loads in flight
        const int ws = nf == 1 ? 3 : nf == 2 ? 2 : nf <= 4 ? 1 : 0, at = 8 * (tid & ((32 << ws) - 1)), step = 256 << ws;
#pragma unroll 1
        for (int f = tid >> (5 + ws); f < nf; f += CONS_WARPS >> ws) {
            unsigned m = (unsigned)nd.fresh;
            for (int q = f; q > 0; --q) m &= m - 1;
            const int col = __ffs(m) - 1, k = nseq == 1 ? 0 : col % nseq;
            const int token = st->pf_end > 0 ? c.tokens[(size_t)(seq0 + k) * c.max_seq + nd.pos[col]] : ctl.newest[k];
            const __nv_bfloat16 *erow = M.tok_embed + (size_t)min(max(token, 0), c.vocab - 1) * c.d;
            // (tensors start on 16-byte boundaries, ada_model_set_tensor, and a row is a multiple of 64 elements)
            auto load = [&](const __nv_bfloat16 *p, int n) { return __ldg(reinterpret_cast<const uint4 *>(p + n)); };
            const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
            uint4 ev = at < c.d ? load(erow, at) : zero, gv = at < c.d ? load(g0, at) : zero;
#pragma unroll 1
            for (int n0 = 0; n0 < c.d; n0 += step) {
                const int n = n0 + at, nn = n + step;
                const uint32_t e[4] = {ev.x, ev.y, ev.z, ev.w}, g[4] = {gv.x, gv.y, gv.z, gv.w};
                ev = nn < c.d ? load(erow, nn) : zero;
                gv = nn < c.d ? load(g0, nn) : zero;
                float v[8], q[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) { v[i] = bf16_of_word(e[i >> 1], i); q[i] = __fmul_rn(v[i], v[i]); }
                // sum of the squares of sixteen neighbours, as a tree
                float sq = ((q[0] + q[1]) + (q[2] + q[3])) + ((q[4] + q[5]) + (q[6] + q[7]));
                sq += __shfl_xor_sync(0xffffffffu, sq, 1);
                if (n < c.d) {
                    float4 *o = reinterpret_cast<float4 *>(c.resid + (size_t)col * c.d + n);
                    o[0] = make_float4(v[0], v[1], v[2], v[3]);
                    o[1] = make_float4(v[4], v[5], v[6], v[7]);
#pragma unroll
                    for (int i = 0; i < 8; i += 2) xfrag_store2(A.XA, n + i, col, v[i] * bf16_of_word(g[i >> 1], i), v[i + 1] * bf16_of_word(g[i >> 1], i + 1));
                    if ((tid & 1) == 0) A.ssq_a[(size_t)(n >> 4) * MAX_COLS + col] = sq;
                }
            }
        }
    }
    // the release orders what all threads wrote (through the barrier); the producers pass a proxy fence behind their acquire of it
    bar_consumers();
    if (tid == 0) asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(&pub->seq), "r"(pub_no) : "memory");
}

// Every role of every CTA passes here; returns the action and (for a new step) the descriptor.
template <int ROLE>
__device__ __forceinline__ int control_point(const MegaArgs &A, const Shared &S, int kind, int e, unsigned &pub_no, StepDesc &d,
                                             int &steps_started) {
    Smem *sm = S.sm;
    ++pub_no;
    const Pub *pub = reinterpret_cast<Pub *>(A.pub) + (pub_no & 1);
    int action;
    // the new step descriptor is copied into the role's shared copy `d` by one thread (by every lane of a
    // producer warp: same values), and checked before anything is indexed with it
    auto fetch = [&]() -> int {
        int act = aborted(S) ? ACT_STOP : *(volatile const int *)&pub->action;
        if (act == ACT_NEWSTEP || act == ACT_CONTINUE) {   // a step that goes on may have lost the columns of sequences that left it
            const volatile int *src = reinterpret_cast<const volatile int *>(&pub->d);
            int *dst = reinterpret_cast<int *>(&d);
#pragma unroll
            for (int i = 0; i < (int)(sizeof(StepDesc) / 4); ++i) dst[i] = src[i];
            bool bad = d.n_cols < 1 || d.n_cols > MAX_COLS || d.pmax < 0 || d.pmax >= A.c.max_seq;
#pragma unroll
            for (int i = 0; i < MAX_COLS; ++i) bad = bad || d.pos[i] < 0 || d.pos[i] >= A.c.max_seq;
#pragma unroll
            for (int i = 0; i < MAX_SEQS; ++i) bad = bad || d.seq_pmax[i] >= A.c.max_seq;
            if (bad) act = ACT_STOP;   // cannot happen unless memory was corrupted; never index with it
        }
        // The two record slots alternate.  A role that fell two control points behind would find its slot
        // already rewritten for a later one: a record is used only if its number is still the expected one
        // after it has been copied.
        if (!aborted(S) && ld_acquire(&pub->seq) != pub_no) {
            raise_error(S, ERR_BAD_STATE);
            act = ACT_STOP;
        }
        return act;
    };
    if (ROLE == 2) {
        if (blockIdx.x == 0) {
            control_cta0(A, sm, kind, e, pub_no, d, steps_started);
            bar_consumers();   // every thread is done with the old descriptor before thread 0 replaces it
        }
        if (threadIdx.x == 0) {
            grid_wait(S, &pub->seq, pub_no);
            const bool cap = kind == CTRL_TOP && A.c.capture && !aborted(S);
            const int cap_keep = cap ? *(volatile const int *)&pub->cap_keep : 0, cap_at = cap ? *(volatile const int *)&pub->cap_at : 0,
                      cap_row0 = cap ? *(volatile const int *)&pub->cap_row0 : 0;
            sm->bcast[1] = fetch();   // also checks that the record was still the expected one after it had been read
            sm->bcast[5] = aborted(S) ? 0 : cap_keep;
            sm->bcast[6] = cap_at;
            sm->bcast[7] = cap_row0;
        }
        bar_consumers();
        action = sm->bcast[1];
        // Logits of the verified rows (test hook): every CTA copies its share.  (CTA 0 alone took 80 us for a row of 128256
        // logits, with the whole GPU waiting; shared out it is one round trip to L2.)
        if (kind == CTRL_TOP && A.c.capture) {
            const int keep = sm->bcast[5], V = A.c.vocab;
            for (int j = 0; j < keep; ++j) {
                const float *src = A.c.logit_stage + (size_t)(sm->bcast[7] + j * A.nseq) * V;   // sequence 0's columns
                float *dst = A.c.capture + (size_t)(sm->bcast[6] + j) * V;
                for (int i0 = blockIdx.x * CONS_THREADS + threadIdx.x; i0 < V; i0 += 4 * gridDim.x * CONS_THREADS) {
                    float v[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int i = i0 + u * gridDim.x * CONS_THREADS;
                        v[u] = i < V ? __ldcg(src + i) : 0.f;
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int i = i0 + u * gridDim.x * CONS_THREADS;
                        if (i < V) dst[i] = v[u];
                    }
                }
            }
        }
    } else {
        grid_wait(S, &pub->seq, pub_no);
        action = fetch();
        // What the grid wrote before this control point -- cache rows of the steps before, the next step's input -- is ordered before the
        // bulk copies of the steps after it: those of cache blocks without rows of their own pass wait for no barrier.
        fence_proxy_async();
        // the lanes stop together: one may have seen an error that another has not
        if (__any_sync(0xffffffffu, action == ACT_STOP)) action = ACT_STOP;
        __syncwarp();
    }
    return action;
}

// ---------------------------------------------------------------- attention phase

// Shared memory of the attention phase: the consumers' scratch.
template <int HD> struct AttnSmem {
    float o[CONS_WARPS][8][HD];      // unnormalised outputs of eight query rows by warp, columns rotated by 8 (row % 8)
    float mx[CONS_WARPS][16], l[CONS_WARPS][16];   // row maxima and sums by warp
};
static_assert(sizeof(AttnSmem<128>) <= SCRATCH_BYTES, "attention buffers exceed the consumers' scratch");

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
    __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t *>(&v);
}
// x / group for the q heads per kv head the persistent path admits (1..4) and x < 128, without the
// general integer division (some thirty of those sat on the critical path of every attention item)
__device__ __forceinline__ int div_group(int x, int group) {
    return group == 4 ? x >> 2 : group == 2 ? x >> 1 : group == 1 ? x : (x * 43) >> 7;
}
__device__ __forceinline__ void st_tagged(unsigned long long *p, float v, unsigned tag) { st_relaxed_u64(p, ((unsigned long long)tag << 32) | __float_as_uint(v)); }
__device__ __forceinline__ void st_tagged2(unsigned long long *p, float a, float b, unsigned tag) {   // two tagged words; 16-byte aligned
    const unsigned long long t = (unsigned long long)tag << 32;
    asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(t | __float_as_uint(a)), "l"(t | __float_as_uint(b)) : "memory");
}
__device__ __forceinline__ bool ld_tagged2(const unsigned long long *p, float &a, float &b, unsigned tag) {
    unsigned long long x, y;
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(x), "=l"(y) : "l"(p) : "memory");
    a = __uint_as_float((unsigned)x);
    b = __uint_as_float((unsigned)y);
    return (unsigned)(x >> 32) == tag && (unsigned)(y >> 32) == tag;
}

// The active columns of the launch's k-th sequence as slots (bit j: column j nseq + k), and its 128-position chunks in this step.
__device__ __forceinline__ unsigned seq_slots(const MegaArgs &A, unsigned mask, int k) {
    if (A.nseq == 1) return mask;
    unsigned m = 0;
    for (int j = 0, col = k; col < MAX_COLS; ++j, col += A.nseq) m |= ((mask >> col) & 1u) << j;
    return m;
}
__device__ __forceinline__ int seq_chunks(const MegaArgs &A, const StepDesc &d, unsigned mask, int k) {
    return (d.seq_pmax[k] >= 0 && seq_slots(A, mask, k) != 0) ? d.seq_pmax[k] / ATT_CHUNK + 1 : 0;
}

// A work item: (sequence of the launch, kv head, 128-position chunk anchored at position 0).
struct AttnItem {
    int k, kvh, j, nsb, p_base;   // sequence, kv head, chunk, 64-position sub-blocks, first position
    unsigned slots;               // the sequence's active slots
    unsigned tiles;               // query tiles in use: row slot group + head of the sequence's (token, q head) pairs, sixteen to a tile
    bool has_new;                 // holds positions of this pass, whose cache rows this step's QKV phase writes
};
// The items of one CTA in the order in which every role walks them: cta, cta + G, ...; those with rows of this pass last, since
// their cache rows are there only when the QKV phase is complete.
struct AttnWalk {
    int pass, at, n;
    __device__ __forceinline__ AttnWalk(const MegaArgs &A, const StepDesc &d, unsigned mask) : pass(0), at(blockIdx.x), n(0) {
        for (int k = 0; k < A.nseq; ++k) n += A.c.nkv * seq_chunks(A, d, mask, k);
    }
    __device__ __forceinline__ bool next(const MegaArgs &A, const StepDesc &d, unsigned mask, AttnItem &it) {
#pragma unroll 1
        for (; pass < 2; ++pass, at = blockIdx.x)
#pragma unroll 1
            for (; at < n;) {
                int i = at, nchunk = seq_chunks(A, d, mask, 0);
                it.k = 0;
                while (it.k + 1 < A.nseq && i >= A.c.nkv * nchunk) {
                    i -= A.c.nkv * nchunk;
                    nchunk = seq_chunks(A, d, mask, ++it.k);
                }
                nchunk = max(nchunk, 1);
                it.kvh = min(i / nchunk, A.c.nkv - 1);
                it.j = i - it.kvh * nchunk;
                it.slots = seq_slots(A, mask, it.k);
                it.p_base = it.j * ATT_CHUNK;
                it.has_new = d.pos[(__ffs(it.slots) - 1) * A.nseq + it.k] < it.p_base + ATT_CHUNK;   // the lowest position of the pass
                at += gridDim.x;
                if ((int)it.has_new != pass) continue;
                it.nsb = min(ATT_CHUNK / ATT_PAGE, (d.seq_pmax[it.k] - it.p_base) / ATT_PAGE + 1);
                const int lo = (__ffs(it.slots) - 1) * A.c.group, hi = (32 - __clz(it.slots)) * A.c.group - 1;   // first and last row in use
                it.tiles = (lo < 16 ? 1u : 0u) | (hi >= 16 ? 2u : 0u);
                return true;
            }
        return false;
    }
};

// K and V blocks (64 positions of one kv head, one cache page's share) travel through the weight ring, in line between the QKV
// and the O product's weights: per item K of its sub-blocks, then V.  Nine blocks are in flight per CTA instead of the three that
// the activation ring held, and O's weights follow without a gap.
// The rows of the tokens of this pass are written by the QKV epilogues of other CTAs: an item that holds one is fetched once the
// grid has passed the barrier that ends the QKV phase (`bar_target`), every other as soon as the ring has room: its rows were written in
// earlier steps, in front of the control point behind which this producer fenced its copies (control_point).
__device__ __forceinline__ void attn_produce_kv(const MegaArgs &A, const Shared &S, const StepDesc &d, int layer, unsigned mask, unsigned bar_target,
                                                Rings &r, uint64_t pol) {
    const Ctx &c = A.c;
    Smem *sm = S.sm;
    const int lane = threadIdx.x & 31;
    const uint32_t bytes = (uint32_t)(ATT_PAGE * c.hd * 2);
    const __nv_bfloat16 *pool = reinterpret_cast<const __nv_bfloat16 *>(c.kv_pool);
    AttnWalk w(A, d, mask);
    AttnItem it;
    bool synced = false;
#pragma unroll 1
    while (w.next(A, d, mask, it)) {
        if (it.has_new && !synced) {
            grid_wait(S, A.grid_ctr, bar_target);
            fence_proxy_async();
            synced = true;
        }
        const int32_t *pages = c.page_table + (size_t)(A.seq0 + it.k) * c.max_pages + (it.p_base >> c.page_shift);
#pragma unroll 1
        for (int b = 0; b < 2 * it.nsb; ++b) {
            const int which = b >= it.nsb, page = pages[which ? b - it.nsb : b];
            const uint32_t ws = r.w % NW;
            mbar_wait(S, &sm->w_empty[ws], ((r.w / NW) & 1) ^ 1);
            ++r.w;
            if (lane == 0) {
                if (!aborted(S)) {
                    const size_t blk = ((((size_t)page * c.L + layer) * 2 + which) * c.nkv + it.kvh) * ((size_t)ATT_PAGE * c.hd);
                    mbar_expect_tx(&sm->w_full[ws], bytes);
                    bulk_g2s(sm->w[ws], pool + blk, bytes, &sm->w_full[ws], pol);
                }
                w_issued_set(sm, r.w);
            }
        }
    }
}
// The items' query fragments come through the activation ring, one stage per item: the tiles in use, 64 hd bytes each.
// `after_first` as for gemm_produce_x.
template <class Hook>
__device__ __forceinline__ void attn_produce_q(const MegaArgs &A, const Shared &S, const StepDesc &d, unsigned mask, unsigned bar_target, Rings &r, uint64_t pol,
                                               Hook &&after_first) {
    const Ctx &c = A.c;
    Smem *sm = S.sm;
    const uint32_t tile_bytes = (uint32_t)c.hd * 64;
    AttnWalk w(A, d, mask);
    AttnItem it;
    bool synced = false;
#pragma unroll 1
    while (w.next(A, d, mask, it)) {
        mbar_wait(S, &sm->x_empty[r.xs], r.xp ^ 1);
        const bool first = !synced;
        if (first) {
            grid_wait(S, A.grid_ctr, bar_target);
            fence_proxy_async();
            synced = true;
        }
        if ((threadIdx.x & 31) == 0 && !aborted(S)) {
            const unsigned char *src = reinterpret_cast<const unsigned char *>(A.qfrag) + (size_t)(it.k * c.nkv + it.kvh) * 2 * tile_bytes + (it.tiles == 2u ? tile_bytes : 0u);
            const uint32_t bytes = it.tiles == 3u ? 2 * tile_bytes : tile_bytes;
            mbar_expect_tx(&sm->x_full[r.xs], bytes);
            bulk_g2s(sm->x[r.xs], src, bytes, &sm->x_full[r.xs], pol);
        }
        if (first) after_first();
        r.next_x();
    }
}

// Consumers: causal attention of every active column over the cache, which by now holds the rows of this pass too (the QKV
// epilogue wrote them).  The queries arrive rotated, scaled and split into bf16 high / low parts, laid out as tensor-core A
// fragments.
//
// An item's 128 positions are eight slices of sixteen.  Where its queries fit one tile of sixteen rows (plain decoding, few tokens
// in flight) each warp takes a slice; where they span two, warp (tile, quarter) takes slices quarter and quarter + 4 of that tile.
// Where a CTA has several items of one tile each, two groups of four warps work on different ones, a warp on slices quarter and
// quarter + 4: an item is a chain of latencies (5 us for 1 us of work), and two chains run side by side.
// Either way a row's numbers are formed alike: the maximum over the chunk first (exchanged through shared memory), weights
// exp(score - maximum), one product per slice, slices s and s + 4 added, then (0 + 1) + (2 + 3).  So a token's attention does not
// depend on which other tokens ride along.  (Running maxima per warp over two sub-blocks left half of the warps idle in the
// one-tile case and cost two more meetings.)
//
// The chunk partials travel as 8-byte words that carry the phase number beside the value: whoever sees the tag sees the
// value, so no fence, counter and second look stand between writing and reading them; all CTAs share the merging (a range of
// the launch's (token, q head, feature pair)s each), in one round trip per eight chunks.  Who merges does not change what is computed.
template <int HD>
__device__ __forceinline__ void attn_consume(const MegaArgs &A, const Shared &S, const StepDesc &d, unsigned mask, unsigned tag, Rings &r) {
    // consumers' barrier of the warps that share an item
    auto meet = [](bool dual, int grp) {
        if (dual) asm volatile("bar.sync %0, 128;" ::"r"(2 + grp) : "memory");
        else bar_consumers();
    };
    const Ctx &c = A.c;
    Smem *sm = S.sm;
    AttnSmem<HD> *as = reinterpret_cast<AttnSmem<HD> *>(sm->scratch);
    constexpr int KSQ = HD / 16, NT = HD / 8;
    constexpr int TS = HD + 2;                             // tagged words per chunk partial: output, max, sum
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int group = c.group, nseq = A.nseq;
    auto words = [&](int col, int h, int chunk) { return A.attn_tag + (((size_t)col * c.nq + h) * c.n_chunks + chunk) * TS; };
    uint32_t known = r.w;
    AttnWalk walk(A, d, mask);
    AttnItem it;
    // Two items at a time: this CTA has more than one, and every sequence's queries fit one tile.  8B shape at 3000 positions (192
    // items) 16.0 -> 14.8 us a layer, 13B with four sequences (640) 30.7 -> 27.7.  With 64 features a head an item is half the work
    // and two one after the other are faster (1B, eight sequences, 128 to 192 items: 10.1 against 11.1 us).
    const int grp = warp >> 2;
    bool dual = walk.n > (int)(blockIdx.x + (HD == 64 ? 2 : 1) * gridDim.x);
    for (int k = 0; k < nseq; ++k) {
        const unsigned sl = seq_slots(A, mask, k);
        if (sl) dual = dual && ((__ffs(sl) - 1) * group >= 16 || (32 - __clz(sl)) * group <= 16);
    }
    // Every row of the step has a single chunk: its item finishes it, there is nothing to merge (1B shape at 60 positions 7.2 -> 6.6 us a layer).
    const bool one_chunk = d.pmax < ATT_CHUNK;
    int turn = 0;   // group whose item it is
#pragma unroll 1
    while (walk.next(A, d, mask, it)) {
        const bool one_tile = it.tiles != 3u, solo = one_tile && !dual;   // solo: eight warps on one tile
        const int mt = one_tile ? (int)(it.tiles >> 1) : grp, qr = warp & 3;
        const int w0 = solo ? 0 : 4 * grp;                                // the first of the warps whose slices make up this warp's tile
        const bool lead = warp == (dual ? 4 * grp : 0);                   // releases the item's K and V blocks
        const uint32_t k_stage = r.w, v_stage = r.w + it.nsb;
        r.w += 2 * it.nsb;
        if (dual) {
            const bool other = turn != grp;
            turn ^= 1;
            if (other) {   // the other group's item; activation stages are waited for and released by every warp
                mbar_wait(S, &sm->x_full[r.xs], r.xp);
                if (lane == 0) mbar_arrive(&sm->x_empty[r.xs]);
                r.next_x();
                continue;
            }
        }
        // last position that rows lane / 4 and lane / 4 + 8 of the tile see (-1: no token)
        int lim[2];
#pragma unroll
        for (int rh = 0; rh < 2; ++rh) {
            const int slot = div_group(mt * 16 + (lane >> 2) + rh * 8, group);
            lim[rh] = slot < 8 && ((it.slots >> slot) & 1u) ? d.pos[slot * nseq + it.k] : -1;
        }
        mbar_wait(S, &sm->x_full[r.xs], r.xp);
        if (tid == 0) trace(S, EV_ATT, 2);   // queries ready
        const unsigned char *qs = sm->x[r.xs] + (one_tile ? 0 : mt) * (HD * 64) + lane * 32;
        float s[2][2][4], m[2] = {-INFINITY, -INFINITY};   // scores [slice][n-tile][fragment], row maxima
        const int sb0 = solo ? grp : 0, n_sl = solo ? (sb0 < it.nsb ? 1 : 0) : it.nsb;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
#pragma unroll
            for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                for (int i = 0; i < 4; ++i) s[u][nt][i] = -INFINITY;
            if (u >= n_sl) continue;
            w_wait(S, k_stage + sb0 + u, known);
            float sh[2][4], sl[2][4];
#pragma unroll
            for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                for (int i = 0; i < 4; ++i) { sh[nt][i] = 0.f; sl[nt][i] = 0.f; }
            const int id = lane >> 3, pl = 16 * qr + (lane & 7) + 8 * (id >> 1);
            const unsigned char *krow = sm->w[(k_stage + sb0 + u) % NW] + pl * (HD * 2);
#pragma unroll
            for (int k0 = 0; k0 < KSQ; k0 += 4) {   // four k-steps of loads in flight, then their multiply-adds
                uint4 qh[4], ql[4];
                uint32_t kf[4][4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int ks = k0 + q;
                    qh[q] = *reinterpret_cast<const uint4 *>(qs + ks * 1024);
                    ql[q] = *reinterpret_cast<const uint4 *>(qs + ks * 1024 + 16);
                    ldmatrix_x4(kf[q], krow + ((((2 * ks) | (id & 1)) ^ (pl & 7)) << 4));
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint32_t ah[4] = {qh[q].x, qh[q].y, qh[q].z, qh[q].w}, al[4] = {ql[q].x, ql[q].y, ql[q].z, ql[q].w};
                    mma16816(sh[0], ah, kf[q][0], kf[q][1]);
                    mma16816(sh[1], ah, kf[q][2], kf[q][3]);
                    mma16816(sl[0], al, kf[q][0], kf[q][1]);
                    mma16816(sl[1], al, kf[q][2], kf[q][3]);
                }
            }
            const int p0 = it.p_base + (sb0 + u) * ATT_PAGE + 16 * qr + 2 * (lane & 3);
#pragma unroll
            for (int nt = 0; nt < 2; ++nt)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    s[u][nt][i] = p0 + 8 * nt + (i & 1) <= lim[i >> 1] ? sh[nt][i] + sl[nt][i] : -INFINITY;
                    m[i >> 1] = fmaxf(m[i >> 1], s[u][nt][i]);
                }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm->x_empty[r.xs]);
        r.next_x();
        // ---- the chunk's row maxima
#pragma unroll
        for (int rh = 0; rh < 2; ++rh) {
            m[rh] = fmaxf(m[rh], __shfl_xor_sync(0xffffffffu, m[rh], 1));
            m[rh] = fmaxf(m[rh], __shfl_xor_sync(0xffffffffu, m[rh], 2));
            if ((lane & 3) == 0) as->mx[warp][(lane >> 2) + 8 * rh] = m[rh];
        }
        meet(dual, grp);   // (A) scores done: maxima in place, K blocks free; and everybody has left the item before
        if (lead && lane < it.nsb) mbar_arrive(&sm->w_empty[(k_stage + lane) % NW]);
        float l[2] = {0.f, 0.f};
        uint32_t ph[2][4], plo[2][4];   // weights of the two slices as A fragments, high and low parts
#pragma unroll
        for (int rh = 0; rh < 2; ++rh) {
            const int row = (lane >> 2) + 8 * rh;
            float mm = -INFINITY;
#pragma unroll
            for (int w = 0; w < 4; ++w) mm = fmaxf(mm, as->mx[w0 + w][row]);
            if (solo) {
#pragma unroll
                for (int w = 4; w < CONS_WARPS; ++w) mm = fmaxf(mm, as->mx[w][row]);
            }
            m[rh] = mm;
            float ls[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                float p[4] = {0.f, 0.f, 0.f, 0.f};
                if (u < n_sl && mm != -INFINITY) {
                    p[0] = __expf(s[u][0][2 * rh] - mm); p[1] = __expf(s[u][0][2 * rh + 1] - mm);
                    p[2] = __expf(s[u][1][2 * rh] - mm); p[3] = __expf(s[u][1][2 * rh + 1] - mm);
                }
                ls[u] = (p[0] + p[1]) + (p[2] + p[3]);
                ls[u] += __shfl_xor_sync(0xffffffffu, ls[u], 1);
                ls[u] += __shfl_xor_sync(0xffffffffu, ls[u], 2);
                // A fragment of P: a0/a1 = n-tile 0 (rows r / r+8), a2/a3 = n-tile 1
                const __nv_bfloat162 h0 = __floats2bfloat162_rn(p[0], p[1]), h1 = __floats2bfloat162_rn(p[2], p[3]);
                ph[u][rh] = *reinterpret_cast<const uint32_t *>(&h0);
                ph[u][2 + rh] = *reinterpret_cast<const uint32_t *>(&h1);
                plo[u][rh] = pack_bf16(p[0] - __low2float(h0), p[1] - __high2float(h0));
                plo[u][2 + rh] = pack_bf16(p[2] - __low2float(h1), p[3] - __high2float(h1));
            }
            l[rh] = solo ? ls[0] : ls[0] + ls[1];
        }
        // ---- outputs of this warp's slice(s)
        float o[NT][4];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int i = 0; i < 4; ++i) o[nt][i] = 0.f;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            if (u >= n_sl) continue;
            w_wait(S, v_stage + sb0 + u, known);
            const int id = lane >> 3, pl = 16 * qr + (lane & 7) + 8 * (id & 1);
            const unsigned char *vrow = sm->w[(v_stage + sb0 + u) % NW] + pl * (HD * 2);
#pragma unroll
            for (int n0 = 0; n0 < NT / 2; n0 += 4) {
                uint32_t vf[4][4];
#pragma unroll
                for (int q = 0; q < 4; ++q) ldmatrix_x4_trans(vf[q], vrow + ((((2 * (n0 + q)) | (id >> 1)) ^ (pl & 7)) << 4));
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int np = n0 + q;
                    float a[2][4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) a[0][i] = a[1][i] = 0.f;
                    mma16816(a[0], ph[u], vf[q][0], vf[q][1]);
                    mma16816(a[1], ph[u], vf[q][2], vf[q][3]);
                    mma16816(a[0], plo[u], vf[q][0], vf[q][1]);
                    mma16816(a[1], plo[u], vf[q][2], vf[q][3]);
#pragma unroll
                    for (int i = 0; i < 4; ++i) { o[2 * np][i] += a[0][i]; o[2 * np + 1][i] += a[1][i]; }
                }
            }
        }
        if (tid == 0) trace(S, EV_ATT, 5);   // products done
        // ---- slices added, eight rows of the tile(s) at a time, and published
        if ((lane & 3) == 0) {
            as->l[warp][lane >> 2] = l[0];
            as->l[warp][(lane >> 2) + 8] = l[1];
            if (warp == w0 && !one_chunk) {   // the maximum's word (the next item's maxima may already be on their way when the sums are read)
#pragma unroll
                for (int rh = 0; rh < 2; ++rh)
                    if (lim[rh] >= it.p_base) {
                        const int row = 16 * mt + (lane >> 2) + 8 * rh, slot = div_group(row, group);
                        st_tagged(words(slot * nseq + it.k, it.kvh * group + row - slot * group, it.j) + HD, m[rh], tag);
                    }
            }
        }
        bool freed = false;
#pragma unroll
        for (int rh = 0; rh < 2; ++rh) {
            // a half of the rows without a token (in any tile in use) is skipped, by all warps alike
            unsigned rows = 0;   // bit t: half rh of tile t holds a token
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                const int lo = div_group(16 * t + 8 * rh, group), hi = div_group(16 * t + 8 * rh + 7, group);
                rows |= ((it.slots & ((2u << min(hi, 30)) - (1u << min(lo, 30)))) != 0 ? 1u : 0u) << t;
            }
            rows &= it.tiles;
            if (rows == 0) continue;
            if (freed) meet(dual, grp);   // everybody has read the half before
            {
                float *dst = as->o[warp][lane >> 2];
#pragma unroll
                for (int nt = 0; nt < NT; ++nt)
                    *reinterpret_cast<float2 *>(dst + ((nt * 8 + 2 * (lane & 3) + 8 * (lane >> 2)) & (HD - 1))) = make_float2(o[nt][2 * rh], o[nt][2 * rh + 1]);
            }
            meet(dual, grp);   // (B) outputs in place
            if (!freed) {      // V blocks free
                if (lead && lane < it.nsb) mbar_arrive(&sm->w_empty[(v_stage + lane) % NW]);
                freed = true;
            }
            const int n_el = (one_tile ? 1 : 2) * 8 * (HD / 2);
#pragma unroll 1
            for (int e = dual ? tid & 127 : tid; e < n_el; e += dual ? 128 : CONS_THREADS) {
                const int dim = (e & (HD / 2 - 1)) * 2, rr = (e / (HD / 2)) & 7, t = one_tile ? mt : e / (HD / 2) >> 3;
                const int row = 16 * t + 8 * rh + rr, slot = div_group(row, group);
                if (slot >= 8 || !((it.slots >> slot) & 1u)) continue;
                const int col = slot * nseq + it.k;
                if (d.pos[col] < it.p_base) continue;
                const int wq = solo ? 0 : dual ? w0 : 4 * t, at = (dim + 8 * rr) & (HD - 1);
                float2 q[4];
                float ql[4];
#pragma unroll
                for (int w = 0; w < 4; ++w) {
                    q[w] = *reinterpret_cast<const float2 *>(&as->o[wq + w][rr][at]);
                    ql[w] = as->l[wq + w][8 * rh + rr];
                    if (solo) {
                        const float2 b = *reinterpret_cast<const float2 *>(&as->o[w + 4][rr][at]);
                        q[w].x += b.x; q[w].y += b.y;
                        ql[w] += as->l[w + 4][8 * rh + rr];
                    }
                }
                const float ox = (q[0].x + q[1].x) + (q[2].x + q[3].x), oy = (q[0].y + q[1].y) + (q[2].y + q[3].y), den = (ql[0] + ql[1]) + (ql[2] + ql[3]);
                const int h = it.kvh * group + row - slot * group;
                if (one_chunk) {
                    xfrag_store2(A.XO, h * HD + dim, col, ox / den, oy / den);
                } else {
                    unsigned long long *out = words(col, h, it.j);
                    st_tagged2(out + dim, ox, oy, tag);
                    if (dim == 0) st_tagged(out + HD + 1, den, tag);
                }
            }
        }
        if (tid == 0) trace(S, EV_ITEM, it.j);
    }
    if (one_chunk) return;
    // ---- this CTA's share of the merging: two features of one (column, q head) per thread and pass; the chunk
    // partials are folded in ascending order, eight at a time with all their loads in flight, by the running-max rule
    const unsigned total = (unsigned)(__popc(mask) * c.nq * (HD / 2));
    const int u1 = (int)(total * (blockIdx.x + 1) / gridDim.x);
#pragma unroll 1
    for (int u = (int)(total * blockIdx.x / gridDim.x) + tid; u < u1; u += CONS_THREADS) {
        const int row = u / (HD / 2), dim = (u % (HD / 2)) * 2, h = row % c.nq;
        int nth = row / c.nq, col = 0;   // the nth active column
        for (unsigned mm = mask; mm; mm &= mm - 1)
            if (nth-- == 0) { col = __ffs(mm) - 1; break; }
        const int nch = d.pos[col] / ATT_CHUNK + 1;
        const unsigned long long *part = words(col, h, 0);
        float Mx = -INFINITY, den = 0.f, ax = 0.f, ay = 0.f;
#pragma unroll 1
        for (int k0 = 0; k0 < nch; k0 += 8) {
            float ml[8], ll[8], ox[8], oy[8];
            unsigned long long t0 = 0;
            for (uint32_t n = 0;; ++n) {
                bool ok = true;
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    ml[q] = -INFINITY; ll[q] = 0.f; ox[q] = 0.f; oy[q] = 0.f;
                    if (k0 + q < nch) {
                        const bool a = ld_tagged2(part + (size_t)(k0 + q) * TS + HD, ml[q], ll[q], tag);
                        const bool b = ld_tagged2(part + (size_t)(k0 + q) * TS + dim, ox[q], oy[q], tag);
                        ok = ok && a && b;
                    }
                }
                if (ok) break;
                if ((n & 15u) == 15u || S.wait_ns < SHORT_LIMIT_NS) {   // bounded like every other wait on another CTA
                    if (aborted(S)) break;
                    if (*(volatile int *)S.err != 0) { *(volatile int *)&S.sm->abort = 1; break; }
                    const unsigned long long t = gtime();
                    if (t0 == 0) t0 = t;
                    else if (t - t0 > S.wait_ns) { raise_error(S, ERR_TIMEOUT_GRID); break; }
                }
                __nanosleep(32);
            }
            float Mn = Mx;
#pragma unroll
            for (int q = 0; q < 8; ++q) Mn = fmaxf(Mn, ml[q]);
            if (Mn == -INFINITY) continue;
            const float sc = Mx == -INFINITY ? 0.f : __expf(Mx - Mn);
            den *= sc; ax *= sc; ay *= sc;
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (ml[q] != -INFINITY) {
                    const float w = __expf(ml[q] - Mn);
                    den = __fmaf_rn(ll[q], w, den);
                    ax = __fmaf_rn(ox[q], w, ax);
                    ay = __fmaf_rn(oy[q], w, ay);
                }
            Mx = Mn;
        }
        xfrag_store2(A.XO, h * HD + dim, col, ax / den, ay / den);
    }
    if (tid == 0) trace(S, EV_COMBINE, 0);
}

// ---------------------------------------------------------------- the walker

// Phases of a step.  The first six are products; their plans are worked out once per launch (Smem::plan).
enum { PH_QKV = 0, PH_O, PH_GU, PH_DOWN, PH_T, PH_HEAD, PH_PRODUCTS, PH_ATTN = PH_PRODUCTS };
__device__ __forceinline__ int prof_class(int ph) {   // class of ada_debug_profile that the phase's time is booked to
    return ph == PH_QKV ? 2 : ph == PH_ATTN ? 4 : ph == PH_O ? 5 : ph == PH_GU ? 6 : ph == PH_DOWN ? 8 : ph == PH_T ? 10 : 9;
}
// Whole tiles or units of (tile, chunk): cutting tiles costs an exchange of partial sums at the end of the phase (some 0.7 us)
// and saves the stages by which the CTA with most whole tiles exceeds its share, 0.36 us each (less where they are parked): taken from
// four stages on.  Measured, whole -> cut: 13B, four columns, O (8 stages fewer) 12.8 -> 10.4 us, down (22) 28.1 -> 22.9, QKV (5)
// 27.1 -> 26.1; 8B gate-up (14) 40.2 -> 36.9, down (7) 19.5 -> 18.8, QKV (3) 10.8 -> 11.0, O (2) 7.6 -> 7.7; 1B gate-up (4)
// 12.7 -> 11.3, QKV (2) 5.6 -> 6.3.  (13B gate-up, 2 stages, gains all the same: 44.7 -> 43.9.)
constexpr int CUT_STAGES = 4;
__host__ __device__ __forceinline__ Gemm phase_gemm(const MegaArgs &A, int ph, int G) {
    const Ctx &c = A.c;
    Gemm g;
    g.N = ph == PH_QKV ? c.qkv_rows : ph == PH_GU ? 2 * c.dff : ph == PH_HEAD ? c.vocab : c.d;
    g.K = ph == PH_O ? c.nq * c.hd : ph == PH_DOWN ? c.dff : c.d;
    g.pair = ph == PH_GU ? 2 : 1;
    g.half = ph == PH_GU ? c.dff : 0;
    const int T = g.tiles(), nch = (g.K + KC - 1) / KC, most = (T + G - 1) / G * nch, share = (T * nch + G - 1) / G;
    g.split = A.part != nullptr && ph != PH_HEAD && (most - share) * g.pair >= CUT_STAGES;
    return g;
}

// Epilogues of the products: consumer warps, one element (row of the tile, column) per thread and pass; see gemm_consume.
template <int HD> struct Epilogue {
    const MegaArgs &A;
    const Shared &S;
    const StepDesc &d;
    int ph, l;               // phase, 0-based layer
    unsigned vseq;           // phase number whose normalisation factors vec[] has to hold
    bool scaled;             // the product's result is multiplied by them
    float scale;             // head: scale of the logits
    bool inter;              // head: an intermediate one
    bool next_in, final_in;  // down product: prepares the next layer's input, a head's input

    static constexpr int HALF = HD / 2, KSQ = HD / 16;
    __device__ __forceinline__ int seq_of(int col) const { return A.seq0 + (A.nseq == 1 ? 0 : col % A.nseq); }

    // Operands fetched while the weights stream: three words per element.
    //   QKV: rotary factors (cos, sin), cache page; O, down: residual, gain of the next product's input, gain of a head's input
    __device__ __forceinline__ const void *operand(int w, int tile, int row, int col) const {   // (null: not needed)
        const Ctx &c = A.c;
        const int n0 = tile * 16, n = n0 + row;
        if (ph == PH_QKV) {
            if (w == 2) return n0 >= c.nq * HD ? c.page_table + (size_t)seq_of(col) * c.max_pages + (d.pos[col] >> c.page_shift) : nullptr;
            return n0 < (c.nq + c.nkv) * HD ? c.rope_cs + ((size_t)col * HALF + ((n0 & (HD - 1)) >> 1) + (row & 7)) * 2 + w : nullptr;
        }
        if (ph != PH_O && ph != PH_DOWN) return nullptr;
        if (w == 0) return c.resid + (size_t)col * c.d + n;
        if (w == 1) return next_in ? (ph == PH_O ? A.m.ffn_norm[l] : A.m.attn_norm[l + 1]) + (n & ~1) : nullptr;
        return final_in ? A.m.final_norm + (n & ~1) : nullptr;
    }
    __device__ __forceinline__ void pre(int ps, int tile, int row, int col) const {
        uint32_t *stash = stash_of(S.sm, ps);
#pragma unroll
        for (int w = 0; w < 3; ++w) {
            const void *p = operand(w, tile, row, col);
            if (p) cp_async4(stash + w * CONS_THREADS, p);
        }
    }
    __device__ __forceinline__ void operator()(int ps, bool act, int tile, int row, int col, float a0, float a1) const {
        const Ctx &c = A.c;
        const int n0 = tile * 16, n = n0 + row;
        float rs = 1.f;
        if (scaled) { vec_wait(S, vseq); rs = S.sm->vec[col]; }
        uint32_t ops[3] = {0u, 0u, 0u};
        if (ph == PH_QKV || ph == PH_O || ph == PH_DOWN) {
            if (TILES == 1 || ps < STASH_PASSES) {
                cp_async_wait_all();
                const uint32_t *stash = stash_of(S.sm, ps);
#pragma unroll
                for (int w = 0; w < 3; ++w) ops[w] = stash[w * CONS_THREADS];
            } else if (act) {
#pragma unroll
                for (int w = 0; w < 3; ++w) {
                    const uint32_t *p = static_cast<const uint32_t *>(operand(w, tile, row, col));
                    if (p) ops[w] = __ldcg(p);
                }
            }
        }
        a0 *= rs;
        if (ph == PH_GU) {
            a1 *= rs;
            if (act) xfrag_store(A.XH, n, col, a0 / (1.0f + expf(-a0)) * a1);
        } else if (ph == PH_HEAD) {
            // Sampled decoding: logits over the temperature, which are kept, the final head's by column, an intermediate head's by
            // the position of its row (the verification of the token drawn from them needs them again).
            // (max, sum exp, argmax) of the tile's sixteen rows by a butterfly, then into the half-warp's running one of this pass.
            Msa run;
            run.m = -INFINITY; run.s = 0.f; run.i = INT_MAX;
            if (act && n < c.vocab) {
                const float z = a0 * scale;
                if (A.sampling && inter) A.q_stage[((size_t)seq_of(col) * DRAFT_SLOTS + (d.pos[col] & 7)) * c.vocab + n] = z;
                else if (A.sampling || A.store_logits) c.logit_stage[(size_t)col * c.vocab + n] = z;
                run.m = z; run.s = 1.f; run.i = n;
            }
#pragma unroll
            for (int off = 1; off < 16; off <<= 1) {
                Msa o;
                o.m = __shfl_xor_sync(0xffffffffu, run.m, off);
                o.s = __shfl_xor_sync(0xffffffffu, run.s, off);
                o.i = __shfl_xor_sync(0xffffffffu, run.i, off);
                run = msa_merge(run, o);
            }
            if (row == 0 && act) {
                Msa *mine = head_state() + 16 * ps + (threadIdx.x >> 4);
                *mine = msa_merge(*mine, run);
            }
        } else if (ph == PH_T) {
            if (act) xfrag_store(A.XT, n, col, a0);
        } else if (ph == PH_QKV) {
            const float other = __shfl_xor_sync(0xffffffffu, a0, 8);   // the partner of a rotation
            const int qd = c.nq * HD, kvd = c.nkv * HD;
            if (!act || n0 >= c.qkv_rows) return;
            if (n0 < qd + kvd) {
                const float co = __uint_as_float(ops[0]), si = __uint_as_float(ops[1]);
                const int dim = ((n0 & (HD - 1)) >> 1) + (row & 7) + (row >> 3) * HALF;   // rows r and r + 8 hold features j and j + hd/2
                const float y = a0 * co + (row < 8 ? -other : other) * si;
                if (n0 < qd) {
                    const int h = n0 / HD, kvh = div_group(h, c.group), k = A.nseq == 1 ? 0 : col % A.nseq, slot = A.nseq == 1 ? col : col / A.nseq;
                    const int qcol = slot * c.group + (h - kvh * c.group);   // row of the sequence's (token, q head) pairs
                    const int qrow = qcol & 15, m = qcol >> 4, ks = dim >> 4, kk = dim & 15;
                    const int ln = (qrow & 7) * 4 + ((kk & 7) >> 1), reg = (qrow >> 3) + 2 * (kk >> 3);
                    const float yq = y * rsqrtf((float)HD);
                    const __nv_bfloat16 hi = __float2bfloat16_rn(yq);
                    __nv_bfloat16 *f = reinterpret_cast<__nv_bfloat16 *>(A.qfrag) + (((((size_t)k * c.nkv + kvh) * 2 + m) * KSQ + ks) * 32 + ln) * 16 + reg * 2 + (kk & 1);
                    f[0] = hi;
                    f[8] = __float2bfloat16_rn(yq - __bfloat162float(hi));
                } else {
                    cache_row(ops[2], 0, (n0 - qd) / HD, d.pos[col], dim, y);
                }
            } else {
                const int nv = n - qd - kvd;
                cache_row(ops[2], 1, nv / HD, d.pos[col], nv & (HD - 1), a0);
            }
        } else {   // O and down: residual add, inputs of the products that follow, partial sums of squares
            const float v = act ? __uint_as_float(ops[0]) + a0 : 0.f;
            float sq = v * v;
            sq += __shfl_xor_sync(0xffffffffu, sq, 8);
            sq += __shfl_xor_sync(0xffffffffu, sq, 1);
            sq += __shfl_xor_sync(0xffffffffu, sq, 2);
            sq += __shfl_xor_sync(0xffffffffu, sq, 4);
            if (!act) return;
            c.resid[(size_t)col * c.d + n] = v;
            if (next_in) xfrag_store(ph == PH_O ? A.XB : A.XA, n, col, v * bf16_of_word(ops[1], n));
            if (final_in) xfrag_store(A.XF, n, col, v * bf16_of_word(ops[2], n));
            if (row == 0) (ph == PH_O ? A.ssq_b : A.ssq_a)[(size_t)tile * MAX_COLS + col] = sq;
        }
    }
    __device__ __forceinline__ void cache_row(uint32_t page, int which, int kvh, int pos, int dim, float v) const {   // one element of a K or V row
        const Ctx &c = A.c;
        const size_t blk = ((((size_t)page * c.L + l) * 2 + which) * c.nkv + kvh) * ((size_t)ATT_PAGE * HD) + (size_t)(pos & (ATT_PAGE - 1)) * HD;
        reinterpret_cast<__nv_bfloat16 *>(c.kv_pool)[blk + ((((dim >> 3) ^ (pos & 7)) << 3) | (dim & 7))] = __float2bfloat16_rn(v);
    }
    // running (max, sum exp, argmax) of every half-warp and pass: (tile slot, column) u of gemm_consume is half-warp u % 16 of pass u / 16
    __device__ __forceinline__ Msa *head_state() const { return reinterpret_cast<Msa *>(S.sm->scratch + RED_BYTES); }
    __device__ __forceinline__ void head_begin() const {   // (each by the thread that uses it)
        if ((threadIdx.x & 15) == 0)
            for (int ps = 0; ps < MAX_COLS / 2; ++ps) {
                Msa &m = head_state()[16 * ps + (threadIdx.x >> 4)];
                m.m = -INFINITY; m.s = 0.f; m.i = INT_MAX;
            }
    }
    // the CTA's (max, sum exp, argmax) of every column in use: the column's half-warps (tile slots) in ascending order
    __device__ __forceinline__ void head_end(const Plan &pl, unsigned mask) const {
        bar_consumers();
        if (threadIdx.x < MAX_COLS && ((mask >> threadIdx.x) & 1u)) {
            const int sh = element_shift(Groups(pl).left), ci = __popc(mask & ((1u << threadIdx.x) - 1u));
            Msa a; a.m = -INFINITY; a.s = 0.f; a.i = INT_MAX;
            for (int w = 0; w < 1 << sh; ++w) a = msa_merge(a, head_state()[(ci << sh) + w]);
            float *o = A.head_part + ((size_t)blockIdx.x * MAX_COLS + threadIdx.x) * 4;
            o[0] = a.m; o[1] = a.s; o[2] = __int_as_float(a.i);
        }
    }
};

// ROLE 0: producer warp of weights and K / V blocks, 1: of activations and queries, 2: consumer warps.
//
// A step is a sequence of phases; every role walks it with one loop whose body holds each piece of code once (one product, one
// attention, one control point) and takes from the phase number what differs.
template <int ROLE, int HD>
__device__ __forceinline__ void run(const MegaArgs &A, Shared &S) {
    const Ctx &c = A.c;
    const MegaModel &M = A.m;
    Smem *sm = S.sm;
    const int G = gridDim.x;
    const int L = c.L, d_model = c.d, ntd = d_model / 16;
    const uint64_t pol = ROLE == 0 ? policy_evict_first() : policy_evict_last();
    Rings r;
    unsigned bar_no = 0, pub_no = 0;   // phases and control points behind this role
    int steps_started = 0;
    // The step descriptor lives in shared memory, one copy per role (the roles pass a control point at
    // different times): indexed by a run-time column it would otherwise sit in local memory, whose
    // cached lines do not survive the acquire of a grid barrier -- every first touch after a barrier
    // then costs a round trip to L2 on the critical path.
    StepDesc &d = *reinterpret_cast<StepDesc *>(sm->desc[ROLE]);
    if (ROLE != 2 || threadIdx.x == 0) {
        d.n_cols = 0; d.newest_mask = 0; d.head_mask = 0; d.pmax = 0; d.fresh = 0; d.run_final = 1;
#pragma unroll
        for (int i = 0; i < MAX_COLS; ++i) { d.first_layer[i] = NO_LAYER; d.pos[i] = 0; }
#pragma unroll
        for (int i = 0; i < MAX_SEQS; ++i) d.seq_pmax[i] = -1;
    }
    if (ROLE == 2) bar_consumers(); else __syncwarp();

    // Phase times: a phase ends when the whole grid has reported it.  The activation producer of CTA 0 sees that first (it waits for
    // it before it fetches the next input, and books after that).  The consumers do not wait for it, and a CTA without a tile of a
    // product passes it in no time: booked by them, the 1B shape's down product took 2 us of its 9.
    if (ROLE == 1) sm->t_booked = gtime();
    int behind = -1;   // class of the phase whose end has not been booked yet
    auto book = [&](int cls) {
        if (ROLE == 1 && blockIdx.x == 0 && (threadIdx.x & 31) == 0 && cls >= 0) {
            const unsigned long long t = gtime();
            // reductions, not read-modify-write: nobody waits for a load from L2 at every phase
            atomicAdd(reinterpret_cast<unsigned long long *>(&c.st->st.phase_ns[cls]), t - sm->t_booked);
            atomicAdd(reinterpret_cast<unsigned long long *>(&c.st->st.phase_count[cls]), 1ull);
            sm->t_booked = t;
        }
    };

    int ctl = CTRL_START, e = 0;   // the control point ahead; 1-based layer of its head
    int step_i = 0, l = 0, ph = PH_QKV;
#pragma unroll 1
    for (;;) {
        if (ROLE == 2 && blockIdx.x == 0) consumers_meet(S, A.grid_ctr, bar_no * (unsigned)G);   // CTA 0 reads every CTA's head partials
        if (ROLE == 1 && blockIdx.x == 0) {
            grid_wait(S, A.grid_ctr, bar_no * (unsigned)G);
            book(behind);
            behind = -1;
        }
        const int action = control_point<ROLE>(A, S, ctl, e, pub_no, d, steps_started);
        book(0);
        if (action == ACT_NEWSTEP) {
            l = 0;
            S.tr_on = step_i >= A.trace_step0 && step_i < A.trace_step1;
            ++step_i;
        } else if (action == ACT_CONTINUE) {
            l = e;   // exit layers are below the last one
        } else {
            if (ROLE == 2 && TILES == 1 && (threadIdx.x & 31) == 0) atomicAdd(reinterpret_cast<unsigned long long *>(&c.st->st.parked), (unsigned long long)r.parked);
            return;
        }
        ph = PH_QKV;
        // ---- the phases up to the next control point
#pragma unroll 1
        for (;;) {
            const bool final_head = ph == PH_HEAD && l == L;   // heads: l counts the layers that are complete
            const bool inter = (ph == PH_HEAD || ph == PH_T) && !final_head;
            const unsigned mask = active_mask(d, final_head ? L - 1 : inter ? l - 1 : l);
            const unsigned cmask = inter ? (unsigned)d.head_mask & mask : mask;
            if (ph == PH_ATTN) {
                if (ROLE == 0) attn_produce_kv(A, S, d, l, mask, bar_no * (unsigned)G, r, pol);
                if (ROLE == 1) attn_produce_q(A, S, d, mask, bar_no * (unsigned)G, r, pol, [&]() { book(behind); });
                if (ROLE == 2) {
                    // (a CTA without an item must not report the phase before the one in front of it is complete)
                    if (AttnWalk(A, d, mask).n <= (int)blockIdx.x) consumers_meet(S, A.grid_ctr, bar_no * (unsigned)G);
                    attn_consume<HD>(A, S, d, mask, bar_no + 1, r);
                }
            } else {
                // ---- a product.  QKV is finished in its epilogue: q rotated, scaled and stored as tensor-core fragments for the
                // attention phase; k rotated, v as it is, both rounded to bf16 and written straight into their cache
                // rows (Algorithm 1: "update KV cache at layer l by processing all tokens in P[l] in parallel").
                // The rows of every q and k head come reordered so that a 16-row tile holds the features
                // [8 t, 8 t + 8) and [hd/2 + 8 t, hd/2 + 8 t + 8): the two partners (i, i + hd/2) of a rotation
                // are then rows r and r + 8 of one tile, which two lanes of a warp finish, eight lanes apart.
                const Plan pl = sm->plan[ph];
                const bool with_T = inter && M.has_T[l];
                const unsigned vseq = bar_no + 1;
                // the product's result is multiplied by the normalisation factors of its input's rows
                const bool scaled = ph == PH_QKV || ph == PH_GU || ph == PH_T || (ph == PH_HEAD && !with_T);
                if (ROLE == 0) {
                    const CUtensorMap *W = M.maps + (ph == PH_HEAD ? MAPS_PER_LAYER * L : ph == PH_T ? MAPS_PER_LAYER * L + 1 + l
                                                     : MAPS_PER_LAYER * l + (ph == PH_QKV ? 0 : ph == PH_O ? 1 : ph == PH_GU ? 2 : 4));
                    gemm_produce_w(S, pl, W, ph == PH_GU && M.gu_two[l] ? W + 1 : nullptr, c.dff, r, pol);
                }
                if (ROLE == 1) {
                    const __nv_bfloat16 *X = ph == PH_QKV ? A.XA : ph == PH_O ? A.XO : ph == PH_GU ? A.XB : ph == PH_DOWN ? A.XH : ph == PH_HEAD && with_T ? A.XT : A.XF;
                    gemm_produce_x(S, pl, reinterpret_cast<const uint4 *>(X), Cols(cmask), r, pol,
                                   [&]() {
                                       book(behind);
                                       if (scaled) rstd_produce(sm, ph == PH_GU ? A.ssq_b : A.ssq_a, ntd, d_model, c.eps, vseq);
                                   },
                                   [&]() {   // the input must not be fetched before the phase that wrote it is complete
                                       grid_wait(S, A.grid_ctr, bar_no * (unsigned)G);
                                       fence_proxy_async();
                                       if ((threadIdx.x & 31) == 0) trace(S, EV_PHASE_BEGIN, prof_class(ph));
                                   });
                }
                if (ROLE == 2) {
                    const Epilogue<HD> epi{A, S, d, ph, l, vseq, scaled,
                                           final_head ? (A.sampling ? A.inv_temp : 1.0f) : inter ? M.head_scale[l] * (A.sampling ? A.inv_temp : 1.0f) : 1.0f, inter,
                                           ph == PH_O || l + 1 < L, ph == PH_DOWN && (l + 1 == L || M.exit_at[l + 1] != 0)};
                    // (an idle CTA must not report a phase before the one in front of it is complete: the counter would run ahead)
                    if (Groups(pl).left <= 0) consumers_meet(S, A.grid_ctr, bar_no * (unsigned)G);
                    if (ph == PH_HEAD) epi.head_begin();
                    gemm_consume<TILES == 1>(S, pl, Cols(cmask), cmask, A.part, vseq, blockIdx.x, r, epi, A.park);
                    if (ph == PH_HEAD) epi.head_end(pl, cmask);
                }
            }
            if (ROLE == 2) consumers_arrive(S, A.grid_ctr, prof_class(ph));
            behind = prof_class(ph);
            ++bar_no;
            // ---- what comes next
            if (ph == PH_HEAD) {
                ctl = final_head ? CTRL_TOP : CTRL_HEAD;
                e = l;
                break;
            }
            if (ph == PH_QKV) ph = PH_ATTN;
            else if (ph == PH_ATTN) ph = PH_O;
            else if (ph == PH_O) ph = PH_GU;
            else if (ph == PH_GU) ph = PH_DOWN;
            else if (ph == PH_T) ph = PH_HEAD;
            else {   // a layer is complete: an intermediate head (Section 2.1) and the early-prediction rule (Eq. 1), the next layer, or the final head
                ++l;
                if (l < L && M.exit_at[l] != 0 && ((unsigned)d.head_mask & mask) != 0) ph = M.has_T[l] ? PH_T : PH_HEAD;   // newest tokens that reached it and may exit early
                else if (l < L) ph = PH_QKV;
                else if (d.run_final) ph = PH_HEAD;   // final head for every column, then verification (Eq. 2 at temperature zero) in the control point
                else { ctl = CTRL_TOP; e = 0; break; }
            }
        }
    }
}

#if ADA_TILES == 1
// Repack on load.  Destination row `prow` of the fused q | k | v matrix: v rows are copied as they are; inside
// every q and k head the rows are reordered so that the 16-row tile t of the head holds the features
// [8 t, 8 t + 8) in its rows 0..7 and [hd/2 + 8 t, hd/2 + 8 t + 8) in its rows 8..15.  The two partners
// (i, i + hd/2) of a rotation then sit in rows r and r + 8 of one tensor-core tile, i.e. in two lanes of one warp of the
// QKV epilogue.  d must be a multiple of 8 and every pointer 16-byte aligned.
__global__ void k_repack_qkv(const __nv_bfloat16 *__restrict__ wq, const __nv_bfloat16 *__restrict__ wk, const __nv_bfloat16 *__restrict__ wv,
                             __nv_bfloat16 *__restrict__ dst, int nq, int nkv, int hd, int d) {
    const int prow = blockIdx.x, qd = nq * hd, kvd = nkv * hd;
    const __nv_bfloat16 *src;
    if (prow < qd + kvd) {
        const __nv_bfloat16 *w = prow < qd ? wq : wk;
        const int rr = prow < qd ? prow : prow - qd;
        const int h = rr / hd, pr = rr - h * hd, t = pr >> 4, r = pr & 15;
        src = w + (size_t)(h * hd + t * 8 + (r & 7) + (r >> 3) * (hd / 2)) * d;
    } else {
        src = wv + (size_t)(prow - qd - kvd) * d;
    }
    const uint4 *s4 = reinterpret_cast<const uint4 *>(src);
    uint4 *d4 = reinterpret_cast<uint4 *>(dst + (size_t)prow * d);
    for (int i = threadIdx.x; i < d / 8; i += blockDim.x) d4[i] = s4[i];
}

// Arms the prompt passes of the persistent kernel for one sequence (KV cache <- LM(x), first line of Algorithm 1).
__global__ void k_prefill_arm(Ctx c, int seq, int n_prompt) {
    DevState *st = c.st;
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    st->pf_pos = 0;
    st->pf_end = n_prompt;
    st->done[seq] = 0;
    st->n_done = 0;
    st->len[seq] = 0;
    st->base[seq] = 0;
    st->tape_n = 0;
    st->tape_i = 0;
    for (int l = 0; l < c.L; ++l) c.fill[(size_t)seq * c.L + l] = 0;
}

#endif

// Warps 0-7 consume, warp 8 produces weights and K / V blocks, warp 9 activations and queries; warps 10 and 11 only complete the producers'
// warp group, which hands registers to the consumers.  (At 168 registers a thread -- three warps on a quarter of the SM --
// the consumers kept loop variables in local memory, whose L1 lines do not survive the acquires of the grid barrier: a round trip to
// L2 for each on the critical path of a phase.  One column tile: at 200 / 104 nothing is spilled; 216 / 72 spills 24 bytes in the
// producers (8B down 18.5 -> 18.9 us, the other phases alike; 64 bytes, when it was 64, cost 0.5 to 2 % of a request).  Three tiles: the
// consumers' sums need more; 216 / 72 (which spills 200 bytes in the producers) 58 us a gate / up product of the 13B shape, 200 / 104 67; requests 183.3 ms, 208 / 88 185, 200 / 104 187.5.)
constexpr int MEGA_THREADS = CONS_THREADS + 128;
constexpr int REGS_CONSUME = TILES == 1 ? 200 : 216, REGS_PRODUCE = TILES == 1 ? 104 : 72;
constexpr int MEGA_REGS = CONS_THREADS * REGS_CONSUME + 128 * REGS_PRODUCE;   // the block must have been launched with as many

template <int HD>
__global__ void __launch_bounds__(MEGA_THREADS, 1) k_decode_persistent(const __grid_constant__ MegaArgs A) {
    extern __shared__ unsigned char smem_raw[];
    Smem *sm = smem_base(smem_raw);
    smem_init(sm);
    if (threadIdx.x >= 32 && threadIdx.x < 32 + PH_PRODUCTS) {
        const int ph = threadIdx.x - 32;
        sm->plan[ph] = make_plan(phase_gemm(A, ph, gridDim.x), blockIdx.x, gridDim.x);
    }
    const int warp = threadIdx.x >> 5;
    if (TILES == 1 && warp == CONS_WARPS + 2) {   // tensor memory for parked weight stages
        park_alloc(sm);
        tc_fence_before();
    }
    __syncthreads();
    if (TILES == 1) tc_fence_after();
    Shared S{sm, A.err, A.trace, 0, A.wait_ns};
    if (warp < CONS_WARPS) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REGS_CONSUME));
        run<2, HD>(A, S);
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_PRODUCE));
        if (warp == CONS_WARPS) run<0, HD>(A, S);
        else if (warp == CONS_WARPS + 1) run<1, HD>(A, S);
    }
    if (TILES == 1) tc_fence_before();
    settle_on_abort(S);   // (meets the whole block)
    if (TILES == 1 && warp == CONS_WARPS + 2) {
        __syncwarp();
        tc_fence_after();
        park_free(sm);
    }
}

}  // namespace ADA_MG
}  // namespace ada
