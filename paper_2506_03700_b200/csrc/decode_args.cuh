// Arguments of the persistent decode kernels, whatever the number of their token columns.
#pragma once

#include <cuda.h>

#include "kernels.cuh"

namespace ada {

// Optional event trace (test hook): records (globaltimer ns, code) pairs while `tr_on` is set.
// Every CTA writes its own region of the buffer, so that recording costs a shared-memory counter
// and one store.
struct Trace {
    unsigned long long *buf;   // [grid][cap][2], or nullptr
    unsigned *count;           // [grid]
    unsigned cap;              // events per CTA
};

constexpr int ATT_PAGE = 64;   // cache positions per attention sub-block (= KV page size on this path)
constexpr int ERR_BAD_STATE = 3;
// Random numbers per sequence position: [0] draw at the last layer, [1] acceptance test of Eq. 2, [2] resampling after a
// rejection, [3 + e] draw at the e-th exit layer of the call.
constexpr int SAMPLE_NU = 8;
constexpr int DRAFT_SLOTS = 8;   // tokens in flight per sequence whose drafts are kept (by position modulo this)

// What the phases need to know of the model.  It travels as a kernel argument: the constant bank answers at once, where a
// pointer read from global memory was a round trip to L2 in front of the loads that depend on it (the L1 copy does not
// survive the acquire of a grid barrier).
struct MegaModel {
    // per layer: wqkv (the fused q | k | v matrix with the rows of every q and k head reordered for the rotation, see the QKV
    // phase), wo, wgu (gate stacked over up, or gate alone where gu_two is set), wup, wdown; then the LM head; then T per 1-based layer
    const CUtensorMap *maps;
    const __nv_bfloat16 *tok_embed, *final_norm;
    const __nv_bfloat16 *attn_norm[ADA_MAX_LAYERS], *ffn_norm[ADA_MAX_LAYERS];
    float head_scale[ADA_MAX_LAYERS + 1];        // by 1-based layer
    unsigned char exit_at[ADA_MAX_LAYERS + 1];   // 1 + the index of 1-based layer e among the call's exit layers if the call consults its head, else 0
    unsigned char has_T[ADA_MAX_LAYERS + 1];     // that head has a transformation of its own
    unsigned char gu_two[ADA_MAX_LAYERS];        // gate and up are separate tensors
};
enum { MAPS_PER_LAYER = 5 };

struct MegaArgs {
    Ctx c;
    MegaModel m;
    __nv_bfloat16 *XA, *XB, *XO, *XH, *XF, *XT;   // GEMM inputs in fragment layout (see stream.cuh)
    float *ssq_a, *ssq_b;      // [d/16][columns] partial sums of squares of the residual (per 16-feature tile, per column)
    uint32_t *qfrag;           // [sequence][nkv][2][hd/16][32][8]: rotated, scaled queries as tensor-core A fragments (bf16 high parts, then low parts)
    float *head_part;          // [grid][columns][4]
    const double *rope_freq;   // [hd/2]: base^(-2i/hd), computed once on the host
    unsigned long long *part;  // [grid][8 k-splits][column tiles][256]: tagged partial sums of weight tiles split between two CTAs (null: none)
    unsigned long long *attn_tag;   // [columns][nq][c.n_chunks][hd + 2]: chunk partials as tagged words (see attn_consume), for the chunks that
                               // the call can reach; zeroed before each launch
    unsigned *grid_ctr;
    void *pub;                 // Pub[2] of the kernel launched
    int *err;
    int step_budget;           // steps this launch may start
    int seq0, nseq;            // the launch decodes sequences seq0 .. seq0 + nseq - 1 of the session together, nseq slots <= the kernel's columns (slots = max_early + 1):
                               // slot j of sequence k of them is token column j nseq + k (neighbouring columns are then of equal age, and a
                               // pass that carries the newest tokens only fetches few column pairs); they share every weight stream
    unsigned long long wait_ns;   // a single device-side wait gives up after this long
    int park;                  // weight stages that a warp parks in tensor memory at a time, at most
    int store_logits;
    // Sampled decoding (Eq. 1 with a drawn token, Eq. 2 with its acceptance test and the resampling): off = greedy
    int sampling;
    float inv_temp;            // 1 / temperature: every head's logits are multiplied by it
    const float *uniforms;     // [batch][max_seq][SAMPLE_NU]: the random numbers of the token at each sequence position
    float *q_stage;            // [batch][8][vocab]: logits of the intermediate head that drew the token after position p, slot p % 8
    float4 *qinfo;             // [batch][8]: (max logit, sum of exp, probability of the drawn token) of that head
    Trace trace;               // test hook: event trace of the steps [trace_step0, trace_step1) of this launch
    int trace_step0, trace_step1;
};

}  // namespace ada
