// Student + teacher forward of the self-distillation objective (App. D.3 "Training Objectives"): the
// student attends under the eviction mask, the teacher sees the full causal context; same model, same
// tokens, same q, k, v.
//
// The causal key set of a query splits into the keys the student still sees and the keys that were
// evicted before the query.  Attention over a union of disjoint key sets is the merge of the attention
// over each: with lse = log(e^lse_a + e^lse_b),  out = e^(lse_a - lse) out_a + e^(lse_b - lse) out_b.
// So the teacher costs one more forward over the EVICTED keys only (metadata for key slots that become
// visible at their eviction step and stay, kvs_mask_meta_evicted), which reads the student's rows and merges
// them with its own as it writes them (MERGE in kvs_fwd.cu): every (query, key) pair of a FULL or EMPTY tile
// is scored once for both streams, only tiles that are PARTIAL for the student are visited by both passes.
// Both passes are the forward kernel (two query heads of a group share every K/V tile).  A fused kernel with both accumulators of one head in tensor
// memory was measured first: 512 columns hold S twice and the two outputs of ONE head, so a CTA cannot
// keep two query tiles in flight, its eight softmax warps move through load / maximum / exponentials /
// store in lockstep and the special-function unit idles half the time; it was slower than two plain
// forwards and is not kept.
#include "kvs_common.cuh"

using namespace kvs;

extern "C" int kvs_attn_fwd_dual(const void* q, const void* k, const void* v, const void* meta_student, const void* meta_evicted,
                                 int batch, int total_tokens, int max_seqlen, int Hq, int Hkv, int head_dim, float softmax_scale,
                                 void* out_student, float* lse_student, void* out_teacher, float* lse_teacher, kvs_stream_t stream) {
    if (!meta_student || !meta_evicted) return KVS_ERR_INVALID_ARG;
    if (out_student == out_teacher || lse_student == lse_teacher) return KVS_ERR_INVALID_ARG;
    int rc = kvs_attn_fwd(q, k, v, meta_student, batch, total_tokens, max_seqlen, Hq, Hkv, head_dim, softmax_scale, out_student,
                          lse_student, stream);
    if (rc != KVS_OK) return rc;
    // the part of the teacher's context that the student no longer sees, merged with the student's on its way out
    return attn_fwd_merged(q, k, v, meta_evicted, batch, total_tokens, max_seqlen, Hq, Hkv, head_dim, softmax_scale, out_student, lse_student,
                           out_teacher, lse_teacher, stream);
}
