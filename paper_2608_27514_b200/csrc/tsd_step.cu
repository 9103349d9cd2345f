// The whole verification step in one call (Section 3.3): verify attention, vocabulary pass, acceptance.
//
// The attention reads none of what the vocabulary pass writes, so the two may run side by side: the vocabulary
// pass lets its successor start once all its blocks run, and the attention takes the SMs as the first rows are finished
// instead of waiting for the last one; the acceptance waits for both.  Done where attention has fewer work items
// than the GPU has SMs (256 draft rows, 32 heads, 768 cached keys, 64 items: the step takes 32.9 us; attention first and the
// vocabulary pass beside it 33.5; one after the other 40.8).  With more items than SMs neither leaves SMs
// free before its end, and what starts early there upsets the balance: 1024 rows, 256 items, 95.2 us side by side
// and 89.8 us one after the other.
//
// The acceptance is brought up while the last rows are finished and asks for the trees ahead of time.
#include "tsd_common.cuh"

extern "C" int tsd_verify_step(const tsd_step_args* x, tsd_stream_t stream) {
  if (!x) return TSD_ERR_INVALID_ARG;
  const tsd_layout* L = x->layout;
  int rc = tsd::check_attention_args(L, x->mask, x->q, x->q_stride[0], x->q_stride[1], x->q_stride[2], x->k_cache,
                                     x->v_cache, x->c_stride[0], x->c_stride[1], x->c_stride[2], x->k_draft, x->v_draft,
                                     x->d_stride[0], x->d_stride[1], x->d_stride[2], x->out, x->o_stride[0],
                                     x->o_stride[1], x->o_stride[2], x->sm_scale, x->attn_workspace);
  if (rc != TSD_OK) return rc;
  const int64_t tiles = (int64_t)L->batch * L->n_q_heads * tsd::mask_dims(*L).n_qt;
  const bool beside = tiles < 148;
  const tsd::AttnArgs a = {*L, static_cast<const int32_t*>(x->mask), x->q, x->k_cache, x->v_cache, x->k_draft, x->v_draft,
                           x->out, x->attn_lse, x->q_stride[0], x->q_stride[1], x->q_stride[2], x->c_stride[0],
                           x->c_stride[1], x->c_stride[2], x->d_stride[0], x->d_stride[1], x->d_stride[2], x->o_stride[0],
                           x->o_stride[1], x->o_stride[2], x->sm_scale, x->attn_workspace, x->attn_workspace_bytes,
                           x->status, stream, beside};
  const tsd::TopkArgs t = {x->logits, x->logits_dtype, x->n_rows, x->vocab, x->row_stride, x->k, x->conf, x->topk_idx,
                           x->topk_prob, x->lse, x->topk_workspace, x->topk_workspace_bytes, stream,
                           beside ? tsd::kNextAtOnce : tsd::kNextAtTail};
  const tsd::AcceptArgs c = {L->batch, L->n_branches, L->n_branches, L->rows_per_branch, x->parent, x->state, x->mask_id,
                             x->conf, x->topk_idx, x->k, x->tau, x->rule, x->search, x->edge_valid, x->prefix_len,
                             x->accepted_node, x->accepted_len, x->n_new_tokens, x->unmask_flag, x->unmask_tok, x->status,
                             stream};
  if ((rc = tsd::check_topk(t)) != TSD_OK || (rc = tsd::check_accept_exact(c)) != TSD_OK) return rc;
  if (beside) {
    if ((rc = tsd::launch_topk(t)) != TSD_OK) return rc;
    if ((rc = tsd::launch_attention(a, x->flags)) != TSD_OK) return rc;
  } else {
    if ((rc = tsd::launch_attention(a, x->flags)) != TSD_OK) return rc;
    if ((rc = tsd::launch_topk(t)) != TSD_OK) return rc;
  }
  return tsd::launch_accept_exact(c);
}
