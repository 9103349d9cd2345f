// The whole verification step in one call (Section 3.3): verify attention, vocabulary pass, acceptance.
//
// The attention reads none of what the vocabulary pass writes, so the two may run side by side; the acceptance waits
// for both.  Done where attention has fewer work items than the GPU has SMs, in one of two ways:
//  * Attention first, the vocabulary pass beside it once all blocks of the attention run, where all blocks of the
//    pass fit on the SMs that attention leaves free (two of 512 threads each), so that none of them is late: 128 rows of 126464
//    and 32 items 23.5 -> 20.9 us, 128 of 32000 and 16 items of 81 key tiles 27.5 -> 22.5, 160 of 126464 and 28 items 26.9
//    -> 23.5 (all against the second way).  64 rows of 152064 in 4 segments each beside 112 blocks would take 29.7 instead of
//    27.1.  The fp32 attention shares its SMs: where its blocks are no more than the SMs and the logits are below 4 MB (128 rows,
//    4 heads, 256 cached keys, in a graph; vocabulary first and attention first: of 2048 13.1 and 11.7 us, of 4096 13.3 and 12.2, of
//    8192 (4.2 MB) 13.5 and 13.7, of 12288 14.5 and 14.8, of 20480 15.4 and 15.7, of 32768 16.3 and 16.7).
//  * The vocabulary pass first: the attention takes the SMs as the first rows are finished instead of waiting for the
//    last one (256 draft rows, 32 heads, 768 cached keys, 64 items: the step takes 32.5 us; attention first 33.9; one
//    after the other 40.8).
// With more items than SMs the two run one after the other.  Some SMs idle in the attention's last round there too (256 items: 108
// blocks take two and 40 take one), but side by side was slower: 1024 rows, 256 items, 95.2 us and 89.8 one after
// the other; which of the kernels loses the time has not been looked into.
//
// The acceptance is brought up while the last rows are finished and asks for the trees ahead of time.
#include "tsd_common.cuh"

static bool attention_first(const tsd_step_args& x, const tsd::AttnArgs& a, const tsd::TopkArgs& t) {
  const tsd_layout& L = a.L;
  if (!(x.flags & TSD_ATTN_FORCE_SIMT) && tsd::attention_tc_supported(a))
    return tsd::topk_threads(t) <= 1024 * (tsd::kPlanSms - tsd::attention_tc_blocks(L));
  const int64_t attn_rows = (int64_t)L.batch * L.n_q_heads * L.n_branches * L.rows_per_branch;  // 8 per block at most
  const int64_t logit_bytes = x.n_rows * x.vocab * (x.logits_dtype == TSD_F32 ? 4 : 2);
  return attn_rows <= 8 * tsd::kPlanSms && tsd::topk_threads(t) <= 1024 * tsd::kPlanSms && logit_bytes < (4 << 20);
}

extern "C" int tsd_verify_step(const tsd_step_args* x, tsd_stream_t stream) {
  if (!x) return TSD_ERR_INVALID_ARG;
  const tsd_layout* L = x->layout;
  int rc = tsd::check_attention_args(L, x->mask, x->q, x->q_stride[0], x->q_stride[1], x->q_stride[2], x->k_cache,
                                     x->v_cache, x->c_stride[0], x->c_stride[1], x->c_stride[2], x->k_draft, x->v_draft,
                                     x->d_stride[0], x->d_stride[1], x->d_stride[2], x->out, x->o_stride[0],
                                     x->o_stride[1], x->o_stride[2], x->sm_scale, x->attn_workspace);
  if (rc != TSD_OK) return rc;
  tsd::AttnArgs a = {*L, static_cast<const int32_t*>(x->mask), x->q, x->k_cache, x->v_cache, x->k_draft, x->v_draft,
                           x->out, x->attn_lse, x->q_stride[0], x->q_stride[1], x->q_stride[2], x->c_stride[0],
                           x->c_stride[1], x->c_stride[2], x->d_stride[0], x->d_stride[1], x->d_stride[2], x->o_stride[0],
                           x->o_stride[1], x->o_stride[2], x->sm_scale, x->attn_workspace, x->attn_workspace_bytes,
                           x->status, stream, false, false};
  tsd::TopkArgs t = {x->logits, x->logits_dtype, x->n_rows, x->vocab, x->row_stride, x->k, x->conf, x->topk_idx,
                           x->topk_prob, x->lse, x->topk_workspace, x->topk_workspace_bytes, stream,
                           tsd::kNextAtTail, false};
  const tsd::AcceptArgs c = {L->batch, L->n_branches, L->n_branches, L->rows_per_branch, x->parent, x->state, x->mask_id,
                             x->conf, x->topk_idx, x->k, x->tau, x->rule, x->search, x->edge_valid, x->prefix_len,
                             x->accepted_node, x->accepted_len, x->n_new_tokens, x->unmask_flag, x->unmask_tok, x->status,
                             stream};
  if ((rc = tsd::check_topk(t)) != TSD_OK || (rc = tsd::check_accept_exact(c)) != TSD_OK) return rc;
  if (x->n_rows > (int64_t)L->batch * L->n_branches * L->rows_per_branch) return TSD_ERR_INVALID_ARG;  // conf, topk_* hold one row each
  // without a vocabulary pass in between there is nothing that the attention might run beside but what came before the step
  const bool beside = x->n_rows > 0 && (int64_t)L->batch * L->n_q_heads * tsd::mask_dims(*L).n_qt < tsd::kPlanSms;
  if (beside && attention_first(*x, a, t)) {
    a.next_at_once = t.concurrent = true;
  } else if (beside) {
    t.launch_next = tsd::kNextAtOnce;
    a.concurrent = true;
    if ((rc = tsd::launch_topk(t)) != TSD_OK) return rc;
    if ((rc = tsd::launch_attention(a, x->flags)) != TSD_OK) return rc;
    return tsd::launch_accept_exact(c);
  }
  if ((rc = tsd::launch_attention(a, x->flags)) != TSD_OK) return rc;
  if ((rc = tsd::launch_topk(t)) != TSD_OK) return rc;
  return tsd::launch_accept_exact(c);
}
