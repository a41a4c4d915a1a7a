// The entry points with their arguments in one struct (ism.h, ism_call_*): a
// foreign call with some twenty arguments costs a Python binding more than the
// launches behind it: a prefill_append call took 82 us of host time, 8.6 of
// them in the library.
#include "ism_internal.cuh"

namespace {

template <class Call>
ism_attn_shape_t shape_of(const Call& c) {
  return ism_attn_shape_t{c.num_heads_q, c.num_heads_kv, c.head_dim, c.dtype, (float)c.softmax_scale};
}

template <class Call>
const ism_rope_t* rope_of(const Call& c) {
  return c.form & ISM_CALL_ROPE ? &c.rope : nullptr;
}

ism_status_t null_call() {
  ism::set_error("call is NULL");
  return ISM_ERR_INVALID_ARG;
}

}  // namespace

extern "C" {

ism_status_t ism_call_fwd(const ism_pass_call_t* call) {
  if (!call) return null_call();
  const ism_pass_call_t& c = *call;
  const ism_attn_shape_t sh = shape_of(c);
  const ism_rope_t* rope = rope_of(c);
  if (c.form & ISM_CALL_E4M3)
    return ism_attn_fwd_e4m3(&c.segs, &sh, c.q, c.k, c.v, (float)c.q_descale, (float)c.k_descale, (float)c.v_descale,
                             c.o, c.lse, c.workspace, c.workspace_bytes, c.stream);
  if (c.plan)
    return rope ? ism_attn_fwd_rope_planned(&c.segs, &sh, c.plan, &c.plan_info, c.q, c.k, c.v, rope, c.q_rot, c.k_rot,
                                            c.o, c.lse, c.stream)
                : ism_attn_fwd_planned(&c.segs, &sh, c.plan, &c.plan_info, c.q, c.k, c.v, c.o, c.lse, c.stream);
  return rope ? ism_attn_fwd_rope(&c.segs, &sh, c.q, c.k, c.v, rope, c.q_rot, c.k_rot, c.o, c.lse, c.workspace,
                                  c.workspace_bytes, c.stream)
              : ism_attn_fwd(&c.segs, &sh, c.q, c.k, c.v, c.o, c.lse, c.workspace, c.workspace_bytes, c.stream);
}

ism_status_t ism_call_bwd(const ism_pass_call_t* call) {
  if (!call) return null_call();
  const ism_pass_call_t& c = *call;
  const ism_attn_shape_t sh = shape_of(c);
  const ism_rope_t* rope = rope_of(c);
  if (c.plan)
    return rope ? ism_attn_bwd_rope_planned(&c.segs, &sh, c.plan, &c.plan_info, c.q, c.k, c.v, c.o, c.lse, c.dout,
                                            rope, c.dq, c.dk, c.dv, c.workspace, c.workspace_bytes, c.stream)
                : ism_attn_bwd_planned(&c.segs, &sh, c.plan, &c.plan_info, c.q, c.k, c.v, c.o, c.lse, c.dout, c.dq,
                                       c.dk, c.dv, c.workspace, c.workspace_bytes, c.stream);
  return rope ? ism_attn_bwd_rope(&c.segs, &sh, c.q, c.k, c.v, c.o, c.lse, c.dout, rope, c.dq, c.dk, c.dv,
                                  c.workspace, c.workspace_bytes, c.stream)
              : ism_attn_bwd(&c.segs, &sh, c.q, c.k, c.v, c.o, c.lse, c.dout, c.dq, c.dk, c.dv, c.workspace,
                             c.workspace_bytes, c.stream);
}

ism_status_t ism_call_pass_sizes(const ism_pass_call_t* call, int32_t backward, size_t* bytes) {
  if (!call) return null_call();
  const ism_attn_shape_t sh = shape_of(*call);
  if (!backward) return ism_attn_fwd_workspace_size(&call->segs, &sh, bytes);
  const ism_status_t r = ism_attn_bwd_workspace_size(&call->segs, &sh, bytes);
  return r != ISM_OK ? r : ism_attn_bwd_workspace_size_min(&call->segs, &sh, bytes ? bytes + 1 : nullptr);
}

ism_status_t ism_call_append(const ism_append_call_t* call) {
  if (!call) return null_call();
  const ism_append_call_t& c = *call;
  const ism_attn_shape_t sh = shape_of(c);
  const ism_rope_t* rope = rope_of(c);
  if (c.form & ISM_CALL_PAGED) {
    if (rope)
      return ism_attn_prefill_append_paged_rope(&sh, c.batch, c.q_new, c.k_new, c.v_new, c.l_new, c.new_seg_end_host,
                                                c.new_seg_type_host, c.n_new_segs, c.k_cache, c.v_cache, c.num_pages,
                                                c.page_size, c.block_table, c.block_table_host, c.max_pages,
                                                c.cache_len, c.cache_len_host, rope, c.o_new, c.lse_new, c.workspace,
                                                c.workspace_bytes, c.stream);
    return ism_attn_prefill_append_paged(&sh, c.batch, c.q_new, c.k_new, c.v_new, c.l_new, c.new_seg_end_host,
                                         c.new_seg_type_host, c.n_new_segs, c.k_cache, c.v_cache, c.num_pages,
                                         c.page_size, c.block_table, c.block_table_host, c.max_pages, c.cache_len,
                                         c.cache_len_host, c.o_new, c.lse_new, c.workspace, c.workspace_bytes,
                                         c.stream);
  }
  const float dq = (float)c.q_descale, dk = (float)c.k_descale, dv = (float)c.v_descale;
  if (c.form & ISM_CALL_E4M3) {
    if (rope)
      return ism_attn_prefill_append_e4m3_rope(&sh, c.batch, c.q_new, c.k_new, c.v_new, c.l_new, c.new_seg_end_host,
                                               c.new_seg_type_host, c.n_new_segs, c.k_cache, c.v_cache,
                                               c.cache_capacity, c.cache_len, c.cache_len_host, dq, dk, dv, rope,
                                               c.o_new, c.lse_new, c.workspace, c.workspace_bytes, c.stream);
    return ism_attn_prefill_append_e4m3(&sh, c.batch, c.q_new, c.k_new, c.v_new, c.l_new, c.new_seg_end_host,
                                        c.new_seg_type_host, c.n_new_segs, c.k_cache, c.v_cache, c.cache_capacity,
                                        c.cache_len, c.cache_len_host, dq, dk, dv, c.o_new, c.lse_new, c.workspace,
                                        c.workspace_bytes, c.stream);
  }
  if (rope)
    return ism_attn_prefill_append_rope(&sh, c.batch, c.q_new, c.k_new, c.v_new, c.l_new, c.new_seg_end_host,
                                        c.new_seg_type_host, c.n_new_segs, c.k_cache, c.v_cache, c.cache_capacity,
                                        c.cache_len, c.cache_len_host, rope, c.o_new, c.lse_new, c.workspace,
                                        c.workspace_bytes, c.stream);
  return ism_attn_prefill_append(&sh, c.batch, c.q_new, c.k_new, c.v_new, c.l_new, c.new_seg_end_host,
                                 c.new_seg_type_host, c.n_new_segs, c.k_cache, c.v_cache, c.cache_capacity,
                                 c.cache_len, c.cache_len_host, c.o_new, c.lse_new, c.workspace, c.workspace_bytes,
                                 c.stream);
}

}  // extern "C"
