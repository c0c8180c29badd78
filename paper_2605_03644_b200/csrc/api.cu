// Version and error strings of the adapshot C ABI, and the calls of a whole pass in one.
#include "common.cuh"

extern "C" const char* adapshot_strerror(int code) {
  switch (code) {
    case ADAPSHOT_OK: return "ok";
    case ADAPSHOT_EINVAL: return "invalid argument (null pointer, non-positive size or unsupported flag)";
    case ADAPSHOT_ESHAPE: return "unsupported shape (head_dim, head ratio, probe list or k out of range)";
    case ADAPSHOT_EALIGN: return "pointer or stride not 16-byte aligned";
    case ADAPSHOT_ECAPACITY: return "capacity too small (ctx_cap, workspace or static scratch)";
    case ADAPSHOT_EUNSUPPORTED: return "dtype or mode not supported by this build";
    case ADAPSHOT_ECUDA: return "a CUDA runtime or driver call failed";
    case ADAPSHOT_EINDEX: return "shot id outside the pool";
    case ADAPSHOT_ETIMEOUT: return "a device pipeline wait exceeded its limit";
    default: return "unknown adapshot error code";
  }
}

extern "C" int adapshot_version(void) { return ADAPSHOT_VERSION_NUMBER; }

extern "C" int adapshot_reuse_pass(const adapshot_pass_t* p, void* stream) {
  if (p == nullptr || p->layer_end == nullptr || p->q == nullptr || p->kq == nullptr || p->vq == nullptr ||
      p->out == nullptr || p->n_chunks <= 0 || p->variant < ADAPSHOT_PASS_FULL || p->variant > ADAPSHOT_PASS_FUSED)
    return ADAPSHOT_EINVAL;
  int rc = adapshot_select(p->pool, p->q_emb, p->B, p->k, p->sel_idx, p->sel_score, p->ws_select, p->ws_select_bytes,
                           p->status, stream);
  if (rc == ADAPSHOT_OK && p->variant == ADAPSHOT_PASS_FUSED)
    rc = adapshot_assemble_kv(p->model, p->pool, p->sel_idx, p->B, p->k, 0, 1, nullptr, nullptr, p->ctx_cap, p->ctx_off, 0,
                              p->status, stream);
  int lb = 0;
  for (int i = 0; rc == ADAPSHOT_OK && i < p->n_chunks; ++i) {
    const int le = p->layer_end[i];
    if (p->variant != ADAPSHOT_PASS_FUSED) {
      const uint32_t flags = (i > 0 ? ADAPSHOT_ASSEMBLE_KEEP_PLAN : 0u) |
                             (p->variant == ADAPSHOT_PASS_VPOOL ? ADAPSHOT_ASSEMBLE_K_ONLY : 0u);
      rc = adapshot_assemble_kv(p->model, p->pool, p->sel_idx, p->B, p->k, lb, le, p->k_ctx, p->v_ctx, p->ctx_cap,
                                p->ctx_off, flags, p->status, stream);
      if (rc != ADAPSHOT_OK) break;
    }
    if (p->variant == ADAPSHOT_PASS_FULL)
      rc = adapshot_query_attn(p->model, p->k_ctx, p->v_ctx, p->ctx_cap, p->ctx_off, p->B, p->k, p->probe_nshots, p->P,
                               p->q[i], p->kq[i], p->vq[i], p->Tq, lb, le, p->out[i], nullptr, 0, p->ws_attn,
                               p->ws_attn_bytes, p->status, stream);
    else if (p->variant == ADAPSHOT_PASS_VPOOL)
      rc = adapshot_query_attn_vpool(p->model, p->pool, p->sel_idx, p->k_ctx, p->ctx_cap, p->ctx_off, p->B, p->k,
                                     p->probe_nshots, p->P, p->q[i], p->kq[i], p->vq[i], p->Tq, lb, le, p->out[i],
                                     nullptr, 0, p->ws_attn, p->ws_attn_bytes, p->status, stream);
    else
      rc = adapshot_query_attn_fused(p->model, p->pool, p->sel_idx, p->ctx_off, p->ctx_cap, p->B, p->k, p->probe_nshots,
                                     p->P, p->q[i], p->kq[i], p->vq[i], p->Tq, lb, le, p->out[i], nullptr, 0,
                                     p->ws_attn, p->ws_attn_bytes, p->status, stream);
    lb = le;
  }
  if (rc != ADAPSHOT_OK) return rc;
  return adapshot_entropy(p->logits, p->logits_dtype, p->B * p->P, p->V, p->logits_stride, p->H, p->tau, p->P,
                          p->first_ok, p->ws_entropy, p->ws_entropy_bytes, p->status, stream);
}
