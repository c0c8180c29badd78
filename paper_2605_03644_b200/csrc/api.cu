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

namespace {

// Whether [a, a + na) and [b, b + nb) share a byte.
bool meet(const void* a, size_t na, const void* b, size_t nb) {
  const uintptr_t x = reinterpret_cast<uintptr_t>(a), y = reinterpret_cast<uintptr_t>(b);
  return a != nullptr && b != nullptr && x < y + nb && y < x + na;
}

// Logits up to this size run beside the attention.  Two launches and their drain are 5 us: passes over eight short shots 33.5 -> 28.2 us,
// one layer of one query with four or seven probes 130.3 -> 124.7 and 93.2 -> 88.3 (0.3 to 2 MB of logits), 28 probes of four
// queries (7 MB) 252 -> 250; from 56 probes (14 MB, 0.5 ms) on the difference is below the runs' own, and reading them (57 MB, 13 us)
// is bound by bandwidth on either side.
constexpr size_t kBesideBytes = 16u << 20;

// Whether the entropy of a pass may run beside its last attention call instead of behind it: a valid call whose logits, states
// and results share no memory with what that attention call still reads (the pool among it, where it takes tiles from there) or
// writes.  Calls in turn may share it, one workspace for every step for instance.
bool entropy_beside(const adapshot_pass_t* p, AdsEntropyJob* job) {
  if (p->model == nullptr || p->B <= 0 || p->P <= 0 || p->Tq <= 0 || p->V <= 0) return false;
  if (ads_entropy_job(p->logits, p->logits_dtype, p->B * p->P, p->V, p->logits_stride, p->H, p->tau, p->P, p->first_ok,
                      p->ws_entropy, p->ws_entropy_bytes, job) != ADAPSHOT_OK)
    return false;
  const size_t rows = (size_t)p->B * p->P, row_q = (size_t)p->model->n_q_heads * p->model->head_dim * 2;
  const size_t logit_bytes = ((rows - 1) * (size_t)p->logits_stride + p->V) * (job->f32 ? 4 : 2);
  if (logit_bytes > kBesideBytes) return false;
  const struct { const void* at; size_t n; } mine[4] = {
      {p->logits, logit_bytes},
      {p->ws_entropy, (size_t)job->blocks * 3 * sizeof(float)},
      {p->H, rows * sizeof(float)},
      {p->first_ok, (size_t)p->B * sizeof(int32_t)}};
  const int last = p->n_chunks - 1;
  const int nl = p->layer_end[last] - (last > 0 ? p->layer_end[last - 1] : 0);
  if (nl <= 0) return false;
  const size_t tok = rows * nl * (size_t)p->Tq, row_kv = (size_t)p->model->n_kv_heads * p->model->head_dim * 2;
  const size_t cache = (size_t)p->B * nl * (size_t)p->ctx_cap * row_kv;
  const size_t pool_bytes = (size_t)p->model->n_layers * (size_t)p->pool->pool_tokens * row_kv;
  for (const auto& m : mine) {
    if (meet(m.at, m.n, p->ws_attn, p->ws_attn_bytes) || meet(m.at, m.n, p->out[last], tok * row_q) ||
        meet(m.at, m.n, p->q[last], tok * row_q) || meet(m.at, m.n, p->kq[last], tok * row_kv) ||
        meet(m.at, m.n, p->vq[last], tok * row_kv) || meet(m.at, m.n, p->sel_idx, (size_t)p->B * p->k * 4) ||
        meet(m.at, m.n, p->ctx_off, (size_t)p->B * (p->k + 1) * 8) || meet(m.at, m.n, p->status, 4))
      return false;
    if (p->variant != ADAPSHOT_PASS_FUSED && meet(m.at, m.n, p->k_ctx, cache)) return false;
    if (p->variant == ADAPSHOT_PASS_FULL && meet(m.at, m.n, p->v_ctx, cache)) return false;
    if (p->variant != ADAPSHOT_PASS_FULL &&
        (meet(m.at, m.n, p->pool->v, pool_bytes) || meet(m.at, m.n, p->pool->shot_off, ((size_t)p->pool->n_shots + 1) * 8)))
      return false;
    if (p->variant == ADAPSHOT_PASS_FUSED && meet(m.at, m.n, p->pool->k, pool_bytes)) return false;
  }
  return true;
}

}  // namespace

extern "C" int adapshot_reuse_pass(const adapshot_pass_t* p, void* stream) {
  if (p == nullptr || p->layer_end == nullptr || p->q == nullptr || p->kq == nullptr || p->vq == nullptr ||
      p->out == nullptr || p->n_chunks <= 0 || p->variant < ADAPSHOT_PASS_FULL || p->variant > ADAPSHOT_PASS_FUSED)
    return ADAPSHOT_EINVAL;
  int rc = adapshot_select(p->pool, p->q_emb, p->B, p->k, p->sel_idx, p->sel_score, p->ws_select, p->ws_select_bytes,
                           p->status, stream);
  if (rc == ADAPSHOT_OK && p->variant == ADAPSHOT_PASS_FUSED)
    rc = adapshot_assemble_kv(p->model, p->pool, p->sel_idx, p->B, p->k, 0, 1, nullptr, nullptr, p->ctx_cap, p->ctx_off, 0,
                              p->status, stream);
  AdsPass pass = {};
  double theta[64];
  if (p->model != nullptr && (p->model->head_dim == 64 || p->model->head_dim == 128)) {      // (anything else is refused below)
    ads_rope_theta(p->model->rope_base, p->model->head_dim, theta);
    pass.theta = theta;
  }
  // The logits are an input of the call: where nothing forbids it, their entropy runs in blocks of the last attention call's small
  // kernels (the states beside the preparation, the rule beside the merge) instead of two launches behind it.
  AdsEntropyJob job;
  const bool beside = rc == ADAPSHOT_OK && entropy_beside(p, &job);
  int lb = 0;
  for (int i = 0; rc == ADAPSHOT_OK && i < p->n_chunks; ++i) {
    const int le = p->layer_end[i];
    pass.ent = beside && i + 1 == p->n_chunks ? &job : nullptr;
    if (p->variant != ADAPSHOT_PASS_FUSED) {
      const uint32_t flags = (i > 0 ? ADAPSHOT_ASSEMBLE_KEEP_PLAN : 0u) |
                             (p->variant == ADAPSHOT_PASS_VPOOL ? ADAPSHOT_ASSEMBLE_K_ONLY : 0u);
      rc = ads_assemble_kv(p->model, p->pool, p->sel_idx, p->B, p->k, 0, lb, le, p->k_ctx, p->v_ctx, p->ctx_cap,
                           p->ctx_off, flags, p->status, stream, &pass);
      if (rc != ADAPSHOT_OK) break;
    }
    if (p->variant == ADAPSHOT_PASS_FULL)
      rc = ads_query_attn(p->model, p->k_ctx, p->v_ctx, p->ctx_cap, p->ctx_off, p->B, p->k, p->probe_nshots, p->P,
                          p->q[i], p->kq[i], p->vq[i], p->Tq, lb, le, p->out[i], nullptr, 0, p->ws_attn,
                          p->ws_attn_bytes, p->status, stream, &pass);
    else if (p->variant == ADAPSHOT_PASS_VPOOL)
      rc = ads_query_attn_vpool(p->model, p->pool, p->sel_idx, p->k_ctx, p->ctx_cap, p->ctx_off, p->B, p->k,
                                p->probe_nshots, p->P, p->q[i], p->kq[i], p->vq[i], p->Tq, lb, le, p->out[i], nullptr,
                                0, p->ws_attn, p->ws_attn_bytes, p->status, stream, &pass);
    else
      rc = ads_query_attn_fused(p->model, p->pool, p->sel_idx, p->ctx_off, p->ctx_cap, p->B, p->k, p->probe_nshots,
                                p->P, p->q[i], p->kq[i], p->vq[i], p->Tq, lb, le, p->out[i], nullptr, 0, p->ws_attn,
                                p->ws_attn_bytes, p->status, stream, &pass);
    lb = le;
  }
  if (rc != ADAPSHOT_OK || beside) return rc;
  return adapshot_entropy(p->logits, p->logits_dtype, p->B * p->P, p->V, p->logits_stride, p->H, p->tau, p->P,
                          p->first_ok, p->ws_entropy, p->ws_entropy_bytes, p->status, stream);
}
