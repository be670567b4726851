// efim_append_prefill_attn: causal attention of the new `inc` tokens over the
// cached `<P>prefix<S>suffix<M>` keys and over each other (EFIM Sec. 1, Sec. 2.2).
// Host side: validates, plans the work list from the host length mirrors, copies
// it into the workspace and launches the tensor-core kernel (prefill_tc.cu).
#include <cstring>
#include <memory>
#include "kv_append.cuh"
#include "prefill_tc.cuh"
#include "mbar.cuh"

extern "C" size_t efim_prefill_workspace_bytes(const efim_cache_desc* cache, const efim_batch_desc* batch) {
  if (efim::check_cache(cache) != EFIM_OK || efim::check_batch(cache, batch, true) != EFIM_OK) return 0;
  if (batch->batch == 0 || batch->total_new_tokens == 0) return 0;
  return efim::pf::make_plan(cache, batch).total();
}

extern "C" int32_t efim_prefill_launch_count(const efim_cache_desc* cache, const efim_batch_desc* batch) {
  if (efim::check_cache(cache) != EFIM_OK || efim::check_batch(cache, batch, true) != EFIM_OK) return 0;
  if (batch->batch == 0 || batch->total_new_tokens == 0) return 0;
  const efim::pf::Plan pl = efim::pf::make_plan(cache, batch);
  return pl.n_items == 0 ? 0 : (pl.s_max > 1 ? 2 : 1);
}

namespace {
// Head of a host plan blob; the work list and the per-sequence split sizes follow it.
struct PlanHeader {
  uint32_t magic;
  int32_t batch, total_new_tokens, Hq, Hkv, D, n_items, s_max;
  uint64_t lengths_hash;                 // of the host mirrors the plan was made from
  uint64_t items_bytes, split_bytes, part_lse_bytes, part_o_bytes;
};
constexpr uint32_t PLAN_MAGIC = 0x4d494645u;      // "EFIM"
constexpr size_t PLAN_HEAD_BYTES = 256;

uint64_t lengths_hash(const efim_batch_desc* b) {
  uint64_t h = 1469598103934665603ull;
  for (int s = 0; s < b->batch; ++s) {
    h = (h ^ (uint32_t)b->h_cached_len[s]) * 1099511628211ull;
    h = (h ^ (uint32_t)b->h_new_len[s]) * 1099511628211ull;
  }
  return h;
}
bool batch_has_work(const efim_batch_desc* b) { return b->batch != 0 && b->total_new_tokens != 0; }

// Writes header and lists of a plan whose list sizes are already known (`sized`).
void fill_plan(const efim_cache_desc* cache, const efim_batch_desc* batch, const efim::pf::Plan* sized, void* h_plan) {
  using namespace efim;
  PlanHeader hd{};
  hd.magic = PLAN_MAGIC;
  hd.batch = batch->batch;
  hd.total_new_tokens = batch->total_new_tokens;
  hd.Hq = cache->num_q_heads;
  hd.Hkv = cache->num_kv_heads;
  hd.D = cache->head_dim;
  hd.lengths_hash = lengths_hash(batch);
  if (sized) {
    unsigned char* body = static_cast<unsigned char*>(h_plan) + PLAN_HEAD_BYTES;
    const size_t items_end = (size_t)sized->n_items * sizeof(pf::WorkItem), split_end = batch->batch * sizeof(int32_t);
    memset(body + items_end, 0, sized->items_bytes - items_end);
    memset(body + sized->items_bytes + split_end, 0, sized->split_bytes - split_end);
    pf::fill_lists(cache, batch, *sized, reinterpret_cast<pf::WorkItem*>(body),
                   reinterpret_cast<int32_t*>(body + sized->items_bytes));
    hd.n_items = sized->n_items;
    hd.s_max = sized->s_max;
    hd.items_bytes = sized->items_bytes;
    hd.split_bytes = sized->split_bytes;
    hd.part_lse_bytes = sized->part_lse_bytes;
    hd.part_o_bytes = sized->part_o_bytes;
  }
  memset(h_plan, 0, PLAN_HEAD_BYTES);
  memcpy(h_plan, &hd, sizeof(hd));
}
}  // namespace

extern "C" size_t efim_prefill_plan_bytes(const efim_cache_desc* cache, const efim_batch_desc* batch) {
  if (efim::check_cache(cache) != EFIM_OK || efim::check_batch(cache, batch, true) != EFIM_OK) return 0;
  if (!batch_has_work(batch)) return PLAN_HEAD_BYTES;
  const efim::pf::Plan pl = efim::pf::make_plan(cache, batch);
  return PLAN_HEAD_BYTES + pl.items_bytes + pl.split_bytes;
}

extern "C" efim_status efim_prefill_plan(const efim_cache_desc* cache, const efim_batch_desc* batch, void* h_plan,
                                         size_t plan_bytes) {
  using namespace efim;
  efim_status st = check_cache(cache);
  if (st != EFIM_OK) return st;
  st = check_batch(cache, batch, true);
  if (st != EFIM_OK) return st;
  if (!h_plan || plan_bytes < PLAN_HEAD_BYTES) return EFIM_ERR_INVALID_ARG;
  if (!batch_has_work(batch)) {
    fill_plan(cache, batch, nullptr, h_plan);
    return EFIM_OK;
  }
  const pf::Plan sized = pf::make_plan(cache, batch);
  if (plan_bytes < PLAN_HEAD_BYTES + sized.items_bytes + sized.split_bytes) return EFIM_ERR_WORKSPACE;
  fill_plan(cache, batch, &sized, h_plan);
  return EFIM_OK;
}

namespace {
// New tokens' k/v rows that the attention kernel itself puts into the pages.
struct NewRows {
  const void *k, *v;
};

// The host checks of what a plan is run on.  They come before a call's first launch: a call that is refused has enqueued
// nothing, so it may be repeated, also where its append would have rotated the queries in place.
efim_status check_run(const efim_rope_desc* rope, const efim::pf::Plan& pl, const void* d_q, const void* d_out,
                      const void* d_workspace, size_t workspace_bytes) {
  if (!d_q || !d_out) return EFIM_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(d_q) | reinterpret_cast<uintptr_t>(d_out)) & 15) return EFIM_ERR_INVALID_ARG;
  if (!d_workspace || workspace_bytes < pl.total()) return EFIM_ERR_WORKSPACE;
  if (reinterpret_cast<uintptr_t>(d_workspace) & 255) return EFIM_ERR_INVALID_ARG;
  if (rope && rope->d_cos_sin && (rope->max_position <= 0 || (reinterpret_cast<uintptr_t>(rope->d_cos_sin) & 15)))
    return EFIM_ERR_INVALID_ARG;
  return EFIM_OK;
}

// Runs a plan on what check_run has passed.  `rope` with a table: the query rows are rotated as the kernel
// loads them.  `h_lists`: the lists to copy to the head of the workspace (null: an earlier call has left
// them there); `list`: the work list, if it travels in the launch parameters instead.
efim_status run_plan(const efim_cache_desc* cache, const efim_batch_desc* batch, const efim_rope_desc* rope,
                     const efim::pf::Plan& pl, const void* h_lists, const efim::pf::InlineList* list, const NewRows* append,
                     const void* d_q, void* d_out, float* d_lse, float sm_scale, void* d_workspace, int32_t* d_status,
                     void* stream) {
  using namespace efim;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  char* ws = static_cast<char*>(d_workspace);
  pf::Params p{};
  p.q = static_cast<const uint16_t*>(d_q);
  p.out = static_cast<uint16_t*>(d_out);
  p.lse = d_lse;
  p.cached_len = batch->d_cached_len;
  p.q_indptr = batch->d_q_indptr;
  p.block_table = batch->d_block_table;
  p.items = reinterpret_cast<const pf::WorkItem*>(ws);
  p.split_tokens = reinterpret_cast<const int32_t*>(ws + pl.items_bytes);
  p.part_lse = reinterpret_cast<float*>(ws + pl.items_bytes + pl.split_bytes);
  p.part_o = reinterpret_cast<float*>(ws + pl.items_bytes + pl.split_bytes + pl.part_lse_bytes);
  p.status = d_status;
  p.batch = batch->batch;
  p.total_new_tokens = batch->total_new_tokens;
  p.Hq = cache->num_q_heads;
  p.Hkv = cache->num_kv_heads;
  p.G = cache->num_q_heads / cache->num_kv_heads;
  p.max_pages_per_seq = batch->max_pages_per_seq;
  p.num_pages = cache->num_pages;
  p.s_max = pl.s_max;
  const float scale = sm_scale > 0.f ? sm_scale : 1.0f / sqrtf((float)cache->head_dim);
  p.scale_log2 = scale * 1.4426950408889634f;
  p.wait_ns = WAIT_LIMIT_NS;
  if (rope && rope->d_cos_sin) {
    p.cos_sin = rope->d_cos_sin;
    p.max_position = rope->max_position;
    p.interleaved = rope->interleaved;
  }
  if (append) {
    p.k_new = static_cast<const uint16_t*>(append->k);
    p.v_new = static_cast<const uint16_t*>(append->v);
    p.k_pool = static_cast<uint16_t*>(cache->d_k_pool);
    p.v_pool = static_cast<uint16_t*>(cache->d_v_pool);
  }
  // work list + per-sequence split sizes go to the head of the workspace in one copy
  if (h_lists) EFIM_CUDA_TRY(cudaMemcpyAsync(ws, h_lists, pl.items_bytes + pl.split_bytes, cudaMemcpyHostToDevice, s));
  return pf::launch(cache, p, pl, list, s);
}

// Runs the plan in a blob of efim_prefill_plan().  `before`: an append, checked, that goes before the attention.
efim_status run_planned(const efim_cache_desc* cache, const efim_batch_desc* batch, const efim_rope_desc* rope,
                        const efim::Append* before, const void* h_plan, size_t plan_bytes, int32_t lists_resident,
                        const void* d_q, void* d_out, float* d_lse, float sm_scale, void* d_workspace, size_t workspace_bytes,
                        int32_t* d_status, void* stream) {
  using namespace efim;
  efim_status st = check_cache(cache);
  if (st != EFIM_OK) return st;
  st = check_batch(cache, batch, true);
  if (st != EFIM_OK) return st;
  if (!h_plan || plan_bytes < PLAN_HEAD_BYTES) return EFIM_ERR_INVALID_ARG;
  PlanHeader hd;
  memcpy(&hd, h_plan, sizeof(hd));
  // the plan must be the one made for this cache shape and these lengths
  if (hd.magic != PLAN_MAGIC || hd.batch != batch->batch || hd.total_new_tokens != batch->total_new_tokens ||
      hd.Hq != cache->num_q_heads || hd.Hkv != cache->num_kv_heads || hd.D != cache->head_dim ||
      hd.lengths_hash != lengths_hash(batch) || plan_bytes < PLAN_HEAD_BYTES + hd.items_bytes + hd.split_bytes)
    return EFIM_ERR_INVALID_ARG;
  if (!batch_has_work(batch) || hd.n_items == 0) return EFIM_OK;
  pf::Plan pl{};
  pl.n_items = hd.n_items;
  pl.s_max = hd.s_max;
  pl.items_bytes = hd.items_bytes;
  pl.split_bytes = hd.split_bytes;
  pl.part_lse_bytes = hd.part_lse_bytes;
  pl.part_o_bytes = hd.part_o_bytes;
  st = check_run(rope, pl, d_q, d_out, d_workspace, workspace_bytes);
  if (st != EFIM_OK) return st;
  if (before && (st = append_launch(cache, batch, *before, d_status, stream)) != EFIM_OK) return st;
  return run_plan(cache, batch, rope, pl, lists_resident ? nullptr : static_cast<const unsigned char*>(h_plan) + PLAN_HEAD_BYTES,
                  nullptr, nullptr, d_q, d_out, d_lse, sm_scale, d_workspace, d_status, stream);
}

// Plans, then runs.  Lists of up to InlineItems::MAX items travel in the launch parameters: no
// copy stands between the append and the attention kernel (append and attention of 16 tokens over 240 in
// one call 15.2 -> 10.7 us; the kernel leaves the list in the workspace all the same).
// `before`: an append, checked, that goes before the attention; it is launched between the plan, which says how large the
// workspace has to be, and the lists, which are written meanwhile.  `append`: rows the attention kernel is to put into the
// pages itself, where the plan allows it; else they are appended by a kernel of their own before it.
efim_status plan_and_run(const efim_cache_desc* cache, const efim_batch_desc* batch, const efim_rope_desc* rope,
                         const efim::Append* before, const NewRows* append, const void* d_q, void* d_out, float* d_lse,
                         float sm_scale, void* d_workspace, size_t workspace_bytes, int32_t* d_status, void* stream) {
  using namespace efim;
  efim_status st = check_cache(cache);
  if (st != EFIM_OK) return st;
  st = check_batch(cache, batch, true);
  if (st != EFIM_OK) return st;
  if (!batch_has_work(batch)) return EFIM_OK;
  const pf::Plan pl = pf::make_plan(cache, batch);
  if (pl.n_items == 0) return EFIM_OK;
  const bool in_params = pl.n_items <= pf::InlineItems::MAX && batch->batch <= pf::InlineSplit::MAX_BATCH;
  const bool aligned = !append || ((reinterpret_cast<uintptr_t>(append->k) | reinterpret_cast<uintptr_t>(append->v)) & 15) == 0;
  Append own;
  if (append && !(in_params && pl.s_max == 1 && aligned)) {  // (the kernel that appends is one of those with the list in its parameters)
    own = Append{rope, nullptr, nullptr, false, append->k, append->v};
    st = append_check(cache, batch, own);
    if (st != EFIM_OK) return st;
    before = &own;
    append = nullptr;
  }
  st = check_run(rope, pl, d_q, d_out, d_workspace, workspace_bytes);
  if (st != EFIM_OK) return st;
  if (before && (st = append_launch(cache, batch, *before, d_status, stream)) != EFIM_OK) return st;
  if (in_params) {
    pf::InlineList list;
    pf::fill_lists(cache, batch, pl, list.items.items, list.split.keys);
    return run_plan(cache, batch, rope, pl, nullptr, &list, append, d_q, d_out, d_lse, sm_scale, d_workspace, d_status,
                    stream);
  }
  const std::unique_ptr<unsigned char[]> lists(new unsigned char[pl.items_bytes + pl.split_bytes]);
  pf::fill_lists(cache, batch, pl, reinterpret_cast<pf::WorkItem*>(lists.get()),
                 reinterpret_cast<int32_t*>(lists.get() + pl.items_bytes));
  return run_plan(cache, batch, rope, pl, lists.get(), nullptr, nullptr, d_q, d_out, d_lse, sm_scale, d_workspace, d_status,
                  stream);
}

bool overlap(const void* a, size_t a_bytes, const void* b, size_t b_bytes) {
  const uintptr_t x = reinterpret_cast<uintptr_t>(a), y = reinterpret_cast<uintptr_t>(b);
  return a && b && x < y + b_bytes && y < x + a_bytes;
}

// Whether a step's new rows may be appended by the attention kernel: one sequence brings all of them (another one might
// count them among its cached tokens, in pages that both share), as one query tile per kv head (so nobody else reads what
// a CTA appends), with at most a CTA per SM; and what the kernel writes does not lie on the rows (a CTA may store its output
// before another one has read its k and v, which an append of its own has all read by then).  One tile: its second stream has no
// query rows to fetch and appends meanwhile.  With two tiles, or more than 128 tokens, two kernels are faster - one kernel against
// two, tokens over 0 at 4/4 heads x 64: 16 6.3 and 9.3 us, 128 11.5 and 13.5, 192 18.7 and 14.1, 256 22.7 and 15.9; at 8/8 x 128:
// 128 17.1 and 18.7, 256 34.7 and 20.8; at 32/8 x 128: 32 10.7 and 16.3, 64 18.6 and 16.1.
bool appends_in_attention(const efim_cache_desc* cache, const efim_batch_desc* batch, const NewRows& rows, const void* d_out,
                          const float* d_lse) {
  if (efim::check_cache(cache) != EFIM_OK || efim::check_batch(cache, batch, true) != EFIM_OK) return false;
  const size_t tokens = (size_t)batch->total_new_tokens, row_bytes = tokens * cache->num_kv_heads * cache->head_dim * 2;
  const size_t out_bytes = tokens * cache->num_q_heads * cache->head_dim * 2, lse_bytes = tokens * cache->num_q_heads * sizeof(float);
  for (const void* r : {rows.k, rows.v})
    if (overlap(r, row_bytes, d_out, out_bytes) || overlap(r, row_bytes, d_lse, lse_bytes)) return false;
  const long long G = cache->num_q_heads / cache->num_kv_heads;
  int with_work = 0;
  for (int s = 0; s < batch->batch; ++s) {
    if (batch->h_new_len[s] * G > efim::pf::BM) return false;
    with_work += batch->h_new_len[s] > 0;
  }
  return with_work == 1 && cache->num_kv_heads <= efim::sm_count();
}
// Whether the append kernel rotates a step's query rows, and leaves them where their outputs go: a work item has its rows in shared
// memory before it writes them, and no other one computes with them (the chunks of a cut key range write partials, and the merge
// comes after all of them).  Copies of 32 rows that reach past an item's last one may read rows that another CTA is writing: nothing
// of theirs is stored, nor does it steer a step.  Not where the output lies on the rows that the append reads, beyond row for row on q itself.  The
// attention kernel can rotate rows as it loads them, but its CTAs' warps wait for that, 12,300 cycles per item.  One-call steps with it
// and with the append: 16 prompts of 1-3.5k tokens 869 and 827 us, 53 x 1-406 over 100-549 at 24/8 100 and 75, 40 x 10-22 over
// 24-125 at 40/8 39 and 30, 39 x 1-5 over 0 at 16/1 12.3 and 9.2, 9 x 1 over 193-632 at 32/8 x 64 10.9 and 10.7.
bool rotates_into_out(const efim_cache_desc* cache, const efim_batch_desc* batch, const efim_rope_desc* rope, const NewRows& rows,
                      const void* d_q, const void* d_out) {
  if (!rope || !rope->d_cos_sin || !d_q || !d_out || efim::check_cache(cache) != EFIM_OK) return false;
  if (efim::check_batch(cache, batch, false) != EFIM_OK) return false;
  if ((reinterpret_cast<uintptr_t>(d_q) | reinterpret_cast<uintptr_t>(d_out)) & 15) return false;
  const size_t row = (size_t)cache->head_dim * 2, tokens = (size_t)batch->total_new_tokens;
  const size_t q_bytes = tokens * cache->num_q_heads * row, kv_bytes = tokens * cache->num_kv_heads * row;
  return !overlap(rows.k, kv_bytes, d_out, q_bytes) && !overlap(rows.v, kv_bytes, d_out, q_bytes) &&
         (d_q == d_out || !overlap(d_q, q_bytes, d_out, q_bytes));
}
}  // namespace

extern "C" efim_status efim_append_prefill_attn_planned(const efim_cache_desc* cache, const efim_batch_desc* batch,
                                                        const void* h_plan, size_t plan_bytes,
                                                        int32_t lists_resident, const void* d_q, void* d_out,
                                                        float* d_lse, float sm_scale, void* d_workspace,
                                                        size_t workspace_bytes, int32_t* d_status, void* stream) {
  return run_planned(cache, batch, nullptr, nullptr, h_plan, plan_bytes, lists_resident, d_q, d_out, d_lse, sm_scale,
                     d_workspace, workspace_bytes, d_status, stream);
}

// Plan and run in one call.
extern "C" efim_status efim_append_prefill_attn(const efim_cache_desc* cache, const efim_batch_desc* batch,
                                                const void* d_q, void* d_out, float* d_lse, float sm_scale,
                                                void* d_workspace, size_t workspace_bytes, int32_t* d_status,
                                                void* stream) {
  return plan_and_run(cache, batch, nullptr, nullptr, nullptr, d_q, d_out, d_lse, sm_scale, d_workspace, workspace_bytes,
                      d_status, stream);
}

// Steps 1 and 2 of a turn: the new tokens' k/v go into the pages (k rotated), then the new queries - rotated by the append
// into d_out, or by the attention kernel as it loads them (rotates_into_out, appends_in_attention) - attend over everything before
// them.
extern "C" efim_status efim_append_prefill_step(const efim_cache_desc* cache, const efim_batch_desc* batch,
                                                const efim_rope_desc* rope, const void* d_q, const void* d_k_new,
                                                const void* d_v_new, void* d_out, float* d_lse, float sm_scale,
                                                const void* h_plan, size_t plan_bytes, int32_t lists_resident,
                                                void* d_workspace, size_t workspace_bytes, int32_t* d_status,
                                                void* stream) {
  if ((d_k_new == nullptr) != (d_v_new == nullptr)) return EFIM_ERR_INVALID_ARG;
  const NewRows rows{d_k_new, d_v_new};
  if (d_k_new && !h_plan && appends_in_attention(cache, batch, rows, d_out, d_lse))
    return plan_and_run(cache, batch, rope, nullptr, &rows, d_q, d_out, d_lse, sm_scale, d_workspace, workspace_bytes, d_status,
                        stream);
  efim::Append rows_first{rope, nullptr, nullptr, false, d_k_new, d_v_new};
  if (d_k_new) {
    if (rotates_into_out(cache, batch, rope, rows, d_q, d_out)) {
      rows_first.q = d_q;
      rows_first.q_out = d_out;
      rows_first.every_row = true;
      d_q = d_out;
      rope = nullptr;
    }
    const efim_status st = efim::append_check(cache, batch, rows_first);
    if (st != EFIM_OK) return st;
  }
  const efim::Append* before = d_k_new ? &rows_first : nullptr;
  if (h_plan)
    return run_planned(cache, batch, rope, before, h_plan, plan_bytes, lists_resident, d_q, d_out, d_lse, sm_scale,
                       d_workspace, workspace_bytes, d_status, stream);
  return plan_and_run(cache, batch, rope, before, nullptr, d_q, d_out, d_lse, sm_scale, d_workspace, workspace_bytes, d_status,
                      stream);
}
