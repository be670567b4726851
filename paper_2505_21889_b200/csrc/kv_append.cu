// efim_kv_append: rotary embedding of the new tokens' q/k fused with the scatter
// of k/v into the paged cache (EFIM Sec. 1: only the `inc` tokens are new and
// they follow `<P>prefix<S>suffix<M>`, so token i of sequence s has position
// cached_len[s] + i).  Pure streaming: every byte is read once and written once.
#include "kv_append.cuh"
#include <math.h>

namespace efim {

struct KvAppendParams {
  const uint16_t* q;        // [T][Hq][D], may be null
  uint16_t* q_out;          // where the rotated rows go: q itself or beside it
  const uint16_t* k_new;    // [T][Hkv][D]
  const uint16_t* v_new;
  uint16_t* k_pool;         // [pages][Hkv][P][D]
  uint16_t* v_pool;
  const int32_t* cached_len;
  const int32_t* q_indptr;
  const int32_t* block_table;
  const float* cos_sin;     // [max_position][D] or null
  int32_t* status;
  int batch, max_pages_per_seq, total_new_tokens;
  int num_pages, Hq, Hkv, max_position, interleaved;
  int early_next;           // let the next kernel start its set-up while this one runs
};

// WPT warps per new token, 256 threads per CTA.  A lane keeps one position along the head
// dimension (vector j, and for the rotate-half pairing its partner j + D/16), so its
// cos/sin values are loaded once, and walks the heads - q heads (rotated in place), then
// k heads (rotated into the page slot) - two at a time so that several 16-byte loads are
// in flight per lane; v is copied straight into the page slot.  Few tokens (a decode step): eight
// warps per token, because then the time is one token's latency.  Many: as few as its rows keep busy,
// from one to four (append_launch), so that every SM is full of independent streams.
//
// Bound: HBM with many tokens, else a chain of dependent loads.  A token's rows do not depend on where it goes, so the first
// of them (all, with few tokens) are on their way before its sequence is looked up; the warp's lanes look that up together,
// 32 candidates a trip, and bring the lengths along in the last one; page id and rotary row are fetched side by side.
// Rotated rows come past L1, as v's do, where they are fetched ahead with q among them, else by ordinary loads.  Past L1 everywhere:
// k and v alone of 2,336 tokens at 32/32 heads 10.1 us instead of 8.9, of 25,600 at 32/32 132.6 and 130.6, and with a warp a token
// 16,384 at 4/4 x 64 9.5 and 8.7.  Ordinary loads everywhere: some appends alone are shorter (2,336 at 32/32 13.5 -> 12.6), but one-call
// steps of 9 x 500-900 tokens at 28/4 are 82.9 us instead of 79.3, of 9 x 200-400 at 32/32 64.1 and 59.5.
constexpr int KV_APPEND_THREADS = 256;

// EVERY_ROW: query rows whose keys have no place are written all the same, zeros where the table has no row.  (A lane has read
// its vectors of a row before it writes them, so in place too.)
template <int D, int WPT, bool EVERY_ROW>
__global__ void __launch_bounds__(KV_APPEND_THREADS, 4) kv_append_kernel(const KvAppendParams p) {
  constexpr int VEC = D / 8;            // 16-byte vectors per head row
  constexpr int HALF = VEC / 2;
  constexpr int LANES = 32 * WPT;       // lanes working on one token
  constexpr int COPIES = WPT == 1 ? 4 : 2;   // vectors of a straight copy in flight per lane
  constexpr bool AHEAD = WPT > 1;       // first rows fetched before the look-up
  const int lane = threadIdx.x % LANES, wl = threadIdx.x & 31;
  const int t = blockIdx.x * (KV_APPEND_THREADS / LANES) + threadIdx.x / LANES;
  pdl_wait();
  if (p.early_next) pdl_launch();
  if (t >= p.total_new_tokens) return;
  const uint4* kin = reinterpret_cast<const uint4*>(p.k_new + (size_t)t * p.Hkv * D);
  const uint4* vin = reinterpret_cast<const uint4*>(p.v_new + (size_t)t * p.Hkv * D);
  const uint4* qin = p.q ? reinterpret_cast<const uint4*>(p.q + (size_t)t * p.Hq * D) : nullptr;
  const int nq = p.q ? p.Hq : 0, nh = nq + p.Hkv, n_vec = p.Hkv * VEC;
  // rotated heads: this lane's position j and first head, heads that the token's lanes cover at once
  const bool halves = !p.interleaved;
  const int per_head = halves ? HALF : VEC, HP = LANES / per_head;
  const int j = lane % per_head, h0 = lane / per_head;
  auto row_of = [&](int h) -> const uint4* { return h < nq ? qin + h * VEC : kin + (h - nq) * VEC; };
  uint4 v[COPIES], a[2], b[2];
  auto fetch_copy = [&](const uint4* src, int u0) {
#pragma unroll
    for (int i = 0; i < COPIES; ++i)
      if (u0 + LANES * i < n_vec) v[i] = ldg_stream(src + u0 + LANES * i);
  };
  auto fetch_heads = [&](int h) {       // vectors of heads h and h + HP
#pragma unroll
    for (int i = 0; i < 2; ++i)
      if (h + i * HP < nh) {
        const uint4* row = row_of(h + i * HP) + j;
        if (AHEAD && p.q) {
          a[i] = ldg_stream(row);
          if (halves) b[i] = ldg_stream(row + HALF);
        } else {
          a[i] = *row;
          if (halves) b[i] = row[HALF];
        }
      }
  };
  if constexpr (AHEAD) {
    if (p.cos_sin) fetch_heads(h0);
    fetch_copy(vin, lane);
  }
  // sequence of this token: the last one that starts at or before t, one of [lo, lo + n)
  int lo = 0, n = p.batch;
  while (n > 32) {
    const int step = (n + 31) / 32;
    const bool le = wl * step < n && *(p.q_indptr + lo + wl * step) <= t;
    const int i = 31 - __clz((int)(__ballot_sync(0xffffffffu, le) | 1u));
    n = min(step, n - i * step);
    lo += i * step;
  }
  int first = 0, cached = 0;
  if (wl < n) {
    first = *(p.q_indptr + lo + wl);
    cached = *(p.cached_len + lo + wl);
  }
  const int i_seq = 31 - __clz((int)(__ballot_sync(0xffffffffu, wl < n && first <= t) | 1u));
  const int pos = __shfl_sync(0xffffffffu, cached, i_seq) + t - __shfl_sync(0xffffffffu, first, i_seq);
  const int page_idx = pos >> 4;
  const bool in_table = !p.cos_sin || (pos >= 0 && pos < p.max_position);
  int err = 0, page = 0;
  if (pos < 0 || page_idx >= p.max_pages_per_seq || !in_table) {
    if (lane == 0 && p.status) atomicOr(p.status, EFIM_DEV_BAD_POSITION);
    if (!EVERY_ROW) return;
    err = EFIM_DEV_BAD_POSITION;
  } else {
    page = *(p.block_table + (size_t)(lo + i_seq) * p.max_pages_per_seq + page_idx);
  }
  // rotary values: position j of the row's halves (8 of either), or the 4 pairs of vector j
  float c[8], sn[8];
  if (p.cos_sin && (!EVERY_ROW || in_table)) {
    const float* cs = p.cos_sin + (size_t)pos * D + j * (halves ? 8 : 4);      // cos[0..D/2) then sin[0..D/2)
    *reinterpret_cast<float4*>(c) = __ldg(reinterpret_cast<const float4*>(cs));
    *reinterpret_cast<float4*>(sn) = __ldg(reinterpret_cast<const float4*>(cs + D / 2));
    if (halves) {
      *reinterpret_cast<float4*>(c + 4) = __ldg(reinterpret_cast<const float4*>(cs + 4));
      *reinterpret_cast<float4*>(sn + 4) = __ldg(reinterpret_cast<const float4*>(cs + D / 2 + 4));
    }
  }
  if (page < 0 || page >= p.num_pages) {
    if (lane == 0 && p.status) atomicOr(p.status, EFIM_DEV_BAD_PAGE);
    if (!EVERY_ROW) return;
    err = EFIM_DEV_BAD_PAGE;
  }
  const size_t pool_tok = ((size_t)page * p.Hkv) * 16 * D + (size_t)(pos & 15) * D;   // + h * 16 * D
  uint4* q_out = reinterpret_cast<uint4*>(const_cast<uint16_t*>(EVERY_ROW ? p.q_out : p.q) + (size_t)t * p.Hq * D);
  // straight copy of a [Hkv][D] row into the page slot; its first vectors have been fetched
  auto copy_row = [&](const uint4* src, uint16_t* pool) {
    for (int u0 = lane; u0 < n_vec; u0 += COPIES * LANES) {
      if (!AHEAD || u0 != lane) fetch_copy(src, u0);
#pragma unroll
      for (int i = 0; i < COPIES; ++i) {
        const int u = u0 + LANES * i;
        if (u < n_vec) *reinterpret_cast<uint4*>(pool + pool_tok + (size_t)(u / VEC) * 16 * D + (u % VEC) * 8) = v[i];
      }
    }
  };
  if (!EVERY_ROW || !err) copy_row(vin, p.v_pool);
  if (!p.cos_sin) {
    if (EVERY_ROW && err) return;
    if constexpr (AHEAD) fetch_copy(kin, lane);
    copy_row(kin, p.k_pool);
    return;
  }
  for (int h = h0; h < nh; h += 2 * HP) {
    if (!AHEAD || h != h0) fetch_heads(h);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int hh = h + i * HP;
      if (hh < nh && (!EVERY_ROW || hh < nq || !err)) {
        uint4* dst = hh < nq ? q_out + hh * VEC : reinterpret_cast<uint4*>(p.k_pool + pool_tok + (size_t)(hh - nq) * 16 * D);
        if (EVERY_ROW && !in_table) {
          dst[j] = make_uint4(0, 0, 0, 0);
          if (halves) dst[j + HALF] = make_uint4(0, 0, 0, 0);
        } else if (halves) {
          rotate8(a[i], b[i], c, sn);
          dst[j] = a[i];
          dst[j + HALF] = b[i];
        } else {
          rotate4_interleaved(a[i], c, sn);
          dst[j] = a[i];
        }
      }
    }
  }
}
}  // namespace efim

extern "C" efim_status efim_rope_table_build(double base, int32_t head_dim, int32_t max_position, float* h_out) {
  if (!h_out || head_dim <= 0 || (head_dim & 1) || max_position <= 0 || !(base > 0.0)) return EFIM_ERR_INVALID_ARG;
  const int half = head_dim / 2;
  for (int f = 0; f < half; ++f) {
    const double theta = pow(base, -2.0 * (double)f / (double)head_dim);
    for (int p = 0; p < max_position; ++p) {
      const double ang = (double)p * theta;
      h_out[(size_t)p * head_dim + f] = (float)cos(ang);
      h_out[(size_t)p * head_dim + half + f] = (float)sin(ang);
    }
  }
  return EFIM_OK;
}

extern "C" efim_status efim_kv_append(const efim_cache_desc* cache, const efim_batch_desc* batch,
                                      const efim_rope_desc* rope, void* d_q, const void* d_k_new,
                                      const void* d_v_new, int32_t* d_status, void* stream) {
  const efim::Append a{rope, d_q, d_q, false, d_k_new, d_v_new};
  const efim_status st = efim::append_check(cache, batch, a);
  return st != EFIM_OK ? st : efim::append_launch(cache, batch, a, d_status, stream);
}

efim_status efim::append_check(const efim_cache_desc* cache, const efim_batch_desc* batch, const Append& a) {
  efim_status st = efim::check_cache(cache);
  if (st != EFIM_OK) return st;
  st = efim::check_batch(cache, batch, false);
  if (st != EFIM_OK) return st;
  if (batch->batch == 0 || batch->total_new_tokens == 0) return EFIM_OK;
  if (!a.k_new || !a.v_new) return EFIM_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(a.k_new) | reinterpret_cast<uintptr_t>(a.v_new) | reinterpret_cast<uintptr_t>(a.q)) & 15)
    return EFIM_ERR_INVALID_ARG;
  if (a.rope && a.rope->d_cos_sin && (a.rope->max_position <= 0 || (reinterpret_cast<uintptr_t>(a.rope->d_cos_sin) & 15)))
    return EFIM_ERR_INVALID_ARG;
  return EFIM_OK;
}

efim_status efim::append_launch(const efim_cache_desc* cache, const efim_batch_desc* batch, const Append& a, int32_t* d_status,
                                void* stream) {
  if (batch->batch == 0 || batch->total_new_tokens == 0) return EFIM_OK;
  efim::KvAppendParams p{};
  p.q = static_cast<const uint16_t*>(a.q);
  p.q_out = static_cast<uint16_t*>(a.q_out);
  p.k_new = static_cast<const uint16_t*>(a.k_new);
  p.v_new = static_cast<const uint16_t*>(a.v_new);
  p.k_pool = static_cast<uint16_t*>(cache->d_k_pool);
  p.v_pool = static_cast<uint16_t*>(cache->d_v_pool);
  p.cached_len = batch->d_cached_len;
  p.q_indptr = batch->d_q_indptr;
  p.block_table = batch->d_block_table;
  p.cos_sin = nullptr;
  if (a.rope && a.rope->d_cos_sin) {
    p.cos_sin = a.rope->d_cos_sin;
    p.max_position = a.rope->max_position;
    p.interleaved = a.rope->interleaved;
  }
  p.status = d_status;
  p.batch = batch->batch;
  p.max_pages_per_seq = batch->max_pages_per_seq;
  p.total_new_tokens = batch->total_new_tokens;
  p.num_pages = cache->num_pages;
  p.Hq = cache->num_q_heads;
  p.Hkv = cache->num_kv_heads;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  // Warps per token: 8, and 4, while every token's CTA is resident at once (a token's latency is the time); beyond that as many as
  // its rows - q's where there are any - keep busy for a few vectors each.  Microseconds with 1 / 2 / 4 / 8 (in brackets with 8 below
  // 1,024 tokens, 4 below 4,096, 2 below 16,384 and look-ups before the rows): 64 tokens at 32/8 heads x 128 4.9 / 3.5 / 3.2 / 3.2 [3.2],
  // 960 5.0 / 4.3 / 4.4 / 4.7 [5.4], 2,336 6.8 / 7.1 / 7.9 / 9.4 [8.0], 25,600 99.0 / 97.7 / 99.1 / 110 [99.5]; 2,336 at 4/4 x 64 3.3 / 3.3 /
  // 4.2 / 6.6 [4.4], 8,192 4.9 / 7.0 / 11.7 / 19.6 [7.5]; 4,096 at 32/32 x 128 34.9 / 32.2 / 31.9 / 31.7 [34.0], 25,600 199 / 199 / 195 / 194
  // [201]; k and v alone of 16,384 at 28/4 10.0 / 13.4 / 22.3 / 38.5 [10.5].
  const int T = batch->total_new_tokens, resident = 4 * efim::sm_count();
  const int vectors = ((p.q ? p.Hq : 0) + 2 * p.Hkv) * (cache->head_dim / 8);   // of the rows that a token moves
  const int wpt = T <= resident ? 8 : T <= 2 * resident || vectors >= 1024 ? 4 : vectors >= 384 || T <= 4 * resident ? 2 : 1;
  const unsigned grid = (unsigned)(((long long)T * wpt * 32 + efim::KV_APPEND_THREADS - 1) / efim::KV_APPEND_THREADS);
  // With at most a CTA per SM the next kernel may start early (a step of 64 rows with its decode
  // attention 128 -> 121 us).  Beside more CTAs the attention kernel's, which take an SM each, are dealt
  // out to whichever SMs run dry first, and the launch lost more than the set-up it hid (append +
  // attention of 64 mixed rows 349 -> 391 us, 16 rows at 32/32 heads 336 -> 351).
  p.early_next = grid <= (unsigned)efim::sm_count();
#define EFIM_KV_APPEND_LAUNCH(D_, W_, A_) \
  EFIM_CUDA_TRY(efim::launch_pdl(efim::kv_append_kernel<D_, W_, A_>, dim3(grid), dim3(efim::KV_APPEND_THREADS), 0, s, p))
#define EFIM_KV_APPEND_WARPS(D_, A_)                  \
  do {                                                \
    if (wpt == 1) EFIM_KV_APPEND_LAUNCH(D_, 1, A_);      \
    else if (wpt == 2) EFIM_KV_APPEND_LAUNCH(D_, 2, A_); \
    else if (wpt == 4) EFIM_KV_APPEND_LAUNCH(D_, 4, A_); \
    else EFIM_KV_APPEND_LAUNCH(D_, 8, A_);               \
  } while (0)
  if (cache->head_dim == 128) {
    if (a.every_row) EFIM_KV_APPEND_WARPS(128, true);
    else EFIM_KV_APPEND_WARPS(128, false);
  } else {
    if (a.every_row) EFIM_KV_APPEND_WARPS(64, true);
    else EFIM_KV_APPEND_WARPS(64, false);
  }
#undef EFIM_KV_APPEND_WARPS
#undef EFIM_KV_APPEND_LAUNCH
  return EFIM_OK;
}
