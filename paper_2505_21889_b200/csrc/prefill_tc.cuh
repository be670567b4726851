// Internal interface of the tensor-core append-prefill kernel.
#pragma once
#include <cuda.h>
#include "common.cuh"

namespace efim {
namespace pf {

constexpr int BM = 128;        // query rows per tile (one TMEM lane each)
constexpr int PT = 128;        // keys per tile of the work list (8 pages)
constexpr int NQ = 2;          // query tiles per CTA sharing one K/V stream
// Keys per step of the kernel's inner loop.  A stream keeps its scores S (fp32, BN columns), its
// probabilities P (bf16, BN / 2 columns) and its O (fp32, D columns) in tensor memory side by side;
// two streams share the 512 columns, so at head_dim 128 2 * (1.5 * BN + 128) <= 512 and, in whole pages,
// BN = 80.  With P in columns of its own the scores of the next step can be computed while this step's
// are being exponentiated.  At head_dim 64 there is room for 128 keys, but 80 are faster there too (4 x
// 3,000 tokens over 2k keys at 32/8 heads: 604 us with 128, 587 with 96, 557 with 80, 642 with 64).
constexpr int BN = 80;
constexpr int THREADS = 384;   // 2 softmax warpgroups + 1 service warpgroup (2 TMA warps, 2 MMA warps)
// Register split (setmaxnreg): the block launches with 168 registers per thread
// (65536 / 384, rounded to 8) = 64512 in total; 2 x 128 x 216 + 128 x 72 and 2 x 128 x 208 + 128 x 88 use them all
// (the sum must not exceed the launch total: an increase beyond it would wait forever).  At head_dim 128 with 208 / 88 the
// softmax warps spill seven words a step (16 prompts of 1-3.5k tokens 975 -> 1,012 us, 8 x 3,200 tokens over 5k 2.51 -> 2.55 ms);
// 224 / 56: the service warps spill (1,027 us, 2.72 ms).  At head_dim 64 216 / 72 and 208 / 88 need the same spills, and 37 x 128
// tokens over 4,000 keys at 4/4 heads take 40.6 and 39.2 us, 26 x 1-132 over 6-15k at 32/8 297.6 and 295.3.
template <int D> constexpr int REGS_SOFTMAX = D == 128 ? 216 : 208;
template <int D> constexpr int REGS_SERVICE = D == 128 ? 72 : 88;

// One work item: packed rows [row0, row0 + 256) of (seq, kv head) against the keys of the
// 128-key tiles [tile_begin, tile_end).  Packed row R = token * G + head-in-group.  The sequence's
// lengths and first query row ride along (the planner has them from the host mirrors),
// so that a CTA's first dependent chain is "item -> block table / query rows" instead of
// "item -> lengths -> block table / query rows".
struct WorkItem {
  int32_t seq;
  int16_t kvh;
  int16_t chunk;               // >= 0: write a partial for this KV chunk; -1: final output
  int32_t row0, tile_begin, tile_end;
  int32_t cached, new_len;     // cached_len[seq], new_len[seq]
  int32_t tok0;                // q_indptr[seq]
};
static_assert(sizeof(WorkItem) == 32, "work items are read as two 16-byte vectors");

struct Params {
  const uint16_t* q;           // [T][Hq][D]
  uint16_t* out;               // [T][Hq][D]
  float* lse;                  // [T][Hq] or null
  const int32_t* cached_len;
  const int32_t* q_indptr;
  const int32_t* block_table;
  const WorkItem* items;
  WorkItem* items_out;         // where to leave lists that came in the launch parameters, or null
  int32_t* split_out;
  const int32_t* split_tokens; // [batch] keys per KV chunk of a split sequence, 0 = not split
  float* part_o;               // [T][Hq][s_max][D]
  float* part_lse;             // [T][Hq][s_max]  base-2
  int32_t* status;
  int batch, total_new_tokens;
  int Hq, Hkv, G, max_pages_per_seq, num_pages, s_max;
  float scale_log2;
  unsigned long long wait_ns;  // limit of every device-side wait
  // rotation of the query rows as they are loaded (null: q is already rotated)
  const float* cos_sin;        // [max_position][D] (and of the new k)
  int max_position, interleaved;
  int early_next;              // let the next kernel start its set-up while this one runs
  // the new tokens' k/v, put into their page slots by this kernel (null: they are there already); every item is all
  // the rows of its (sequence, kv head) then, and of one sequence
  const uint16_t *k_new, *v_new;   // [T][Hkv][D]
  uint16_t *k_pool, *v_pool;   // [pages][Hkv][16][D]
  uint32_t g_mul;              // floor(2^32 / G) + 1 (0: G = 1), see token_of
  int q_tma, out_tma;          // 32 rows are whole tokens (G divides 32): they move as boxes of 64 dims
};

struct Plan {
  int n_items;
  int s_max;                   // largest KV split count (1 = no partials, no merge)
  long long chunk_tiles;       // key tiles per KV chunk aimed at
  size_t items_bytes, split_bytes, part_lse_bytes, part_o_bytes;
  size_t total() const { return items_bytes + split_bytes + part_lse_bytes + part_o_bytes; }
};

// Lists that travel in the launch parameters: the work items and the split sizes of the sequences.  Calls of
// 8 rows at 32/8 or 16 at 4/4 heads (64 items) take 12.3 and 10.2 us that way, 16.4 and 14.4 with a copied
// list, of 32 rows at 32/8 (256 items) 25.0 against 28.0; beyond that the planning on the host (60 us at 512
// items) hides the copy, while room for 640 items costs every call 0.7 us more on the host.  A sequence with
// work has at least one item, so both lists get the same size.
struct NoList {};
struct InlineItems {
  static constexpr int MAX = 256;
  WorkItem items[MAX];
};
struct InlineSplit {
  static constexpr int MAX_BATCH = 256;
  int32_t keys[MAX_BATCH];
};
struct InlineList {
  InlineItems items;
  InlineSplit split;
};
inline const InlineItems& items_of(const InlineList& l) { return l.items; }
inline const NoList& items_of(const NoList& l) { return l; }

// Host: choose the cut and size the lists; then write them.
Plan make_plan(const efim_cache_desc* c, const efim_batch_desc* b);
void fill_lists(const efim_cache_desc* c, const efim_batch_desc* b, const Plan& pl, WorkItem* items, int32_t* split_tokens);

// `list`: the work list if it is to travel in the launch parameters, else null (it is in the workspace).
efim_status launch(const efim_cache_desc* c, const Params& p, const Plan& pl, const InlineList* list, cudaStream_t s);

// Tensor map of a page pool (one box = the 16 slots x head_dim of one (page, kv head)), kept per
// host thread; null if it cannot be encoded.  Valid until the thread's next call: copy it.
const CUtensorMap* pool_map(void* pool, int pages, int Hkv, int D);

}  // namespace pf
}  // namespace efim
