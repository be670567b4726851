// Internal interface of the append kernel.
#pragma once
#include "common.cuh"

namespace efim {

// Arguments of an append: efim_kv_append's, with the rotated query rows going to `q_out`: `q` itself, or an array of its own (16-byte
// aligned).  `every_row`: the rows of tokens whose keys are reported and dropped are written too - rotated, or zero where the rotary
// table has no row - as an attention that takes them from there needs; else they stay as they are.
struct Append {
  const efim_rope_desc* rope;
  const void* q;
  void* q_out;
  bool every_row;
  const void *k_new, *v_new;
};
// Host checks of the arguments; and the launch, of arguments that have passed them.
efim_status append_check(const efim_cache_desc* cache, const efim_batch_desc* batch, const Append& a);
efim_status append_launch(const efim_cache_desc* cache, const efim_batch_desc* batch, const Append& a, int32_t* d_status,
                          void* stream);

}  // namespace efim
