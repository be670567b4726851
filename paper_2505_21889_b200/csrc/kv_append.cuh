// Internal interface of the append kernel.
#pragma once
#include "common.cuh"

namespace efim {

// efim_kv_append, with the rotated query rows going to `d_q_out`: `d_q` itself, or an array of its own (16-byte aligned).  There
// every row is written, also of tokens whose keys are reported and dropped: rotated, or zero where the rotary table has no row.
efim_status append_run(const efim_cache_desc* cache, const efim_batch_desc* batch, const efim_rope_desc* rope, const void* d_q,
                       void* d_q_out, const void* d_k_new, const void* d_v_new, int32_t* d_status, void* stream);

}  // namespace efim
