// efim_decode_attn: split-KV paged decode attention with a log-sum-exp merge
// (decode of the generated middle, EFIM Sec. 2.2 / Fig. 4).  Bandwidth-bound: every K/V
// byte of the visible context is read once, whatever the number of query heads that share it.
//
// One CTA = (query row, kv head [x tile of at most 16 query heads], key chunk).  Each of its 4
// warps walks whole pages (16 tokens) round-robin, staged into shared memory by one bulk-tensor
// copy per K page and V page.  A page is one 16-row tile of the warp's matrix instructions
// (mma.sync m16n8k16, bf16 in, fp32 accumulation), with the query heads along n:
//   S^T [16 tokens][heads]  = K [16][D] Q^T [D][heads]
//   O^T [D][heads]         += V^T [D][16] P^T [16][heads]
// The softmax runs on the S^T fragments (a lane holds 2 tokens x 2 heads, so 4 exponentials a
// page); P^T is the same fragments transposed by movmatrix.  P keeps its fp32 precision: it enters
// the second product as three bf16 terms (hi + mid + lo, 24 significant bits in all).
//
// Bound: HBM.  A page's 16 tokens are exactly one m-tile and there is nothing to share between
// pages, so warp-level instructions fit where a 128-row tcgen05 tile would be mostly padding; one
// page costs a warp about 160 instructions for any group of up to 8 heads, against some 600 for
// 4 heads on fp32 FMAs (which bound groups of 5 and more, and through the power limit long steps
// of 4).  Split kernel, before -> after: 64 rows x 1-16k keys at 28/4 heads 233 -> 113 us (3.1 ->
// 6.5 TB/s), 256 rows x 4-32k at 32/8 3.2-3.4 -> 2.58 ms (7.1 TB/s), 16 rows x 2-8k at 32/32 179 ->
// 173 us, 16 rows x 2-2.9k at 32/8 41 -> 28 us.
#include "decode_attn.cuh"
#include "mbar.cuh"
#include "prefill_tc.cuh"
#include <algorithm>
#include <cfloat>
#include <atomic>

namespace efim {

// ---- shared-memory staging of whole pages -------------------------------------------
// Every warp owns a ring of dec_stages pages (K + V), keeps them in flight without holding them
// in registers and consumes them in order; an mbarrier per stage counts the copied bytes.  64 KB
// of ring per CTA, three CTAs (12 warps, 192 KB in flight) per SM.
constexpr int DEC_WARPS = 4;
constexpr int DEC_THREADS = 32 * DEC_WARPS;
constexpr int DEC_CTAS_PER_SM = 3;
__host__ __device__ constexpr int dec_stages(int D) { return D == 128 ? 2 : 4; }
__host__ __device__ constexpr int dec_ring_bytes(int D) { return DEC_WARPS * dec_stages(D) * 2 * 16 * D * 2; }

// One (page, kv head) of a pool into shared memory as [slot / 8][dim / 64][slot % 8][64 dims],
// 16-byte chunk c of a 128-byte row at chunk position c ^ (slot & 7): ldmatrix reads it without
// bank conflicts, plain or transposed.
__device__ __forceinline__ void dec_load_page(uint32_t dst, const CUtensorMap* map, uint32_t bar, int page_head) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %3, %3, %3, %4}], "
      "[%2];" ::"r"(dst),
      "l"(map), "r"(bar), "r"(0), "r"(page_head)
      : "memory");
}
// byte offset of 16-byte chunk `c` (0 .. D/8-1) of slot `t` in a staged page
template <int D>
__device__ __forceinline__ uint32_t dec_page_off(int t, int c) {
  return (uint32_t)((t >> 3) * (D * 16) + (c >> 3) * 1024 + (t & 7) * 128 + (((c & 7) ^ (t & 7)) << 4));
}
__device__ __forceinline__ void ldsm4(uint32_t addr, uint32_t* r) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void ldsm4_t(uint32_t addr, uint32_t* r) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ uint32_t movm_t(uint32_t v) {
  uint32_t r;
  asm("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(r) : "r"(v));
  return r;
}
// c += a b, a 16 x 16 (row), b 16 x 8 (col), bf16 in, fp32 accumulation
__device__ __forceinline__ void mma16816(float* c, const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ float dec_ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Rotation of one 16-byte vector (8 bf16) of a head row, exactly as efim_kv_append does it
// (fp32 FMA, one rounding to bf16).  Rotate-half pairing: `mine` is vector j of the row,
// `other` vector j ^ (D/16); the first half of the row gets a c - b s, the second b c + a s.
// Interleaved pairing: the pairs (2f, 2f+1) sit inside the vector and `other` is not used.
__device__ __forceinline__ uint4 dec_rotate_vec(uint4 mine, uint4 other, const float* cs, int D, int j, int interleaved) {
  uint32_t* m = reinterpret_cast<uint32_t*>(&mine);
  const uint32_t* o = reinterpret_cast<const uint32_t*>(&other);
  if (!interleaved) {
    const int half = D / 16;
    const bool first = j < half;
    const float* c = cs + (j % half) * 8;
    const float* sn = c + D / 2;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float m0 = bf16lo(m[i]), m1 = bf16hi(m[i]), o0 = bf16lo(o[i]), o1 = bf16hi(o[i]);
      const float c0 = __ldg(c + 2 * i), c1 = __ldg(c + 2 * i + 1), s0 = __ldg(sn + 2 * i), s1 = __ldg(sn + 2 * i + 1);
      const float r0 = first ? fmaf(m0, c0, -(o0 * s0)) : fmaf(m0, c0, o0 * s0);
      const float r1 = first ? fmaf(m1, c1, -(o1 * s1)) : fmaf(m1, c1, o1 * s1);
      m[i] = pack_bf16x2(r0, r1);
    }
  } else {
    const float* c = cs + j * 4;
    const float* sn = c + D / 2;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float a = bf16lo(m[i]), b = bf16hi(m[i]);
      const float ci = __ldg(c + i), si = __ldg(sn + i);
      m[i] = pack_bf16x2(fmaf(a, ci, -(b * si)), fmaf(b, ci, a * si));
    }
  }
  return mine;
}

// Four dimensions of the weighted mean of keys [begin, end) of one (row, kv head) when some of their values
// are infinite or NaN: every visible key has a positive weight, so a dimension is NaN if it holds a NaN or
// infinities of both signs, else the infinity it holds.  (P enters the products as three terms, of which the
// lower two may be 0 or negative, and 0 or a negative times infinity beside the first term's is NaN.)
// `v_last`: the new token's values, where key `last` is one that may not be in its page yet, else null.
// Out of line and rare: only threads whose sums came out as NaN under a sound row sum come here.
__device__ __noinline__ float4 mean_of_unbounded(const uint16_t* v_pool, const int32_t* bt, int num_pages, int Hkv, int kvh,
                                                 int D, int d, int begin, int end, const uint16_t* v_last, int last) {
  uint32_t nan = 0, pos = 0, neg = 0;                        // a bit per dimension
  for (int key = begin; key < end; ++key) {
    const uint16_t* v;
    if (v_last && key == last) {
      v = v_last + d;
    } else {
      const int pid = *(bt + (key >> 4));
      if (pid < 0 || pid >= num_pages) continue;             // rejected pages have no keys
      v = v_pool + (((size_t)pid * Hkv + kvh) * 16 + (key & 15)) * D + d;
    }
    const uint2 w = *reinterpret_cast<const uint2*>(v);
    const uint16_t u[4] = {(uint16_t)w.x, (uint16_t)(w.x >> 16), (uint16_t)w.y, (uint16_t)(w.y >> 16)};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if ((u[i] & 0x7fff) > 0x7f80) nan |= 1u << i;
      if (u[i] == 0x7f80) pos |= 1u << i;
      if (u[i] == 0xff80) neg |= 1u << i;
    }
  }
  float r[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const bool p = pos >> i & 1, n = neg >> i & 1;
    r[i] = (nan >> i & 1) || p == n ? NAN : (p ? INFINITY : -INFINITY);
  }
  return make_float4(r[0], r[1], r[2], r[3]);
}

// NT tiles of 8 query heads per CTA (heads beyond the group's are zero queries, dropped at the end).
template <int D, int NT, bool FUSED>
__global__ void __launch_bounds__(DEC_THREADS, DEC_CTAS_PER_SM)
decode_splitkv_kernel(const DecodeParams p, const __grid_constant__ CUtensorMap map_k,
                      const __grid_constant__ CUtensorMap map_v) {
  constexpr int ST = dec_stages(D);
  constexpr int VEC = D / 8;            // 16-byte vectors per head row
  constexpr int KS = D / 16;            // k-steps of S^T, m-tiles of O^T
  constexpr int GP = 8 * NT;            // heads with padding
  constexpr int PAGE_BYTES = 16 * D * 2;
  constexpr int XD = D + 4;             // floats per row of the warps' exchange buffer (padded: no bank conflicts)
  static_assert(DEC_WARPS * GP * XD * 4 <= dec_ring_bytes(D), "the exchange buffer re-uses the ring");

  extern __shared__ uint8_t dec_smem[];                  // ring, 1024-byte aligned below
  __shared__ __align__(8) uint64_t s_bar[DEC_WARPS][ST];
  __shared__ __align__(16) uint16_t s_q[GP][D + 8];      // query rows (rotated in a fused step)
  __shared__ float s_m[DEC_WARPS][GP], s_l[DEC_WARPS][GP];

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int r = blockIdx.x;
  const int G = p.Hq / p.Hkv;
  const int gsplit = (G + p.group_tile - 1) / p.group_tile;
  const int kvh = blockIdx.y / gsplit;
  const int g0 = (blockIdx.y % gsplit) * p.group_tile;
  const int ng = min(p.group_tile, G - g0);
  const int c = blockIdx.z;
  const uint32_t ring0 = (smem_u32(dec_smem) + 1023u) & ~1023u;
  uint8_t* ring_gen = dec_smem + (ring0 - smem_u32(dec_smem));
  if (tid == 0) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_k) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map_v) : "memory");
  }
  if (lane == 0) {
    for (int sg = 0; sg < ST; ++sg) mbar_init(smem_u32(&s_bar[warp][sg]), 1);
    mbar_fence_init();
  }
  __syncwarp();
  pdl_wait();
  pdl_launch();
  // The first block-table entries of every warp are fetched before the row's length is known
  // (any entry of the row may be read; those past the length are dropped below), so that the
  // two loads share one round trip: a short step's time is mostly this ramp.
  const int32_t* bt = p.block_table + (size_t)r * p.max_pages_per_seq;
  const int first_pg = ((c * p.chunk_tokens) >> 4) + warp;
  const int my_pg = first_pg + DEC_WARPS * lane;
  const int pid_early = my_pg < p.max_pages_per_seq ? *(bt + my_pg) : -1;
  int len = *(p.row_len + r);
  // longer than the launch was planned for (max_ctx_len) or than the block table can address:
  // clamp and report.  A fused step then has no valid position for its new token and runs as a
  // plain decode over the clamped range.
  bool append = FUSED;
  if (len > p.key_cap) {
    len = p.key_cap;
    append = false;
    if (tid == 0 && p.status) atomicOr(p.status, EFIM_DEV_BAD_POSITION);
  }
  const int begin = c * p.chunk_tokens;
  const int head0 = kvh * G + g0;
  // fused step: the new token sits at position len - 1; its rotation needs a table row
  const float* cs_row = nullptr;
  bool skip_row = false;
  if (FUSED && append && len > 0 && p.cos_sin) {
    if (len - 1 >= p.max_position) {
      // no table row for the new token's position: report it and skip the row (nothing is
      // appended; the output is zero, lse -inf)
      if (tid == 0 && p.status) atomicOr(p.status, EFIM_DEV_BAD_POSITION);
      skip_row = true;
    } else {
      cs_row = p.cos_sin + (size_t)(len - 1) * D;
    }
  }
  if (begin >= len || skip_row) {
    // nothing to attend in this chunk.  A row without any key (or a skipped one) still gets a
    // defined result: directly, or as an empty partial for every chunk the merge will read.
    if (p.n_chunks == 1) {
      if (len <= 0 || skip_row) {
        for (int i = tid; i < ng * D; i += DEC_THREADS) p.out[((size_t)r * p.Hq + head0) * D + i] = 0;
        if (p.lse && tid < ng) p.lse[(size_t)r * p.Hq + head0 + tid] = -INFINITY;
      }
    } else if (skip_row && begin < len) {
      for (int i = tid; i < ng * D; i += DEC_THREADS) {
        const size_t row_head = (size_t)r * p.Hq + head0 + i / D;
        p.part_o[(row_head * p.n_chunks + c) * D + i % D] = 0.f;
        if (i % D == 0) p.part_lse[row_head * p.n_chunks + c] = -INFINITY;
      }
    }
    return;
  }
  const int end = min(len, begin + p.chunk_tokens);

  // ---- this warp's pages: first_pg, first_pg + 4, ... ; start their copies before anything else
  const int last_pg = (end - 1) >> 4;
  const int n_pages = first_pg <= last_pg ? (last_pg - first_pg) / DEC_WARPS + 1 : 0;
  const uint32_t ring = ring0 + warp * (ST * 2 * PAGE_BYTES);
  // page ids of the next 32 pages of this warp, one per lane (refilled every 32 pages)
  int pid_cache = (lane < n_pages) ? pid_early : -1;
  auto issue = [&](int i) {             // start the copies of this warp's i-th page into stage i % ST
    const int pid = __shfl_sync(0xffffffffu, pid_cache, i & 31);
    const bool ok = pid >= 0 && pid < p.num_pages;
    if (lane == 0) {
      const uint32_t bar = smem_u32(&s_bar[warp][i % ST]);
      if (ok) {
        const uint32_t dst = ring + (i % ST) * 2 * PAGE_BYTES;
        mbar_expect_tx(bar, 2 * PAGE_BYTES);
        dec_load_page(dst, &map_k, bar, pid * p.Hkv + kvh);
        dec_load_page(dst + PAGE_BYTES, &map_v, bar, pid * p.Hkv + kvh);
      } else {
        mbar_arrive(bar);                                                // nothing to copy
        if (p.status) atomicOr(p.status, EFIM_DEV_BAD_PAGE);
      }
    }
    return ok;
  };
  uint32_t ok_bits = 0;                 // which of the in-flight pages are valid (bit = stage)
#pragma unroll
  for (int i = 0; i < ST; ++i)
    if (i < n_pages && issue(i)) ok_bits |= 1u << i;

  // ---- query rows: through shared memory (rotated there) into B fragments, dims 2q, 2q+1 (+8) of
  // head lane / 4 for every k-step, kept in registers
  for (int i = tid; i < GP * VEC; i += DEC_THREADS) {
    const int g = i / VEC, j = i % VEC;
    uint4 w = make_uint4(0, 0, 0, 0);
    if (g < ng) {
      const uint4* qrow = reinterpret_cast<const uint4*>(p.q + ((size_t)r * p.Hq + head0 + g) * D);
      w = *(qrow + j);
      if (FUSED && cs_row) w = dec_rotate_vec(w, *(qrow + (j ^ (VEC / 2))), cs_row, D, j, p.interleaved);
    }
    *reinterpret_cast<uint4*>(&s_q[g][j * 8]) = w;
  }
  __syncthreads();
  const int hq = lane >> 2, tq = lane & 3;
  uint32_t qf[NT][KS][2];
#pragma unroll
  for (int n = 0; n < NT; ++n)
#pragma unroll
    for (int k = 0; k < KS; ++k) {
      qf[n][k][0] = *reinterpret_cast<const uint32_t*>(&s_q[n * 8 + hq][k * 16 + 2 * tq]);
      qf[n][k][1] = *reinterpret_cast<const uint32_t*>(&s_q[n * 8 + hq][k * 16 + 8 + 2 * tq]);
    }
  float o[NT][KS][4];                   // O^T fragments: dims 16 k + hq (+8), heads 8 n + 2 tq + {0, 1}
#pragma unroll
  for (int n = 0; n < NT; ++n)
#pragma unroll
    for (int k = 0; k < KS; ++k)
#pragma unroll
      for (int e = 0; e < 4; ++e) o[n][k][e] = 0.f;
  // of heads 8 n + 2 tq + {0, 1}; the sum over this lane's tokens.  The reference is finite from the start:
  // a key whose score is -inf then has the probability 0, also before any other key was seen.
  float m_ref[NT][2], l_part[NT][2];
#pragma unroll
  for (int n = 0; n < NT; ++n)
#pragma unroll
    for (int e = 0; e < 2; ++e) { m_ref[n][e] = -FLT_MAX; l_part[n][e] = 0.f; }

  // ldmatrix row addresses of this lane inside a staged page: K (tokens along m), V (dims along m)
  const uint32_t k_lane = (uint32_t)(((lane >> 3) & 1) * (D * 16) + (lane & 7) * 128 + (((lane >> 4) ^ (lane & 7)) << 4));
  const uint32_t v_lane = (uint32_t)((lane >> 4) * (D * 16) + (lane & 7) * 128 + ((((lane >> 3) & 1) ^ (lane & 7)) << 4));
  int gave_up_at = -1;                  // page index at which a stage wait expired

  for (int i = 0; i < n_pages; ++i) {
    const int pg = first_pg + DEC_WARPS * i;
    const int sg = i % ST;
    const bool page_ok = (ok_bits >> sg) & 1u;
    // ---- wait for the stage (bounded; on expiry flag and stop walking)
    {
      const bool ok = mbar_wait_bounded(smem_u32(&s_bar[warp][sg]), (i / ST) & 1, p.wait_ns, nullptr,
                                        lane == 0 ? p.status : nullptr);
      if (__any_sync(0xffffffffu, !ok)) {
        gave_up_at = i;
        break;
      }
    }
    const uint32_t k_page = ring + sg * 2 * PAGE_BYTES, v_page = k_page + PAGE_BYTES;
    if (page_ok) {
      const int left = end - (pg << 4);                     // keys of this page the chunk may see
      if (FUSED && append && pg == ((len - 1) >> 4)) {
        // The page of the new token: whatever the copy brought for its slot is replaced, in
        // shared memory, by the token's rotated k and its v; the CTA of the kv head's first
        // group tile also puts them into the pools.  (Other CTAs that read this page patch
        // their own copy the same way, so nobody depends on when the pool is written.)
        if (lane < VEC) {
          const int j = lane, slot = (len - 1) & 15;
          const uint4* krow = reinterpret_cast<const uint4*>(p.k_new + ((size_t)r * p.Hkv + kvh) * D);
          const uint4* vrow = reinterpret_cast<const uint4*>(p.v_new + ((size_t)r * p.Hkv + kvh) * D);
          uint4 kv = *(krow + j);
          if (cs_row) kv = dec_rotate_vec(kv, *(krow + (j ^ (VEC / 2))), cs_row, D, j, p.interleaved);
          const uint4 vv = *(vrow + j);
          uint8_t* kpage = ring_gen + (k_page - ring0);
          *reinterpret_cast<uint4*>(kpage + dec_page_off<D>(slot, j)) = kv;
          *reinterpret_cast<uint4*>(kpage + PAGE_BYTES + dec_page_off<D>(slot, j)) = vv;
          if (g0 == 0) {
            const int pid = *(bt + pg);
            const size_t off = (((size_t)pid * p.Hkv + kvh) * 16 + slot) * D + j * 8;
            *reinterpret_cast<uint4*>(p.k_pool_w + off) = kv;
            *reinterpret_cast<uint4*>(p.v_pool_w + off) = vv;
          }
        }
        __syncwarp();
      }
      if (left < 16) {
        // values of slots past the context are anything (NaN included): P is 0 there, 0 * NaN is not
        uint8_t* vpage = ring_gen + (v_page - ring0);
        for (int idx = left * VEC + lane; idx < 16 * VEC; idx += 32)
          *reinterpret_cast<uint4*>(vpage + dec_page_off<D>(idx / VEC, idx % VEC)) = make_uint4(0, 0, 0, 0);
        __syncwarp();
      }
      // ---- S^T: lane's tokens hq and hq + 8, heads 8 n + 2 tq + {0, 1}; two chains of k-steps
      float s[NT][4], s2[NT][4];
#pragma unroll
      for (int n = 0; n < NT; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) { s[n][e] = 0.f; s2[n][e] = 0.f; }
#pragma unroll
      for (int k = 0; k < KS; k += 2) {
        uint32_t a[4], b[4];
        ldsm4((k_page + k_lane + (k >> 2) * 1024) ^ ((k & 3) << 5), a);
        ldsm4((k_page + k_lane + (k >> 2) * 1024) ^ (((k & 3) + 1) << 5), b);
#pragma unroll
        for (int n = 0; n < NT; ++n) {
          mma16816(s[n], a, qf[n][k][0], qf[n][k][1]);
          mma16816(s2[n], b, qf[n][k + 1][0], qf[n][k + 1][1]);
        }
      }
      float mx[NT][2];
      bool grow = false;
#pragma unroll
      for (int n = 0; n < NT; ++n) {
#pragma unroll
        for (int e = 0; e < 4; ++e) s[n][e] = (s[n][e] + s2[n][e]) * p.scale_log2;
        if (left < 16) {
          if (hq >= left) s[n][0] = s[n][1] = -INFINITY;
          if (hq + 8 >= left) s[n][2] = s[n][3] = -INFINITY;
        }
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          mx[n][e] = fmaxf(s[n][e], s[n][e + 2]);
          grow |= mx[n][e] > m_ref[n][e] + 8.f;
        }
      }
      // Lazy rescale: the reference maximum of a head only moves when a score exceeds it by more
      // than 2^8 (always on the first page), so the lanes need not agree on every page's maximum.
      if (__any_sync(0xffffffffu, grow)) {
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            float x = mx[n][e];
#pragma unroll
            for (int off = 4; off < 32; off <<= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, off));
            const float m_new = fmaxf(m_ref[n][e], x);
            const float alpha = dec_ex2(m_ref[n][e] - m_new);
            m_ref[n][e] = m_new;
            l_part[n][e] *= alpha;
#pragma unroll
            for (int k = 0; k < KS; ++k) { o[n][k][e] *= alpha; o[n][k][e + 2] *= alpha; }
          }
      }
      // ---- P^T: exponentials, split into three bf16 terms, transposed into B fragments
      uint32_t pb[NT][3][2];
#pragma unroll
      for (int n = 0; n < NT; ++n) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float x0 = dec_ex2(s[n][2 * h] - m_ref[n][0]), x1 = dec_ex2(s[n][2 * h + 1] - m_ref[n][1]);
          l_part[n][0] += x0;
          l_part[n][1] += x1;
#pragma unroll
          for (int t = 0; t < 3; ++t) {
            const uint32_t w = pack_bf16x2(x0, x1);
            pb[n][t][h] = movm_t(w);
            x0 -= bf16lo(w);
            x1 -= bf16hi(w);
          }
        }
      }
      // ---- O^T
#pragma unroll
      for (int k = 0; k < KS; ++k) {
        uint32_t a[4];
        ldsm4_t((v_page + v_lane + (k >> 2) * 1024) ^ ((k & 3) << 5), a);
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
          for (int t = 0; t < 3; ++t) mma16816(o[n][k], a, pb[n][t][0], pb[n][t][1]);
      }
    }
    __syncwarp();                                     // everyone is done with the stage
    // ---- refill the stage with the page ST ahead
    const int nxt = i + ST;
    if (nxt < n_pages) {
      if ((nxt & 31) == 0) pid_cache = (nxt + lane < n_pages) ? *(bt + first_pg + DEC_WARPS * (nxt + lane)) : -1;
      ok_bits &= ~(1u << sg);
      if (issue(nxt)) ok_bits |= 1u << sg;
    }
  }

  if (gave_up_at >= 0) {
    // copies issued for the stages still in flight must land before the CTA's shared memory
    // is used for anything else or handed to another CTA
    for (int k = gave_up_at; k < min(gave_up_at + ST, n_pages); ++k)
      mbar_drain(smem_u32(&s_bar[warp][k % ST]), (k / ST) & 1);
  }
  // ---- fold the lanes' sums, then the 4 warps (their rings are quiet: the exchange buffer takes their place)
#pragma unroll
  for (int n = 0; n < NT; ++n)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
#pragma unroll
      for (int off = 4; off < 32; off <<= 1) l_part[n][e] += __shfl_xor_sync(0xffffffffu, l_part[n][e], off);
      if (lane < 4) {
        s_l[warp][n * 8 + 2 * lane + e] = l_part[n][e];
        s_m[warp][n * 8 + 2 * lane + e] = m_ref[n][e];
      }
    }
  __syncthreads();
  float* xo = reinterpret_cast<float*>(ring_gen);           // [warp][head][XD]
#pragma unroll
  for (int n = 0; n < NT; ++n)
#pragma unroll
    for (int k = 0; k < KS; ++k)
#pragma unroll
      for (int e = 0; e < 4; ++e)
        xo[(warp * GP + n * 8 + 2 * tq + (e & 1)) * XD + k * 16 + hq + (e >> 1) * 8] = o[n][k][e];
  __syncthreads();
  for (int idx = tid; idx < ng * (D / 4); idx += DEC_THREADS) {
    const int g = idx / (D / 4), d = (idx % (D / 4)) * 4;
    float M = s_m[0][g];
#pragma unroll
    for (int w = 1; w < DEC_WARPS; ++w) M = fmaxf(M, s_m[w][g]);
    float L = 0.f;
    float4 O = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int w = 0; w < DEC_WARPS; ++w) {
      const float sc = exp2f(s_m[w][g] - M);
      const float4 x = *reinterpret_cast<const float4*>(xo + (w * GP + g) * XD + d);
      L = fmaf(s_l[w][g], sc, L);
      O.x = fmaf(x.x, sc, O.x);
      O.y = fmaf(x.y, sc, O.y);
      O.z = fmaf(x.z, sc, O.z);
      O.w = fmaf(x.w, sc, O.w);
    }
    const float inv = L == 0.f ? 0.f : 1.f / L;             // no key of weight, or every page rejected: 0, -inf
    const float lse2 = L == 0.f ? -INFINITY : M + log2f(L); // (a sum of NaN stays NaN)
    if (L > 0.f && (O.x != O.x || O.y != O.y || O.z != O.z || O.w != O.w)) {
      const float4 x = mean_of_unbounded(p.v_pool, bt, p.num_pages, p.Hkv, kvh, D, d, begin, end,
                                         FUSED && append ? p.v_new + ((size_t)r * p.Hkv + kvh) * D : nullptr, len - 1);
      if (O.x != O.x) O.x = x.x;
      if (O.y != O.y) O.y = x.y;
      if (O.z != O.z) O.z = x.z;
      if (O.w != O.w) O.w = x.w;
    }
    const size_t row_head = (size_t)r * p.Hq + head0 + g;
    if (p.n_chunks == 1) {
      *reinterpret_cast<uint2*>(p.out + row_head * D + d) =
          make_uint2(pack_bf16x2(O.x * inv, O.y * inv), pack_bf16x2(O.z * inv, O.w * inv));
      if (p.lse && d == 0) p.lse[row_head] = lse2 * 0.6931471805599453f;
    } else {
      *reinterpret_cast<float4*>(p.part_o + (row_head * p.n_chunks + c) * D + d) =
          make_float4(O.x * inv, O.y * inv, O.z * inv, O.w * inv);
      if (d == 0) p.part_lse[row_head * p.n_chunks + c] = lse2;
    }
  }
}

// Merge the chunk partials of one (row, head): lse = log2 sum 2^lse_c,
// o = sum 2^(lse_c - lse) o_c.  WPR warps share one (row, head), each taking every WPR-th block of
// four chunks; lanes over head_dim.  Latency-bound on short steps: one warp for few chunks, four
// from 9 chunks on, where one warp's chain of dependent loads showed.  Launched programmatically, it is
// resident when the split kernel ends (1.7 us of a step of 1 row x 2.3k keys, 1 us at 16 rows).
template <int D, int WPR>
__global__ void __launch_bounds__(128) decode_merge_kernel(const DecodeParams p) {
  constexpr int EPL = D / 32;
  constexpr int RPB = 4 / WPR;                     // (row, head) pairs per CTA
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int part = warp % WPR;
  const size_t row_head = (size_t)blockIdx.x * RPB + warp / WPR;
  __shared__ float s_acc[WPR > 1 ? 4 : 1][WPR > 1 ? D + 1 : 1];
  // The row's length is an input of the step: the split kernel does not write it, and everything before
  // that kernel has completed, so it is looked up before the wait (in L2, where what has completed is
  // visible).  With the first partial rows fetched beside the maximum's lse values: steps of 1 to 64 rows in
  // chunks 0.7-1.0 us shorter (1 row x 2.3k keys 6.5 us, 16 rows x 2-2.9k 29.5).
  int nc = 0;
  if (row_head < (size_t)p.R * p.Hq) {
    const int len = min(__ldcg(p.row_len + row_head / p.Hq), p.key_cap);
    nc = min((len + p.chunk_tokens - 1) / p.chunk_tokens, p.n_chunks);
  }
  pdl_wait();
  pdl_launch();
  if (row_head >= (size_t)p.R * p.Hq) return;      // (WPR = 4: the whole CTA)
  const float* pl = p.part_lse + row_head * p.n_chunks;
  const float* po = p.part_o + row_head * p.n_chunks * D + lane * EPL;
  float L = 0.f, acc[EPL];
#pragma unroll
  for (int e = 0; e < EPL; ++e) acc[e] = 0.f;
  // partial rows c0 .. c0+3 and their lse values; the first four go out together with the maximum's loads
  float w[4];
  __align__(16) float v[4][EPL];
  auto fetch = [&](int c0) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (c0 + i < nc) {
        w[i] = pl[c0 + i];
        if constexpr (EPL == 4) {
          *reinterpret_cast<float4*>(v[i]) = *reinterpret_cast<const float4*>(po + (size_t)(c0 + i) * D);
        } else {
          *reinterpret_cast<float2*>(v[i]) = *reinterpret_cast<const float2*>(po + (size_t)(c0 + i) * D);
        }
      }
    }
  };
  fetch(4 * part);
  float M = -INFINITY;
  for (int c0 = 0; c0 < nc; c0 += 32)
    if (c0 + lane < nc) M = max_nan(M, pl[c0 + lane]);          // a NaN chunk makes the row NaN
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) M = max_nan(M, __shfl_xor_sync(0xffffffffu, M, d));
  if (!(M == -INFINITY)) {                         // else a row without keys, or every chunk came back empty
    for (int c0 = 4 * part; c0 < nc; c0 += 4 * WPR) {
      if (c0 != 4 * part) fetch(c0);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (c0 + i < nc) {
          const float wi = exp2f(w[i] - M);
          L += wi;
#pragma unroll
          for (int e = 0; e < EPL; ++e) acc[e] = fmaf(wi, v[i][e], acc[e]);
        }
      }
    }
  }
  if constexpr (WPR > 1) {
#pragma unroll
    for (int e = 0; e < EPL; ++e) s_acc[warp][lane * EPL + e] = acc[e];
    if (lane == 0) s_acc[warp][D] = L;
    __syncthreads();
    if (part != 0) return;
#pragma unroll
    for (int w = 1; w < WPR; ++w) {
      L += s_acc[w][D];
#pragma unroll
      for (int e = 0; e < EPL; ++e) acc[e] += s_acc[w][lane * EPL + e];
    }
  }
  const float inv = L == 0.f ? 0.f : 1.f / L;
  uint16_t* out = p.out + row_head * D + lane * EPL;
  if constexpr (EPL == 4) {
    *reinterpret_cast<uint2*>(out) = make_uint2(pack_bf16x2(acc[0] * inv, acc[1] * inv), pack_bf16x2(acc[2] * inv, acc[3] * inv));
  } else {
    *reinterpret_cast<uint32_t*>(out) = pack_bf16x2(acc[0] * inv, acc[1] * inv);
  }
  if (p.lse && lane == 0) p.lse[row_head] = L == 0.f ? -INFINITY : (M + log2f(L)) * 0.6931471805599453f;
}

// fp32 partials of `row_chunks` (row, chunk) pairs
static size_t part_o_size(long long row_chunks, int Hq, int D) { return (size_t)row_chunks * Hq * D * sizeof(float); }
static size_t part_lse_size(long long row_chunks, int Hq) { return ((size_t)row_chunks * Hq * sizeof(float) + 255) / 256 * 256; }

DecodePlan plan_decode(int rows, int Hq, int Hkv, int D, int max_len) {
  DecodePlan pl;
  const int G = Hq / Hkv;
  // Up to 16 query heads share one CTA's walk over the K/V pages; larger groups are cut evenly.
  pl.gsplit = (G + 15) / 16;
  pl.group_tile = (G + pl.gsplit - 1) / pl.gsplit;
  pl.gsplit = (G + pl.group_tile - 1) / pl.group_tile;
  if (max_len < 1) max_len = 1;
  // A CTA pays a few microseconds before its pages stream, and CTAs beyond the ones that are
  // resident together (slots) wait for a whole CTA to end: chunks of 2048 keys when even those
  // make several waves, else as many chunks as one wave holds, but neither shorter than 256 keys
  // (the merge then costs more than the split gains) nor longer than 1024 (ragged rows).  Steps of
  // 32/8 heads in microseconds at 256 / 384 / 768 / 1024 / 2048 keys: 1 row x 2.3k keys 9.0 / 10.1 /
  // 13.1 / 15.4 / 25; 4 rows x 2-2.9k 15.8 / 15.6 / 16.5 / 17.5 / 27; 16 rows 35.3 / 35.2 / 33.7 /
  // 31.4 / 34.4; 64 rows x 4-32k - / 636 / 611 / 603 / 596.
  // (decode_workspace_bound below follows these rules.)
  const long long slots = (long long)sm_count() * DEC_CTAS_PER_SM;
  const long long units = (long long)rows * Hkv * pl.gsplit;
  long long chunk = 2048;
  if (units * ((max_len + 2047) / 2048) < 4 * slots) {
    const long long n = std::max<long long>(1, slots / units);
    chunk = std::min<long long>(1024, std::max<long long>(256, (max_len + n - 1) / n));
    // Partials that the fixed array of efim_decode_attn_static holds, where longer chunks allow it: the two
    // entry points give the same bits, and the array's one takes whatever fits with chunks of 2048 keys.
    const long long per_chunk = (long long)rows * Hq * (D + 1) * (long long)sizeof(float);
    const long long n_fit = std::max<long long>(1, ((long long)DEC_STATIC_BYTES - 512) / per_chunk);
    if ((max_len + chunk - 1) / chunk > n_fit) chunk = std::min<long long>(2048, (max_len + n_fit - 1) / n_fit);
  }
  chunk = (chunk + 63) / 64 * 64;
  pl.chunk_tokens = (int)chunk;
  pl.n_chunks = (max_len + pl.chunk_tokens - 1) / pl.chunk_tokens;
  pl.part_o_bytes = pl.n_chunks > 1 ? part_o_size((long long)rows * pl.n_chunks, Hq, D) : 0;
  pl.part_lse_bytes = pl.n_chunks > 1 ? part_lse_size((long long)rows * pl.n_chunks, Hq) : 0;
  return pl;
}

// The most that a plan for at most `rows` rows of at most `max_len` keys needs.  The plans themselves are not
// monotone (32/8 heads, 2,048 keys: 221 rows 7.3 MB, 256 rows none), and a serving loop that sizes its
// workspace once has to get by as rows leave it.
static size_t decode_workspace_bound(int rows, int Hq, int Hkv, int D, int max_len) {
  if (max_len <= 256) return 0;                              // never cut
  const DecodePlan pl = plan_decode(rows, Hq, Hkv, D, max_len);
  const long long slots = (long long)sm_count() * DEC_CTAS_PER_SM, per_row = (long long)Hkv * pl.gsplit, r = rows;
  auto chunks = [&](long long keys) { return (max_len + keys - 1) / keys; };
  auto bytes = [&](long long row_chunks) { return part_o_size(row_chunks, Hq, D) + part_lse_size(row_chunks, Hq); };
  // (row, chunk) pairs of less than several waves: one wave of 256 to 1024 keys each, or chunks of 1024 keys that
  // are at most twice as many as the chunks of 2048 they replace - in either case what fits the static array
  const long long one_wave = std::min(r * chunks(256), slots / per_row);
  const long long of_1024 = std::min(r * chunks(1024), 2 * (4 * slots - 1) / per_row);
  return std::max(std::min(bytes(std::max(one_wave, of_1024)), DEC_STATIC_BYTES), bytes(r * chunks(2048)));
}

// The kernel's shared-memory size has to be raised once per device.
template <int D, int NT, bool FUSED>
static efim_status dec_raise_smem_limit() {
  constexpr int kMaxDevices = 64;
  static std::atomic<bool> done[kMaxDevices];
  int dev = 0;
  EFIM_CUDA_TRY(cudaGetDevice(&dev));
  if (dev >= 0 && dev < kMaxDevices && done[dev].load(std::memory_order_acquire)) return EFIM_OK;
  EFIM_CUDA_TRY(cudaFuncSetAttribute(decode_splitkv_kernel<D, NT, FUSED>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     dec_ring_bytes(D) + 1024));
  if (dev >= 0 && dev < kMaxDevices) done[dev].store(true, std::memory_order_release);
  return EFIM_OK;
}

template <int D, int NT, bool FUSED>
static efim_status launch_split(const efim_cache_desc* cache, const DecodeParams& p, dim3 grid, cudaStream_t s) {
  const CUtensorMap* pk = pf::pool_map(cache->d_k_pool, cache->num_pages, cache->num_kv_heads, D);
  if (!pk) return EFIM_ERR_CUDA;
  const CUtensorMap mk = *pk;
  const CUtensorMap* pv = pf::pool_map(cache->d_v_pool, cache->num_pages, cache->num_kv_heads, D);
  if (!pv) return EFIM_ERR_CUDA;
  const efim_status st = dec_raise_smem_limit<D, NT, FUSED>();
  if (st != EFIM_OK) return st;
  EFIM_CUDA_TRY(launch_pdl(decode_splitkv_kernel<D, NT, FUSED>, grid, dim3(DEC_THREADS), dec_ring_bytes(D) + 1024, s, p,
                           mk, *pv));
  return EFIM_OK;
}

template <int D>
static efim_status launch_decode_d(const efim_cache_desc* cache, const DecodeParams& p, const DecodePlan& pl,
                                   cudaStream_t s) {
  dim3 grid(p.R, p.Hkv * pl.gsplit, pl.n_chunks);
  efim_status st;
  if (pl.group_tile <= 8)
    st = p.fused ? launch_split<D, 1, true>(cache, p, grid, s) : launch_split<D, 1, false>(cache, p, grid, s);
  else
    st = p.fused ? launch_split<D, 2, true>(cache, p, grid, s) : launch_split<D, 2, false>(cache, p, grid, s);
  if (st != EFIM_OK) return st;
  if (pl.n_chunks > 1) {
    const size_t row_heads = (size_t)p.R * p.Hq;
    if (pl.n_chunks > 8)
      EFIM_CUDA_TRY(launch_pdl(decode_merge_kernel<D, 4>, dim3((unsigned)row_heads), dim3(128), 0, s, p));
    else
      EFIM_CUDA_TRY(launch_pdl(decode_merge_kernel<D, 1>, dim3((unsigned)((row_heads + 3) / 4)), dim3(128), 0, s, p));
  }
  return EFIM_OK;
}

static efim_status launch_decode(const efim_cache_desc* cache, const DecodeParams& p, const DecodePlan& pl,
                                 cudaStream_t s) {
  if (p.R == 0) return EFIM_OK;
  if ((long long)p.R * p.Hq > 2147483647LL || p.Hkv * pl.gsplit > 65535 || pl.n_chunks > 65535) return EFIM_ERR_UNSUPPORTED;
  return cache->head_dim == 128 ? launch_decode_d<128>(cache, p, pl, s) : launch_decode_d<64>(cache, p, pl, s);
}

}  // namespace efim

extern "C" size_t efim_decode_workspace_bytes(const efim_cache_desc* cache, int32_t batch, int32_t max_ctx_len) {
  if (efim::check_cache(cache) != EFIM_OK || batch <= 0) return 0;
  return efim::decode_workspace_bound(batch, cache->num_q_heads, cache->num_kv_heads, cache->head_dim, max_ctx_len);
}

extern "C" int32_t efim_decode_launch_count(const efim_cache_desc* cache, int32_t batch, int32_t max_ctx_len) {
  if (efim::check_cache(cache) != EFIM_OK || batch <= 0) return 0;
  const efim::DecodePlan pl = efim::plan_decode(batch, cache->num_q_heads, cache->num_kv_heads, cache->head_dim,
                                                max_ctx_len);
  return pl.n_chunks > 1 ? 2 : 1;
}

efim_status efim::decode_run(const efim_cache_desc* cache, int32_t batch, const int32_t* d_ctx_len,
                             int32_t max_ctx_len, const int32_t* d_block_table, int32_t max_pages_per_seq,
                             const efim_rope_desc* rope, const void* d_k_new, const void* d_v_new, bool fused,
                             const void* d_q, void* d_out, float* d_lse, float sm_scale, void* d_workspace,
                             size_t workspace_bytes, int32_t* d_status, void* stream, WorkspaceSource ws_source) {
  efim_status st = efim::check_cache(cache);
  if (st != EFIM_OK) return st;
  if (batch < 0 || max_pages_per_seq <= 0) return EFIM_ERR_INVALID_ARG;
  if (batch == 0) return EFIM_OK;
  if (!d_ctx_len || !d_block_table || !d_q || !d_out) return EFIM_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(d_q) | reinterpret_cast<uintptr_t>(d_out)) & 15) return EFIM_ERR_INVALID_ARG;
  const long long cap = (long long)max_pages_per_seq * cache->page_size;
  if (max_ctx_len <= 0) max_ctx_len = (int32_t)(cap > 2147483647LL ? 2147483647LL : cap);
  if (max_ctx_len > cap) return EFIM_ERR_OUT_OF_RANGE;
  const efim::DecodePlan pl = efim::plan_decode(batch, cache->num_q_heads, cache->num_kv_heads, cache->head_dim,
                                                max_ctx_len);
  const size_t need = pl.part_o_bytes + pl.part_lse_bytes;
  if (need > 0) {
    if (ws_source) {
      st = ws_source(&d_workspace, &workspace_bytes);
      if (st != EFIM_OK) return st;
    }
    if (!d_workspace || workspace_bytes < need) return EFIM_ERR_WORKSPACE;
    if (reinterpret_cast<uintptr_t>(d_workspace) & 255) return EFIM_ERR_INVALID_ARG;
  }
  efim::DecodeParams p{};
  p.q = static_cast<const uint16_t*>(d_q);
  p.row_len = d_ctx_len;
  p.block_table = d_block_table;
  p.out = static_cast<uint16_t*>(d_out);
  p.lse = d_lse;
  p.v_pool = static_cast<const uint16_t*>(cache->d_v_pool);
  p.part_lse = static_cast<float*>(d_workspace);
  p.part_o = need ? reinterpret_cast<float*>(static_cast<char*>(d_workspace) + pl.part_lse_bytes) : nullptr;
  p.status = d_status;
  p.R = batch;
  p.Hq = cache->num_q_heads;
  p.Hkv = cache->num_kv_heads;
  p.max_pages_per_seq = max_pages_per_seq;
  p.num_pages = cache->num_pages;
  p.group_tile = pl.group_tile;
  p.chunk_tokens = pl.chunk_tokens;
  p.n_chunks = pl.n_chunks;
  p.key_cap = (int)std::min<long long>((long long)pl.n_chunks * pl.chunk_tokens, cap);
  p.wait_ns = efim::WAIT_LIMIT_NS;
  const float scale = sm_scale > 0.f ? sm_scale : 1.0f / sqrtf((float)cache->head_dim);
  p.scale_log2 = scale * 1.4426950408889634f;
  if (fused) {
    if (!d_k_new || !d_v_new) return EFIM_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(d_k_new) | reinterpret_cast<uintptr_t>(d_v_new)) & 15) return EFIM_ERR_INVALID_ARG;
    p.fused = 1;
    p.k_new = static_cast<const uint16_t*>(d_k_new);
    p.v_new = static_cast<const uint16_t*>(d_v_new);
    p.k_pool_w = static_cast<uint16_t*>(cache->d_k_pool);
    p.v_pool_w = static_cast<uint16_t*>(cache->d_v_pool);
    if (rope && rope->d_cos_sin) {
      if (rope->max_position <= 0 || (reinterpret_cast<uintptr_t>(rope->d_cos_sin) & 15)) return EFIM_ERR_INVALID_ARG;
      p.cos_sin = rope->d_cos_sin;
      p.max_position = rope->max_position;
      p.interleaved = rope->interleaved;
    }
  }
  return efim::launch_decode(cache, p, pl, static_cast<cudaStream_t>(stream));
}

extern "C" efim_status efim_decode_attn(const efim_cache_desc* cache, int32_t batch, const int32_t* d_ctx_len,
                                        int32_t max_ctx_len, const int32_t* d_block_table,
                                        int32_t max_pages_per_seq, const void* d_q, void* d_out, float* d_lse,
                                        float sm_scale, void* d_workspace, size_t workspace_bytes,
                                        int32_t* d_status, void* stream) {
  return efim::decode_run(cache, batch, d_ctx_len, max_ctx_len, d_block_table, max_pages_per_seq, nullptr, nullptr,
                      nullptr, false, d_q, d_out, d_lse, sm_scale, d_workspace, workspace_bytes, d_status, stream);
}

extern "C" efim_status efim_decode_step(const efim_cache_desc* cache, int32_t batch, const int32_t* d_ctx_len,
                                        int32_t max_ctx_len, const int32_t* d_block_table,
                                        int32_t max_pages_per_seq, const efim_rope_desc* rope, const void* d_q,
                                        const void* d_k_new, const void* d_v_new, void* d_out, float* d_lse,
                                        float sm_scale, void* d_workspace, size_t workspace_bytes,
                                        int32_t* d_status, void* stream) {
  return efim::decode_run(cache, batch, d_ctx_len, max_ctx_len, d_block_table, max_pages_per_seq, rope, d_k_new,
                      d_v_new, true, d_q, d_out, d_lse, sm_scale, d_workspace, workspace_bytes, d_status, stream);
}
