// Tensor-core append-prefill attention for sm_100a (EFIM Sec. 1, Sec. 2.2: the new
// `inc` queries attend causally over the cached `<P>prefix<S>suffix<M>` keys and
// over each other).
//
// A work item is up to 256 packed query rows (row = token * G + head-in-group) of one
// (sequence, kv head) as two 128-row tiles; a CTA walks items and streams each one's visible K/V range in
// steps of 80 keys (5 pages):
//   warps 8,11 TMA producers (K tiles / V tiles): walk the block table, one tiled bulk-tensor
//             copy per page (16 slots x all dims of the kv head) into rings of 3 entries each
//             (8 at head_dim 64; 128B swizzle); warp 8 also claims the CTA's next item
//   warp 10   issues the tcgen05.mma for S_t = Q_t K^T into TMEM
//   warp 9    issues the tcgen05.mma for O_t += P_t V (P read from TMEM)
//   warps 0-7 two softmax groups ("streams"), one TMEM lane (row) per thread: S from TMEM, mask,
//             exp2 against the row's reference maximum, P (bf16) to TMEM beside S; final
//             normalisation and store
// Hand-offs are mbarriers; every wait is bounded and on expiry sets
// EFIM_DEV_TIMEOUT and lets all roles run out their (fixed) loop counts.
//
// Bound: with two query tiles the tensor core (2,048 cycles per 128 keys) and the exponential unit
// (128 x 256 of them, 16 per clock: 2,048 cycles) alike; with one tile the K/V bytes.  P used to
// take the place of S, so a stream's next scores had to wait for PV of this step (3,490 cycles per 128
// keys); with P in columns of its own they wait for nothing but their reader.  That, no row
// maximum per step after the first ones and the streams started half a step apart took 10 % off 8 x
// 3,200 tokens over 5k keys at 32/8 heads, 6 % off 8 x 128 over 8k and off prompts of 1-3.5k tokens, 3 %
// off 64 mixed rows at 28/4.
#include "prefill_tc.cuh"
#include "mbar.cuh"
#include <cfloat>
#include <vector>
#include <algorithm>
#include <functional>
#include <atomic>
#include <type_traits>

namespace efim {
namespace pf {

// ------------------------------------------------------------------ PTX wrappers
// Bounded wait (limit p.wait_ns): on expiry the CTA-wide abort flag goes up, after which
// every wait returns at once, and the timeout is recorded in the status word.
__device__ __forceinline__ void mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int32_t* status,
                                          unsigned long long limit_ns) {
  if (__builtin_expect(mbar_try(bar, parity), 1)) return;      // (what follows is laid out behind the loops)
  mbar_wait_bounded(bar, parity, limit_ns, abort_flag, status);
}
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// One lane of a converged warp.  (Asked for this way the compiler keeps an MMA's descriptors in uniform
// registers: an issuing thread then needs 48 cycles or less per tcgen05.mma, against 60 behind `lane == 0`;
// 16 rows x 2-8k keys at 32/32 heads 331 -> 318 us for append and attention.)
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
  return p != 0;
}
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// same with the A operand (P, bf16) read from tensor memory
__device__ __forceinline__ void umma_bf16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc,
                                             uint32_t accumulate) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d_tmem),
      "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// One (page, kv head) of a pool: coordinates (dim % 64, slot % 8, dim / 64, slot / 8, page * Hkv + head);
// the first four are always 0 here (the box covers them whole).
__device__ __forceinline__ void tma_load_page(uint32_t dst, const CUtensorMap* map, uint32_t bar, int page_head) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %3, %3, %3, %4}], "
      "[%2];" ::"r"(dst),
      "l"(map), "r"(bar), "r"(0), "r"(page_head)
      : "memory");
}

// tcgen05.ld / tcgen05.st of N consecutive columns of this warp's 32 lanes (cut into the widths the
// instructions have).
#define EFIM_R4(o) "=r"((r)[o]), "=r"((r)[o + 1]), "=r"((r)[o + 2]), "=r"((r)[o + 3])
#define EFIM_R16(o) EFIM_R4(o), EFIM_R4(o + 4), EFIM_R4(o + 8), EFIM_R4(o + 12)
#define EFIM_W4(o) "r"((r)[o]), "r"((r)[o + 1]), "r"((r)[o + 2]), "r"((r)[o + 3])
#define EFIM_W16(o) EFIM_W4(o), EFIM_W4(o + 4), EFIM_W4(o + 8), EFIM_W4(o + 12)
#define EFIM_L16 "%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15"
#define EFIM_S16 "%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16"
template <int N>
__device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t* r) {
  if constexpr (N >= 32) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {" EFIM_L16
                 ",%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                 : EFIM_R16(0), EFIM_R16(16)
                 : "r"(taddr));
    tmem_ld<N - 32>(taddr + 32, r + 32);
  } else if constexpr (N >= 16) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {" EFIM_L16 "}, [%16];" : EFIM_R16(0) : "r"(taddr));
    tmem_ld<N - 16>(taddr + 16, r + 16);
  } else if constexpr (N >= 4) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];" : EFIM_R4(0) : "r"(taddr));
    tmem_ld<N - 4>(taddr + 4, r + 4);
  } else {
    static_assert(N == 0, "columns are read in multiples of 4");
  }
}
template <int N>
__device__ __forceinline__ void tmem_st(uint32_t taddr, const uint32_t* r) {
  if constexpr (N >= 32) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {" EFIM_S16
                 ",%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr),
                 EFIM_W16(0), EFIM_W16(16)
                 : "memory");
    tmem_st<N - 32>(taddr + 32, r + 32);
  } else if constexpr (N >= 16) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {" EFIM_S16 "};" ::"r"(taddr), EFIM_W16(0) : "memory");
    tmem_st<N - 16>(taddr + 16, r + 16);
  } else if constexpr (N >= 8) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr), EFIM_W4(0),
                 EFIM_W4(4)
                 : "memory");
    tmem_st<N - 8>(taddr + 8, r + 8);
  } else if constexpr (N >= 2) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1,%2};" ::"r"(taddr), "r"(r[0]), "r"(r[1]) : "memory");
    tmem_st<N - 2>(taddr + 2, r + 2);
  } else {
    static_assert(N == 0, "columns are written in multiples of 2");
  }
}
#undef EFIM_R4
#undef EFIM_R16
#undef EFIM_W4
#undef EFIM_W16
#undef EFIM_L16
#undef EFIM_S16

__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// Waits for this thread's tcgen05.ld; the registers they fill are named so that no use of them can be
// moved before the wait (it costs no instruction).
template <int N>
__device__ __forceinline__ void tmem_wait_ld(uint32_t* r) {
  tmem_wait_ld();
#pragma unroll
  for (int i = 0; i < N; ++i) asm volatile("" : "+r"(r[i]));
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// two-wide fp32 arithmetic (one issue slot for two lanes of work)
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// Instruction descriptor: bf16 x bf16 -> fp32, M = 128, N = n, A K-major, B K- or MN-major.
__host__ __device__ constexpr uint32_t instr_desc(int n, int b_mn_major) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(b_mn_major) << 16) |
         (static_cast<uint32_t>(n >> 3) << 17) | (static_cast<uint32_t>(BM >> 4) << 24);
}

// barrier slots (8 bytes each) inside the BAR_OFF block, per stream or per ring entry
enum {
  BAR_Q = 0,         // query tile is in shared memory
  BAR_S = 2,         // scores of a step are in tensor memory
  BAR_SFREE = 4,     // ... and have been read by the softmax warps
  BAR_P = 6,         // probabilities of a step are in tensor memory (and O has been rescaled if need be)
  BAR_PV = 8,        // PV of a step has finished
  BAR_IFULL = 10,    // a work item is in the mailbox
  BAR_IEMPTY = 12,   // ... and has been read by the warps
  BAR_PAIR = 14,     // the two softmax warps that share 32 TMEM lanes
  BAR_ALL = 18,      // all softmax warps
  BAR_CLAIM = 19,    // the answer to a claim is in shared memory
  BAR_KFULL = 20, BAR_KEMPTY = 28, BAR_VFULL = 36, BAR_VEMPTY = 44,
  BAR_NEW = 52,      // the item's new k/v are in their pages
  BAR_COUNT = 53
};

// Shared-memory plan.  A query tile is [64-element half][128 rows][128 bytes]; a K or V tile
// is [8-key group][64-element half][8 keys][128 bytes], which is what one copy per page
// writes (a page is two key groups).  In both, 16-byte chunk c of row r is stored at chunk
// position c ^ (r & 7) (the 128B swizzle the tensor-map copies and the MMA descriptors use).
// K and V tiles have rings of their own: every ring barrier is waited on by one warp, phase after
// phase, from the CTA's first item to its last.  Three entries each at head_dim 128: more do not fit beside the output rows
// (and without those four each, or four of K, were no faster: 8 x 3,200 tokens over 5k keys 2,512 and 2,511 us against
// 2,484, 8 x 128 over 8k 150.5 and 152.5 against 149).
template <int D>
struct Smem {
  static constexpr int HALVES = D / 64;
  static constexpr int HALF_BYTES = 128 * 128;                  // 16 KB
  static constexpr int Q_BYTES = HALVES * HALF_BYTES;
  static constexpr int GROUP_BYTES = HALVES * 1024;             // 8 keys of a K/V tile, all dims
  static constexpr int PAGE_BYTES = 2 * GROUP_BYTES;            // one page = one copy
  static constexpr int KV_BYTES = BN / 16 * PAGE_BYTES;         // 20 KB at head_dim 128, 10 KB at 64
  static constexpr int NK = D == 128 ? 3 : 8, NV = NK;            // ring entries
  static constexpr int Q_OFF = 0;
  static constexpr int KV_OFF = Q_OFF + NQ * Q_BYTES;
  static constexpr int STAGE_OFF = KV_OFF + (NK + NV) * KV_BYTES;          // output rows on their way out, 4 KB per warp
  static constexpr int BAR_OFF = STAGE_OFF + 8 * 4096;
  static constexpr int TMEM_SLOT_OFF = BAR_OFF + BAR_COUNT * 8, ABORT_OFF = TMEM_SLOT_OFF + 8;
  static constexpr int ITEM_OFF = (ABORT_OFF + 8 + 15) / 16 * 16;          // mailbox: two work items
  static constexpr int CLAIM_OFF = ITEM_OFF + 2 * 48;                     // answer to a claim
  // Exchange of the 32-row shape: the four quarters' O in the query tiles' space, (reference, sum) here.
  static_assert(4 * 32 * D * 4 <= NQ * Q_BYTES, "the quarters' states must fit in the query tiles");
  static constexpr int ML_OFF = CLAIM_OFF + 16;
  static constexpr int TOTAL = ML_OFF + 4 * 32 * 8 + 1024;                // + alignment slack
  static_assert(TOTAL <= 227 * 1024, "shared memory of a CTA");
  // tensor memory: [S | P] of each stream, then O of each
  static constexpr int SP_COLS = 128;
  static_assert(BN + BN / 2 <= SP_COLS && NQ * (SP_COLS + D) <= 512, "tensor memory has 512 columns");
};
// A step's probabilities are taken relative to the reference maximum of the steps before; a row whose
// sum of one step leaves this range (2^8) takes its exact maximum as the new reference and redoes the
// step.  So no probability that enters PV is above 2^8 (O stays finite for |v| up to 2^120 / keys), and a
// key far above the ones before it has the probability 1, which bf16 holds exactly: with 2^40 here the
// outputs of peaked rows (scores of 8 sigma) were off by 2.0e-3 to 2.25e-3 (2-norm) instead of 1.7e-3.
constexpr float SUM_LIMIT = 256.f;
// The reference is the row's exact maximum over the first EXACT_STEPS steps of a stream, or over the first one
// where two query tiles see more than EXACT_MAX_STEPS steps.  The key at the reference is weighted without
// rounding and short rows live on their heaviest keys: with one step everywhere, 16 tokens over 240 at 4/4 x 64
// were off by 2.10e-3 instead of 2.00e-3 (2-norm, scores of 1 sigma), 60 over 1,000 at 32/8 by 2.293e-3 instead
// of 2.252e-3.  It costs a rescale of O (16 prompts of 1-3.5k tokens 1009 -> 1015 us; in every row block 3 %); in long
// rows the heaviest key is hardly ever among the first 160.
constexpr int EXACT_STEPS = 2, EXACT_MAX_STEPS = 12;

// Moves a row's reference `m_ref` up to the score `mx`; returns the factor that O and the row's sum take on.
// A reference starts at -FLT_MAX and stays finite where the row has seen no key or infinitely low scores
// only: those keys' probabilities are 0 against it, and the first finite score to come is above it or
// overflows its step's sum.
__device__ __forceinline__ float move_reference(float& m_ref, float mx) {
  const float m_new = fmaxf(m_ref, mx);
  const float alpha = m_new == m_ref ? 1.f : ex2(m_ref - m_new);
  m_ref = m_new;
  return alpha;
}

// O row of every lane of the warp *= alpha (the rare rescale of the 32-row shape; kept out
// of line so that its 32 registers do not count against the loop that calls it).
template <int D>
__device__ __noinline__ void rescale_o_row(uint32_t o_addr, float alpha) {
#pragma unroll
  for (int c0 = 0; c0 < D; c0 += 32) {
    uint32_t o[32];
    tmem_ld<32>(o_addr + c0, o);
    tmem_wait_ld<32>(o);
#pragma unroll
    for (int c = 0; c < 32; ++c) o[c] = __float_as_uint(__uint_as_float(o[c]) * alpha);
    tmem_st<32>(o_addr + c0, o);
  }
}

// One arrival for a whole warp, after every lane has done its part.
__device__ __forceinline__ void warp_arrive(uint32_t bar, int lane) {
  __syncwarp();
  if (lane == 0) mbar_arrive(bar);
}

// Largest of N scores (4 chains).
template <int N>
__device__ __forceinline__ float row_max(const uint32_t* s) {
  float mx[4];
#pragma unroll
  for (int a = 0; a < 4; ++a) mx[a] = __uint_as_float(s[a]);
#pragma unroll
  for (int c = 4; c < N; c += 4)
#pragma unroll
    for (int a = 0; a < 4; ++a) mx[a] = fmaxf(mx[a], __uint_as_float(s[c + a]));
  return fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
}
// w = bf16 pairs of p_c = 2^(scale s_c + neg_m), returns their sum (fp32).  The sum runs two-wide, the
// multiply-add one at a time (two-wide: 8 x 3,200 tokens over 5k 2.61 instead of 2.45 ms; a sum of
// single adds: 2.57).
template <int N>
__device__ __forceinline__ float row_exp(const uint32_t* s, float scale, float neg_m, uint32_t* w) {
  uint64_t ls[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
  for (int e = 0; e < N / 2; ++e) {
    const float p0 = ex2(fmaf(__uint_as_float(s[2 * e]), scale, neg_m));
    const float p1 = ex2(fmaf(__uint_as_float(s[2 * e + 1]), scale, neg_m));
    ls[e & 3] = add2(ls[e & 3], pack2(p0, p1));
    w[e] = pack_bf16x2(p0, p1);
  }
  float lo, hi;
  unpack2(add2(add2(ls[0], ls[1]), add2(ls[2], ls[3])), lo, hi);
  return lo + hi;
}

// 32 query rows (lane i knows row i: its index `th` in the packed [token * Hq + head] rows, or -1 for
// a row past the sequence, and its position) into rows row0 .. row0+31 of a shared-memory query tile
// (swizzled), zeros for absent rows; with a rotary table every row is rotated by its position on the
// way (the arithmetic of efim_kv_append).  The warp reads whole rows, 32 * 16 bytes of them per
// instruction: with a row per lane every instruction touched 32 lines (16 prompts of 1-3.5k tokens,
// whose CTAs have some 16 steps, lost 13 us to that).
template <int D>
__device__ __noinline__ void q_rows_rotated_to_smem(const uint4* q, const float* cos_sin, int max_position, int interleaved,
                                                    int32_t* status, uint8_t* tile, int row0, int lane, int th, int pos) {
  using L = Smem<D>;
  constexpr int VEC = D / 8, RPI = 32 / VEC;                 // 16-byte vectors per row, rows per instruction
  const int c = lane % VEC, sub = lane / VEC;
  if (th >= 0 && pos >= max_position) {                      // no table row: reported, attends with a zero query (finite)
    if (status) atomicOr(status, EFIM_DEV_BAD_POSITION);
    th = -1;
  }
  // The loads of two instructions' rows are on their way together (a store between them would keep the second's back), and both
  // halves of a row go through the same code: the warp's lanes hold vectors of either.  One at a time, a branch per half: 16
  // prompts of 1-3.5k tokens 1,022 us for append and attention, 53 x 1-406 over 100-549 at 24/8 heads 119, 16 over 240 at
  // 4/4 x 64 7.8; this: 920, 97, 7.5; with a branch per half 945, 101, 8.0, and four at a time 995, 95, -.  (20 x 1 over 0 at 32/32:
  // 33.9; 36 with groups without rows rotated too; 32.)
  constexpr int AT_ONCE = 2;
  const int cs_off = interleaved ? c * 4 : (c % (VEC / 2)) * 8;
  const uint32_t flip = c < VEC / 2 ? 0x80000000u : 0u;
  uint32_t have = __ballot_sync(0xffffffffu, th >= 0);
#pragma unroll 1
  for (int i0 = 0; i0 < VEC; i0 += AT_ONCE, have >>= AT_ONCE * RPI) {
    uint4 v[AT_ONCE], o[AT_ONCE];
#pragma unroll
    for (int b = 0; b < AT_ONCE; ++b) v[b] = make_uint4(0, 0, 0, 0);
    if (have & ((1u << AT_ONCE * RPI) - 1)) {               // (none in most of a block of one token's rows)
      float4 cf[AT_ONCE][2], sf[AT_ONCE][2];
#pragma unroll
      for (int b = 0; b < AT_ONCE; ++b) {
        const int t = __shfl_sync(0xffffffffu, th, (i0 + b) * RPI + sub), ps = __shfl_sync(0xffffffffu, pos, (i0 + b) * RPI + sub);
        o[b] = v[b];
        cf[b][0] = cf[b][1] = sf[b][0] = sf[b][1] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (t >= 0) {
          const uint4* src = q + (size_t)t * VEC;
          const float4* cs = reinterpret_cast<const float4*>(cos_sin + (size_t)ps * D + cs_off);
          v[b] = src[c];
          cf[b][0] = cs[0];
          sf[b][0] = cs[D / 8];
          if (!interleaved) {
            o[b] = src[c ^ (VEC / 2)];
            cf[b][1] = cs[1];
            sf[b][1] = cs[D / 8 + 1];
          }
        }
      }
#pragma unroll
      for (int b = 0; b < AT_ONCE; ++b) {
        const float *cp = reinterpret_cast<const float*>(cf[b]), *sp = reinterpret_cast<const float*>(sf[b]);
        if (interleaved) rotate4_interleaved(v[b], cp, sp);
        else rotate_half(v[b], o[b], cp, sp, flip);
      }
    }
#pragma unroll
    for (int b = 0; b < AT_ONCE; ++b) {
      const int r = row0 + (i0 + b) * RPI + sub;
      *reinterpret_cast<uint4*>(tile + (c >> 3) * L::HALF_BYTES + r * 128 + (((c & 7) ^ (r & 7)) << 4)) = v[b];
    }
  }
}
template <int D>
__device__ __forceinline__ void q_rows_to_smem(const Params& p, uint8_t* smem_gen, int tile_off, uint32_t smem_base, int row0,
                                               int lane, int th, int pos) {
  using L = Smem<D>;
  constexpr int VEC = D / 8, RPI = 32 / VEC;
  if (p.cos_sin != nullptr) {
    q_rows_rotated_to_smem<D>(reinterpret_cast<const uint4*>(p.q), p.cos_sin, p.max_position, p.interleaved, p.status,
                              smem_gen + tile_off, row0, lane, th, pos);
    return;
  }
  const int c = lane % VEC, sub = lane / VEC;
#pragma unroll 1                                            // (see the note on cold code at softmax_item)
  for (int i = 0; i < VEC; ++i) {
    const int t = __shfl_sync(0xffffffffu, th, i * RPI + sub);
    const int r = row0 + i * RPI + sub;
    const uint4* src = reinterpret_cast<const uint4*>(p.q) + (size_t)max(t, 0) * VEC + c;
    const uint32_t dst = smem_base + tile_off + (c >> 3) * L::HALF_BYTES + r * 128 + (((c & 7) ^ (r & 7)) << 4);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(t >= 0 ? 16 : 0) : "memory");
  }
}

// The N new k (rotated) and v rows of one (sequence, kv head) into their page slots, by 128 threads: the arithmetic and
// the checks of efim_kv_append.  Afterwards they may be read by bulk-tensor copies.
template <int D>
__device__ __noinline__ void append_rows(const uint4* k_new, const uint4* v_new, uint4* k_pool, uint4* v_pool, const int32_t* bt,
                                         const float* cos_sin, int max_position, int interleaved, int32_t* status, int max_pages,
                                         int num_pages, int Hkv, int kvh, int C, int N, int tok0, int t) {
  constexpr int VEC = D / 8;
  for (int u = t; u < N * VEC; u += 128) {
    const int i = u / VEC, j = u % VEC, pos = C + i;
    int err = 0, page = -1;
    if ((pos >> 4) >= max_pages || (cos_sin && pos >= max_position)) {
      err = EFIM_DEV_BAD_POSITION;
    } else {
      page = bt[pos >> 4];
      if (page < 0 || page >= num_pages) err = EFIM_DEV_BAD_PAGE;
    }
    if (err) {
      if (j == 0 && status) atomicOr(status, err);
      continue;
    }
    const size_t src = ((size_t)(tok0 + i) * Hkv + kvh) * VEC;
    uint4 k = k_new[src + j];
    const uint4 v = v_new[src + j];
    if (cos_sin) {
      const float* cs = cos_sin + (size_t)pos * D;
      if (!interleaved) {
        uint4 o = k_new[src + (j ^ (VEC / 2))];
        const float* cp = cs + (j % (VEC / 2)) * 8;
        float cf[8], sf[8];
        *reinterpret_cast<float4*>(cf) = *reinterpret_cast<const float4*>(cp);
        *reinterpret_cast<float4*>(cf + 4) = *reinterpret_cast<const float4*>(cp + 4);
        *reinterpret_cast<float4*>(sf) = *reinterpret_cast<const float4*>(cp + D / 2);
        *reinterpret_cast<float4*>(sf + 4) = *reinterpret_cast<const float4*>(cp + D / 2 + 4);
        if (j < VEC / 2) rotate8(k, o, cf, sf);
        else rotate8(o, k, cf, sf);
      } else {
        float cf[4], sf[4];
        *reinterpret_cast<float4*>(cf) = *reinterpret_cast<const float4*>(cs + j * 4);
        *reinterpret_cast<float4*>(sf) = *reinterpret_cast<const float4*>(cs + D / 2 + j * 4);
        rotate4_interleaved(k, cf, sf);
      }
    }
    const size_t dst = (((size_t)page * Hkv + kvh) * 16 + (pos & 15)) * VEC + j;
    k_pool[dst] = k;
    v_pool[dst] = v;
  }
  __threadfence();
  asm volatile("fence.proxy.async;" ::: "memory");           // the copies read what ordinary stores wrote
}

// Two softmax groups ("streams") run per CTA.  With more than 128 rows, stream t
// owns query tile t and both walk every step of BN keys.  With 128 rows or fewer there is
// one query tile; stream 0 takes the even steps and stream 1 the odd ones, each
// with its own reference, sum and O, and the two states are merged at the end -
// the tensor core then still works on one stream while the other does its softmax.
//
// SHAPE_ONE: one query tile (33..128 rows); SHAPE_TWO: two query tiles; SHAPE_TINY: at most 32 rows (one-token
// rows of a mixed batch, short `inc`s): the one query tile holds the rows four times, once per 32-lane
// quarter, and the softmax warp of quarter w takes keys 20w..20w+19 (BN / 4) of every step with a
// reference, sum and O of its own - a quarter of the exponentials per thread and step, so the
// two alternating streams turn a step round in about half the time; the eight states of a row
// (2 streams x 4 quarters) are merged at the end.
enum { SHAPE_ONE = 0, SHAPE_TWO = 1, SHAPE_TINY = 2 };

// A work item as the roles use it.  Every value is the same in all lanes, and the compiler has to know it: loop
// bounds, ring positions and with them the MMAs' descriptors stay in uniform registers only then.  (The same holds
// for the warp's index, which the roles branch on: taken from threadIdx as it is, the loops were compiled for
// diverging lanes - twice the convergence instructions, and 8 x 3,200 tokens over 5k keys at 32/8 heads took 2.81 ms,
// 8 x 128 over 8k 165 us, against 2.51 ms and 150 us.)
struct Work {
  int seq, kvh, chunk, row0, C, tok0, rows_total;
  int key0, kv_cap, nt;        // keys [key0, kv_cap): the tiles of the item, up to what its last row sees; steps of BN keys
  int shape;
  __device__ __forceinline__ int steps(int st) const {
    return shape == SHAPE_TWO ? nt : (st == 0 ? (nt + 1) >> 1 : nt >> 1);
  }
};
__device__ __forceinline__ int uniform(int x) {
  return static_cast<int>(__reduce_or_sync(0xffffffffu, static_cast<unsigned>(x)));
}
// Token of packed row R (R / G, without a division).
__device__ __forceinline__ int token_of(const Params& p, int R) {
  if (p.g_mul == 0) return R;
  const int t = static_cast<int>(__umulhi(static_cast<unsigned>(R), p.g_mul));
  return t * p.G > R ? t - 1 : t;
}
__device__ __forceinline__ Work work_of(const WorkItem& it, const Params& p) {
  Work w;
  w.seq = uniform(it.seq);
  const int kc = uniform((int)(uint16_t)it.kvh | (int)it.chunk << 16);
  w.kvh = (int)(int16_t)(kc & 0xffff);
  w.chunk = kc >> 16;
  w.row0 = uniform(it.row0);
  w.C = uniform(it.cached);
  w.tok0 = uniform(it.tok0);
  w.rows_total = uniform(it.new_len) * p.G;
  const int rows_here = min(NQ * BM, w.rows_total - w.row0);
  const int i_last = token_of(p, w.row0 + rows_here - 1);    // last token of this item
  w.key0 = uniform(it.tile_begin) * PT;
  w.kv_cap = min(w.C + i_last + 1, uniform(it.tile_end) * PT);
  w.nt = (w.kv_cap - w.key0 + BN - 1) / BN;
  w.shape = rows_here > BM ? SHAPE_TWO : (rows_here <= 32 ? SHAPE_TINY : SHAPE_ONE);
  return w;
}

// What every role of a CTA knows.
template <int D>
struct Cta {
  using L = Smem<D>;
  const Params& p;
  uint32_t smem_base;
  uint8_t* smem_gen;
  volatile int* abort_flag;
  const CUtensorMap *map_q, *map_out;
  uint32_t tmem_S, tmem_P, tmem_O;       // S of stream t at columns t * SP_COLS, P (bf16 pairs) behind it; O of stream t at t * D
  int lane;
  __device__ __forceinline__ uint32_t bar(int i) const { return smem_base + L::BAR_OFF + 8u * i; }
  // The loop of a wait stands behind the code that it is called from at head_dim 128 only: at 64 a step of two tiles took 11 % longer
  // so (37 x 256 tokens over 4,000 keys at 4/4 heads 71.6 us, with the loop in place and the other register split 65.6).
  __device__ __forceinline__ void wait(int b, uint32_t parity) const {
    if constexpr (D == 128) mbar_wait(bar(b), parity, abort_flag, p.status, p.wait_ns);
    else mbar_wait_bounded(bar(b), parity, p.wait_ns, abort_flag, p.status);
  }
};

// The item after the present one, from the mailbox that warp 8 fills; false: there is none, or the CTA has given up.
// Every warp but warp 8 reads every slot, so a slot is free again after 11 arrivals.
struct Mailbox {
  int slot = 0;
  uint32_t phase = 0;
  template <int D>
  static __device__ __forceinline__ uint4* at(const Cta<D>& c, int slot) {
    return reinterpret_cast<uint4*>(c.smem_gen + Smem<D>::ITEM_OFF) + 3 * slot;
  }
  template <int D>
  __device__ __forceinline__ void put(const Cta<D>& c, const Work& w) {    // by warp 8; seq -1: no more items
    c.wait(BAR_IEMPTY + slot, phase ^ 1);
    if (c.lane == 0) {
      uint4* dst = at(c, slot);
      dst[0] = make_uint4(w.seq, (uint32_t)(uint16_t)w.kvh | (uint32_t)w.chunk << 16, w.row0, w.C);
      dst[1] = make_uint4(w.tok0, w.rows_total, w.key0, w.kv_cap);
      dst[2] = make_uint4((uint32_t)w.nt << 2 | (uint32_t)w.shape, 0, 0, 0);
      mbar_arrive(c.bar(BAR_IFULL + slot));
    }
    __syncwarp();
    if (++slot == 2) { slot = 0; phase ^= 1; }
  }
  template <int D>
  __device__ __forceinline__ bool next(const Cta<D>& c, Work& w) {
    c.wait(BAR_IFULL + slot, phase);
    const uint4* src = at(c, slot);
    const uint4 a = src[0], b = src[1];
    const int ns = uniform(src[2].x), seq = uniform(a.x), kc = uniform(a.y);
    const bool gone = __any_sync(0xffffffffu, *c.abort_flag != 0);
    warp_arrive(c.bar(BAR_IEMPTY + slot), c.lane);
    if (++slot == 2) { slot = 0; phase ^= 1; }
    w.seq = seq;
    w.kvh = (int)(int16_t)(kc & 0xffff);
    w.chunk = kc >> 16;
    w.row0 = uniform(a.z);
    w.C = uniform(a.w);
    w.tok0 = uniform(b.x);
    w.rows_total = uniform(b.y);
    w.key0 = uniform(b.z);
    w.kv_cap = uniform(b.w);
    w.nt = ns >> 2;
    w.shape = ns & 3;
    return !gone && seq >= 0;
  }
};

// Claim of one more item: a CTA of this launch that has not started is taken out of it and its block index handed over
// (cluster launch control); the answer is written to shared memory.
__device__ __forceinline__ void claim_next(uint32_t answer, uint32_t bar) {
  asm volatile("clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.b128 [%0], [%1];" ::"r"(answer),
               "r"(bar)
               : "memory");
}
__device__ __forceinline__ int claimed_block(uint32_t answer) {   // -1: there was none left
  uint32_t ok, x;
  asm volatile(
      "{\n.reg .b128 a;\n.reg .pred p;\n"
      "ld.shared.b128 a, [%2];\n"
      "clusterlaunchcontrol.query_cancel.is_canceled.pred.b128 p, a;\n"
      "selp.u32 %0, 1, 0, p;\nmov.u32 %1, 0;\n"
      "@p clusterlaunchcontrol.query_cancel.get_first_ctaid::x.b32.b128 %1, a;\n}\n"
      : "=r"(ok), "=r"(x)
      : "r"(answer)
      : "memory");
  return ok ? static_cast<int>(x) : -1;
}

// This lane's query row of tile `qt`, quarter `w` (SHAPE_TINY: the same 32 rows in every quarter).
struct Row {
  bool valid;
  int pos, th;                 // position; index of the (token, head) row in q, out and lse, -1 for a row past the sequence
  __device__ __forceinline__ Row(const Params& p, const Work& it, int qt, int w, int lane) {
    const int R = it.row0 + (it.shape == SHAPE_TINY ? lane : qt * BM + w * 32 + lane);
    valid = R < it.rows_total;
    const int i_tok = valid ? token_of(p, R) : 0;
    pos = it.C + i_tok;
    th = valid ? (it.tok0 + i_tok) * p.Hq + it.kvh * p.G + (R - i_tok * p.G) : -1;
  }
};
// 32 rows x 64 dims between a [token][head][dim] array and shared memory (128-byte swizzle): one box is the G heads of
// 32 / G tokens.  Coordinates (dim % 64, dim / 64, head, token); tokens past the end read as zeros.
__device__ __forceinline__ void tma_load_rows(uint32_t dst, const CUtensorMap* map, uint32_t bar, int half, int head, int token) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];" ::"r"(dst),
      "l"(map), "r"(bar), "r"(0), "r"(half), "r"(head), "r"(token)
      : "memory");
}
__device__ __forceinline__ void tma_store_rows(uint32_t src, const CUtensorMap* map, int half, int head, int token) {
  asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%1, {%2, %3, %4, %5}], [%0];" ::"r"(src), "l"(map),
               "r"(0), "r"(half), "r"(head), "r"(token)
               : "memory");
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}

// The query rows of a tile, by the four warps of a stream, each its 32-lane quarter.  Where 32 rows are whole tokens they
// are copied as boxes: per-lane copies kept the softmax warps for 2,300 cycles per item of prompts.  (Rows past the sequence then
// hold what follows it; nothing of theirs is stored, nor heard by the steps.)
template <int D>
__device__ __forceinline__ void fetch_q(const Cta<D>& c, const Work& it, int qt, int w) {
  using L = Smem<D>;
  if (c.p.q_tma) {
    if (c.lane == 0) {
      const uint32_t bar = c.bar(BAR_Q + qt), dst = c.smem_base + L::Q_OFF + qt * L::Q_BYTES + w * 4096;
      const int token = it.tok0 + token_of(c.p, it.row0 + (it.shape == SHAPE_TINY ? 0 : qt * BM + w * 32));
      mbar_expect_tx(bar, L::HALVES * 4096);
#pragma unroll
      for (int h = 0; h < L::HALVES; ++h) tma_load_rows(dst + h * L::HALF_BYTES, c.map_q, bar, h, it.kvh * c.p.G, token);
    }
    __syncwarp();
    return;
  }
  const Row r(c.p, it, qt, w, c.lane);
  q_rows_to_smem<D>(c.p, c.smem_gen, L::Q_OFF + qt * L::Q_BYTES, c.smem_base, w * 32, c.lane, r.th, r.pos);
}
template <int D>
__device__ __forceinline__ void publish_q(const Cta<D>& c, int qt) {
  if (c.p.q_tma) return;                                    // (the copies complete the barrier)
  asm volatile("cp.async.wait_all;" ::: "memory");
  fence_async_smem();
  warp_arrive(c.bar(BAR_Q + qt), c.lane);
}

// 64 columns (from `col` on) of this warp's 32 output rows, or of a chunk's partials; `th` as in Row, `whole`: all 32
// rows are of the sequence, from `token` on.  The rows leave through 4 KB of shared memory, as one box, or else 128 bytes
// of four rows per instruction.  (With a row per lane every store touched 32 lines: 4,200 cycles per item of
// prompts.  Boxes against instructions only: 16 prompts of 1-3.5k tokens 935 and 954 us.)
template <int D>
__device__ __forceinline__ void store_cols(const Cta<D>& c, const Work& it, int warp, int token, int th, bool whole, int col,
                                           const float* f) {
  const Params& p = c.p;
  const uint32_t off = Smem<D>::STAGE_OFF + warp * 4096;
  auto slot_of = [&](int row, int j) {
    return reinterpret_cast<uint4*>(c.smem_gen + off + row * 128 + ((j ^ (row & 7)) << 4));
  };
  const int j = c.lane & 7, sub = c.lane >> 3;
  if (c.lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");     // (what left last has been read)
  __syncwarp();
  if (it.chunk < 0) {
#pragma unroll
    for (int i = 0; i < 8; ++i)
      *slot_of(c.lane, i) = make_uint4(pack_bf16x2(f[8 * i], f[8 * i + 1]), pack_bf16x2(f[8 * i + 2], f[8 * i + 3]),
                                       pack_bf16x2(f[8 * i + 4], f[8 * i + 5]), pack_bf16x2(f[8 * i + 6], f[8 * i + 7]));
    if (whole && p.out_tma) {
      fence_async_smem();
      __syncwarp();
      if (c.lane == 0) tma_store_rows(c.smem_base + off, c.map_out, col / 64, it.kvh * p.G, token);
    } else {
      __syncwarp();
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int t = __shfl_sync(0xffffffffu, th, i * 4 + sub);
        const uint4 x = *slot_of(i * 4 + sub, j);
        if (t >= 0) *reinterpret_cast<uint4*>(p.out + (size_t)t * D + col + j * 8) = x;
      }
    }
  } else {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
#pragma unroll
      for (int i = 0; i < 8; ++i)
        *slot_of(c.lane, i) = make_uint4(__float_as_uint(f[32 * h + 4 * i]), __float_as_uint(f[32 * h + 4 * i + 1]),
                                         __float_as_uint(f[32 * h + 4 * i + 2]), __float_as_uint(f[32 * h + 4 * i + 3]));
      __syncwarp();
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int t = __shfl_sync(0xffffffffu, th, i * 4 + sub);
        const uint4 x = *slot_of(i * 4 + sub, j);
        if (t >= 0) *reinterpret_cast<uint4*>(p.part_o + ((size_t)t * p.s_max + it.chunk) * D + col + h * 32 + j * 4) = x;
      }
      __syncwarp();
    }
  }
}
__device__ __forceinline__ void store_lse(const Params& p, int th, int chunk, float lse2) {
  if (th < 0) return;
  if (chunk >= 0) {
    p.part_lse[(size_t)th * p.s_max + chunk] = lse2;
  } else if (p.lse) {
    p.lse[th] = lse2 * 0.6931471805599453f;
  }
}

// The states (reference, sum) of a row's two streams: the lane of stream 0 and the one of stream 1 that share the TMEM
// lane swap theirs through two dead columns of P.  Afterwards the partner's O may be read too (its PV MMAs are done).
struct Pair {
  float M, L, w0, w1;          // common reference and sum, weights of the two O
};
template <int D>
__device__ __forceinline__ Pair meet_partner(const Cta<D>& c, int st, int w, uint32_t lane_addr, float m_ref, float l_sum,
                                             uint32_t& pair_phase) {
  using L = Smem<D>;
  const uint32_t mine[2] = {__float_as_uint(m_ref), __float_as_uint(l_sum)};
  tmem_st<2>(c.tmem_P + lane_addr + st * L::SP_COLS, mine);
  tmem_wait_st();
  tc_fence_before();
  warp_arrive(c.bar(BAR_PAIR + w), c.lane);
  c.wait(BAR_PAIR + w, pair_phase);
  pair_phase ^= 1;
  tc_fence_after();
  uint32_t o[4];
  tmem_ld<4>(c.tmem_P + lane_addr + (st ^ 1) * L::SP_COLS, o);
  tmem_wait_ld<4>(o);
  const float m0 = st == 0 ? m_ref : __uint_as_float(o[0]), l0 = st == 0 ? l_sum : __uint_as_float(o[1]);
  const float m1 = st == 1 ? m_ref : __uint_as_float(o[0]), l1 = st == 1 ? l_sum : __uint_as_float(o[1]);
  Pair r;
  r.M = fmaxf(m0, m1);
  r.w0 = l0 == 0.f ? 0.f : ex2(m0 - r.M);
  r.w1 = l1 == 0.f ? 0.f : ex2(m1 - r.M);
  r.L = l0 * r.w0 + l1 * r.w1;
  return r;
}
// Before either of a pair may go on and let its stream's O be overwritten, both have read what they need.
template <int D>
__device__ __forceinline__ void leave_partner(const Cta<D>& c, int w, uint32_t& pair_phase) {
  tc_fence_before();
  warp_arrive(c.bar(BAR_PAIR + w), c.lane);
  c.wait(BAR_PAIR + w, pair_phase);
  pair_phase ^= 1;
  tc_fence_after();
}

// ------------------------------------------------------------------ softmax groups
// One item of at most 32 rows; `n`: steps of this stream so far.
template <int D>
__device__ __forceinline__ void softmax_tiny(const Cta<D>& c, const Work& it, int st, int w, uint32_t& n, uint32_t& pair_phase,
                                             uint32_t& all_phase) {
  using L = Smem<D>;
  const Params& p = c.p;
  const int my_cnt = it.steps(st);
  const Row row(p, it, 0, w, c.lane);
  const int vis = row.valid ? min(row.pos + 1, it.kv_cap) : it.kv_cap;
  constexpr int KQ = BN / 4;                              // keys of a step this warp scores
  const uint32_t lane_addr = (uint32_t)(w * 32) << 16;
  const uint32_t s_addr = c.tmem_S + lane_addr + st * L::SP_COLS;
  const uint32_t p_addr = c.tmem_P + lane_addr + st * L::SP_COLS;
  const uint32_t o_addr = c.tmem_O + lane_addr + st * D;
  // P of this quarter's rows is zero but for the quarter's own keys: cleared once here, the steps
  // write only columns KQ / 2 * w ...
  {
    const uint32_t z[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
#pragma unroll
    for (int i = 0; i < BN / 2; i += 8) tmem_st<8>(p_addr + i, z);
    tmem_wait_st();
  }
  float m_ref = row.valid ? -FLT_MAX : FLT_MAX, l_sum = 0.f;
  for (int k = 0; k < my_cnt; ++k, ++n) {
    c.wait(BAR_S + st, n & 1);
    tc_fence_after();
    uint32_t s[KQ];
    tmem_ld<KQ>(s_addr + KQ * w, s);
    tmem_wait_ld<KQ>(s);
    tc_fence_before();
    warp_arrive(c.bar(BAR_SFREE + st), c.lane);
    const int kv0 = it.key0 + (2 * k + st) * BN + KQ * w;
    if (__any_sync(0xffffffffu, kv0 + KQ > vis)) {
#pragma unroll
      for (int i = 0; i < KQ; ++i)
        if (kv0 + i >= vis) s[i] = 0xff800000u;           // -inf
    }
    float alpha = 1.f;                                    // what O and the sum so far are scaled by
    if (k < EXACT_STEPS) alpha = move_reference(m_ref, row_max<KQ>(s) * p.scale_log2);
    uint32_t v[KQ / 2];
    float sum = row_exp<KQ>(s, p.scale_log2, -m_ref, v);
    if (k > 0) {
      c.wait(BAR_PV + st, (n - 1) & 1);                   // P of the step before is consumed
      tc_fence_after();
      const bool redo = row.valid && !(sum <= SUM_LIMIT);   // (a row past the sequence asks for nothing: see softmax_item)
      if (__any_sync(0xffffffffu, redo || (row.valid && alpha != 1.f))) {
        if (redo) alpha = move_reference(m_ref, row_max<KQ>(s) * p.scale_log2);
        l_sum *= alpha;
        rescale_o_row<D>(o_addr, alpha);
        if (__any_sync(0xffffffffu, redo)) sum = row_exp<KQ>(s, p.scale_log2, -m_ref, v);
      }
    }
    tmem_st<KQ / 2>(p_addr + KQ / 2 * w, v);
    tmem_wait_st();
    tc_fence_before();
    warp_arrive(c.bar(BAR_P + st), c.lane);
    l_sum += sum;
  }
  // ---- the two streams' states of a quarter meet in tensor memory, the four quarters' in the query tiles' space
  // (all MMAs that read the queries are done): [quarter][row][D], 16-byte chunk j of a row at j ^ (row & 7)
  if (my_cnt > 0) c.wait(BAR_PV + st, (n - 1) & 1);
  tc_fence_after();
  float* x = reinterpret_cast<float*>(c.smem_gen + L::Q_OFF);
  float2* xml = reinterpret_cast<float2*>(c.smem_gen + L::ML_OFF);       // [quarter][row]
  auto chunk_at = [&](int q, int j) { return reinterpret_cast<float4*>(x + (q * 32 + c.lane) * D) + (j ^ (c.lane & 7)); };
  if (it.nt > 1) {
    const Pair pr = meet_partner(c, st, w, lane_addr, m_ref, l_sum, pair_phase);
#pragma unroll 1
    for (int c0 = 0; c0 < D / 2; c0 += 32) {
      const int col = st * (D / 2) + c0;
      uint32_t o0[32], o1[32];
      tmem_ld<32>(c.tmem_O + lane_addr + col, o0);
      tmem_ld<32>(c.tmem_O + lane_addr + D + col, o1);
      tmem_wait_ld<32>(o0);
      tmem_wait_ld<32>(o1);
      float f[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        f[i] = pr.w0 == 0.f ? 0.f : __uint_as_float(o0[i]) * pr.w0;      // (an O without weight may hold anything)
        f[i] = pr.w1 == 0.f ? f[i] : fmaf(__uint_as_float(o1[i]), pr.w1, f[i]);
      }
#pragma unroll
      for (int i = 0; i < 32; i += 4) *chunk_at(w, (col + i) / 4) = make_float4(f[i], f[i + 1], f[i + 2], f[i + 3]);
    }
    if (st == 0) xml[w * 32 + c.lane] = make_float2(pr.L == 0.f ? -INFINITY : pr.M, pr.L);
    leave_partner(c, w, pair_phase);
  } else if (st == 0) {
    const bool have = !(l_sum == 0.f);                     // (a sum of NaN is handed on, not dropped)
#pragma unroll 1
    for (int c0 = 0; c0 < D; c0 += 32) {
      uint32_t o[32];
      tmem_ld<32>(o_addr + c0, o);
      tmem_wait_ld<32>(o);
#pragma unroll
      for (int i = 0; i < 32; i += 4)
        *reinterpret_cast<uint4*>(chunk_at(w, (c0 + i) / 4)) = have ? make_uint4(o[i], o[i + 1], o[i + 2], o[i + 3]) : make_uint4(0, 0, 0, 0);
    }
    xml[w * 32 + c.lane] = make_float2(have ? m_ref : -INFINITY, l_sum);
  }
  warp_arrive(c.bar(BAR_ALL), c.lane);
  c.wait(BAR_ALL, all_phase);
  all_phase ^= 1;
  {
    constexpr int DS = D / 8;                              // dims this thread finishes
    const int d0 = (st * 4 + w) * DS;
    float M = -INFINITY, Lt = 0.f, acc[DS];
#pragma unroll
    for (int q = 0; q < 4; ++q) M = fmaxf(M, xml[q * 32 + c.lane].x);
#pragma unroll
    for (int i = 0; i < DS; ++i) acc[i] = 0.f;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float2 ml = xml[q * 32 + c.lane];
      const float wq = ml.y == 0.f ? 0.f : ex2(ml.x - M);
      Lt = fmaf(ml.y, wq, Lt);
#pragma unroll
      for (int i = 0; i < DS; i += 4) {
        const float4 v = *chunk_at(q, (d0 + i) / 4);
        acc[i] = fmaf(v.x, wq, acc[i]);
        acc[i + 1] = fmaf(v.y, wq, acc[i + 1]);
        acc[i + 2] = fmaf(v.z, wq, acc[i + 2]);
        acc[i + 3] = fmaf(v.w, wq, acc[i + 3]);
      }
    }
    const float inv = Lt == 0.f ? 0.f : 1.f / Lt;
#pragma unroll
    for (int i = 0; i < DS; ++i) acc[i] *= inv;
    if (row.th >= 0) {
      if (it.chunk < 0) {
        uint4* dst = reinterpret_cast<uint4*>(p.out + (size_t)row.th * D + d0);
#pragma unroll
        for (int i = 0; i < DS; i += 8)
          dst[i / 8] = make_uint4(pack_bf16x2(acc[i], acc[i + 1]), pack_bf16x2(acc[i + 2], acc[i + 3]),
                                  pack_bf16x2(acc[i + 4], acc[i + 5]), pack_bf16x2(acc[i + 6], acc[i + 7]));
      } else {
        float4* dst = reinterpret_cast<float4*>(p.part_o + ((size_t)row.th * p.s_max + it.chunk) * D + d0);
#pragma unroll
        for (int i = 0; i < DS; i += 4) dst[i / 4] = make_float4(acc[i], acc[i + 1], acc[i + 2], acc[i + 3]);
      }
      if (d0 == 0) store_lse(p, row.th, it.chunk, Lt == 0.f ? -INFINITY : M + log2f(Lt));
    }
  }
  // the space may be filled with the next item's queries (by copies of the async proxy)
  fence_async_smem();
  warp_arrive(c.bar(BAR_ALL), c.lane);
  c.wait(BAR_ALL, all_phase);
  all_phase ^= 1;
}

// One item of more than 32 rows, one query tile or two (DUAL); `n`: steps of this stream so far.  Looks the next item up
// and gets its query rows on their way; returns false if there is none.
// A step is some 500 instructions that two warps per scheduler stream through, and a tenth of the stalls are instruction
// fetches: code that a step rarely or never runs is kept small (rolled loops) and out of its way (__builtin_expect,
// in the waits too).  Copy loop and epilogue rolled, then the hints: 8 x 128 tokens over 8k 154.7 -> 146.5 -> 145.6 us,
// 8 x 3,200 over 5k 2,497 -> 2,471 -> 2,441.
template <int D, bool DUAL>
__device__ __forceinline__ bool softmax_item(const Cta<D>& c, const Work& it, Work& next, Mailbox& mail, int st, int w,
                                             uint32_t& n, uint32_t& pair_phase) {
  using L = Smem<D>;
  const Params& p = c.p;
  const uint32_t lane_addr = (uint32_t)(w * 32) << 16;      // tile row == TMEM lane
  const uint32_t s_addr = c.tmem_S + lane_addr + st * L::SP_COLS;
  const uint32_t p_addr = c.tmem_P + lane_addr + st * L::SP_COLS;
  const uint32_t o_addr = c.tmem_O + lane_addr + st * D;
  const int my_cnt = it.steps(st);
  const Row row(p, it, DUAL ? st : 0, w, c.lane);
  // keys this row sees; a row past the sequence is shown all of the item's, each with probability 0 (with 0 keys it would
  // take the masking path on every step and slow its group)
  const int vis = row.valid ? min(row.pos + 1, it.kv_cap) : it.kv_cap;
  const int exact = !DUAL || it.nt <= EXACT_MAX_STEPS ? EXACT_STEPS : 1;
  const int kv_first = it.key0 + (DUAL ? 0 : st * BN), kv_step = DUAL ? BN : 2 * BN;
  // (a row past the sequence holds zeros or what follows the sequence: against this reference its probabilities are zero)
  float m_ref = row.valid ? -FLT_MAX : FLT_MAX, l_sum = 0.f;
  for (int k = 0; k < my_cnt; ++k, ++n) {
    c.wait(BAR_S + st, n & 1);
    tc_fence_after();
    uint32_t s[BN];
    // The scores come in two parts, the exponentials of the first running under the second's load, and P is
    // stored before its sum is checked: what a stream cannot overlap with itself is what its step takes
    // (8 x 128 tokens over 8k 155 -> 145 us for append and attention, 8 x 3,200 over 5k 2.59 -> 2.55 ms, 64
    // mixed rows 312 -> 306; first parts of 32 and 64 keys: 156 and 145 us, 2.71 and 2.56 ms).
    constexpr int LA = 48;
    tmem_ld<LA>(s_addr, s);
    tmem_wait_ld<LA>(s);
    tmem_ld<BN - LA>(s_addr + LA, s + LA);
    const int kv0 = kv_first + k * kv_step;
    const bool edge = __any_sync(0xffffffffu, kv0 + BN > vis);
    if (__builtin_expect(edge, 0)) {
      tmem_wait_ld<BN - LA>(s + LA);
#pragma unroll
      for (int i = 0; i < BN; ++i)
        if (kv0 + i >= vis) s[i] = 0xff800000u;             // -inf
    }
    // The first steps' exact maximum is the row's reference; later steps only check that their sum stays
    // in range (SUM_LIMIT), so they have no row maximum to take before their first exponential.
    auto freed = [&]() {
      tmem_wait_ld<BN - LA>(s + LA);
      tc_fence_before();
      warp_arrive(c.bar(BAR_SFREE + st), c.lane);           // the next step's scores may be computed
    };
    if (__builtin_expect(edge || k < exact, 0)) freed();
    // alpha: what O and the sum so far are scaled by.  A moved reference lowers the limit, so that the one
    // test below finds it (a second condition there: 8 x 128 tokens over 8k 150.0 -> 152.6 us).
    float alpha = 1.f, limit = SUM_LIMIT;
    if (__builtin_expect(k < exact, 0)) {
      alpha = move_reference(m_ref, row_max<BN>(s) * p.scale_log2);
      if (alpha != 1.f) limit = -1.f;
    }
    uint32_t v[BN / 2];                                     // P as bf16 pairs
    const float neg_m = -m_ref;
    float sum = row_exp<LA>(s, p.scale_log2, neg_m, v);
    if (__builtin_expect(!(edge || k < exact), 1)) freed();
    sum += row_exp<BN - LA>(s + LA, p.scale_log2, neg_m, v + LA / 2);
    if (k > 0) {
      c.wait(BAR_PV + st, (n - 1) & 1);                     // P of the step before is consumed
      tc_fence_after();
    }
    tmem_st<BN / 2>(p_addr, v);
    if (__builtin_expect(__any_sync(0xffffffffu, !(sum <= limit)) && k > 0, 0)) {
      // (O is quiet: PV(k-1) has finished and PV(k) waits for this warp)
      // A row past the sequence holds whatever follows it and asks for nothing.  (With its sums heard like the others', NaN in the
      // queries behind a sequence of 36 tokens over 16k at 32/8 heads made its attention 41.5 us instead of 30.3; now 30.6.
      // A limit of its own for every lane instead, in the test above: prompts of 1-3.5k tokens 0.7 % slower.)
      const bool redo = row.valid && !(sum <= SUM_LIMIT);
      if (__any_sync(0xffffffffu, row.valid && !(sum <= limit))) {
        if (redo) alpha = move_reference(m_ref, row_max<BN>(s) * p.scale_log2);
        l_sum *= alpha;
        rescale_o_row<D>(o_addr, alpha);
        if (__any_sync(0xffffffffu, redo)) {
          sum = row_exp<BN>(s, p.scale_log2, -m_ref, v);
          tmem_wait_st();                                   // two stores to the same columns are not ordered by themselves
          tmem_st<BN / 2>(p_addr, v);
        }
      }
    }
    tmem_wait_st();
    tc_fence_before();
    warp_arrive(c.bar(BAR_P + st), c.lane);
    l_sum += sum;
  }
  // ---- The next item's query rows are on their way under the last PV.  A tile's space is free once the scores of
  // its last step have come: those of this stream, or, where both streams read the one tile, of the stream
  // that has the last step (QK MMAs complete in order).
  const bool more = mail.next(c, next);
  int q_next = -1;
  if (more) {
    if (DUAL ? st == 0 : st == ((it.nt - 1) & 1)) q_next = 0;
    else if (next.shape == SHAPE_TWO) q_next = 1;
    if (q_next >= 0) fetch_q(c, next, q_next, w);
  }
  if (my_cnt > 0) {
    c.wait(BAR_PV + st, (n - 1) & 1);
    tc_fence_after();
  }
  if (q_next >= 0) publish_q(c, q_next);
  // ---- epilogue: PV of the next item's first step waits for its P, and with it for the loads of O here
  const bool whole = __all_sync(0xffffffffu, row.valid);
  const int token = it.tok0 + token_of(p, it.row0 + (DUAL ? st * BM : 0) + w * 32);
  if (!DUAL && it.nt > 1) {
    // both streams have a state of every row: each finishes half of the columns (at head_dim 64 stream 0 all)
    const Pair pr = meet_partner(c, st, w, lane_addr, m_ref, l_sum, pair_phase);
    const float inv = pr.L == 0.f ? 0.f : 1.f / pr.L;
    const float a0 = pr.w0 * inv, a1 = pr.w1 * inv;
    if (D == 128 || st == 0) {
      const int col = D == 128 ? st * 64 : 0;
      uint32_t o0[64], o1[64];
      tmem_ld<64>(c.tmem_O + lane_addr + col, o0);
      tmem_ld<64>(c.tmem_O + lane_addr + D + col, o1);
      tmem_wait_ld<64>(o0);
      tmem_wait_ld<64>(o1);
      float f[64];
#pragma unroll
      for (int i = 0; i < 64; ++i) f[i] = fmaf(__uint_as_float(o1[i]), a1, __uint_as_float(o0[i]) * a0);
      store_cols<D>(c, it, st * 4 + w, token, row.th, whole, col, f);
    }
    if (st == 0) store_lse(p, row.th, it.chunk, pr.L == 0.f ? -INFINITY : pr.M + log2f(pr.L));
    leave_partner(c, w, pair_phase);
  } else if (my_cnt > 0) {
    const float inv = l_sum == 0.f ? 0.f : 1.f / l_sum;
#pragma unroll 1
    for (int c0 = 0; c0 < D; c0 += 64) {
      uint32_t o[64];
      tmem_ld<64>(o_addr + c0, o);
      tmem_wait_ld<64>(o);
      float f[64];
#pragma unroll
      for (int i = 0; i < 64; ++i) f[i] = __uint_as_float(o[i]) * inv;
      store_cols<D>(c, it, st * 4 + w, token, row.th, whole, c0, f);
    }
    store_lse(p, row.th, it.chunk, l_sum == 0.f ? -INFINITY : m_ref + log2f(l_sum));
    tc_fence_before();
  }
  return more;
}

template <int D, bool APPEND>
__device__ __forceinline__ void softmax_role(const Cta<D>& c, Work it, int warp) {
  const int st = warp >> 2, w = warp & 3;                   // stream, 32-lane quarter
  Mailbox mail;
  uint32_t n = 0, pair_phase = 0, all_phase = 0;            // steps of this stream so far; phases of the exchange barriers
  if (it.shape == SHAPE_TWO || st == 0) {
    fetch_q(c, it, st, w);
    publish_q(c, st);
  }
  for (;;) {
    if (APPEND && st == 1) {
      const Params& p = c.p;
      append_rows<D>(reinterpret_cast<const uint4*>(p.k_new), reinterpret_cast<const uint4*>(p.v_new),
                     reinterpret_cast<uint4*>(p.k_pool), reinterpret_cast<uint4*>(p.v_pool),
                     p.block_table + (size_t)it.seq * p.max_pages_per_seq, p.cos_sin, p.max_position, p.interleaved, p.status,
                     p.max_pages_per_seq, p.num_pages, p.Hkv, it.kvh, it.C, token_of(p, it.rows_total), it.tok0, w * 32 + c.lane);
      warp_arrive(c.bar(BAR_NEW), c.lane);
    }
    Work next;
    bool more;
    if (it.shape == SHAPE_TINY) {
      softmax_tiny(c, it, st, w, n, pair_phase, all_phase);
      more = mail.next(c, next);
      if (more && (next.shape == SHAPE_TWO || st == 0)) {
        fetch_q(c, next, st, w);
        publish_q(c, st);
      }
    } else {
      more = it.shape == SHAPE_TWO ? softmax_item<D, true>(c, it, next, mail, st, w, n, pair_phase)
                                   : softmax_item<D, false>(c, it, next, mail, st, w, n, pair_phase);
    }
    if (!more) break;
    it = next;
  }
  asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
  tc_fence_before();
}

// ------------------------------------------------------------------ TMA producers
// Every bulk-tensor copy costs its issuing warp ~65 cycles (one box per page: 16 slots x all dims
// of one kv head).  Warp 8 loads the K tiles and warp 11 the V tiles; warp 8 also claims the items.
template <int D, bool K_ROLE, bool APPEND, typename List>
__device__ __forceinline__ void producer_role(const Cta<D>& c, const CUtensorMap& map, const List& list, Work it) {
  using L = Smem<D>;
  const Params& p = c.p;
  constexpr int n_ring = K_ROLE ? L::NK : L::NV;            // (the ring's constants fold into each copy)
  constexpr uint32_t my_off = K_ROLE ? L::KV_OFF : L::KV_OFF + L::NK * L::KV_BYTES;
  constexpr int full = K_ROLE ? BAR_KFULL : BAR_VFULL, empty = K_ROLE ? BAR_KEMPTY : BAR_VEMPTY;
  const int lane = c.lane, page_l = lane;
  Mailbox mail;                                             // of warp 11; warp 8 keeps the place it writes in it
  int slot = 0, n_steps = 0;
  uint32_t phase = 0, claim_phase = 0, new_phase = 0;
  // A work list that came in the launch parameters is left in the workspace like any other: a call that plans for itself may be
  // followed by planned calls with resident lists.  A CTA's first item is written here, a claimed one by warp 8 as it
  // claims it.  (By warp 8 at the head of each item's copies, the steps of two-tile items took 6 % longer than in the kernel for
  // resident lists: 8 x 128 tokens over 8k planned in the call 130 us against 121, now 121.  All by block 0: 121 too, but 14
  // x 8-14 over 0 at 32/8 x 64 7.8 us instead of 6.8.)
  if constexpr (!K_ROLE && std::is_same<List, InlineItems>::value) {
    if (lane == 0) p.items_out[blockIdx.x] = list.items[blockIdx.x];
  }
  for (;;) {
    const int32_t* bt = p.block_table + (size_t)it.seq * p.max_pages_per_seq + (it.key0 >> 4);
    const int n_pages = (it.kv_cap - it.key0 + 15) >> 4;    // pages this item reads
    // page id of this lane in step jj: -2 if the lane fetches none (lanes beyond the step's visible
    // pages; the last test only matters for a plan that does not belong to this block table), -1 for
    // any negative entry
    auto lookup = [&](int jj) {
      const int pg = jj * (BN / 16) + page_l;
      if (page_l >= BN / 16 || pg >= n_pages || (it.key0 >> 4) + pg >= p.max_pages_per_seq) return -2;
      return max(bt[pg], -1);
    };
    // the block-table read is a dependent global load in front of every copy: fetch it two steps ahead
    int pid_a = lookup(0), pid_b = lookup(1);
    // Another item is claimed when the copies of the last but one step are due: the rings then hold the steps before,
    // which covers the claim, the item and its first pages.  (Claimed earlier, the last items of a launch would be
    // bound to CTAs that are still busy.)
    const int claim_at = max(it.nt - 2, 0);
    // APPEND: step that holds the first key this kernel appends, and the pages it appends to, one per lane from lane 8 on
    // (128 new tokens lie in 9 pages at most).
    const int first_new = APPEND ? (it.C - it.key0) / BN : -1;
    int new_page = -1;
    if constexpr (APPEND) {
      const int pg = (it.C >> 4) + lane - 8;
      if (lane >= 8 && pg * 16 < it.kv_cap && pg < p.max_pages_per_seq) new_page = p.block_table[(size_t)it.seq * p.max_pages_per_seq + pg];
    }
    for (int jj = 0; jj < it.nt; ++jj) {
      const int pid = pid_a;
      pid_a = pid_b;
      pid_b = lookup(jj + 2);
      const bool ok = pid >= 0 && pid < p.num_pages;
      const bool bad = pid != -2 && !ok;                    // an id outside the pool: reported, never dereferenced
      const uint32_t okmask = __ballot_sync(0xffffffffu, ok);
      const bool any_bad = __any_sync(0xffffffffu, bad);
      const uint32_t bytes = __popc(okmask) * (uint32_t)L::PAGE_BYTES;
      if (K_ROLE && jj == claim_at && lane == 0) {
        mbar_expect_tx(c.bar(BAR_CLAIM), 16);
        claim_next(c.smem_base + L::CLAIM_OFF, c.bar(BAR_CLAIM));
      }
      c.wait(empty + slot, phase ^ 1);
      if constexpr (APPEND) {
        bool held = jj >= first_new;
        if (!held) {                                        // (a table may name a page twice: for cached keys and for new ones)
          const int key = lane < 8 ? pid : new_page;
          const uint32_t twins = __match_any_sync(0xffffffffu, key >= 0 ? key : -3 - lane) >> 8;
          held = __any_sync(0xffffffffu, lane < 8 && twins != 0);
        }
        if (held) {
          c.wait(BAR_NEW, new_phase);
          asm volatile("fence.proxy.async;" ::: "memory");
        }
      }
      const uint32_t dst_off = my_off + slot * L::KV_BYTES + page_l * L::PAGE_BYTES;
      if (any_bad) {
        // the page's 16 keys are replaced by zeros (score 0, value 0), so the tile holds nothing
        // undefined; written with ordinary stores, made visible to the tensor core's reads
        if (bad) {
          if (K_ROLE && p.status) atomicOr(p.status, EFIM_DEV_BAD_PAGE);
          uint4* z = reinterpret_cast<uint4*>(c.smem_gen + dst_off);
          for (int i = 0; i < L::PAGE_BYTES / 16; ++i) z[i] = make_uint4(0, 0, 0, 0);
          fence_async_smem();
        }
        __syncwarp();
      }
      if (lane == 0) mbar_expect_tx(c.bar(full + slot), bytes);
      __syncwarp();
      if (ok) tma_load_page(c.smem_base + dst_off, &map, c.bar(full + slot), pid * p.Hkv + it.kvh);
      if (++slot == n_ring) { slot = 0; phase ^= 1; }
    }
    n_steps += it.nt;
    if (APPEND) new_phase ^= 1;                             // (the last step holds new keys: it has been waited for)
    bool more;
    if constexpr (K_ROLE) {
      c.wait(BAR_CLAIM, claim_phase);
      claim_phase ^= 1;
      const bool gone = __any_sync(0xffffffffu, *c.abort_flag != 0);
      const int block = gone ? -1 : uniform(claimed_block(c.smem_base + L::CLAIM_OFF));
      fence_async_smem();                                   // the answer has been read: the next one may be written
      more = block >= 0;
      if (more) {
        if constexpr (std::is_same<List, InlineItems>::value) {
          const WorkItem w = list.items[block];
          if (lane == 0) p.items_out[block] = w;
          it = work_of(w, p);
        } else {
          it = work_of(p.items[block], p);
        }
      } else {
        it.seq = -1;
      }
      mail.put(c, it);
    } else {
      more = mail.next(c, it);
    }
    if (!more) break;
  }
  // if the CTA gave up, let copies that are still in flight land before shared memory goes away
  if (*c.abort_flag) {
    for (int jj = max(0, n_steps - n_ring); jj < n_steps; ++jj) mbar_drain(c.bar(full + jj % n_ring), (jj / n_ring) & 1);
  }
}

// ------------------------------------------------------------------ MMA issuers
// Issuing an MMA costs its thread nearly as long as the tensor core needs to run it,
// so the work is split: warp 9 issues the PV MMAs of both streams, warp 10 the QK
// MMAs.  QK(k+1) of a stream needs S(k) read (barrier SFREE), PV(k) needs P(k) written:
// neither waits for the other, so the tensor core has a stream's next scores ready when
// its softmax warps come back for them.
//
// Descriptors: the high word is fixed (SBO = distance between 8-row groups: 1024 in a
// query tile, GROUP_BYTES in a K/V tile; version 1; 128B swizzle); the low word is
// (address >> 4) | LBO << 16, so stepping through a tile is one add.
template <int D>
struct Desc {
  static constexpr uint32_t HI_Q = (1024u >> 4) | (1u << 14) | (2u << 29);
  static constexpr uint32_t HI_KV = ((uint32_t)Smem<D>::GROUP_BYTES >> 4) | (1u << 14) | (2u << 29);
  static constexpr uint32_t LBO_K = 1u << 16;                                      // K-major: LBO unused
  static constexpr uint32_t LBO_V = (1024u >> 4) << 16;                            // MN-major: next 64 dims
  static __device__ __forceinline__ uint64_t q(uint32_t lo) { return (static_cast<uint64_t>(HI_Q) << 32) | lo; }
  static __device__ __forceinline__ uint64_t kv(uint32_t lo) { return (static_cast<uint64_t>(HI_KV) << 32) | lo; }
};

template <int D>
struct PvIssuer {
  using L = Smem<D>;
  static constexpr uint32_t V_OFF = L::KV_OFF + L::NK * L::KV_BYTES;
  const Cta<D>& c;
  int slot = 0;
  uint32_t phase = 0, n[2] = {0, 0};                        // ring position; steps of each stream so far

  // O_st (+)= P_st V of the step in ring entry `slot`; P from TMEM
  __device__ __forceinline__ void issue(int st, uint32_t first) {
    const uint32_t v_lo = (((c.smem_base + V_OFF) >> 4) | Desc<D>::LBO_V) + slot * (L::KV_BYTES >> 4);
    constexpr uint32_t IDESC = instr_desc(D, 1);
#pragma unroll
    for (int k = 0; k < BN / 16; ++k)
      umma_bf16_ts(c.tmem_O + st * D, c.tmem_P + st * L::SP_COLS + k * 8, Desc<D>::kv(v_lo + k * (L::PAGE_BYTES >> 4)), IDESC,
                   (!first || k > 0) ? 1u : 0u);
  }
  // V rows past the visible range hold stale or foreign data; P is 0 there but
  // 0 * NaN would poison O, so clear them before the step's values are used.
  __device__ __forceinline__ void clear_tail(const Work& it, int step) {
    const int keys = it.kv_cap - it.key0 - step * BN;
    if (keys < BN) {
      uint8_t* vb = c.smem_gen + V_OFF + slot * L::KV_BYTES;
      const int first = max(keys, 0);
      const int chunks = (BN - first) * 8;                  // 16-byte chunks to clear per 64-dim half
#pragma unroll
      for (int h = 0; h < L::HALVES; ++h)
        for (int idx = c.lane; idx < chunks; idx += 32) {
          const int key = first + (idx >> 3);
          *reinterpret_cast<uint4*>(vb + (key >> 3) * L::GROUP_BYTES + h * 1024 + (key & 7) * 128 + ((idx & 7) << 4)) =
              make_uint4(0, 0, 0, 0);
        }
      fence_async_smem();
      __syncwarp();
    }
  }
  template <bool DUAL>
  __device__ __forceinline__ void item(const Work& it) {
    const int cnt0 = it.steps(0), cnt1 = it.steps(1);
    for (int k = 0; k < cnt0; ++k) {
#pragma unroll
      for (int st = 0; st < 2; ++st) {
        if (k >= (st == 0 ? cnt0 : cnt1)) continue;
        const bool last_user = !DUAL || st == 1;            // last stream to touch this V tile
        if (!DUAL || st == 0) {
          c.wait(BAR_VFULL + slot, phase);
          clear_tail(it, DUAL ? k : 2 * k + st);
        }
        c.wait(BAR_P + st, n[st] & 1);
        ++n[st];
        tc_fence_after();
        if (elect_one()) {
          issue(st, k == 0);
          if (last_user) tc_commit(c.bar(BAR_VEMPTY + slot));
          tc_commit(c.bar(BAR_PV + st));
        }
        __syncwarp();
        if (last_user && ++slot == L::NV) { slot = 0; phase ^= 1; }
      }
    }
  }
};

template <int D>
struct QkIssuer {
  using L = Smem<D>;
  const Cta<D>& c;
  int slot = 0;
  uint32_t phase = 0, n[2] = {0, 0}, q_phase[2] = {0, 0};
  bool apart = false;                                       // the streams run half a step apart already

  __device__ __forceinline__ void issue(int st, int tile) {
    const uint32_t k_lo = (((c.smem_base + L::KV_OFF) >> 4) | Desc<D>::LBO_K) + slot * (L::KV_BYTES >> 4);
    const uint32_t a_lo = (((c.smem_base + L::Q_OFF) >> 4) | Desc<D>::LBO_K) + tile * (L::Q_BYTES >> 4);
    constexpr uint32_t IDESC = instr_desc(BN, 0);
#pragma unroll
    for (int k = 0; k < D / 16; ++k) {
      const uint32_t off_q = ((k >> 2) * L::HALF_BYTES + (k & 3) * 32) >> 4;
      const uint32_t off_k = ((k >> 2) * 1024 + (k & 3) * 32) >> 4;
      umma_bf16(c.tmem_S + st * L::SP_COLS, Desc<D>::q(a_lo + off_q), Desc<D>::kv(k_lo + off_k), IDESC, k > 0 ? 1u : 0u);
    }
  }
  template <bool DUAL>
  __device__ __forceinline__ void item(const Work& it) {
    const int cnt0 = it.steps(0), cnt1 = it.steps(1);
    // The streams share the tensor core and the exponential unit, so they should run half a step
    // apart: stream 1 starts when stream 0 has its first probabilities.  (Started together they
    // stay together: 2,236 cycles per step against 1,796.)  From one item of two tiles to the next they stay
    // apart by themselves; where an item's end brings them together they are set apart again.  (The first wait makes the
    // second one's phase the next to come; it cannot move on meanwhile: stream 0's next scores are issued here.)
    const bool set_apart = !(DUAL && apart);
    const uint32_t p0 = n[0] & 1;
    if (set_apart && n[0] > 0) c.wait(BAR_P + 0, p0 ^ 1);
    for (int k = 0; k < cnt0; ++k) {
#pragma unroll
      for (int st = 0; st < 2; ++st) {
        if (k >= (st == 0 ? cnt0 : cnt1)) continue;
        const bool last_user = !DUAL || st == 1;            // last stream to touch this K tile
        if (k == 0 && (DUAL || st == 0)) {
          c.wait(BAR_Q + st, q_phase[st]);
          q_phase[st] ^= 1;
        }
        if (!DUAL || st == 0) c.wait(BAR_KFULL + slot, phase);
        if (n[st] > 0) c.wait(BAR_SFREE + st, (n[st] - 1) & 1);
        if (k == 0 && st == 1 && set_apart) c.wait(BAR_P + 0, p0);
        ++n[st];
        tc_fence_after();
        if (elect_one()) {
          issue(st, DUAL ? st : 0);
          tc_commit(c.bar(BAR_S + st));
          if (last_user) tc_commit(c.bar(BAR_KEMPTY + slot));
        }
        __syncwarp();
        if (last_user && ++slot == L::NK) { slot = 0; phase ^= 1; }
      }
    }
    apart = DUAL;
  }
};

// A CTA walks items: its own block index's first, then, one at a time, those of blocks of the launch that have not
// started yet, until none is left - so the hardware's order and balance stay, and what a fresh CTA costs outside its
// steps is paid once: the next item's pages are copied while the present one's last steps run, its query rows under
// the last PV, its first scores under the epilogue.  A CTA per item spent 14,000 cycles of each outside the steps (of
// 2,000): launch gap, set-up, query rows and first pages in front, the last PV, the output and the exit behind.  From one item
// to the next it is 4,300 to 4,600 (prompts: look-up 400, query boxes 470 and 210, last PV 250, output 2,560, wait for the
// first scores 640), 8,800 where the query rows come per lane and 16,300 where they are rotated as they come.  Append and attention,
// one CTA per item -> now: 16 prompts of 1-3.5k tokens 1,017 -> 898 us, 16 x 8-112 tokens over 1-3.4k planned in the call 69 -> 64,
// 64 mixed rows at 28/4 heads 316 -> 302, 16 x 32-256 over 2-8k at 32/32 317 -> 308, 8 x 3,200 over 5k 2,555 -> 2,450.
// The work list: in the workspace (List = NoList), or, a short one planned inside the call, in the launch
// parameters (List = InlineItems) - which saves the copy between the append and this kernel.
// APPEND: the softmax warps of stream 1 first put the item's new k/v rows into their pages, and the copies of those pages
// wait for them: a step of a few short rows is one launch instead of two (16 tokens over 240 at 4/4 heads x 64 9.85 ->
// 7.35 us, now 7.5 with the rows' pages compared).  A kernel of its own: in the others' place it cost their steps 5 %.
template <int D, typename List, bool APPEND>
__global__ void __launch_bounds__(THREADS, 1)
prefill_tc_kernel(const Params p, const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                  const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_out,
                  const __grid_constant__ List list) {
  using L = Smem<D>;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem_gen + L::TMEM_SLOT_OFF);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem_gen + L::ABORT_OFF);
  auto bar = [&](int i) { return smem_base + L::BAR_OFF + 8u * i; };
  const int tid = threadIdx.x, warp = uniform(tid >> 5), lane = tid & 31;

  if (tid == 0) {
    for (int t = 0; t < NQ; ++t) {
      mbar_init(bar(BAR_Q + t), 4);                        // one arrival per softmax warp
      mbar_init(bar(BAR_S + t), 1);
      mbar_init(bar(BAR_SFREE + t), 4);
      mbar_init(bar(BAR_P + t), 4);
      mbar_init(bar(BAR_PV + t), 1);
      mbar_init(bar(BAR_IFULL + t), 1);
      mbar_init(bar(BAR_IEMPTY + t), 11);
    }
    for (int s = 0; s < 4; ++s) mbar_init(bar(BAR_PAIR + s), 2);
    mbar_init(bar(BAR_ALL), 8);
    mbar_init(bar(BAR_CLAIM), 1);
    mbar_init(bar(BAR_NEW), 4);
    for (int s = 0; s < L::NK; ++s) {
      mbar_init(bar(BAR_KFULL + s), 1);
      mbar_init(bar(BAR_KEMPTY + s), 1);
      mbar_init(bar(BAR_VFULL + s), 1);
      mbar_init(bar(BAR_VEMPTY + s), 1);
    }
    *abort_flag = 0;
    mbar_fence_init();
  }
  if (warp == 9) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(const_cast<uint32_t*>(tmem_slot))),
                 "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = uniform(*tmem_slot);
  const Cta<D> c{p, smem_base, smem_gen, abort_flag, &map_q, &map_out, tmem, tmem + BN, tmem + NQ * L::SP_COLS, lane};

  // Programmatic launch: up to here a CTA has touched nothing but itself; every warp that reads or writes global
  // memory waits for the kernel before (which may be one that leaves its list in this workspace).
  WorkItem raw;                                               // 32 bytes: two vector loads, no dependent load after them
  if constexpr (std::is_same<List, InlineItems>::value) {
    if (warp != 9 && warp != 10) pdl_wait();
    raw = list.items[blockIdx.x];
  } else {
    pdl_wait();
    const uint4* src = reinterpret_cast<const uint4*>(p.items + blockIdx.x);
    uint4* dst = reinterpret_cast<uint4*>(&raw);
    dst[0] = src[0];
    dst[1] = src[1];
  }
  Work it = work_of(raw, p);
  // Register split: every warp of a warpgroup runs the same setmaxnreg; the service
  // group releases first what the two softmax groups then take.  (Nothing may come between this and a role's code: past a
  // point where the two branches meet the compiler plans with fewer registers, and the steps spilled 1.4 KB.)
  if (warp < 8) {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REGS_SOFTMAX<D>));
    softmax_role<D, APPEND>(c, it, warp);
  } else {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_SERVICE<D>));
    if (warp == 8) {
      if (p.early_next) pdl_launch();
      producer_role<D, true, APPEND>(c, map_k, list, it);
    } else if (warp == 11) {
      if (p.early_next) pdl_launch();
      producer_role<D, false, APPEND>(c, map_v, list, it);
    } else if (warp == 9) {
      PvIssuer<D> pv{c};
      Mailbox mail;
      do {
        if (it.shape == SHAPE_TWO) pv.template item<true>(it);
        else pv.template item<false>(it);
      } while (mail.next(c, it));
      tc_fence_before();
    } else {
      QkIssuer<D> qk{c};
      Mailbox mail;
      do {
        if (it.shape == SHAPE_TWO) qk.template item<true>(it);
        else qk.template item<false>(it);
      } while (mail.next(c, it));
      tc_fence_before();
    }
  }
  __syncthreads();
  if (*abort_flag) {
    // a wait expired: roles ran out of step, copies and MMAs may still be in flight; give
    // them a generous moment to finish before TMEM and shared memory are released
    for (int i = 0; i < 2000; ++i) __nanosleep(1000);
    __syncthreads();
  }
  if (warp == 9) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
  }
}

// Merge the KV-chunk partials of split sequences.  A warp takes MERGE_ROWS consecutive heads of one token (a divisor of all), with
// the partial rows of AT_ONCE chunks in flight.  `split`: keys per chunk of every sequence, 0 = not split - in the workspace (NoList)
// or in the launch parameters (InlineSplit), in which case the kernel leaves it in the workspace too.
//
// Bound: the partials' bytes, which the kernel before has left in L2, behind a chain of dependent look-ups.  The lanes look
// a token's sequence up together, 32 candidates a trip, and bring its lengths along in the last one; with a warp per row
// that bisected q_indptr and then read one value after the other, a chain of ten trips in each of 8 waves of CTAs,
// the merge of 960 tokens at 32/8 heads in two chunks took 25 us; now 6.2, and 64 mixed rows at 28/4, cut into 516 items on trial
// (the planner leaves 500; 304 us), 307 us instead of 355 for the layer.
//
// Rows of a warp and chunks in flight.  Up to 32 rows an SM there are warps enough resident for a row each, with eight chunks in flight
// (2 x 1-2 tokens over 8-10k at 4/4 heads x 64 attention and merge 10.7 us, four rows a warp 14.2 [a warp per row, bisecting, 12.0]); up
// to 80 a row each, with four, which leaves room for more warps; beyond that looking up is what there is to save: four heads, or two.
// Append, attention and merge with 1 x 4 / 2 x 4 / 4 x 2 [as in the brackets above]: 2 x 150-160 over 9-12k at 16/1 (4,900 rows)
// 38.0 / 38.9 / 40.3 [37.9], 6 x 20-30 over 3-8k at 32/8 x 64 (4,900) 27.5 / 28.0 / 28.8 [28.3], 12 x 10-60 over 0.5-4k at 16/1 (7,600)
// 26.0 / 26.6 / 27.9 [29.6], 4 x 60-110 over 5-9k at 32/8 (10,100) 73.3 / 74.2 / 75.3 [73.2], 10 x 20-60 over 0.8-3k at 28/4 (11,700)
// 36.0 / 33.0 / 32.1 [39.6], 12 x 10-60 over 0.5-4k at 32/8 (15,100) 58.5 / 57.9 / 57.3 [64.4].  An odd number of heads: one row, four
// chunks at any size (eight: 4 x 500-620 tokens over 3-4k at 5/1 36.9 us instead of 35.3, 4 x 100-300 over 5-9k at 9/3 45.5 and 42.2).
constexpr int MERGE_WARPS = 8;
template <int D, int MERGE_ROWS, int AT_ONCE, typename Split>
__global__ void __launch_bounds__(32 * MERGE_WARPS) prefill_merge_kernel(const Params p, const __grid_constant__ Split split) {
  constexpr int EPL = D / 32;                               // dims of a lane
  constexpr bool inl = std::is_same<Split, InlineSplit>::value;
  const int lane = threadIdx.x & 31;
  const size_t th = ((size_t)blockIdx.x * MERGE_WARPS + (threadIdx.x >> 5)) * MERGE_ROWS;    // this warp's rows: heads of one token
  // (everything before the attention kernel has completed, and that kernel writes partials only: the
  // look-ups need not wait for it.  Read in L2, where what has completed is visible.)
  int st = 0, nc = 0;
  if (th < (size_t)p.total_new_tokens * p.Hq) {
    const int t = (int)(th / p.Hq);
    int lo = 0, n = p.batch;                                // the last sequence that starts at or before t is one of [lo, lo + n)
    while (n > 32) {
      const int step = (n + 31) / 32, probe = lo + lane * step;
      const bool le = lane * step < n && __ldcg(p.q_indptr + probe) <= t;
      const int i = 31 - __clz((int)(__ballot_sync(0xffffffffu, le) | 1u));
      n = min(step, n - i * step);
      lo += i * step;
    }
    int first = 0x7fffffff, cached = 0, keys = 0;
    if (lane < n) {
      first = __ldcg(p.q_indptr + lo + lane);
      cached = __ldcg(p.cached_len + lo + lane);
      if constexpr (inl) keys = split.keys[lo + lane];
      else keys = __ldcg(p.split_tokens + lo + lane);
    }
    const int i = 31 - __clz((int)(__ballot_sync(0xffffffffu, first <= t) | 1u));
    st = __shfl_sync(0xffffffffu, keys, i);
    const int pos = __shfl_sync(0xffffffffu, cached, i) + t - __shfl_sync(0xffffffffu, first, i);
    if (st > 0) nc = min(p.s_max, (pos + 1 + st - 1) / st);
  }
  pdl_wait();
  pdl_launch();
  if constexpr (inl) {
    if (blockIdx.x == 0)
      for (int i = threadIdx.x; i < p.batch; i += 32 * MERGE_WARPS) p.split_out[i] = split.keys[i];
  }
  if (nc == 0) return;                                      // written directly by the main kernel
  // rows r of chunks c0 .. c0 + AT_ONCE - 1
  const float* po = p.part_o + th * p.s_max * D + lane * EPL;
  __align__(16) float v[AT_ONCE][MERGE_ROWS][EPL];
  auto fetch = [&](int c0) {
#pragma unroll
    for (int c = 0; c < AT_ONCE; ++c)
#pragma unroll
      for (int r = 0; r < MERGE_ROWS; ++r) {
        if (c0 + c >= nc) continue;
        const float* src = po + ((size_t)r * p.s_max + c0 + c) * D;
        if constexpr (EPL == 4) {
          *reinterpret_cast<float4*>(v[c][r]) = __ldcg(reinterpret_cast<const float4*>(src));
        } else {
          *reinterpret_cast<float2*>(v[c][r]) = __ldcg(reinterpret_cast<const float2*>(src));
        }
      }
  };
  // lane 16 h + c: the lse of chunk c (at most 16) of rows h and h + 2
  const int my_c = lane & 15, my_r = lane >> 4;
  float lse[2];
#pragma unroll
  for (int j = 0; j < 2; ++j)
    lse[j] = my_c < nc && my_r + 2 * j < MERGE_ROWS ? __ldcg(p.part_lse + (th + my_r + 2 * j) * p.s_max + my_c) : -INFINITY;
  fetch(0);
  float M[2], L[2], w[2];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    M[j] = lse[j];
#pragma unroll
    for (int d = 8; d > 0; d >>= 1) M[j] = max_nan(M[j], __shfl_xor_sync(0xffffffffu, M[j], d));   // a NaN chunk makes the row NaN
    w[j] = M[j] == -INFINITY ? 0.f : exp2f(lse[j] - M[j]);                                       // 0 beyond the last chunk
    L[j] = w[j];
#pragma unroll
    for (int d = 8; d > 0; d >>= 1) L[j] += __shfl_xor_sync(0xffffffffu, L[j], d);
  }
  float acc[MERGE_ROWS][EPL];
#pragma unroll
  for (int r = 0; r < MERGE_ROWS; ++r)
#pragma unroll
    for (int e = 0; e < EPL; ++e) acc[r][e] = 0.f;
  for (int c0 = 0; c0 < nc; c0 += AT_ONCE) {
    if (c0 > 0) fetch(c0);
#pragma unroll
    for (int c = 0; c < AT_ONCE; ++c)
#pragma unroll
      for (int r = 0; r < MERGE_ROWS; ++r) {
        const float wc = __shfl_sync(0xffffffffu, w[r >> 1], (r & 1) * 16 + ((c0 + c) & 15));
#pragma unroll
        for (int e = 0; e < EPL; ++e) acc[r][e] = c0 + c < nc ? fmaf(wc, v[c][r][e], acc[r][e]) : acc[r][e];
      }
  }
#pragma unroll
  for (int r = 0; r < MERGE_ROWS; ++r) {
    const float Lr = __shfl_sync(0xffffffffu, L[r >> 1], (r & 1) * 16), Mr = __shfl_sync(0xffffffffu, M[r >> 1], (r & 1) * 16);
    const float inv = Lr == 0.f ? 0.f : 1.f / Lr;
    if (Lr == 0.f) {                                        // (no chunk has a weight: what their partials hold is not looked at)
#pragma unroll
      for (int e = 0; e < EPL; ++e) acc[r][e] = 0.f;
    }
    uint16_t* out = p.out + (th + r) * D + lane * EPL;
    if constexpr (EPL == 4) {
      *reinterpret_cast<uint2*>(out) = make_uint2(pack_bf16x2(acc[r][0] * inv, acc[r][1] * inv), pack_bf16x2(acc[r][2] * inv, acc[r][3] * inv));
    } else {
      *reinterpret_cast<uint32_t*>(out) = pack_bf16x2(acc[r][0] * inv, acc[r][1] * inv);
    }
    if (p.lse && lane == 0) p.lse[th + r] = Lr == 0.f ? -INFINITY : (Mr + log2f(Lr)) * 0.6931471805599453f;
  }
}

// ------------------------------------------------------------------ host side
namespace {
// Cost of a work item in tenths of a microsecond: a 128-key tile with two query tiles is bound by the softmax / tensor
// pipeline, with one by its K/V bytes; every item pays for what lies between it and the one before on its CTA (what a
// CTA pays before its first one is the same for every cut); a split adds the partials' round trip and the merge.  Of 16
// batches, with the costs of a kernel of one item per CTA (18, 12, 95 instead of 16, 10, 40) -> with these: two of 13 drawn ones
// 125 -> 119 and 62.4 -> 60.3 us, 64 mixed rows 303.9 -> 302.3, 16 x 32-256 over 2-8k at 32/32 heads 306.9 -> 305.7, the
// others the same.  (18, 12, 40: 16 x 8-112 tokens over 1-3.4k are cut too fine, 65 -> 92 us.)
constexpr long long COST_TILE_DUAL = 16, COST_TILE_SINGLE = 10, COST_CTA = 40, COST_PARTIAL = 8, COST_MERGE = 40;
// Weights of a tile in the launch order of a few waves (see fill_lists).
constexpr long long ORDER_TILE_DUAL = 21, ORDER_TILE_SINGLE = 9;

// A run of consecutive work items that differ in the kv head only.
struct Block {
  int32_t seq, row0, tile_begin, tile_end;
  int16_t chunk;
  int32_t cost;                // place in the launch order
};

// Walks the blocks of a batch whose sequences' K/V ranges are cut into chunks of about `chunk_tiles`
// tiles (at most 16 per sequence): f(seq, row0, rows of the block, tile_begin, tile_end, chunk or -1);
// returns the largest number of chunks, writes keys per chunk of every cut sequence to `split`.
template <typename F>
int walk_blocks(const efim_cache_desc* c, const efim_batch_desc* b, long long chunk_tiles, int32_t* split, F&& f) {
  const long long G = c->num_q_heads / c->num_kv_heads;
  int s_max = 1;
  for (int s = 0; s < b->batch; ++s) {
    const long long N = b->h_new_len[s], C = b->h_cached_len[s];
    if (split) split[s] = 0;
    if (N <= 0) continue;
    const long long rows = N * G;
    const long long kt_max = (C + N + PT - 1) / PT;
    long long S = 1, ct = kt_max;
    if (chunk_tiles < kt_max) {
      S = std::min<long long>(16, (kt_max + chunk_tiles - 1) / chunk_tiles);
      ct = (kt_max + S - 1) / S;                             // tiles per chunk
      S = (kt_max + ct - 1) / ct;
      if (S > 1 && split) split[s] = (int32_t)(ct * PT);
      s_max = std::max<int>(s_max, (int)S);
    }
    for (long long row0 = 0; row0 < rows; row0 += NQ * BM) {
      const long long rows_here = std::min<long long>(rows - row0, NQ * BM);
      const long long kt = (C + (row0 + rows_here - 1) / G + 1 + PT - 1) / PT;
      for (long long tb = 0, ch = 0; tb < kt; tb += ct, ++ch)
        f(s, (int32_t)row0, (int)rows_here, (int32_t)tb, (int32_t)std::min(kt, tb + ct), (int)(S > 1 ? ch : -1));
    }
  }
  return s_max;
}

// Finish time of the launch with that cut: the hardware hands CTAs, longest first, to whichever SM is
// free.  `best`: the earliest finish known; a cut whose lower bound is no better is not simulated, and a simulation
// ends where it is no better any more.
long long estimate_makespan(const efim_cache_desc* c, const efim_batch_desc* b, long long chunk_tiles, int n_sm,
                            long long best, std::vector<int32_t>& cost, std::vector<int32_t>& sm) {
  cost.clear();
  long long total = 0, longest = 0;
  const int s_max = walk_blocks(c, b, chunk_tiles, nullptr, [&](int, int32_t, int rows, int32_t tb, int32_t te, int ch) {
    const long long x = COST_CTA + (te - tb) * (rows > BM ? COST_TILE_DUAL : COST_TILE_SINGLE) + (ch >= 0 ? COST_PARTIAL : 0);
    cost.push_back((int32_t)std::min<long long>(x, 1 << 30));
    total += x;
    longest = std::max(longest, x);
  });
  const long long Hkv = c->num_kv_heads;
  const long long merge = s_max > 1 ? COST_MERGE : 0;
  const long long bound = std::max(longest, (total * Hkv + n_sm - 1) / n_sm) + merge;
  if (bound >= best || (long long)cost.size() * Hkv <= n_sm) return bound;
  std::sort(cost.begin(), cost.end(), std::greater<int32_t>());
  // The first items go to one SM each: their finish times, the last of them first, are a min-heap as they stand.
  sm.resize((size_t)n_sm);
  size_t i0 = 0;
  long long h0 = 0;
  for (int k = n_sm; k-- > 0;) {
    sm[(size_t)k] = cost[i0];
    if (++h0 == Hkv) { h0 = 0; ++i0; }
  }
  long long end = sm[(size_t)n_sm - 1];
  for (; i0 < cost.size(); ++i0, h0 = 0)
    for (; h0 < Hkv; ++h0) {
      const int32_t v = sm[0] + cost[i0];                    // the earliest SM takes the item: sift it down
      if (v > end) {
        end = v;
        if (end + merge >= best) return end + merge;         // (no better than the best, whatever follows)
      }
      size_t i = 0;
      for (size_t k = 1; k < sm.size(); k = 2 * i + 1) {
        if (k + 1 < sm.size() && sm[k + 1] < sm[k]) ++k;
        if (sm[k] >= v) break;
        sm[i] = sm[k];
        i = k;
      }
      sm[i] = v;
    }
  return end + merge;
}
}  // namespace

Plan make_plan(const efim_cache_desc* c, const efim_batch_desc* b) {
  const int Hkv = c->num_kv_heads;
  long long n_blocks = 0, tiles_total = 0;
  constexpr long long NO_CUT = 1LL << 40;
  walk_blocks(c, b, NO_CUT, nullptr, [&](int, int32_t, int, int32_t tb, int32_t te, int) {
    ++n_blocks;
    tiles_total += (long long)(te - tb) * Hkv;
  });
  // Few long items cannot fill the SMs, or leave a ragged last wave: try cutting the K/V range of every
  // sequence into chunks that would give between half a CTA and 4 CTAs per SM if they came out even
  // (each at least 3 tiles long) and keep the cut, or none, with the earliest estimated finish.  (Cuts for
  // less than one CTA per SM matter: ragged sequences round up, and a few CTAs too many are a second
  // wave: 4 x 8-112 tokens over 1-3k keys at 32/8 heads, planned in the call, 62 -> 35 us; 1 x 40 over 4k 22 ->
  // 19; 2 x 32-256 over 2-8k at 32/32 90 -> 80.)
  const int n_sm = sm_count();
  Plan pl{};
  pl.chunk_tiles = NO_CUT;
  pl.s_max = 1;
  if (n_blocks * Hkv < 4LL * n_sm && tiles_total > 0) {
    std::vector<int32_t> cost, sm;
    cost.reserve((size_t)n_blocks * 2);
    long long best = estimate_makespan(c, b, NO_CUT, n_sm, 1LL << 60, cost, sm);
    long long last = 0;
    for (const int k : {4, 5, 6, 7, 8, 10, 12, 16, 24, 32}) {    // CTAs per SM aimed at, in eighths
      const long long ct = std::max<long long>(3, (tiles_total * 8 + (long long)n_sm * k - 1) / ((long long)n_sm * k));
      if (ct == last) continue;
      last = ct;
      const long long t = estimate_makespan(c, b, ct, n_sm, best, cost, sm);
      if (t < best) { best = t; pl.chunk_tiles = ct; }
    }
    if (pl.chunk_tiles != NO_CUT) {
      n_blocks = 0;
      pl.s_max = walk_blocks(c, b, pl.chunk_tiles, nullptr, [&](int, int32_t, int, int32_t, int32_t, int) { ++n_blocks; });
    }
  }
  pl.n_items = (int)(n_blocks * Hkv);
  auto up = [](size_t x) { return (x + 255) / 256 * 256; };
  pl.items_bytes = up((size_t)pl.n_items * sizeof(WorkItem));
  pl.split_bytes = up((size_t)b->batch * sizeof(int32_t));
  const size_t th = (size_t)b->total_new_tokens * c->num_q_heads;
  pl.part_lse_bytes = pl.s_max > 1 ? up(th * pl.s_max * sizeof(float)) : 0;
  pl.part_o_bytes = pl.s_max > 1 ? up(th * pl.s_max * c->head_dim * sizeof(float)) : 0;
  return pl;
}

void fill_lists(const efim_cache_desc* c, const efim_batch_desc* b, const Plan& pl, WorkItem* items, int32_t* split_tokens) {
  const int Hkv = c->num_kv_heads;
  std::vector<Block> blocks;
  blocks.reserve((size_t)pl.n_items / Hkv);
  // A two-tile CTA is bound by its softmax wherever it runs; a one-tile CTA is bound by its K/V
  // bytes and speeds up once SMs fall idle at the end of a launch (0.89 us per tile with 8 to 32 such
  // CTAs on the GPU, 1.5 us with 148), so it is weighted with its lone rate.  The weights were measured on a
  // kernel with P in S's columns, whose two-tile CTAs took 2.1 us a tile (cfg2: 305 us ordered by tile
  // count, 290 by cost at 2.1 : 1.5, 281 at 2.1 : 1.2; 2.1 : 0.9 3-5 % faster still on three of four
  // other draws of cfg2), and not on the present one.
  walk_blocks(c, b, pl.chunk_tiles, split_tokens, [&](int s, int32_t row0, int rows, int32_t tb, int32_t te, int ch) {
    blocks.push_back(Block{s, row0, tb, te, (int16_t)ch,
                           (int32_t)((te - tb) * (rows > BM ? ORDER_TILE_DUAL : ORDER_TILE_SINGLE))});
  });
  std::vector<int32_t> tok0((size_t)b->batch);
  for (int s = 0, t = 0; s < b->batch; t += b->h_new_len[s], ++s) tok0[s] = t;
  auto put = [&](WorkItem*& w, const Block& k, int h) {
    *w = WorkItem{};
    w->seq = k.seq;
    w->kvh = (int16_t)h;
    w->chunk = k.chunk;
    w->row0 = k.row0;
    w->tile_begin = k.tile_begin;
    w->tile_end = k.tile_end;
    w->cached = b->h_cached_len[k.seq];
    w->new_len = b->h_new_len[k.seq];
    w->tok0 = tok0[k.seq];
    ++w;
  };
  WorkItem* w = items;
  if (pl.n_items > 8LL * sm_count()) {
    // Many waves: CTAs that run together should read the same K/V.  Keep the row tiles
    // of one (sequence, kv head) adjacent (longest first inside the group), so the
    // concurrent working set is a few heads' K/V and stays in L2.
    for (size_t i = 0, j = 0; i < blocks.size(); i = j) {
      while (j < blocks.size() && blocks[j].seq == blocks[i].seq) ++j;
      for (int h = 0; h < Hkv; ++h)
        for (size_t k = j; k-- > i;) put(w, blocks[k], h);
    }
  } else {
    // Few waves: costliest first, so the tail of the launch is made of cheap items.  It also puts items of one shape on the two
    // SMs of a TPC, which fetch their instructions together: a two-tile item beside a one-tile item takes 2,540 ns a step, beside
    // another two-tile item 1,470 (16 x 8-112 tokens over 1-3.4k; dealt to SMs in another order 76 us instead of 58).
    std::stable_sort(blocks.begin(), blocks.end(), [](const Block& x, const Block& y) { return x.cost > y.cost; });
    for (const Block& k : blocks)
      for (int h = 0; h < Hkv; ++h) put(w, k, h);
  }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(ptr);
  }
  return fn;
}

// Pool [pages][Hkv][16][D] bf16 as a 5-D tensor (dim % 64, slot % 8, dim / 64, slot / 8,
// page * Hkv + head); one box = the 16 slots x D dims of one (page, head), written to shared
// memory as [slot / 8][dim / 64][slot % 8][64 dims], 128-byte swizzled.
static bool make_pool_map(CUtensorMap* m, void* pool, int pages, int Hkv, int D) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t row = (cuuint64_t)D * 2;
  const cuuint64_t dims[5] = {64, 8, (cuuint64_t)D / 64, 2, (cuuint64_t)pages * Hkv};
  const cuuint64_t strides[4] = {row, 128, 8 * row, 16 * row};
  const cuuint32_t box[5] = {64, 8, (cuuint32_t)D / 64, 2, 1};
  const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, pool, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Rows [tokens][heads][D] bf16 as a 4-D tensor (dim % 64, dim / 64, head, token); one box = 64 dims of the G heads of 32 / G
// tokens, 128-byte swizzled in shared memory.
static bool make_rows_map(CUtensorMap* m, const void* rows, int tokens, int heads, int D, int G) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t row = (cuuint64_t)D * 2;
  const cuuint64_t dims[4] = {64, (cuuint64_t)D / 64, (cuuint64_t)heads, (cuuint64_t)tokens};
  const cuuint64_t strides[3] = {128, row, row * heads};
  const cuuint32_t box[4] = {64, 1, (cuuint32_t)G, (cuuint32_t)(32 / G)};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(rows), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// A model calls this once per layer with the same few pools over and over: the encoded maps
// of the pools seen last are kept per host thread (a map is a pure function of the key).
struct PoolMapEntry {
  void* pool;
  int pages, Hkv, D;
  CUtensorMap map;
};
const CUtensorMap* pool_map(void* pool, int pages, int Hkv, int D) {
  constexpr int kEntries = 16;
  thread_local PoolMapEntry cache[kEntries] = {};
  thread_local int next = 0;
  for (int i = 0; i < kEntries; ++i)
    if (cache[i].pool == pool && cache[i].pages == pages && cache[i].Hkv == Hkv && cache[i].D == D)
      return &cache[i].map;
  PoolMapEntry& e = cache[next];
  next = (next + 1) % kEntries;
  e.pool = nullptr;
  if (!make_pool_map(&e.map, pool, pages, Hkv, D)) return nullptr;
  e.pool = pool;
  e.pages = pages;
  e.Hkv = Hkv;
  e.D = D;
  return &e.map;
}

// The kernel's shared-memory size has to be raised once per device.
template <int D, typename List, bool APPEND>
static efim_status raise_smem_limit() {
  constexpr int kMaxDevices = 64;
  static std::atomic<bool> done[kMaxDevices];
  int dev = 0;
  EFIM_CUDA_TRY(cudaGetDevice(&dev));
  if (dev >= 0 && dev < kMaxDevices && done[dev].load(std::memory_order_acquire)) return EFIM_OK;
  EFIM_CUDA_TRY(cudaFuncSetAttribute(prefill_tc_kernel<D, List, APPEND>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     Smem<D>::TOTAL));
  if (dev >= 0 && dev < kMaxDevices) done[dev].store(true, std::memory_order_release);
  return EFIM_OK;
}

template <int D, typename List>
static efim_status launch_d(const efim_cache_desc* c, const Params& args, const Plan& pl, const List& list, cudaStream_t s) {
  Params p = args;
  // Few waves: the next kernel's set-up hides in the tail (8 x 128 tokens over 8k: 171 -> 169 us).  Many
  // waves: nothing to hide it in, 1 % lost (16 prompts of 1-3.5k tokens 1172 -> 1183 us).
  p.early_next = pl.n_items <= 4 * sm_count();
  constexpr bool inl = std::is_same<List, InlineList>::value;
  p.items_out = inl ? const_cast<WorkItem*>(p.items) : nullptr;
  p.split_out = inl ? const_cast<int32_t*>(p.split_tokens) : nullptr;
  const CUtensorMap* pk = pool_map(c->d_k_pool, c->num_pages, c->num_kv_heads, D);
  if (!pk) return EFIM_ERR_CUDA;
  const CUtensorMap mk = *pk;
  const CUtensorMap* pv = pool_map(c->d_v_pool, c->num_pages, c->num_kv_heads, D);
  if (!pv) return EFIM_ERR_CUDA;
  // Query and output rows as boxes of 32 rows, where those are whole tokens and there are as many.  (Encoding a map takes the
  // host 0.09 us; they are of this call's buffers and not kept.)
  p.g_mul = p.G == 1 ? 0u : (uint32_t)((1ull << 32) / (unsigned)p.G + 1);
  CUtensorMap mq{}, mo{};
  if (p.G <= 32 && 32 % p.G == 0 && (long long)p.total_new_tokens * p.G >= 32) {
    p.q_tma = p.cos_sin == nullptr && make_rows_map(&mq, p.q, p.total_new_tokens, p.Hq, D, p.G);
    p.out_tma = make_rows_map(&mo, p.out, p.total_new_tokens, p.Hq, D, p.G);
  }
  using Items = std::decay_t<decltype(items_of(list))>;
  auto start = [&](auto append) -> efim_status {
    constexpr bool APPEND = decltype(append)::value;
    const efim_status st = raise_smem_limit<D, Items, APPEND>();
    if (st != EFIM_OK) return st;
    EFIM_CUDA_TRY(launch_pdl(prefill_tc_kernel<D, Items, APPEND>, dim3(pl.n_items), dim3(THREADS), Smem<D>::TOTAL, s, p, mk, *pv,
                             mq, mo, items_of(list)));
    return EFIM_OK;
  };
  efim_status st;
  if constexpr (inl) st = p.k_new ? start(std::true_type{}) : start(std::false_type{});
  else st = start(std::false_type{});
  if (st != EFIM_OK) return st;
  if (pl.s_max > 1) {
    const size_t rows = (size_t)p.total_new_tokens * p.Hq;
    using Split = std::conditional_t<inl, InlineSplit, NoList>;
    const Split* split;
    NoList none;
    if constexpr (inl) split = &list.split;
    else split = &none;
    auto merge = [&](auto per_warp, auto at_once) -> efim_status {
      constexpr int ROWS = decltype(per_warp)::value, per_block = MERGE_WARPS * ROWS;
      EFIM_CUDA_TRY(launch_pdl(prefill_merge_kernel<D, ROWS, decltype(at_once)::value, Split>,
                               dim3((unsigned)((rows + per_block - 1) / per_block)), dim3(32 * MERGE_WARPS), 0, s, p, *split));
      return EFIM_OK;
    };
    using One = std::integral_constant<int, 1>;
    using Two = std::integral_constant<int, 2>;
    using Four = std::integral_constant<int, 4>;
    if (rows <= (size_t)32 * sm_count()) return merge(One{}, std::integral_constant<int, 8>{});
    if (rows <= (size_t)80 * sm_count() || p.Hq % 2 != 0) return merge(One{}, Four{});
    return p.Hq % 4 == 0 ? merge(Four{}, Two{}) : merge(Two{}, Four{});
  }
  return EFIM_OK;
}

efim_status launch(const efim_cache_desc* c, const Params& p, const Plan& pl, const InlineList* list, cudaStream_t s) {
  if (pl.n_items == 0) return EFIM_OK;
  if (list) return c->head_dim == 128 ? launch_d<128>(c, p, pl, *list, s) : launch_d<64>(c, p, pl, *list, s);
  return c->head_dim == 128 ? launch_d<128>(c, p, pl, NoList{}, s) : launch_d<64>(c, p, pl, NoList{}, s);
}

}  // namespace pf
}  // namespace efim
