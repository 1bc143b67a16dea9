// The attention pipeline shared by the one-CTA verification kernel and the prefill: S = Q K^T, online softmax,
// O += P V on 128-key tiles.
//
// PAIR = 2: a cluster of two CTAs (tcgen05 cta_group::2) works on 256 stacked query rows, CTA r on the rows r*128..;
// each CTA stages half of every K/V tile (K: 64 of the 128 keys; V: 64 of the 128 value columns) and the pair's MMAs
// (M = 256, issued by the leader CTA) read both halves.  PAIR = 1: one CTA, 128 rows, whole K/V tiles.
//
//   tensor memory per CTA: O [0,128) | S0 [128,256) | S1 [256,384) | P0 [384,448) | P1 [448,512)
//
// Two softmax warpgroups take the key tiles of the same 128 rows in turn (tile t: warpgroup, S buffer and P buffer
// t mod 2), one thread per row.  A thread pulls its whole S row into registers and releases the S buffer at once, so the
// S tiles run two key tiles ahead of the exponentials; P goes to tensor memory 32 keys at a time as it is made.  The row's
// reference maximum is handed from tile to tile through shared memory, each warpgroup keeps its own partial row sum, and
// O is rescaled lazily by whichever warpgroup raises the maximum by more than 2^8.
//
// A worker goes through its segments (the tiles of one problem) without stopping the pipeline: tiles are numbered through
// all of them, and the Q rows, K/V tiles and S MMAs of the next segment proceed under the last tiles of this one.
#ifndef SPECEXT_CORE_CUH_
#define SPECEXT_CORE_CUH_

#include "common.cuh"
#include "pair.cuh"

namespace core {

using namespace sm100;
using namespace pair;

constexpr int kWG = 2;                         // softmax warpgroups
constexpr int kThreads = (kWG + 1) * 128;
constexpr int kProducerWarp = 8, kMmaWarp = 9, kPvWarp = 10, kTreeWarp = 11;
constexpr int kRegsLaunch = 168, kRegsOther = 64, kRegsSoftmax = 216;
static_assert(128 * (kRegsLaunch - kRegsOther) >= kWG * 128 * (kRegsSoftmax - kRegsLaunch),
              "setmaxnreg.inc would wait for registers that are never released");
constexpr float kRescaleThreshold = 8.0f;      // log2 units
constexpr uint32_t kColO = 0, kColS = 128, kColP = 384;
constexpr int kMaxStages = 6;

// Shared-memory layout: Q | K ring | V ring | control block.  Everything is in 64-element column blocks of 128 bytes a
// row (128-byte swizzle).
template <int PAIR, int D>
struct Geo {
  static constexpr int kBlocks = D / 64;
  static constexpr int kKBlk = (SPX_TILE_KEYS / PAIR) * 128;
  static constexpr int kKStage = kKBlk * kBlocks;
  static constexpr int kVBlk = SPX_TILE_KEYS * 128;
  static constexpr int kVStage = PAIR == 2 ? kVBlk : kVBlk * kBlocks;
  static constexpr int kQBytes = 128 * 128 * kBlocks;
  static constexpr bool kWide = kKStage == 32768;            // one CTA with head_dim 128: stages of 32 KB
  // (wide: 16 KB of Q and six stages with 64 rows, 8 KB and six with 32, or 32 KB and five with 128)
  static constexpr int kCtrlOffset = kWide ? 16384 + 6 * 32768 : kQBytes + 11 * 16384;
  int q_blk, nk, nv;
  uint32_t k_off, v_off;
  // rows = AttnPlan::q_rows.  64 or 32 (one CTA, head_dim 128 and at most that many stacked rows): Q takes half the room or less,
  // which is one more stage.  The MMA still reads 128 rows; what lies behind Q is multiplied into rows nobody looks at.  Calls
  // with as few rows may keep 128 all the same, zeros behind the last (see lay_out in api.cu).
  __device__ __forceinline__ explicit Geo(int rows) {
    q_blk = rows * 128;
    nk = kWide ? (rows <= 64 ? 3 : 2) : 5;
    nv = kWide ? 3 : 6;
    k_off = q_blk * kBlocks;
    v_off = k_off + nk * kKStage;
  }
};

struct Ctrl {
  uint64_t k_full[kMaxStages];     // leader: one producer per CTA + bytes
  uint64_t k_empty[kMaxStages];    // each CTA: MMA completion
  uint64_t v_full[kMaxStages];
  uint64_t v_empty[kMaxStages];
  uint64_t q_full;                 // leader: the segment's Q rows have landed
  uint64_t q_empty;                // each CTA: the last S MMA of a segment is complete
  // per warpgroup w, one phase for each of its tiles:
  uint64_t s_full[kWG];            // each CTA: S is complete
  uint64_t s_free[kWG];            // leader: 4 warps per CTA have their S rows in registers
  uint64_t p_full[kWG];            // leader: 4 warps per CTA have stored P
  uint64_t pv_done[kWG];           // each CTA: the PV is complete
  uint64_t m_pub[kWG];             // this CTA: 4 arrivals, reference maxima of the tile are published
  uint64_t o_done;                 // each CTA: the last PV of a segment is complete
  uint64_t o_free;                 // leader: the softmax warps have read O of a segment
  uint64_t epi[2];                 // this CTA: the row sums of a segment are published (alternating by segment)
  uint64_t drain;
  uint64_t anc_ready;              // this CTA: the ancestor masks are in shared memory
  uint64_t v_rag;                  // this CTA: a V part whose tail rows must be cleared has landed (device-side length)
  unsigned long long anc[kSpxMaxTree][2];
  int parent[kSpxMaxTree];
  float m_row[128];                // reference maximum of each row after the latest tile
  float l_x[2][kWG][128];          // end of a segment: each warpgroup's row sums (two, so that the next segment's may be
                                   // written while a slow warp still reads these)
  uint32_t tmem_base;
  int abort_flag;
};
constexpr int kCtrlBytes = 6144;
static_assert(sizeof(Ctrl) <= kCtrlBytes, "control block too large");

template <int PAIR, int D>
constexpr int smem_bytes() {
  return Geo<PAIR, D>::kCtrlOffset + kCtrlBytes + 1024;
}

// ---- forms of the cluster instructions for one CTA and for a pair -----------------------------------------
template <int PAIR>
__device__ __forceinline__ void commit(uint64_t* bar) {
  if constexpr (PAIR == 2) commit_pair(bar); else mma_commit(bar);
}
template <int PAIR>
__device__ __forceinline__ uint32_t leader_addr(uint64_t* bar) {
  return PAIR == 2 ? map_to_cta(smem_u32(bar), 0) : smem_u32(bar);
}
template <int PAIR>
__device__ __forceinline__ void tma_load(uint32_t dst, const CUtensorMap* m, uint32_t bar, int c0, int c1, int c2) {
  if constexpr (PAIR == 2) {
    tma_load_3d_pair(dst, m, bar, c0, c1, c2);
  } else {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(m)), "r"(bar), "r"(c0), "r"(c1), "r"(c2)
        : "memory");
  }
}
template <int PAIR>
__device__ __forceinline__ void tma_load_hint(uint32_t dst, const CUtensorMap* m, uint32_t bar, int c0, int c1, int c2,
                                              uint64_t policy) {
  if constexpr (PAIR == 2) {
    tma_load_3d_pair_hint(dst, m, bar, c0, c1, c2, policy);
  } else {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4, "
        "%5}], [%2], %6;"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(m)), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "l"(policy)
        : "memory");
  }
}

// ---- set-up and end of a CTA ---------------------------------------------------------------------------
// Barriers by the producer warp, tensor memory by the MMA warp, and the cluster barrier (block barrier) that publishes
// them.  None of it touches global memory: it runs ahead of the dependency wait, under the kernel before.
// HANDOVER: segments end with segment_handover (else segment_end).
template <int PAIR, bool HANDOVER = false>
__device__ __forceinline__ void setup(Ctrl* ctl, int warp, int lane) {
  constexpr int kEnd = HANDOVER ? 4 : 4 * kWG;    // warps of a CTA that take part in the end of a segment
  if (warp == kProducerWarp) {
    if (lane < kMaxStages) {
      mbar_init(&ctl->k_full[lane], PAIR);
      mbar_init(&ctl->k_empty[lane], 1);
      mbar_init(&ctl->v_full[lane], PAIR);
      mbar_init(&ctl->v_empty[lane], 1);
    } else if (lane < kMaxStages + kWG) {
      const int i = lane - kMaxStages;
      mbar_init(&ctl->s_full[i], 1);
      mbar_init(&ctl->s_free[i], 4 * PAIR);      // one arrival per warp of the warpgroup, in every CTA
      mbar_init(&ctl->p_full[i], 4 * PAIR);
      mbar_init(&ctl->pv_done[i], 1);
      mbar_init(&ctl->m_pub[i], 4);
    } else if (lane == kMaxStages + kWG) {
      mbar_init(&ctl->q_full, PAIR);
      mbar_init(&ctl->q_empty, 1);
      mbar_init(&ctl->o_done, 1);
      mbar_init(&ctl->o_free, kEnd * PAIR);
      mbar_init(&ctl->epi[0], kEnd);
      mbar_init(&ctl->epi[1], kEnd);
      mbar_init(&ctl->drain, 2);
      mbar_init(&ctl->anc_ready, 1);
      mbar_init(&ctl->v_rag, 1);
      ctl->abort_flag = 0;
    }
    fence_mbar_init();
  } else if (warp == kMmaWarp) {
    if constexpr (PAIR == 2) {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl->tmem_base)),
                   "r"(512u)
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      tmem_alloc(&ctl->tmem_base, 512);
      tmem_relinquish();
    }
  }
  tc_fence_before();
  if constexpr (PAIR == 2) {
    cluster_arrive();
    cluster_wait();
  } else {
    __syncthreads();
  }
  tc_fence_after();
}
// The peer may still signal this CTA's barriers or read its halves, and tensor memory is freed by one warp for all:
// everybody meets once more.  Results written to global memory need no ordering here.
template <int PAIR>
__device__ __forceinline__ void finish(Ctrl* ctl, int warp) {
  tc_fence_before();
  if constexpr (PAIR == 2) cluster_sync_relaxed(); else __syncthreads();
  if (warp == kMmaWarp) {
    tc_fence_after();
    if constexpr (PAIR == 2)
      asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(ctl->tmem_base), "r"(512u) : "memory");
    else
      tmem_dealloc(ctl->tmem_base, 512);
  }
}

// ---- MMA issuers -----------------------------------------------------------------------------------------
// Two threads of the leader CTA issue the S and the PV MMAs.  (A thread that issues an MMA is held until the tensor pipe
// takes it, and its waits, commits and bookkeeping cost it another ~0.5 K cycles a tile: one thread for both kinds left
// the pipe idle that long, 2.1 K cycles a tile against 1.0 K of MMAs.)  `Work` enumerates the segments (`next()`, `n`
// tiles in the current one).
template <int PAIR, int D, class Work>
__device__ __forceinline__ bool issue_s(Ctrl* ctl, unsigned char* base, const Geo<PAIR, D>& geo, Work work,
                                        volatile int* abort_flag) {
  using G = Geo<PAIR, D>;
  const uint32_t tmem = ctl->tmem_base;
  const uint32_t idesc = idesc_bf16_f32(128 * PAIR, SPX_TILE_KEYS, false, false);
  constexpr uint32_t hi = desc_hi(1024);
  const uint32_t q_lo = desc_lo(smem_u32(base), 16), q_blk = geo.q_blk >> 4;
  const uint32_t k_lo = desc_lo(smem_u32(base + geo.k_off), 16);
  int kst = 0, w = 0;
  uint32_t kph = 0, qph = 0, t = 0;
  bool ok = true;
  while (ok && work.next()) {
    ok = wait_c(&ctl->q_full, qph, abort_flag);
    qph ^= 1;
    for (int j = work.n; j > 0 && ok; --j) {
      // the rows of the tile before last are in registers: its S buffer is free
      if (t >= kWG) ok = wait_c(&ctl->s_free[w], (t / kWG - 1) & 1, abort_flag);
      if (ok) ok = wait_c(&ctl->k_full[kst], kph, abort_flag);
      if (!ok) break;
      tc_fence_after();
      const uint32_t kb = k_lo + kst * (G::kKStage >> 4), d = tmem + kColS + w * 128;
#pragma unroll
      for (int kk = 0; kk < D / 16; ++kk) {
        const uint32_t qa = q_lo + (kk >> 2) * q_blk + (kk & 3) * 2;
        const uint32_t ka = kb + (kk >> 2) * (G::kKBlk >> 4) + (kk & 3) * 2;
        if constexpr (PAIR == 2)
          mma_ss_pair(d, qa, hi, ka, hi, idesc, kk > 0 ? 1u : 0u);
        else
          mma_ss2(d, qa, hi, ka, hi, idesc, kk > 0 ? 1u : 0u);
      }
      commit<PAIR>(&ctl->s_full[w]);
      commit<PAIR>(&ctl->k_empty[kst]);
      if (++kst == geo.nk) {
        kst = 0;
        kph ^= 1;
      }
      w ^= 1;
      ++t;
    }
    if (ok) commit<PAIR>(&ctl->q_empty);
  }
  commit<PAIR>(&ctl->drain);
  return ok;
}
template <int PAIR, int D, class Work>
__device__ __forceinline__ bool issue_pv(Ctrl* ctl, unsigned char* base, const Geo<PAIR, D>& geo, Work work,
                                         volatile int* abort_flag) {
  using G = Geo<PAIR, D>;
  const uint32_t tmem = ctl->tmem_base, d = tmem + kColO;
  const uint32_t idesc = idesc_bf16_f32(128 * PAIR, D, false, true);
  constexpr uint32_t hi = desc_hi(1024);
  const uint32_t v_lo = desc_lo(smem_u32(base + geo.v_off), PAIR == 2 ? 16 : G::kVBlk);
  int vst = 0, w = 0;
  uint32_t vph = 0, wph = 0, seg = 0;
  bool ok = true;
  while (ok && work.next()) {
    // every thread is done reading the O of the segment before
    if (seg > 0) ok = wait_c(&ctl->o_free, (seg - 1) & 1, abort_flag);
    ++seg;
    uint32_t acc = 0;
    for (int j = work.n; j > 0 && ok; --j) {
      ok = wait_c(&ctl->v_full[vst], vph, abort_flag);
      if (ok) ok = wait_c(&ctl->p_full[w], wph, abort_flag);
      if (!ok) break;
      tc_fence_after();
      const uint32_t vb = v_lo + vst * (G::kVStage >> 4), pa = tmem + kColP + w * 64;
#pragma unroll
      for (int kk = 0; kk < SPX_TILE_KEYS / 16; ++kk) {
        if constexpr (PAIR == 2)
          mma_ts_pair(d, pa + kk * 8, vb + kk * 128, hi, idesc, kk > 0 ? 1u : acc);
        else
          mma_ts2(d, pa + kk * 8, vb + kk * 128, hi, idesc, kk > 0 ? 1u : acc);
      }
      acc = 1;
      commit<PAIR>(&ctl->pv_done[w]);
      commit<PAIR>(&ctl->v_empty[vst]);
      if (++vst == geo.nv) {
        vst = 0;
        vph ^= 1;
      }
      if ((w ^= 1) == 0) wph ^= 1;
    }
    if (ok) commit<PAIR>(&ctl->o_done);
  }
  // everything issued by both must be complete before tensor memory is released
  commit<PAIR>(&ctl->drain);
  for (int spin = 0; spin < (1 << 22) && !mbar_test_wait(&ctl->drain, 0); ++spin) {}
  return ok;
}

// ---- softmax of one tile by one warpgroup -----------------------------------------------------------------
struct RowCtx {
  Ctrl* ctl;
  uint32_t lane_tmem;      // tensor memory of this warp's 32 rows
  int w, row_t, lane;      // warpgroup, row inside the CTA's 128 rows
  uint32_t s_free, p_full; // cluster addresses of the leader's s_free[w] and p_full[w]
  float scale2;
  bool pad;                // a row behind the last stacked one: its probabilities are zeros
  volatile int* abort_flag;
};

__device__ __forceinline__ void mask_chunk(uint32_t (&v)[32], uint32_t visible) {
#pragma unroll
  for (int k = 0; k < 32; ++k)
    if (!((visible >> k) & 1u)) v[k] = 0xff800000u;    // -inf
}
__device__ __forceinline__ float max_row(const uint32_t (&s0)[32], const uint32_t (&s1)[32], const uint32_t (&s2)[32],
                                         const uint32_t (&s3)[32]) {
  float t0 = -INFINITY, t1 = -INFINITY, t2 = -INFINITY, t3 = -INFINITY;
#pragma unroll
  for (int k = 0; k < 32; k += 2) {
    t0 = fmax3(t0, __uint_as_float(s0[k]), __uint_as_float(s0[k + 1]));
    t1 = fmax3(t1, __uint_as_float(s1[k]), __uint_as_float(s1[k + 1]));
    t2 = fmax3(t2, __uint_as_float(s2[k]), __uint_as_float(s2[k + 1]));
    t3 = fmax3(t3, __uint_as_float(s3[k]), __uint_as_float(s3[k + 1]));
  }
  return fmaxf(fmaxf(t0, t1), fmaxf(t2, t3));
}

// Tile number t (through all segments) of warpgroup t mod 2; `first`: first tile of its segment.  `mask(lo, hi)` gives
// the visible keys of this thread's row as two 64-bit words and is called when need_mask is set.  `sums(c, v, sum)`
// gets each 32-key group's unrounded exponentials and their sum.  m_loc: the reference maximum of this tile, which the
// row sum l is relative to.  O is D columns wide.
template <int D, class MaskFn, class SumFn>
__device__ __forceinline__ bool softmax_tile(const RowCtx& rc, uint32_t t, bool first, bool need_mask, MaskFn&& mask,
                                             SumFn&& sums, float& m_loc, float& l) {
  Ctrl* ctl = rc.ctl;
  const int w = rc.w, wp = w ^ 1;
  const uint32_t s_addr = rc.lane_tmem + kColS + w * 128, p_addr = rc.lane_tmem + kColP + w * 64;
  if (!wait_c(&ctl->s_full[w], (t / kWG) & 1, rc.abort_flag)) return false;
  tc_fence_after();
  uint32_t s0[32], s1[32], s2[32], s3[32];
  tmem_ld32(s_addr, s0);
  tmem_ld32(s_addr + 32, s1);
  tmem_ld32(s_addr + 64, s2);
  tmem_ld32(s_addr + 96, s3);
  // The row's reference maximum after the previous tile (the other warpgroup's) is fetched while the scores are on their
  // way from tensor memory: it was published long before, as a rule.
  float m_cur = -INFINITY;
  if (!first) {
    if (!mbar_wait(&ctl->m_pub[wp], ((t - 1) / kWG) & 1, rc.abort_flag)) return false;
    m_cur = ctl->m_row[rc.row_t];
  }
  tmem_wait_ld();
  tc_fence_before();
  warp_arrive_cluster(rc.s_free, rc.lane);           // the S buffer may take the next tile but one
  if (need_mask) {
    unsigned long long lo, hi;
    mask(lo, hi);
    mask_chunk(s0, static_cast<uint32_t>(lo));
    mask_chunk(s1, static_cast<uint32_t>(lo >> 32));
    mask_chunk(s2, static_cast<uint32_t>(hi));
    mask_chunk(s3, static_cast<uint32_t>(hi >> 32));
  }
  const float m_tile = max_row(s0, s1, s2, s3) * rc.scale2;     // -inf when the row sees nothing here (never on the first tile)

  float m_new = m_cur;
  bool rescale = false;
  if (m_tile > m_cur + kRescaleThreshold || m_cur == -INFINITY) {
    m_new = m_tile;
    rescale = !first;
  }
  ctl->m_row[rc.row_t] = m_new;
  warp_arrive(&ctl->m_pub[w], rc.lane);
  if (m_loc != m_new) {
    l *= (m_loc == -INFINITY) ? 0.f : ex2_approx(m_loc - m_new);
    m_loc = m_new;
  }
  // The PV of this warpgroup's previous tile has read the P buffer.  Waiting for it here, and not behind the first
  // exponentials, also keeps the two warpgroups' exponentials apart: without it they drift into step and queue for the
  // special-function unit together (16K prefill 1648 us against 1589).
  if (t >= kWG && !wait_c(&ctl->pv_done[w], (t / kWG - 1) & 1, rc.abort_flag)) return false;
  if (__any_sync(0xffffffffu, rescale)) {
    // O must hold the sum up to the previous tile and nothing may be accumulating into it
    if (!wait_c(&ctl->pv_done[wp], ((t - 1) / kWG) & 1, rc.abort_flag)) return false;
    tc_fence_after();
    const float alpha = rescale ? ex2_approx(m_cur - m_new) : 1.f;
#pragma unroll 1
    for (int c = 0; c < D / 16; ++c) {
      uint32_t v[16];
      tmem_ld16(rc.lane_tmem + kColO + c * 16, v);
      tmem_wait_ld();
#pragma unroll
      for (int k = 0; k < 16; ++k) v[k] = __float_as_uint(__uint_as_float(v[k]) * alpha);
      tmem_st16(rc.lane_tmem + kColO + c * 16, v);
    }
  }
  tc_fence_after();

  const float neg_m = rc.pad ? -INFINITY : -m_new;
  const uint64_t scale2x2 = pack_f32x2(rc.scale2, rc.scale2), neg_mx2 = pack_f32x2(neg_m, neg_m);
  auto exp_chunk = [&](uint32_t (&v)[32], int c) {
    // two elements per fma and per add (packed fp32 pairs); the exponential itself is per element
    uint64_t acc01 = 0ull, acc23 = 0ull;
#pragma unroll
    for (int k = 0; k < 32; k += 4) {
      float e0, e1, e2, e3;
      unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(v[k]), __uint_as_float(v[k + 1])), scale2x2, neg_mx2), e0, e1);
      unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(v[k + 2]), __uint_as_float(v[k + 3])), scale2x2, neg_mx2), e2, e3);
      e0 = ex2_approx(e0);
      e1 = ex2_approx(e1);
      e2 = ex2_approx(e2);
      e3 = ex2_approx(e3);
      acc01 = add_f32x2(acc01, pack_f32x2(e0, e1));
      acc23 = add_f32x2(acc23, pack_f32x2(e2, e3));
      v[k] = __float_as_uint(e0);
      v[k + 1] = __float_as_uint(e1);
      v[k + 2] = __float_as_uint(e2);
      v[k + 3] = __float_as_uint(e3);
    }
    float gs0, gs1, gs2, gs3;
    unpack_f32x2(acc01, gs0, gs1);
    unpack_f32x2(acc23, gs2, gs3);
    const float gs = (gs0 + gs1) + (gs2 + gs3);
    l += gs;
    sums(c, v, gs);
    uint32_t pk[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) pk[k] = pack_bf16x2(__uint_as_float(v[2 * k]), __uint_as_float(v[2 * k + 1]));
    tmem_st16(p_addr + c * 16, pk);
  };
  exp_chunk(s0, 0);
  exp_chunk(s1, 1);
  exp_chunk(s2, 2);
  exp_chunk(s3, 3);
  tmem_wait_st();
  tc_fence_before();
  warp_arrive_cluster(rc.p_full, rc.lane);
  return true;
}

// The part of softmax_tile that a warp without any valid row keeps: its arrivals, none of them ahead of the phase it
// belongs to.
__device__ __forceinline__ bool skip_tile(const RowCtx& rc, uint32_t t) {
  if (!wait_c(&rc.ctl->s_full[rc.w], (t / kWG) & 1, rc.abort_flag)) return false;
  if (rc.lane == 0) arrive_cluster(rc.s_free);
  if (t >= kWG && !wait_c(&rc.ctl->pv_done[rc.w], (t / kWG - 1) & 1, rc.abort_flag)) return false;
  if (rc.lane == 0) {
    mbar_arrive(&rc.ctl->m_pub[rc.w]);
    arrive_cluster(rc.p_full);
  }
  return true;
}

// End of a segment whose last tile is number `last`: the final reference maximum of the row, the sum of the
// warpgroups' row sums, and O complete.  n_seg: segments finished before this one.
__device__ __forceinline__ bool segment_end(const RowCtx& rc, uint32_t last, uint32_t n_seg, float m_loc, float l,
                                            float& m_fin, float& l_tot) {
  Ctrl* ctl = rc.ctl;
  if (!mbar_wait(&ctl->m_pub[last % kWG], (last / kWG) & 1, rc.abort_flag)) return false;
  m_fin = ctl->m_row[rc.row_t];
  if (m_loc != m_fin) l *= (m_loc == -INFINITY) ? 0.f : ex2_approx(m_loc - m_fin);
  float (*lx)[128] = ctl->l_x[n_seg & 1];
  lx[rc.w][rc.row_t] = l;
  warp_arrive(&ctl->epi[n_seg & 1], rc.lane);
  if (!wait_c(&ctl->o_done, n_seg & 1, rc.abort_flag)) return false;
  tc_fence_after();
  if (!mbar_wait(&ctl->epi[n_seg & 1], (n_seg >> 1) & 1, rc.abort_flag)) return false;
  l_tot = lx[0][rc.row_t] + lx[1][rc.row_t];
  return true;
}

// End of a segment where the next one follows at once: the warpgroup of the last tile ends the segment alone (`last_wg`;
// its m_loc is the final reference maximum), the other one leaves its row sums behind and goes on to the next segment,
// whose first tile is its own.  When both waited for the PV and read half of O each, every segment cost ~5 K cycles on top
// of its tiles.  l_x and epi alternate by segment: the other warpgroup reaches the segment after next only once the PVs of
// the next one run, for which this one has handed O over.
__device__ __forceinline__ bool segment_handover(const RowCtx& rc, uint32_t last, uint32_t n_seg, bool last_wg, float m_loc,
                                                 float l, float& l_tot) {
  Ctrl* ctl = rc.ctl;
  float (*lx)[128] = ctl->l_x[n_seg & 1];
  uint64_t* epi = &ctl->epi[n_seg & 1];
  if (!last_wg) {
    if (!mbar_wait(&ctl->m_pub[last % kWG], (last / kWG) & 1, rc.abort_flag)) return false;
    lx[0][rc.row_t] = l;
    lx[1][rc.row_t] = m_loc;
    warp_arrive(epi, rc.lane);
    return true;
  }
  if (!mbar_wait(epi, (n_seg >> 1) & 1, rc.abort_flag)) return false;
  const float m_o = lx[1][rc.row_t];
  l_tot = l + (m_o == -INFINITY ? 0.f : lx[0][rc.row_t] * ex2_approx(m_o - m_loc));
  if (!wait_c(&ctl->o_done, n_seg & 1, rc.abort_flag)) return false;
  tc_fence_after();
  return true;
}

}  // namespace core

#endif  // SPECEXT_CORE_CUH_
