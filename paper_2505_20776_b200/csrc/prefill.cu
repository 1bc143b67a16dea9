// Prefill (causal self-attention of the prompt) on pairs of SMs, on the pipeline of core.cuh.
//
// A problem is one KV head and one block of tb = 256 / G consecutive prompt tokens: the block's G * tb = 256 stacked
// query rows (row = token * G + head in group) attend to the keys 0 .. end of the block.  Keys are taken in 128-key tiles
// aligned at multiples of 128; the tiles that end at or before the block's first token are fully visible, the last one
// or two ("diagonal") tiles are masked per row (key j is visible to token i iff j <= i).  A problem is processed from its
// first to its last tile by one cluster, so its result is final: O = sum / row sum and lse are written by the kernel
// itself; there are no partial results and no merge.  Problems are dealt to the clusters longest first, in
// boustrophedon order, which balances the triangular work to within one problem; the Q rows and the first S tiles of the
// next problem are fetched and computed under the last tiles of the one before.
//
// What bounds it: the tensor pipe's 1.0 K cycles a tile, the special-function unit's 1.0 K and the power cap together.
// Between problems the warpgroup of the last tile writes O and the other one is already in the next problem (core.cuh,
// segment_handover).  us per call, replayed, against the same loop with one P buffer, Q in tensor memory by plain loads and a
// stop between problems / with both warpgroups ending a problem (32 query / 8 KV heads): 1K tokens 22.6 / 20.5 -> 18.4,
// 2K 52.5 / 45.0 -> 40.6, 4K 135 / 121 -> 115, 16K 1655 / 1628 -> 1600 (1374 TFLOP/s; under the power cap 1825 -> 1720
// before the last step).  Each role waits for the kernel before just ahead of its own first access or bounded wait, with
// its first problem worked out, and an idle thread asks for the first tile in L2 ahead of the wait: one by one 2K 43.6 -> 42.9,
// 1.8K with 64 query heads 66.0 -> 65.4; 16K the same.  Prefetching the tensor maps by the producer costs 0.4 us at 2K and helps
// nowhere.  Slower than that loop are prompts of at most 16 tokens with many KV heads, a single tile on every cluster: 48 heads of
// their own with 8 tokens 5.6 -> 6.2, 32 5.4 -> 5.9, 12 5.3 -> 5.5; 33 tokens 6.4 -> 6.3, 6.1 -> 5.8, 6.3 -> 5.7.
#include "common.cuh"
#include "core.cuh"
#include "tmap.h"

using namespace core;

namespace {

constexpr int D = 128;
constexpr float kLn2 = 0.693147180559945309417f;

struct PrefillArgs {
  __nv_bfloat16* O;
  float* lse;
  int32_t* status;
  long long o_st, o_sh;
  int L, Hkv, G;
  int tb;          // tokens per block = 256 / G
  int nb;          // blocks = ceil(L / tb)
  int n_prob;      // nb * Hkv
  int W;           // clusters
  float scale2;    // softmax_scale * log2(e)
};

struct PrefillMaps {
  CUtensorMap q;         // [L][Hq][128], boxes of the 128 stacked rows of one CTA x 64 elements
  CUtensorMap k, v;      // [L][Hkv][128], boxes 64 x 1 x 64 (K halves) and 64 x 1 x 128 (V halves)
};

// The problems of cluster `cl`: numbered longest first and dealt out back and forth.
struct PrefillWork {
  const PrefillArgs& a;
  int cl, rnd = 0;
  int b, g, n;
  __device__ __forceinline__ PrefillWork(const PrefillArgs& args, int cluster) : a(args), cl(cluster) {}
  __device__ __forceinline__ bool next() {
    for (;; ++rnd) {
      if (rnd * a.W >= a.n_prob) return false;
      const int pos = rnd * a.W + ((rnd & 1) ? a.W - 1 - cl : cl);
      if (pos >= a.n_prob) continue;
      ++rnd;
      b = a.nb - 1 - pos / a.Hkv;
      g = pos % a.Hkv;
      n = (min((b + 1) * a.tb, a.L) + SPX_TILE_KEYS - 1) / SPX_TILE_KEYS;
      return true;
    }
  }
};

__global__ void __launch_bounds__(kThreads, 1)
prefill_kernel(const __grid_constant__ PrefillArgs a, const __grid_constant__ PrefillMaps maps) {
  using G = Geo<2, D>;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* base = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                         ~static_cast<uintptr_t>(1023));
  Ctrl* ctl = reinterpret_cast<Ctrl*>(base + G::kCtrlOffset);
  volatile int* abort_flag = &ctl->abort_flag;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const G geo(128);

  setup<2, true>(ctl, warp, lane);
  const uint32_t rank = cluster_rank();
  PrefillWork work(a, blockIdx.x >> 1);
  // Global memory is read and written, and a bounded wait begun, only once the kernel before has completed: each role waits for
  // that itself.
  pdl_launch_dependents();
  bool ok = true;

  if (warp == kProducerWarp) {
    // ================================ TMA producer of K and V (each CTA loads its halves) =====
    setmaxnreg_dec<kRegsOther>();
    if (lane == 0) {
      const uint32_t kfull0 = leader_addr<2>(&ctl->k_full[0]), vfull0 = leader_addr<2>(&ctl->v_full[0]);
      int kst = 0, vst = 0;
      uint32_t kph = 1, vph = 1;
      bool more = work.next();                           // (worked out ahead of the wait)
      pdl_wait();
      for (; ok && more; more = work.next()) {
        for (int tile = 0; tile < work.n && ok; ++tile) {
          const int key0 = tile * SPX_TILE_KEYS;
          ok = wait_c(&ctl->k_empty[kst], kph, abort_flag);
          if (!ok) break;
          const uint32_t kbar = kfull0 + kst * 8, kdst = smem_u32(base + geo.k_off + kst * G::kKStage);
          arrive_expect_tx_cluster(kbar, G::kKStage);
          tma_load<2>(kdst, &maps.k, kbar, 0, work.g, key0 + 64 * rank);
          tma_load<2>(kdst + G::kKBlk, &maps.k, kbar, 64, work.g, key0 + 64 * rank);
          if (++kst == geo.nk) {
            kst = 0;
            kph ^= 1;
          }
          ok = wait_c(&ctl->v_empty[vst], vph, abort_flag);
          if (!ok) break;
          const uint32_t vbar = vfull0 + vst * 8;
          arrive_expect_tx_cluster(vbar, G::kVStage);
          tma_load<2>(smem_u32(base + geo.v_off + vst * G::kVStage), &maps.v, vbar, 64 * rank, work.g, key0);
          if (++vst == geo.nv) {
            vst = 0;
            vph ^= 1;
          }
        }
      }
      if (*abort_flag) ok = false;                       // (see settle)
    }
  } else if (warp == kMmaWarp) {
    setmaxnreg_dec<kRegsOther>();
    pdl_wait();                                          // (a bounded wait must not count the time of the kernel before)
    if (lane == 0 && rank == 0) ok = issue_s<2, D>(ctl, base, geo, work, abort_flag);
  } else if (warp == kPvWarp) {
    setmaxnreg_dec<kRegsOther>();
    if (lane == 0) {
      // The first tile is asked for in L2 ahead of the dependency wait, by a thread that has nothing else to do yet.  (A prefetch
      // changes no result: what the kernel before may still write to these lines goes through L2 as well.)
      PrefillWork first = work;
      if (first.next()) {
        tma_prefetch_3d(&maps.k, 0, first.g, 64 * rank);
        tma_prefetch_3d(&maps.k, 64, first.g, 64 * rank);
        tma_prefetch_3d(&maps.v, 64 * rank, first.g, 0);
      }
    }
    pdl_wait();
    if (lane == 0 && rank == 0) ok = issue_pv<2, D>(ctl, base, geo, work, abort_flag);
  } else if (warp == kTreeWarp) {
    // ================================ TMA producer of Q =======================================
    setmaxnreg_dec<kRegsOther>();
    if (lane == 0) {
      const uint32_t bar = leader_addr<2>(&ctl->q_full);
      bool more = work.next();
      pdl_wait();
      for (uint32_t seg = 0; ok && more; ++seg, more = work.next()) {
        if (seg > 0) ok = wait_c(&ctl->q_empty, (seg - 1) & 1, abort_flag);
        if (!ok) break;
        // rows rank*128.. of the block: 128/G tokens of all G heads, or half of the heads of the one token (G = 256)
        const int tok = work.b * a.tb + (int)rank * 128 / a.G;
        const int head = work.g * a.G + (int)rank * 128 % a.G;
        arrive_expect_tx_cluster(bar, G::kQBytes);
        tma_load<2>(smem_u32(base), &maps.q, bar, 0, head, tok);
        tma_load<2>(smem_u32(base + geo.q_blk), &maps.q, bar, 64, head, tok);
      }
      if (*abort_flag) ok = false;
    }
  } else {
    // ================================ softmax warps ===========================================
    setmaxnreg_inc<kRegsSoftmax>();
    const int quarter = warp & 3;
    RowCtx rc;
    rc.ctl = ctl;
    rc.w = warp >> 2;
    rc.lane = lane;
    rc.row_t = quarter * 32 + lane;
    rc.lane_tmem = ctl->tmem_base + (static_cast<uint32_t>(quarter * 32) << 16);
    rc.s_free = leader_addr<2>(&ctl->s_free[rc.w]);
    rc.p_full = leader_addr<2>(&ctl->p_full[rc.w]);
    rc.scale2 = a.scale2;
    rc.abort_flag = abort_flag;
    rc.pad = false;                                      // (only the last block has rows behind the last one)
    const uint32_t o_free_l = leader_addr<2>(&ctl->o_free);
    const int rr = (int)rank * 128 + rc.row_t;           // row inside the 256-row block
    uint32_t t0 = 0, seg = 0;                            // tiles and problems before the current problem
    pdl_wait();
    while (ok && work.next()) {
      const int n = work.n;
      const int tok = work.b * a.tb + rr / a.G;          // this row's token
      const bool valid = tok < a.L;
      const int head = work.g * a.G + rr % a.G;
      const int tok_eff = valid ? tok : a.L - 1;         // a padding row sees what the last token sees; it is not stored
      const int block_lo = work.b * a.tb;                // tiles that end at or before this key are fully visible
      float m_loc = -INFINITY, l = 0.f;                  // l is relative to m_loc
      for (int j = (rc.w ^ t0) & 1; j < n && ok; j += kWG) {
        const int key_lo = j * SPX_TILE_KEYS;
        ok = softmax_tile<D>(
            rc, t0 + j, j == 0, key_lo + SPX_TILE_KEYS > block_lo,
            [&](unsigned long long& lo, unsigned long long& hi) {
              // keys key_lo .. key_lo + nvis - 1 are visible (none when the tile lies past this row's token)
              const int nvis = min(SPX_TILE_KEYS, max(0, tok_eff - key_lo + 1));
              lo = nvis >= 64 ? ~0ull : ((1ull << nvis) - 1ull);
              hi = nvis <= 64 ? 0ull : (nvis >= 128 ? ~0ull : ((1ull << (nvis - 64)) - 1ull));
            },
            [](int, const uint32_t (&)[32], float) {}, m_loc, l);
      }
      if (!ok) break;

      // ---- end of the problem: the result is final ----
      const bool last_wg = ((t0 + n - 1) & 1) == (uint32_t)rc.w;
      float l_tot = 1.f;
      ok = segment_handover(rc, t0 + n - 1, seg, last_wg, m_loc, l, l_tot);
      if (!ok) break;
      if (last_wg) {
        const float inv = 1.f / l_tot;
        __nv_bfloat16* out = a.O + (long long)tok * a.o_st + (long long)head * a.o_sh;
#pragma unroll
        for (int c = 0; c < D / 32; ++c) {
          uint32_t v[32];
          tmem_ld32(rc.lane_tmem + kColO + c * 32, v);
          tmem_wait_ld();
          if (c == D / 32 - 1) {
            tc_fence_before();
            warp_arrive_cluster(o_free_l, lane);         // O may be overwritten
          }
          if (valid) {
#pragma unroll
            for (int q8 = 0; q8 < 4; ++q8) {
              uint4 x;
              x.x = pack_bf16x2(__uint_as_float(v[q8 * 8]) * inv, __uint_as_float(v[q8 * 8 + 1]) * inv);
              x.y = pack_bf16x2(__uint_as_float(v[q8 * 8 + 2]) * inv, __uint_as_float(v[q8 * 8 + 3]) * inv);
              x.z = pack_bf16x2(__uint_as_float(v[q8 * 8 + 4]) * inv, __uint_as_float(v[q8 * 8 + 5]) * inv);
              x.w = pack_bf16x2(__uint_as_float(v[q8 * 8 + 6]) * inv, __uint_as_float(v[q8 * 8 + 7]) * inv);
              *reinterpret_cast<uint4*>(out + c * 32 + q8 * 8) = x;
            }
          }
        }
        if (valid) a.lse[(long long)head * a.L + tok] = (m_loc + log2f(l_tot)) * kLn2;
      }
      t0 += n;
      ++seg;
    }
  }

  if (!ok) {
    if (lane == 0) spx_raise(a.status, SPECEXT_ERR_TIMEOUT);
    settle();
  }
  finish<2>(ctl, warp);
}

}  // namespace

// Causal self-attention of L prompt tokens; head_dim 128 and G = Hq / Hkv a power of two <= 256.
cudaError_t spx_launch_prefill(const void* Q, const void* K, const void* V, void* O, float* lse, int L, int Hq, int Hkv,
                               float scale2, long long q_st, long long q_sh, long long kv_sl, long long kv_sh,
                               long long o_st, long long o_sh, int n_sm, int32_t* status, cudaStream_t st) {
  PrefillArgs a;
  a.O = static_cast<__nv_bfloat16*>(O);
  a.lse = lse;
  a.status = status;
  a.o_st = o_st; a.o_sh = o_sh;
  a.L = L; a.Hkv = Hkv; a.G = Hq / Hkv;
  a.tb = 256 / a.G;
  a.nb = (L + a.tb - 1) / a.tb;
  a.n_prob = a.nb * Hkv;
  int W = n_sm / 2;
  if (W > a.n_prob) W = a.n_prob;
  if (W < 1) W = 1;
  a.W = W;
  a.scale2 = scale2;
  PrefillMaps maps;
  const int q_heads = a.G < 128 ? a.G : 128;
  if (!spx_encode_map(&maps.q, Q, D, Hq, q_sh, L, q_st, q_heads, 128 / q_heads) ||
      !spx_encode_map(&maps.k, K, D, Hkv, kv_sh, L, kv_sl, 1, 64) ||
      !spx_encode_map(&maps.v, V, D, Hkv, kv_sh, L, kv_sl, 1, SPX_TILE_KEYS))
    return cudaErrorInvalidValue;
  static SpxOncePerDevice once;
  constexpr int smem = smem_bytes<2, D>();
  const cudaError_t ec = spx_opt_in_smem(prefill_kernel, smem, &once);
  if (ec != cudaSuccess) return ec;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * W);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, prefill_kernel, a, maps);
}
