// Hybrid Tree Attention with one CTA per worker, on the pipeline of core.cuh: split-over-KV partial attention of the
// stacked (query head x tree node) rows of one KV head, in row blocks of 128, against 128-key tiles of the prefix and the
// tree.  Taken for head_dim 64, for at most 128 stacked rows (targets without grouped heads, single-token steps, draft models)
// and, in clusters, for more rows on short prefixes.  (Longer ones with head_dim 128 and more than 128 rows go to the pairs of
// attn_tc2.cu; the line is drawn at cluster_size in api.cu.)
//
// A worker owns a range of (problem, key tile) units; the part of the range inside one problem is a segment and ends with
// one partial result (unnormalised O, reference maximum, row sum) in the workspace.
//
// What bounds it: memory.  A K/V tile of 64 KB is 3.0 K cycles of an SM's share of the copy rate, a softmax warpgroup
// needs ~3.3 K for a tile and two alternate.  Measured (us per call, replayed; before: two row tiles of one CTA, whose
// second softmax warpgroup had nothing to do here and whose S, P and PV of a tile formed one chain):
//   32 heads of their own, 60 nodes, 8K prefix    40.3 -> 27.3   4.9 TB/s of K/V; 16K 64.9 -> 46.5
//   32 query / 8 KV heads, one node, 16K prefix   27.9 -> 19.3   128K 113.8 -> 87.5 = 6.1 TB/s
//   12 heads x 64, 8 nodes, 4K prefix             15.6 -> 9.6
//
// MERGE != 0: the workers of a problem form one cluster and merge their results among themselves (1 through shared memory,
// 2 through L2, 3 through L2 with more than 8 CTAs), so that the call is one kernel: no second launch waiting for the
// slowest block of the first.
//
// Warps: 0-7 softmax (two warpgroups), 8 TMA producer of K and V, 9 issuer of the S MMAs, 10 of the PV MMAs, 11 ancestor
// masks of the tree and TMA producer of Q.  Every wait is bounded; an expired wait raises SPECEXT_ERR_TIMEOUT, and all
// threads reach the final barrier before tensor memory is freed.
//
// The kernel is launched with programmatic stream serialization: barrier set-up, tensor-memory allocation and the
// start-up barrier run while the kernel before it in the stream finishes.  Each role waits for that kernel just before its own
// first read or write of global memory or, if that comes earlier, its first bounded wait, with the place of its first tile
// worked out, and the first tiles are asked for in L2 ahead of the wait.  Between the release and the request for the first K
// tile 1.2 to 2.0 us went by when all threads waited at one place and the producer asked for L2 itself, now 0.5; us per pass,
// launched one by one: four layers at 1K with scores and retrieval 53.0 -> 50.0, two layers of 12 x 64 heads on a 1K cache
// 16.4 -> 15.8, four layers of 32 KV heads at 8K 137.3 -> 135.0, eight layers of 64 query heads at 1.4K 111.1 -> 106.9.  (The
// issuers without that wait, ahead of the release in a wait of about a second at most: 0.1 us a call less with 240 rows at 1K,
// nothing elsewhere; with a limit that starts at the release, a state word of the CTA that every wait looks at, 0.2 us more.)
#include <atomic>

#include "common.cuh"
#include "core.cuh"
#include "tmap.h"

using namespace core;

namespace {

struct VerifyMaps {
  CUtensorMap q, kp, vp, kt, vt;
};

// The segments of a worker's unit range, in order.
template <bool DEVLEN>
struct VerifyWork {
  const AttnPlan& p;
  int u, hi, tph_eff;
  int prob, tile_lo, n;
  SpxSeg sg;
  __device__ __forceinline__ VerifyWork(const AttnPlan& plan, int lo, int hi_, int tph) : p(plan), u(lo), hi(hi_), tph_eff(tph) {}
  // next segment, an empty one (no tile of it exists at the device-side length) included
  __device__ __forceinline__ bool next_any() {
    if (u >= hi) return false;
    prob = u / p.UPP;
    tile_lo = u - prob * p.UPP;
    const int n_units = min(p.UPP - tile_lo, hi - u);
    u += n_units;
    n = n_units;
    if (DEVLEN) {
      sg = spx_segment(p, tile_lo, n_units, tph_eff);
      n = sg.n;
    }
    return true;
  }
  __device__ __forceinline__ bool next() {
    while (next_any())
      if (!DEVLEN || n > 0) return true;
    return false;
  }
  __device__ __forceinline__ int tile(int j) const { return DEVLEN ? spx_seg_tile(p, sg, tile_lo, j) : tile_lo + j; }
};

// End of a worker that is one of the CTAs of a cluster: every CTA has an unnormalised O, a reference maximum and a row sum
// for the same rows.  Each CTA passes its part on, the cluster meets, and each CTA adds up and writes its share of O.  How
// depends on the number of rows of the call.
//
// Up to 32: through the other CTAs' shared memory, the rows dealt in equal runs.  More: through the workspace, that is through
// L2, the columns dealt in units of 8.  Shared memory of another CTA takes stores at ~20 GB/s, 64 KB of 128 rows in 3 us; L2
// costs two of its latencies.  us per call, by shared memory / by L2, when the parts still went where Q and the rings had been
// and the CTAs therefore met twice: 4 rows on 2K 8.0 / 8.5, 12 x 64 heads with 8 rows 7.4 / 7.6, 10 rows of 32 KV heads
// 10.2 / 10.1, 40 rows 8.3 / 7.6, 120 rows at 8K 17.2 / 15.9, 240 rows at 1K 10.6 / 9.7.  Room of its own for the parts (see
// Layout) saves the first meeting, 0.5 to 0.9 us; launched one by one, us per pass: two draft layers of 12 x 64 heads, 8 rows
// 15.8 -> 15.0, one with 1 row 7.3 -> 6.8, 1 row of 32 KV heads on a 1K cache 10.3 -> 9.8, 4 rows 9.6 -> 9.1.
// (Bulk copies between the CTAs instead of stores were slower than either: 8.8, 7.7, 10.5, 8.1, 17.7, 11.2.  Through L2, (m, l)
// passed through shared memory and a CTA's own part of its share kept in tensor memory instead of going through L2 too: 240
// rows at 1K 12.5 -> 13.2 us a call, 60 rows of 32 KV heads at 8K 33.8 -> 34.6.)  The line at 32 rows stands where it was with two
// meetings: more rows need more room than Q gives up.  The other way round where the tiles are many: 60 rows of 32 KV heads at 8K
// are 0.5 us shorter through shared memory.  Each is an instantiation of its own: with both in one kernel a call was 0.1 to 0.3 us
// longer.  The forms through shared memory spill for head_dim 128 and for the device-side length (8 bytes of stack, 328 to 352
// bytes of reloads), in the exchange; those through L2 do not.  (Without clusters the forms without scores spill: 16 bytes of stack
// and 180 of reloads, 8 and 48 with the device-side length.)
struct MergeCtx {
  int cs, rank;            // CTAs of the cluster, this one
  int prob, g, rblk;       // the problem
  int n_rows, log_g;
  float m, l;              // of this thread's row in this CTA
  bool any;                // this CTA had a key tile (else: zeros of weight zero)
};
constexpr int kMaxCluster = 16;
constexpr int kRowsBySmem = kSpxClusterRowsBySmem;

// Shared memory of an instantiation: the pipeline's (core.cuh) and, behind its control block, what the CTAs of a cluster write
// into each other (MERGE 1): c CTAs x ceil(rows / c) parts of rows, at most 36 for up to 32 rows and 8 CTAs, of D floats and
// (m, l).  With head_dim 128 the room comes from Q, which has at most 32 rows there (AttnPlan::q_rows).
template <int D, int MERGE>
struct Layout {
  static constexpr int kCtrl = Geo<1, D>::kCtrlOffset - (MERGE == 1 && D == 128 ? 8192 : 0);
  static constexpr int kExchange = kCtrl + kCtrlBytes;
  static constexpr int kBytes = kExchange + (MERGE == 1 ? 36 * (D * 4 + 8) : 0) + 1024;
  static_assert(kBytes <= 232448, "more shared memory than a CTA can have");
};
static_assert(kRowsBySmem <= 32, "Layout has room for 36 parts");
constexpr float kLn2 = 0.693147180559945309417f;

// This thread's half row of O.
template <int D>
__device__ __forceinline__ void own_half_row(const RowCtx& rc, bool any, uint32_t (&v)[D / 64][32]) {
  if (any) {
#pragma unroll
    for (int c = 0; c < D / 64; ++c) tmem_ld32(rc.lane_tmem + kColO + rc.w * (D / 2) + c * 32, v[c]);
    tmem_wait_ld();
    tc_fence_before();
  } else {
#pragma unroll
    for (int k = 0; k < D / 2; ++k) v[k / 32][k % 32] = 0u;
  }
}

template <int D>
__device__ __forceinline__ void merge_by_smem(const AttnArgs& a, const RowCtx& rc, unsigned char* room, const MergeCtx& mc,
                                              bool ok) {
  cluster_wait();                                                  // every CTA of the cluster has started
  constexpr int kCols = D / 4;                                     // 16-byte columns of a row
  const AttnPlan& p = a.plan;
  const int cs = mc.cs, run = (mc.n_rows + cs - 1) / cs;           // rows of a CTA
  // received: [source CTA][row of the run][column, swizzled by the row so that a warp's rows use all banks]
  float4* part = reinterpret_cast<float4*>(room);
  float2* ml = reinterpret_cast<float2*>(part + cs * run * kCols);
  if (ok && rc.row_t - rc.lane < mc.n_rows) {
    uint32_t v[D / 64][32];
    own_half_row<D>(rc, mc.any, v);
    if (rc.row_t < mc.n_rows) {
      const int owner = rc.row_t / run, slot = mc.rank * run + rc.row_t - owner * run;
      const uint32_t dst = map_to_cta(smem_u32(part + slot * kCols), owner);
#pragma unroll
      for (int c = 0; c < kCols / 2; ++c)
        st_cluster_v4(dst + (((rc.w * (kCols / 2) + c) ^ (rc.row_t & (kCols - 1))) << 4), v[c / 8][c % 8 * 4],
                      v[c / 8][c % 8 * 4 + 1], v[c / 8][c % 8 * 4 + 2], v[c / 8][c % 8 * 4 + 3]);
      if (rc.w == 0) st_cluster_v2(map_to_cta(smem_u32(ml + slot), owner), mc.m, mc.l);
    }
  }
  __syncwarp();
  cluster_sync();
  if (!ok) return;
  const int n_mine = min(run, mc.n_rows - mc.rank * run);
  constexpr int kRowsPerWarp = 32 / kCols;                         // 1, or 2 with head_dim 64
  const int sub = rc.lane / kCols, col = rc.lane - sub * kCols;
  for (int i = (rc.w * 4 + rc.row_t / 32) * kRowsPerWarp + sub; i < n_mine; i += 8 * kRowsPerWarp) {
    const int row = mc.rank * run + i;
    float w[8], M = -INFINITY, Z = 0.f;
    float4 x[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      if (c < cs) {
        w[c] = ml[c * run + i].x;
        x[c] = part[(c * run + i) * kCols + (col ^ (row & (kCols - 1)))];
        M = fmaxf(M, w[c]);
      }
    }
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      if (c < cs) {
        const float f = ex2_approx(w[c] - M);
        Z = fmaf(ml[c * run + i].y, f, Z);
        acc.x = fmaf(f, x[c].x, acc.x);
        acc.y = fmaf(f, x[c].y, acc.y);
        acc.z = fmaf(f, x[c].z, acc.z);
        acc.w = fmaf(f, x[c].w, acc.w);
      }
    }
    const float inv = 1.f / Z;
    const int r = mc.rblk * 128 + row, t = r >> mc.log_g, h = mc.g * p.G + (r & (p.G - 1));
    *reinterpret_cast<uint2*>(a.O + (long long)t * a.o_st + (long long)h * a.o_sh + col * 4) =
        make_uint2(pack_bf16x2(acc.x * inv, acc.y * inv), pack_bf16x2(acc.z * inv, acc.w * inv));
    if (col == 0) a.lse[(long long)h * p.T + t] = (M + log2f(Z)) * kLn2;
  }
}

// MAX: bound on the cluster's size (8 or 16).
template <int D, int MAX>
__device__ __forceinline__ void merge_by_l2(const AttnArgs& a, const RowCtx& rc, const MergeCtx& mc, bool ok) {
  constexpr int kUnits = D / 8;
  const AttnPlan& p = a.plan;
  const int cs = mc.cs;
  // [CTA][D / 4][128 rows] of float4 and [CTA][128 rows] of (m, l)
  float4* part = reinterpret_cast<float4*>(a.ws + p.off_part_o) + (long long)mc.prob * cs * (D / 4) * 128;
  float2* ml = reinterpret_cast<float2*>(a.ws + p.off_part_m) + mc.prob * cs * 128;
  if (ok && rc.row_t - rc.lane < mc.n_rows) {
    uint32_t v[D / 64][32];
    own_half_row<D>(rc, mc.any, v);
    if (rc.row_t < mc.n_rows) {
      uint4* dst = reinterpret_cast<uint4*>(part) + (mc.rank * (D / 4) + rc.w * (D / 8)) * 128 + rc.row_t;
#pragma unroll
      for (int q = 0; q < D / 8; ++q)
        __stcg(dst + q * 128,
               make_uint4(v[q / 8][q % 8 * 4], v[q / 8][q % 8 * 4 + 1], v[q / 8][q % 8 * 4 + 2], v[q / 8][q % 8 * 4 + 3]));
      if (rc.w == 0) __stcg(ml + mc.rank * 128 + rc.row_t, make_float2(mc.m, mc.l));
    }
  }
  __syncwarp();
  cluster_sync();
  if (!ok) return;
  const int groups = (mc.n_rows + 31) / 32;
  // 8 warps over (unit, group of 32 rows), two at a time so that their loads are in flight together
  struct Task {
    int u, row;
    float2 s[MAX];
    float4 x[MAX], y[MAX];
  };
  int group = rc.w * 4 + rc.row_t / 32, u = mc.rank;
  auto load = [&](Task& t) {
    while (group >= groups) {
      group -= groups;
      u += cs;
    }
    t.u = u;
    t.row = group * 32 + rc.lane;
    group += 8;
    if (t.u >= kUnits) return;
    const float4* src = part + t.u * 256 + t.row;
#pragma unroll
    for (int c = 0; c < MAX; ++c) {
      if (c < cs) {
        t.s[c] = __ldcg(ml + c * 128 + t.row);
        t.x[c] = __ldcg(src + c * (D / 4) * 128);
        t.y[c] = __ldcg(src + c * (D / 4) * 128 + 128);
      }
    }
  };
  auto finish = [&](const Task& t) {
    if (t.u >= kUnits || t.row >= mc.n_rows) return;
    float M = -INFINITY, Z = 0.f;
#pragma unroll
    for (int c = 0; c < MAX; ++c)
      if (c < cs) M = fmaxf(M, t.s[c].x);
    float4 acc0 = make_float4(0.f, 0.f, 0.f, 0.f), acc1 = acc0;
#pragma unroll
    for (int c = 0; c < MAX; ++c) {
      if (c < cs) {
        const float f = ex2_approx(t.s[c].x - M);
        Z = fmaf(t.s[c].y, f, Z);
        acc0.x = fmaf(f, t.x[c].x, acc0.x);
        acc0.y = fmaf(f, t.x[c].y, acc0.y);
        acc0.z = fmaf(f, t.x[c].z, acc0.z);
        acc0.w = fmaf(f, t.x[c].w, acc0.w);
        acc1.x = fmaf(f, t.y[c].x, acc1.x);
        acc1.y = fmaf(f, t.y[c].y, acc1.y);
        acc1.z = fmaf(f, t.y[c].z, acc1.z);
        acc1.w = fmaf(f, t.y[c].w, acc1.w);
      }
    }
    const float inv = 1.f / Z;
    const int r = mc.rblk * 128 + t.row, node = r >> mc.log_g, h = mc.g * p.G + (r & (p.G - 1));
    *reinterpret_cast<uint4*>(a.O + (long long)node * a.o_st + (long long)h * a.o_sh + t.u * 8) =
        make_uint4(pack_bf16x2(acc0.x * inv, acc0.y * inv), pack_bf16x2(acc0.z * inv, acc0.w * inv),
                   pack_bf16x2(acc1.x * inv, acc1.y * inv), pack_bf16x2(acc1.z * inv, acc1.w * inv));
    if (t.u == 0) a.lse[(long long)h * p.T + node] = (M + log2f(Z)) * kLn2;
  };
  if constexpr (MAX > 8) {
    // at least 9 CTAs: at most two units each, a task per warp
    Task t0;
    load(t0);
    finish(t0);
  } else {
    Task t0, t1;
    do {
      load(t0);
      load(t1);
      finish(t0);
      finish(t1);
    } while (t1.u < kUnits);
  }
}

template <int D, int MERGE, class Work>
__device__ __forceinline__ bool merge_in_cluster(const AttnArgs& a, const RowCtx& rc, unsigned char* room, const Work& work,
                                                 bool ok, float m_loc, float l) {
  const AttnPlan& p = a.plan;
  MergeCtx mc;
  mc.cs = p.cluster;
  mc.rank = (int)cluster_rank();
  mc.prob = work.prob;
  mc.g = work.prob / p.n_rblk;
  mc.rblk = work.prob - mc.g * p.n_rblk;
  mc.n_rows = min(128, p.rows - mc.rblk * 128);
  mc.log_g = 31 - __clz(p.G);
  mc.any = work.n > 0;
  mc.m = -1e30f;
  mc.l = 0.f;
  if (ok && mc.any) ok = segment_end(rc, work.n - 1, 0, m_loc, l, mc.m, mc.l);
  __syncwarp();
  if constexpr (MERGE == 1) merge_by_smem<D>(a, rc, room, mc, ok);
  else merge_by_l2<D, MERGE == 2 ? 8 : 16>(a, rc, mc, ok);
  return ok;
}

// SCORE: 0 no chunk sums; otherwise the class of the chunk size, so that each variant carries only the code it runs:
// 1 chunks of 32 keys, 2 chunks of 64 or 128 keys, 3 chunks of fewer than 32 keys.
// DEVLEN: the prefix length is read from device memory (a.L_dev) and may be shorter than the planned capacity p.L; the
// instantiation without it carries none of that code.
template <int D, int SCORE, bool DEVLEN, int MERGE>
__global__ void __launch_bounds__(kThreads, 1)
verify_kernel(const __grid_constant__ AttnArgs a, const __grid_constant__ VerifyMaps maps) {
  using G = Geo<1, D>;
  const AttnPlan& p = a.plan;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* base = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                         ~static_cast<uintptr_t>(1023));
  Ctrl* ctl = reinterpret_cast<Ctrl*>(base + Layout<D, MERGE>::kCtrl);
  volatile int* abort_flag = &ctl->abort_flag;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const G geo(p.q_rows);

  const int worker = blockIdx.x;
  const int unit_lo = spx_unit_start(p, worker), unit_hi = spx_unit_start(p, worker + 1);
  setup<1>(ctl, warp, lane);
  if constexpr (MERGE == 1) cluster_arrive_relaxed();    // (waited for before the first write to another CTA)
  // The kernel after this one may be set up while this one runs; this one reads and writes global memory, and begins a bounded
  // wait, only once the kernel before it has completed: each role waits for that itself.
  pdl_launch_dependents();
  bool ok = true;
  int L_eff = p.L;
  VerifyWork<DEVLEN> work(p, unit_lo, unit_hi, p.TPH);
  auto read_length = [&]() {
    if (DEVLEN) {
      L_eff = spx_prefix_len(a);
      work.tph_eff = (L_eff + SPX_TILE_KEYS - 1) / SPX_TILE_KEYS;
    }
  };

  if (warp == kProducerWarp) {
    // ================================ TMA producer of K and V ================================
    setmaxnreg_dec<kRegsOther>();
    if (lane == 0) {
      const uint64_t stream_once = policy_evict_first();
      const uint32_t kfull0 = smem_u32(&ctl->k_full[0]), vfull0 = smem_u32(&ctl->v_full[0]);
      unsigned char* kring = base + geo.k_off;
      unsigned char* vring = base + geo.v_off;
      int kst = 0, vst = 0;
      uint32_t kph = 1, vph = 1, n_rag = 0;
      bool more = false;
      if (!DEVLEN) more = work.next();                   // (worked out ahead of the wait)
      pdl_wait();
      if (DEVLEN) {
        read_length();
        more = work.next();
      }
      for (; ok && more; more = work.next()) {
        const int g = work.prob / p.n_rblk;
        for (int j = 0; j < work.n && ok; ++j) {
          const int tile = work.tile(j);
          const bool is_tree = tile == p.TPH;
          const int key0 = is_tree ? 0 : tile * SPX_TILE_KEYS;
          ok = wait_c(&ctl->k_empty[kst], kph, abort_flag);
          if (!ok) break;
          {
            const uint32_t bar = kfull0 + kst * 8, dst = smem_u32(kring + kst * G::kKStage);
            const CUtensorMap* m = is_tree ? &maps.kt : &maps.kp;
            arrive_expect_tx_cluster(bar, G::kKStage);
#pragma unroll
            for (int ds = 0; ds < G::kBlocks; ++ds) {
              // (no eviction hint with a device-side length: a compact cache is read again at the next draft step)
              if (DEVLEN) tma_load<1>(dst + ds * G::kKBlk, m, bar, 64 * ds, g, key0);
              else tma_load_hint<1>(dst + ds * G::kKBlk, m, bar, 64 * ds, g, key0, stream_once);
            }
          }
          if (++kst == geo.nk) {
            kst = 0;
            kph ^= 1;
          }
          ok = wait_c(&ctl->v_empty[vst], vph, abort_flag);
          if (!ok) break;
          {
            const uint32_t bar = vfull0 + vst * 8;
            unsigned char* dst = vring + vst * G::kVStage;
            const CUtensorMap* m = is_tree ? &maps.vt : &maps.vp;
            const int nk = is_tree ? SPX_TILE_KEYS : L_eff - tile * SPX_TILE_KEYS;
            if (DEVLEN && nk < SPX_TILE_KEYS) {
              // Device-side length: the tensor map spans the whole capacity, so the rows of this tile past the length
              // hold whatever the cache holds (their probabilities are zero, but zero times a NaN is a NaN).  The tile
              // lands on a barrier of its own, its tail rows are cleared (a row of a block is 128 bytes whatever the
              // swizzle), and only then is the stage handed to the MMA issuer.
              mbar_arrive_expect_tx(&ctl->v_rag, G::kVStage);
              for (int ds = 0; ds < G::kBlocks; ++ds) tma_load_3d(dst + ds * G::kVBlk, m, &ctl->v_rag, 64 * ds, g, key0);
              ok = mbar_wait(&ctl->v_rag, n_rag & 1, abort_flag);
              if (!ok) break;
              ++n_rag;
              for (int ds = 0; ds < G::kBlocks; ++ds) {
                uint4* tail = reinterpret_cast<uint4*>(dst + ds * G::kVBlk + nk * 128);
                for (int i = 0; i < (SPX_TILE_KEYS - nk) * 8; ++i) tail[i] = make_uint4(0u, 0u, 0u, 0u);
              }
              asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
              mbar_arrive(&ctl->v_full[vst]);
            } else {
              arrive_expect_tx_cluster(bar, G::kVStage);
#pragma unroll
              for (int ds = 0; ds < G::kBlocks; ++ds) {
                const uint32_t d = smem_u32(dst + ds * G::kVBlk);
                if (DEVLEN) tma_load<1>(d, m, bar, 64 * ds, g, key0);
                else tma_load_hint<1>(d, m, bar, 64 * ds, g, key0, stream_once);
              }
            }
          }
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
    read_length();
    if (lane == 0) ok = issue_s<1, D>(ctl, base, geo, work, abort_flag);
  } else if (warp == kPvWarp) {
    setmaxnreg_dec<kRegsOther>();
    if (lane == 0 && unit_lo < unit_hi) {
      // The first tile is asked for in L2 ahead of the dependency wait, by a thread that has nothing else to do yet; the second one
      // too where a worker has several: 16K 19.6 -> 19.3, 128K 88.3 -> 87.5, but 2K 8.1 -> 8.4.  A prefetch changes no result:
      // what the kernel before may still write to these lines goes through L2 as well.
      // A device-side length is looked at here as it stands (the kernel before may be about to change it, so it decides about
      // this request and nothing else): a cache that is partly filled does not read the rest of its capacity.  us per pass of
      // two calls, no request / asked for whatever the length / as it is, 10 nodes of 32 query / 8 KV heads: 2048 tokens of
      // 8192 24.5 / 26.4 / 24.7, 4096 27.6 / 28.0 / 27.3, all 30.3 / 29.5 / 29.0, 16384 of 16384 46.6 / 42.7 / 42.5.
      const int prob = unit_lo / p.UPP, tile = unit_lo - prob * p.UPP, g = prob / p.n_rblk;
      const int tph_now = DEVLEN ? (spx_prefix_len(a) + SPX_TILE_KEYS - 1) / SPX_TILE_KEYS : p.TPH;
      for (int i = 0; i < (unit_hi - unit_lo >= 6 ? 2 : 1); ++i) {
        if (tile + i > p.TPH) break;
        const bool is_tree = tile + i == p.TPH;
        if (DEVLEN && !is_tree && tile + i >= tph_now) break;
        const int key0 = is_tree ? 0 : (tile + i) * SPX_TILE_KEYS;
#pragma unroll
        for (int ds = 0; ds < G::kBlocks; ++ds) tma_prefetch_3d(is_tree ? &maps.kt : &maps.kp, 64 * ds, g, key0);
#pragma unroll
        for (int ds = 0; ds < G::kBlocks; ++ds) tma_prefetch_3d(is_tree ? &maps.vt : &maps.vp, 64 * ds, g, key0);
      }
    }
    pdl_wait();
    read_length();
    if (lane == 0) ok = issue_pv<1, D>(ctl, base, geo, work, abort_flag);
  } else if (warp == kTreeWarp) {
    // ================================ ancestor masks, TMA producer of Q =======================
    setmaxnreg_dec<kRegsOther>();
    // boxes of 64 elements x G heads x q_rows/G nodes: exactly the stacked rows (G is a power of two), rows past the
    // tree zero-filled
    const uint32_t q_bar = smem_u32(&ctl->q_full);
    auto load_q = [&](int prob) {
      const int g = prob / p.n_rblk, rblk = prob - g * p.n_rblk;
      arrive_expect_tx_cluster(q_bar, geo.q_blk * G::kBlocks);
#pragma unroll
      for (int ds = 0; ds < G::kBlocks; ++ds)
        tma_load<1>(smem_u32(base + ds * geo.q_blk), &maps.q, q_bar, 64 * ds, g * p.G, rblk * p.RB / p.G);
    };
    // the first segment's; later ones below
    bool any = false;
    if (!DEVLEN) any = work.next();
    pdl_wait();
    if (DEVLEN) {
      read_length();
      any = work.next();
    }
    if (lane == 0 && any) load_q(work.prob);
    __syncwarp();
#pragma unroll
    for (int q = 0; q < kSpxMaxTree / 32; ++q) ctl->parent[lane + 32 * q] = lane + 32 * q < p.T ? a.parent[lane + 32 * q] : -1;
    __syncwarp();
    bool bad = false;
#pragma unroll 1
    for (int q = 0; q < kSpxMaxTree / 32; ++q) {
      const int t = lane + 32 * q;
      SpxMask128 m = {0ull, 0ull};
      if (t < p.T) m = spx_walk_up(ctl->parent, p.T, t, bad);
      ctl->anc[t][0] = m.lo;
      ctl->anc[t][1] = m.hi;
    }
    if (bad && blockIdx.x == 0) spx_raise(a.status, SPECEXT_ERR_BAD_TREE);
    warp_arrive(&ctl->anc_ready, lane);
    if (lane == 0) {
      for (uint32_t seg = 0; ok && work.next(); ++seg) {
        ok = wait_c(&ctl->q_empty, seg & 1, abort_flag);
        if (ok) load_q(work.prob);
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
    rc.s_free = smem_u32(&ctl->s_free[rc.w]);
    rc.p_full = smem_u32(&ctl->p_full[rc.w]);
    rc.scale2 = p.scale2;
    rc.abort_flag = abort_flag;
    const int rr = rc.row_t;                             // row inside the row block
    uint32_t t0 = 0, seg = 0;                            // tiles and segments before the current segment
    bool anc_seen = false;
    float m_loc, l;                                      // l is relative to m_loc
    if (rr - lane >= p.rows) {
      // No row block reaches this warp's rows: zeros for the PV MMAs to read there, once.  (Rows of zeros cost the tensor cores
      // next to no power, see lay_out in api.cu.)
      uint32_t z[16];
#pragma unroll
      for (int k = 0; k < 16; ++k) z[k] = 0u;
#pragma unroll
      for (int c = 0; c < 4; ++c) tmem_st16(rc.lane_tmem + kColP + rc.w * 64 + c * 16, z);
      tmem_wait_st();
      tc_fence_before();
    }
    pdl_wait();
    read_length();
    while (ok && work.next_any()) {
      const int prob = work.prob, g = prob / p.n_rblk, rblk = prob - g * p.n_rblk, n = work.n;
      const int r = rblk * p.RB + rr;
      const bool valid = r < p.rows;
      const bool warp_valid = r - lane < p.rows;
      rc.pad = !valid;
      const int slot = worker + prob;
      float* po = a.ws + p.off_part_o + (long long)slot * (D / 4) * p.RB * 4;
      // this warpgroup's half of the output columns, in groups of 16
      constexpr int kGroups = D / 16 / kWG;
      const int c_lo = rc.w * kGroups;
      if (MERGE == 0 && DEVLEN && n == 0) {
        // No tile of this run exists at the device-side length: its slot gets the neutral partial (weight zero in
        // the merge), and no barrier of the pipeline is touched.
        if (valid) {
#pragma unroll 4
          for (int q4 = c_lo * 4; q4 < (c_lo + kGroups) * 4; ++q4)
            *reinterpret_cast<float4*>(po + ((long long)q4 * p.RB + rr) * 4) = make_float4(0.f, 0.f, 0.f, 0.f);
          if (rc.w == 0) {
            a.ws[p.off_part_m + (long long)slot * p.RB + rr] = -1e30f;      // finite: see the merge
            a.ws[p.off_part_l + (long long)slot * p.RB + rr] = 0.f;
          }
        }
        continue;
      }
      const int t_node = valid ? r / p.G : 0;
      m_loc = -INFINITY;
      l = 0.f;
      for (int j = (rc.w ^ t0) & 1; j < n && ok; j += kWG) {
        if (!warp_valid) {
          ok = skip_tile(rc, t0 + j);
          continue;
        }
        const int tile = work.tile(j);
        const bool is_tree = tile == p.TPH;
        const int nkeys = is_tree ? p.T : min(SPX_TILE_KEYS, L_eff - tile * SPX_TILE_KEYS);
        if (is_tree && !anc_seen) {
          ok = mbar_wait(&ctl->anc_ready, 0, abort_flag);
          if (!ok) break;
          anc_seen = true;
        }
        float cg[4];                                     // sums of the tile's four groups of 32 keys
        float* mass = nullptr;
        long long rowbase = 0;
        if (SCORE != 0 && !is_tree) {
          rowbase = ((long long)prob * p.TPH + tile) * p.RB + rr;
          mass = a.ws + p.off_mass + rowbase * p.CPT;
        }
        ok = softmax_tile<D>(
            rc, t0 + j, j == 0, is_tree || nkeys < SPX_TILE_KEYS,
            [&](unsigned long long& lo, unsigned long long& hi) {
              if (is_tree) {               // this node and its ancestors (a padding row sees key 0)
                lo = valid ? ctl->anc[t_node][0] : 1ull;
                hi = valid ? ctl->anc[t_node][1] : 0ull;
              } else {
                lo = nkeys >= 64 ? ~0ull : ((1ull << nkeys) - 1ull);
                hi = nkeys <= 64 ? 0ull : ((1ull << (nkeys - 64)) - 1ull);
              }
            },
            [&](int c, const uint32_t (&v)[32], float sum) {
              if (SCORE == 1 || SCORE == 2) {
                cg[c] = sum;
              } else if (SCORE == 3 && mass) {
                float acc = 0.f;
                float* dst = mass + c * (32 / p.C);      // (one division here, none per store)
#pragma unroll
                for (int k = 0; k < 32; ++k) {
                  acc += __uint_as_float(v[k]);
                  if (((k + 1) & (p.C - 1)) == 0) {
                    *dst++ = acc;
                    acc = 0.f;
                  }
                }
              }
            },
            m_loc, l);
        if (SCORE != 0 && ok && mass) {
          if (SCORE == 1) {
            *reinterpret_cast<float4*>(mass) = make_float4(cg[0], cg[1], cg[2], cg[3]);
          } else if (SCORE == 2) {
            if (p.C == 64)
              *reinterpret_cast<float2*>(mass) = make_float2(cg[0] + cg[1], cg[2] + cg[3]);
            else
              *mass = (cg[0] + cg[1]) + (cg[2] + cg[3]);
          }
          a.ws[p.off_mref + rowbase] = m_loc;
        }
      }
      if (!ok) break;

      if (MERGE != 0) break;                                  // (its end is below: a worker of a cluster has one segment)

      // ---- end of the segment: unnormalised O, reference maximum and row sum to the partial slot ----
      float m_fin, l_tot;
      ok = segment_end(rc, t0 + n - 1, seg, m_loc, l, m_fin, l_tot);
      if (!ok) break;
      if (warp_valid) {
#pragma unroll
        for (int c = 0; c < kGroups; ++c) {
          uint32_t v[16];
          tmem_ld16(rc.lane_tmem + kColO + (c_lo + c) * 16, v);
          tmem_wait_ld();
#pragma unroll
          for (int q4 = 0; q4 < 4; ++q4) {
            const float4 x = make_float4(__uint_as_float(v[q4 * 4]), __uint_as_float(v[q4 * 4 + 1]),
                                         __uint_as_float(v[q4 * 4 + 2]), __uint_as_float(v[q4 * 4 + 3]));
            if (valid) *reinterpret_cast<float4*>(po + ((long long)((c_lo + c) * 4 + q4) * p.RB + rr) * 4) = x;
          }
        }
      }
      if (rc.w == 0 && valid) {                          // rows past the last stacked row are never read
        a.ws[p.off_part_m + (long long)slot * p.RB + rr] = m_fin;
        a.ws[p.off_part_l + (long long)slot * p.RB + rr] = l_tot;
      }
      tc_fence_before();
      warp_arrive(&ctl->o_free, lane);
      t0 += n;
      ++seg;
    }
    if constexpr (MERGE != 0) ok = merge_in_cluster<D, MERGE>(a, rc, base + Layout<D, MERGE>::kExchange, work, ok, m_loc, l);
  }
  if constexpr (MERGE != 0) {
    if (warp >= kProducerWarp) {                         // the meetings of merge_in_cluster
      __syncwarp();
      if (MERGE == 1) cluster_wait();
      cluster_sync();
    }
  }

  if (!ok) {
    if (lane == 0) spx_raise(a.status, SPECEXT_ERR_TIMEOUT);
    settle();
  }
  finish<1>(ctl, warp);
}

template <int D, int SCORE, bool DEVLEN, int MERGE>
cudaError_t launch(const AttnArgs& a, const VerifyMaps& maps, cudaStream_t st) {
  static SpxOncePerDevice once;
  constexpr int smem = Layout<D, MERGE>::kBytes;
  const cudaError_t ec = spx_opt_in_smem(verify_kernel<D, SCORE, DEVLEN, MERGE>, smem, &once, MERGE != 0);
  if (ec != cudaSuccess) return ec;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(a.plan.n_cta);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = a.plan.cluster;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = MERGE != 0 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, verify_kernel<D, SCORE, DEVLEN, MERGE>, a, maps);
}

template <int D, int MERGE>
cudaError_t launch_class(const AttnArgs& a, const VerifyMaps& maps, cudaStream_t st) {
  const AttnPlan& p = a.plan;
  if (a.L_dev) return launch<D, 0, true, MERGE>(a, maps, st);       // never with chunk sums
  if (!p.want_score) return launch<D, 0, false, MERGE>(a, maps, st);
  return p.C == 32 ? launch<D, 1, false, MERGE>(a, maps, st)
         : p.C > 32 ? launch<D, 2, false, MERGE>(a, maps, st)
                    : launch<D, 3, false, MERGE>(a, maps, st);
}

template <int MERGE>
cudaError_t launch_dim(const AttnArgs& a, const VerifyMaps& maps, cudaStream_t st) {
  return a.plan.D == 128 ? launch_class<128, MERGE>(a, maps, st) : launch_class<64, MERGE>(a, maps, st);
}

}  // namespace

// How many clusters of `size` CTAs of this kernel device `dev` (the current one) holds at once, looked up once per device
// and size; 0 when there is no device.
int spx_verify_max_clusters(int dev, int size) {
  static std::atomic<int> known[kSpxMaxDevices][kMaxCluster + 1];
  if (dev < 0 || dev >= kSpxMaxDevices || size < 1 || size > kMaxCluster) return 0;
  int n = known[dev][size].load();
  if (n > 0) return n - 1;
  auto* kernel = verify_kernel<128, 0, false, 3>;
  static SpxOncePerDevice once;
  constexpr int smem = Layout<128, 3>::kBytes;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(size);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = size;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (spx_opt_in_smem(kernel, smem, &once, true) != cudaSuccess || cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
    (void)cudaGetLastError();
    return 0;
  }
  known[dev][size].store(n + 1);
  return n;
}

// Row blocks of 128 (plan.RB); plan.n_cta counts CTAs.
cudaError_t spx_launch_verify(const AttnArgs& a, cudaStream_t st, int* n_launches) {
  const AttnPlan& p = a.plan;
  VerifyMaps maps;
  bool ok = spx_encode_map(&maps.kt, a.Kt, p.D, p.Hkv, a.tkv_sh, p.T, a.tkv_st, 1, SPX_TILE_KEYS);
  ok = ok && spx_encode_map(&maps.vt, a.Vt, p.D, p.Hkv, a.tkv_sh, p.T, a.tkv_st, 1, SPX_TILE_KEYS);
  if (p.L > 0) {
    ok = ok && spx_encode_map(&maps.kp, a.Kp, p.D, p.Hkv, a.kv_sh, p.L, a.kv_sl, 1, SPX_TILE_KEYS);
    ok = ok && spx_encode_map(&maps.vp, a.Vp, p.D, p.Hkv, a.kv_sh, p.L, a.kv_sl, 1, SPX_TILE_KEYS);
  } else {
    maps.kp = maps.kt;
    maps.vp = maps.vt;
  }
  ok = ok && spx_encode_map(&maps.q, a.Q, p.D, p.Hq, a.q_sh, p.T, a.q_st, p.G, p.q_rows / p.G);
  if (!ok) return cudaErrorInvalidValue;
  const int merge = p.cluster == 0 ? 0 : p.rows <= kRowsBySmem ? 1 : p.cluster <= 8 ? 2 : 3;
  cudaError_t e;
  switch (merge) {
    case 0: e = launch_dim<0>(a, maps, st); break;
    case 1: e = launch_dim<1>(a, maps, st); break;
    case 2: e = launch_dim<2>(a, maps, st); break;
    default: e = launch_dim<3>(a, maps, st); break;
  }
  *n_launches += 1;
  return e;
}
