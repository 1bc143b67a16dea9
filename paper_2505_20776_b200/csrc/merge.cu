// Log-sum-exp merge of the per-segment partial results, and the normalisation of the per-chunk
// sums into the head-averaged chunk scores that retrieval ranks.
//
// merge_kernel: for each query row: M = max_s m_s,
// Z = sum_s l_s 2^(m_s - M), lse = (M + log2 Z) ln 2, O = sum_s O~_s 2^(m_s - M) / Z.
//
// score_kernel (and score_beside, in the merge's launch): for every (tree node, chunk) sums over all query heads the chunk's exponential sum
// rescaled from its tile's reference maximum to the row's final lse, i.e. the exactly normalised
// probability mass, and divides by Hq.
#include "common.cuh"
#include "sm100.cuh"

namespace {

constexpr float kLn2 = 0.693147180559945309417f;
constexpr int kMergeSmemCap = 200 * 1024;          // bytes of dynamic shared memory requested only to limit residency
constexpr float kLog2e = 1.44269504088896340736f;
constexpr int kOneWave = 148;                      // blocks, one per SM

// Block = NT / 32 warps; warp w handles two 16-byte column groups (d4, d4 + 1) for 32 consecutive rows of
// one problem, so every partial read is a 512-byte coalesced segment, all reads of a thread are
// independent of each other, and the segment weights are computed once for eight output columns.
template <int B>
__device__ __forceinline__ void merge_batch(const float* __restrict__ pm, const float* __restrict__ pl,
                                            const float* __restrict__ po, long long ostride, int RB, int s, int n,
                                            float& M, float& Z, float4& acc0, float4& acc1) {
  // Segments s .. s+n-1 (n <= B).  Every load of the batch is in flight at once: issued one by one
  // they would each pay the full latency, and a second batch pays it a second time.
  float ms[B], ls[B];
  float4 v0[B], v1[B];
#pragma unroll
  for (int k = 0; k < B; ++k) {
    const bool in = k < n;
    const float4* q = reinterpret_cast<const float4*>(po + (s + k) * ostride);
    ms[k] = in ? __ldcg(pm + (long long)(s + k) * RB) : -INFINITY;
    ls[k] = in ? __ldcg(pl + (long long)(s + k) * RB) : 0.f;
    v0[k] = in ? __ldcg(q) : make_float4(0.f, 0.f, 0.f, 0.f);
    v1[k] = in ? __ldcg(q + RB) : make_float4(0.f, 0.f, 0.f, 0.f);     // next column group: RB float4 further on
  }
  float Mb = M;
#pragma unroll
  for (int k = 0; k < B; ++k) Mb = fmaxf(Mb, ms[k]);
  // (A worker that found no key, because a device-side length was shorter than planned, leaves the
  // neutral partial m = -1e30, l = 0, O = 0: finite, so that no difference of maxima is inf - inf.)
  const float carry = sm100::ex2_approx(M - Mb);    // 0 on the first batch (M = -inf)
  Z *= carry;
  acc0.x *= carry; acc0.y *= carry; acc0.z *= carry; acc0.w *= carry;
  acc1.x *= carry; acc1.y *= carry; acc1.z *= carry; acc1.w *= carry;
  M = Mb;
#pragma unroll
  for (int k = 0; k < B; ++k) {
    const float w = sm100::ex2_approx(ms[k] - M);
    Z = fmaf(ls[k], w, Z);
    acc0.x = fmaf(w, v0[k].x, acc0.x);
    acc0.y = fmaf(w, v0[k].y, acc0.y);
    acc0.z = fmaf(w, v0[k].z, acc0.z);
    acc0.w = fmaf(w, v0[k].w, acc0.w);
    acc1.x = fmaf(w, v1[k].x, acc1.x);
    acc1.y = fmaf(w, v1[k].y, acc1.y);
    acc1.z = fmaf(w, v1[k].z, acc1.z);
    acc1.w = fmaf(w, v1[k].w, acc1.w);
  }
}

// The partial results of a problem: slot of the first one, and how many.
__device__ __forceinline__ int segments_of(const AttnPlan& p, int prob, int& slot0) {
  int c_first, c_last;
  if (p.cpp > 0 && p.UPP >= p.cpp) {               // every one of the problem's cpp workers has a segment
    c_first = prob * p.cpp;
    c_last = c_first + p.cpp - 1;
  } else {
    c_first = spx_unit_owner(p, prob * p.UPP);
    c_last = spx_unit_owner(p, (prob + 1) * p.UPP - 1);
  }
  slot0 = c_first + prob;
  return c_last - c_first + 1;
}

// Chunk scores beside the merge: 256 threads of a block that merges with its others.  A block has one task, 64 rows of one key
// tile (VW chunks); it takes the rows' statistics from the partial results instead of waiting for the lse that the merge writes.
// A thread has one row of every fourth KV head, of two at most.  All sums have a fixed order, as in score_kernel.
constexpr int kScoreRows = 64;
constexpr int kScoreSlices = 256 / kScoreRows, kScoreHeads = 2;
template <int VW>
__device__ __forceinline__ void score_beside(const AttnArgs& a, float (&part)[kScoreSlices][kScoreRows][VW], int tid) {
  const AttnPlan& p = a.plan;
  const int rr = tid & (kScoreRows - 1), slice = tid / kScoreRows;
  const int n_groups = (p.rows + kScoreRows - 1) / kScoreRows;
  const int tile = blockIdx.x / n_groups, group = blockIdx.x - tile * n_groups, r = group * kScoreRows + rr;
  if (tile >= p.TPH) return;                       // a block that only merges
  const int nodes = kScoreRows / p.G, t0 = group * nodes;          // nodes of the group
  const float inv = 1.f / (float)p.Hq;
  const int n_heads = r < p.rows ? (p.Hkv - slice + kScoreSlices - 1) / kScoreSlices : 0;      // heads slice, slice + 4
  sm100::pdl_wait();                               // the attention kernel's results are complete
  float lse2[kScoreHeads];                         // log2 of the row's sum, its maximum included
#pragma unroll
  for (int q = 0; q < kScoreHeads; ++q) {
    lse2[q] = 0.f;
    if (q < n_heads) {
      int slot0;
      const int nseg = segments_of(p, slice + q * kScoreSlices, slot0);
      const float* pm = a.ws + p.off_part_m + (long long)slot0 * p.RB + r;
      const float* pl = a.ws + p.off_part_l + (long long)slot0 * p.RB + r;
      float M = -INFINITY, Z = 0.f;
      for (int s0 = 0; s0 < nseg; s0 += 12) {
        float ms[12], ls[12];
#pragma unroll
        for (int k = 0; k < 12; ++k) {
          ms[k] = s0 + k < nseg ? __ldcg(pm + (s0 + k) * p.RB) : -INFINITY;
          ls[k] = s0 + k < nseg ? __ldcg(pl + (s0 + k) * p.RB) : 0.f;
        }
        float Mb = M;
#pragma unroll
        for (int k = 0; k < 12; ++k) Mb = fmaxf(Mb, ms[k]);
        Z *= sm100::ex2_approx(M - Mb);            // (0 on the first batch)
        M = Mb;
#pragma unroll
        for (int k = 0; k < 12; ++k) Z = fmaf(ls[k], sm100::ex2_approx(ms[k] - M), Z);
      }
      lse2[q] = M + log2f(Z);
    }
  }
  float m[kScoreHeads][VW], ref[kScoreHeads];
#pragma unroll
  for (int q = 0; q < kScoreHeads; ++q) {
    if (q < n_heads) {
      const long long base = ((long long)(slice + q * kScoreSlices) * p.TPH + tile) * p.RB + r;
      const float* src = a.ws + p.off_mass + base * VW;
      if constexpr (VW == 4) {
        const float4 v = __ldcg(reinterpret_cast<const float4*>(src));
        m[q][0] = v.x; m[q][1] = v.y; m[q][2] = v.z; m[q][3] = v.w;
      } else if constexpr (VW == 2) {
        const float2 v = __ldcg(reinterpret_cast<const float2*>(src));
        m[q][0] = v.x; m[q][1] = v.y;
      } else {
        m[q][0] = __ldcg(src);
      }
      ref[q] = __ldcg(a.ws + p.off_mref + base);
    }
  }
  float acc[VW];
#pragma unroll
  for (int k = 0; k < VW; ++k) acc[k] = 0.f;
#pragma unroll
  for (int q = 0; q < kScoreHeads; ++q) {
    if (q < n_heads) {
      const float f = exp2f(ref[q] - lse2[q]);
#pragma unroll
      for (int k = 0; k < VW; ++k) acc[k] = fmaf(m[q][k], f, acc[k]);
    }
  }
#pragma unroll
  for (int k = 0; k < VW; ++k) part[slice][rr][k] = acc[k];
  sm100::named_bar_sync(1, 256);
  for (int o = tid; o < nodes * VW; o += 256) {
    const int tt = o / VW, k = o - tt * VW, node = t0 + tt, c = tile * VW + k;
    if (node < p.T && c < p.NC) {
      float sum = 0.f;
      for (int s = 0; s < kScoreSlices; ++s)
        for (int j = 0; j < p.G; ++j) sum += part[s][tt * p.G + j][k];
      a.chunk_score[(long long)node * p.NC + c] = sum * inv;
    }
  }
}

// VW > 0: blocks of NT + 256 threads in one line, of which the first n_merge (merge_x groups of rows times the blocks that share a
// group's columns) merge with their first NT threads; the other 256 threads add up the chunk scores of task blockIdx.x, if there
// is one.  Those 512 threads have 128 registers each and the merge spills 16 bytes (with 192 for the merge and 64 for the scores,
// setmaxnreg, nothing spills, but a pass with 64 rows and 140 tiles takes 32.7 instead of 32.3 us, 240 rows at 4K 21.2 instead of
// 21.1).
// VW = 0 (one block per SM, see launch_merge: told so, the compiler takes 242 and 107 registers a thread instead of 134 and 64 and
// keeps more of a batch in flight.  us per pass, one by one: one scored call and its retrieval at 12K with 4 rows and chunks of 16
// 35.5 -> 34.3, at 10K with 92 rows 37.2 -> 35.9, two layers at 27K with 8 rows 68.6 -> 66.9, at 36K with 4 rows 74.8 -> 73.0,
// four layers at 5K with chunks of 16 81.9 -> 80.7; no change where the power limit sets the pace.)
template <int B, int NT, int VW>
__global__ void __launch_bounds__(NT + (VW > 0 ? 256 : 0), 1) merge_kernel(const __grid_constant__ AttnArgs a, int merge_x, int n_merge) {
  const AttnPlan& p = a.plan;
  sm100::pdl_launch_dependents();
  if constexpr (VW > 0) {
    __shared__ float part[kScoreSlices][kScoreRows][VW];
    if (threadIdx.x >= NT) {
      score_beside<VW>(a, part, threadIdx.x - NT);
      return;
    }
    if ((int)blockIdx.x >= n_merge) return;
  }
  const int bx = VW > 0 ? (int)blockIdx.x % merge_x : (int)blockIdx.x, by = VW > 0 ? (int)blockIdx.x / merge_x : (int)blockIdx.y;
  // everything that needs no global memory (indices, addresses, the output position) comes before the wait
  const int blocks_per_prob = p.RB / 32;
  const int prob = bx / blocks_per_prob;
  const int rr0 = (bx - prob * blocks_per_prob) * 32;
  const int g = prob / p.n_rblk;
  const int rblk = prob - g * p.n_rblk;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rr = rr0 + lane;
  const int r = rblk * p.RB + rr;
  if (r >= p.rows) return;
  int slot0;
  const int nseg = segments_of(p, prob, slot0);
  const int nd4 = p.D / 4;
  const int d4 = (by * (NT / 32) + warp) * 2;

  const float* pm = a.ws + p.off_part_m + (long long)slot0 * p.RB + rr;
  const float* pl = a.ws + p.off_part_l + (long long)slot0 * p.RB + rr;
  const float* po = a.ws + p.off_part_o + (((long long)slot0 * nd4 + d4) * p.RB + rr) * 4;
  const long long ostride = (long long)nd4 * p.RB * 4;
  const int t = r / p.G, h = g * p.G + r % p.G;
  __nv_bfloat16* out = a.O + (long long)t * a.o_st + (long long)h * a.o_sh + d4 * 4;
  float* lse_out = a.lse + (long long)h * p.T + t;

  sm100::pdl_wait();                               // the partial results of the attention kernel are complete
  float M = -INFINITY, Z = 0.f;
  float4 acc0 = make_float4(0.f, 0.f, 0.f, 0.f), acc1 = acc0;
  for (int s = 0; s < nseg; s += B) merge_batch<B>(pm, pl, po, ostride, p.RB, s, min(B, nseg - s), M, Z, acc0, acc1);

  const float inv = 1.f / Z;
  if (d4 == 0) *lse_out = (M + log2f(Z)) * kLn2;
  __nv_bfloat162 b0 = __floats2bfloat162_rn(acc0.x * inv, acc0.y * inv);
  __nv_bfloat162 b1 = __floats2bfloat162_rn(acc0.z * inv, acc0.w * inv);
  __nv_bfloat162 b2 = __floats2bfloat162_rn(acc1.x * inv, acc1.y * inv);
  __nv_bfloat162 b3 = __floats2bfloat162_rn(acc1.z * inv, acc1.w * inv);
  uint4 pk;
  pk.x = *reinterpret_cast<uint32_t*>(&b0);
  pk.y = *reinterpret_cast<uint32_t*>(&b1);
  pk.z = *reinterpret_cast<uint32_t*>(&b2);
  pk.w = *reinterpret_cast<uint32_t*>(&b3);
  *reinterpret_cast<uint4*>(out) = pk;
}

// Block = the rows of one row block x S slices of the KV heads, for one key tile and one group of VW chunks of it: a thread
// adds up its row over the KV heads of its slice, so that every load of a warp is one contiguous piece and the loads of
// four heads are in flight at once; the G rows of a node and the slices are added through shared memory.  All sums have
// a fixed order, so the result does not depend on the run.
// What bounds it: reading the chunk sums (20 bytes per row and tile of 32-key chunks) from L2, and latency when there are
// few tiles: 2.8 us of a 4K call, 3.2 at 16K, 7.7 at 128K (42 MB, 5.5 TB/s).  A scored call against the form with one node
// per thread, whose loads were strided and waited for one another: 4K 17.2 -> 16.4 us, 16K 28.5 -> 26.8, 64 query heads
// with chunks of 64 53.9 -> 43.5 (there together with the one-piece store of the chunk sums in attn_tc2.cu).
constexpr int kScoreThreads = 512;

template <int VW>
__global__ void __launch_bounds__(kScoreThreads) score_kernel(const __grid_constant__ AttnArgs a) {
  const AttnPlan& p = a.plan;
  __shared__ __align__(16) float part[kScoreThreads][VW];
  sm100::pdl_launch_dependents();
  const int rr = threadIdx.x, slice = threadIdx.y, n_slices = blockDim.y;
  const int tile = blockIdx.x, rblk = blockIdx.z;
  const int c0 = blockIdx.y * VW;                  // first chunk of the group inside the tile
  const int r = rblk * p.RB + rr;
  const int t = r / p.G, i = r - t * p.G;
  float acc[VW];
#pragma unroll
  for (int k = 0; k < VW; ++k) acc[k] = 0.f;
  sm100::pdl_wait();                               // lse and the chunk sums are complete
  if (r < p.rows) {
    for (int g0 = slice; g0 < p.Hkv; g0 += 4 * n_slices) {
      float m[4][VW], ref[4], lse[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int g = g0 + q * n_slices;
        if (g < p.Hkv) {
          const long long base = ((long long)(g * p.n_rblk + rblk) * p.TPH + tile) * p.RB + rr;
          const float* src = a.ws + p.off_mass + base * p.CPT + c0;
          if (VW >= 4) {
#pragma unroll
            for (int e = 0; e < VW / 4; ++e) {
              const float4 v = __ldcg(reinterpret_cast<const float4*>(src) + e);
              m[q][e * 4] = v.x; m[q][(e * 4 + 1) % VW] = v.y; m[q][(e * 4 + 2) % VW] = v.z; m[q][(e * 4 + 3) % VW] = v.w;
            }
          } else if (VW == 2) {
            const float2 v = __ldcg(reinterpret_cast<const float2*>(src));
            m[q][0] = v.x; m[q][1 % VW] = v.y;
          } else {
            m[q][0] = __ldcg(src);
          }
          ref[q] = __ldcg(a.ws + p.off_mref + base);
          lse[q] = __ldcg(a.lse + (long long)(g * p.G + i) * p.T + t);
        }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (g0 + q * n_slices < p.Hkv) {
          const float f = exp2f(ref[q] - lse[q] * kLog2e);
#pragma unroll
          for (int k = 0; k < VW; ++k) acc[k] = fmaf(m[q][k], f, acc[k]);
        }
      }
    }
  }
#pragma unroll
  for (int k = 0; k < VW; ++k) part[slice * p.RB + rr][k] = acc[k];
  __syncthreads();
  const int nodes = p.RB / p.G;                    // nodes of a row block
  const float inv = 1.f / (float)p.Hq;
  for (int o = slice * p.RB + rr; o < nodes * VW; o += n_slices * p.RB) {
    const int tt = o / VW, k = o - tt * VW;
    const int node = rblk * nodes + tt, c = tile * p.CPT + c0 + k;
    if (node < p.T && c < p.NC) {
      float sum = 0.f;
      for (int s = 0; s < n_slices; ++s)
        for (int j = 0; j < p.G; ++j) sum += part[s * p.RB + tt * p.G + j][k];
      a.chunk_score[(long long)node * p.NC + c] = sum * inv;
    }
  }
}

template <int VW>
cudaError_t launch_score(const AttnArgs& a, cudaStream_t st) {
  const AttnPlan& p = a.plan;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(p.TPH, p.CPT / VW, p.n_rblk);
  cfg.blockDim = dim3(p.RB, kScoreThreads / p.RB);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, score_kernel<VW>, a);
}

}  // namespace

namespace {

int score_groups(const AttnPlan& p) { return (p.rows + kScoreRows - 1) / kScoreRows; }

// Whether the chunk scores are added up beside the merge, in one launch, or by a launch of their own that waits for it.
// Beside, the scores wait for the attention kernel only, which saves a launch that waits for another (3 us with its own chain of
// latencies), but a block works out its rows' statistics from all their segments, twelve at a time and one KV head after another:
// as long as every block has one task, a thread has two heads and a head has at most 48 segments.
// Tasks.  One scored call and its retrieval, one by one, own launch / beside, 32 query / 8 KV heads: 60 nodes at 4K (128 tasks)
// 23.4 / 21.9 us, one node at 16K (129) 29.9 / 29.7.  Two tasks a block, in a loop: 60 nodes at 6K 24.9 / 24.1, at 8K 26.9 / 26.3,
// but one node at 32K 38.4 / 40.3, 16 at 30K 39.4 / 40.4; three: 60 nodes at 12K 30.3 / 30.8, one at 50K 49.6 / 51.3; four and more:
// 60 nodes at 16K 4 us longer.  (The loop for several tasks, where every block has one: 60 nodes at 4K 21.13 -> 21.05 without it,
// one at 16K 28.5 -> 28.0.)
// Heads and segments.  Beside over own launch, calls of random shapes back to back, median (tenth, ninetieth percentile): 8 KV
// heads 0.93 (0.89, 1.00) with head_dim 128, 0.99 (0.96, 1.01) with 64; up to 12 segments and 4 heads 0.88, 36 to 48 segments 1.00
// (0.96, 1.03).  Any number of both, in a loop over the heads: 12 KV heads 1.08 (1.05, 1.09), 16 1.07 (1.04, 1.16), 32 1.12; 1 to 4
// with 48 to 59 segments 1.02, 60 and more 1.03 to 1.13.
// (Started beside the merge as a launch of its own, by the merge once the attention kernel was complete: 4K 23.6 -> 27.6.  A launch
// that was not set up ahead comes 4 us after it is asked for.)
bool scores_beside_merge(const AttnPlan& p) {
  return p.cluster == 0 && p.C >= 32 && p.n_rblk == 1 && p.Hkv <= kScoreSlices * kScoreHeads && p.max_segs <= 48 &&
         p.NP * (p.RB / 32) * (p.D / 64) <= kOneWave && p.TPH * score_groups(p) <= kOneWave;
}

// Launched so that its blocks may be resident (waiting) before the attention kernel has finished.
// Blocks become resident wherever an SM has room, so without a limit the SMs that the attention
// kernel leaves first would take eight blocks each and a fraction of the SMs would do all the work:
// an (unused) dynamic shared-memory request caps residency at one block per SM (measured: 1.1 us
// per call faster than two per SM, which in turn was 2 us faster than no cap).
template <int B, int NT, int VW = 0>
cudaError_t launch_merge(const AttnArgs& a, cudaStream_t st) {
  const AttnPlan& p = a.plan;
  static SpxOncePerDevice once;
  const cudaError_t ec = spx_opt_in_smem(merge_kernel<B, NT, VW>, kMergeSmemCap, &once);
  if (ec != cudaSuccess) return ec;
  const int merge_x = p.NP * (p.RB / 32), merge_y = p.D * 4 / NT;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(merge_x, merge_y);
  cfg.blockDim = dim3(NT + (VW > 0 ? 256 : 0));
  if (VW > 0) {
    const int tasks = p.TPH * score_groups(p), n_merge = merge_x * merge_y;
    cfg.gridDim = dim3(tasks > n_merge ? tasks : n_merge);
  }
  cfg.dynamicSmemBytes = kMergeSmemCap;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, merge_kernel<B, NT, VW>, a, merge_x, merge_x * merge_y);
}

}  // namespace

// What follows the attention kernel: the merge of the partial results (unless its clusters have merged them), then the
// chunk scores.
cudaError_t spx_launch_merge(const AttnArgs& a, cudaStream_t st, int* n_launches) {
  const AttnPlan& p = a.plan;
  cudaError_t e = cudaSuccess;
  if (p.want_score && p.NC > 0 && scores_beside_merge(p)) {
    e = p.C == 32   ? launch_merge<12, 256, 4>(a, st)
        : p.C == 64 ? launch_merge<12, 256, 2>(a, st)
                    : launch_merge<12, 256, 1>(a, st);
    *n_launches += 1;
    return e;
  }
  if (p.cluster == 0) {
    // With few segments per row the problems are many (64 query heads: 16 problems of 4 segments, 256 blocks of 256 threads):
    // blocks of 512 threads, all columns of 32 rows, keep the grid to one wave.  64 query heads at 16K 36.5 -> 34.8 us a
    // call, 32 with 100 nodes at 8K 25.4 -> 23.3.
    e = p.max_segs <= 4 && p.D == 128 ? launch_merge<4, 512>(a, st) : launch_merge<12, 256>(a, st);
    *n_launches += 1;
    if (e != cudaSuccess) return e;
  }
  if (p.want_score && p.NC > 0) {
    // With 16 chunks and more in a tile groups of 8: a 32-byte sector of a row's sums is then read by one block and not by two
    // (chunks of 4 at 12K, 32 query / 4 KV heads with 100 nodes 147 -> 142 us a call, 64 / 2 heads with 60 nodes 175 -> 160).  Not where they make
    // fewer than four blocks per SM (60 nodes at 3K 36.8 -> 40.3, 100 nodes of 16 KV heads at 500 tokens 19.4 -> 20.9).
    const long long wide = (long long)p.TPH * (p.CPT / 8) * p.n_rblk;
    e = p.CPT >= 16 && wide >= 4 * 148 ? launch_score<8>(a, st)
        : p.CPT >= 4                   ? launch_score<4>(a, st)
        : p.CPT == 2                   ? launch_score<2>(a, st)
                                       : launch_score<1>(a, st);
    *n_launches += 1;
  }
  return e;
}
