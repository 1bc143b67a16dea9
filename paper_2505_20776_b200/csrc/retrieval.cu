// SelectChunks and UpdateDraftCache kernels.
//
// The ranking key of chunk c is score[c] / len_c, a non-negative fp32 whose bit pattern orders like the value.  A block
// reads every key once, into registers (thread t holds the keys of consecutive chunks; above 16384 chunks 64 of them, which
// is all the registers a thread of 1024 has, so that some are spilled), finds the k-th largest by a
// most-significant-digit radix select (at most 4 passes of 8 bits over shared-memory histograms) and emits the kept
// chunks in ascending order after one block-wide scan: a chunk with a larger key is kept, and of the chunks equal to the
// k-th the lowest-indexed are kept until k are chosen.
//
// What bounds it: latency.  One block barrier per radix pass (every warp scans the histogram for itself) and two for the
// emission; the copy that follows has all its loads in flight at once.  select_gather_kernel, us per call replayed alone
// (draft cache in L2), against the form with two barriers per pass, one emission round per 256 chunks and the selection
// repeated by 256 to 512 blocks: 128 chunks 5.5 -> 5.6, 512 chunks 6.5 -> 5.1, 4096 chunks 29.7 -> 10.2, two layers of
// 12 x 64 heads and 257 chunks 7.9 -> 6.2.  select_kernel above 8192 chunks, against the form that recomputed the keys in
// every pass: 10000 chunks 30.7 -> 11.8, 16384 46.3 -> 14.3 (with 64 keys a thread 39.5), 20000 56.7 -> 42.5, 65536 193 -> 72.
#include "common.cuh"
#include "sm100.cuh"

namespace {

constexpr int kSelThreads = 512;
constexpr int kFusedMaxK = 1024;           // selected indices a fused block keeps in shared memory
constexpr int kFusedMaxChunks = 8192;      // 16 keys a thread; above this the repeated selection costs more than a launch

// Shape of one selection: chunk count, prefix length, chunk size, and the forced chunks (the first n_sink
// and the last n_recent chunks are kept whatever their score; 0 and 0 = the plain top-k).
struct SelShape {
  int NC, L, C, n_sink, n_recent;
};

__device__ __forceinline__ uint32_t chunk_key(const float* __restrict__ score, int c, const SelShape& sh) {
  if (c < sh.n_sink || c >= sh.NC - sh.n_recent) return 0x7F800000u;     // +inf: above every finite key, ties by index
  const int len = (c == sh.NC - 1) ? (sh.L - c * sh.C) : sh.C;
  float x = score[c] / (float)len;
  if (!(x > 0.f)) x = 0.f;                 // -0, negative or NaN rank lowest
  if (x > 3.0e38f) x = 3.0e38f;            // a finite score never reaches the forced chunks' key
  return __float_as_uint(x);
}

template <int NT>
struct SelectSmem {
  uint32_t hist[4][256];                   // one histogram per radix pass: cleared once
  uint32_t warp_tot[NT / 32];
};

// Selection by one block of NT threads over NC <= NT * IPT chunks: writes the keff = min(k, NC) kept chunk indices,
// ascending, to idx_out (global or shared memory).  Every thread of the block must call it.
template <int NT, int IPT>
__device__ __forceinline__ void select_block(SelectSmem<NT>& sm, const float* __restrict__ score, const SelShape& sh,
                                             int keff, int32_t* idx_out) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int c0 = tid * IPT;
  uint32_t key[IPT];
#pragma unroll
  for (int i = 0; i < IPT; ++i) key[i] = c0 + i < sh.NC ? chunk_key(score, c0 + i, sh) : 0u;
  for (int i = tid; i < 4 * 256; i += NT) (&sm.hist[0][0])[i] = 0;
  __syncthreads();

  // ---- radix select of the keff-th largest key --------------------------------------------
  uint32_t prefix = 0, mask = 0, need = keff;        // `need` keys still to take among those matching prefix
  bool all = false;                                  // every key that matches prefix is kept
#pragma unroll 1
  for (int pass = 0; pass < 4 && !all; ++pass) {
    const int shift = 24 - 8 * pass;
#pragma unroll
    for (int i = 0; i < IPT; ++i)
      if (c0 + i < sh.NC && (key[i] & mask) == prefix) atomicAdd(&sm.hist[pass][(key[i] >> shift) & 255u], 1u);
    __syncthreads();
    // bins from high to low: lane owns bins 255-8*lane .. 248-8*lane
    const uint4 h0 = *reinterpret_cast<const uint4*>(&sm.hist[pass][248 - 8 * lane]);
    const uint4 h1 = *reinterpret_cast<const uint4*>(&sm.hist[pass][252 - 8 * lane]);
    const uint32_t local[8] = {h1.w, h1.z, h1.y, h1.x, h0.w, h0.z, h0.y, h0.x};
    const uint32_t tot = ((local[0] + local[1]) + (local[2] + local[3])) + ((local[4] + local[5]) + (local[6] + local[7]));
    uint32_t incl = tot;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    // the lane whose bins hold the need-th key (one of them always does: need <= the number of matching keys)
    const int src = __ffs(__ballot_sync(0xffffffffu, need <= incl)) - 1;
    uint32_t before = incl - tot, bin = 0, left = 0, cnt = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      if (before < need && need <= before + local[i]) {
        bin = 255 - (lane * 8 + i);
        left = need - before;
        cnt = local[i];
      }
      before += local[i];
    }
    bin = __shfl_sync(0xffffffffu, bin, src);
    left = __shfl_sync(0xffffffffu, left, src);
    cnt = __shfl_sync(0xffffffffu, cnt, src);
    prefix |= bin << shift;
    mask |= 255u << shift;
    need = left;
    all = left == cnt;
  }
  // now: a key above prefix (in the digits looked at) is kept, and `need` of those that match it

  // ---- emit in ascending index order --------------------------------------------------------
  uint32_t mine = 0;                                 // keys above | keys that match << 16
#pragma unroll
  for (int i = 0; i < IPT; ++i)
    if (c0 + i < sh.NC) mine += (key[i] & mask) > prefix ? 1u : ((key[i] & mask) == prefix ? 0x10000u : 0u);
  uint32_t incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  if (lane == 31) sm.warp_tot[warp] = incl;
  __syncthreads();
  uint32_t before = incl - mine;                     // (a count before a thread is below 65536: the two halves stay apart)
#pragma unroll
  for (int w = 0; w < NT / 32; ++w)
    if (w < warp) before += sm.warp_tot[w];
  uint32_t gt = before & 0xffffu, eq = before >> 16;
#pragma unroll
  for (int i = 0; i < IPT; ++i) {
    if (c0 + i < sh.NC) {
      const uint32_t kv = key[i] & mask;
      if (kv > prefix || (kv == prefix && eq < need)) idx_out[gt + min(eq, need)] = c0 + i;
      gt += kv > prefix;
      eq += kv == prefix;
    }
  }
}

template <int NT, int IPT>
__global__ void __launch_bounds__(NT) select_kernel(const float* __restrict__ score, const SelShape sh, int k,
                                                    int32_t* __restrict__ idx, int32_t* __restrict__ n_selected) {
  __shared__ __align__(16) SelectSmem<NT> sm;
  sm100::pdl_launch_dependents();
  sm100::pdl_wait();                       // the scores are complete
  const int keff = min(k, sh.NC);
  select_block<NT, IPT>(sm, score, sh, keff, idx);
  if (threadIdx.x == 0) *n_selected = keff;
}

struct GatherArgs {
  const __nv_bfloat16* src[2];
  __nv_bfloat16* dst[2];
  const int32_t* idx;
  const int32_t* n_selected;
  int32_t* n_tokens_out;
  int32_t* status;
  int n_layers, H, D, L, C, NC, max_selected, sub;
  long long s_layer, s_l, s_h;
  // fused selection (select_gather_kernel only)
  const float* score;
  int32_t* idx_out;
  int32_t* n_selected_out;
  int k, n_sink, n_recent;
};

// Copies the tokens [o_lo, o_hi) of kept chunk number i (chunk index c) of one layer of K or V.
__device__ __forceinline__ void gather_part(const GatherArgs& g, int i, int c, int part, int layer, int which) {
  const int len = min(g.C, g.L - c * g.C);
  const int tok_per_part = (g.C + g.sub - 1) / g.sub;
  const int o_lo = part * tok_per_part, o_hi = min(len, o_lo + tok_per_part);
  const int vpr = g.D / 8;                            // 16-byte vectors per head row
  const int vpt = g.H * vpr;                          // per token
  const __nv_bfloat16* src = g.src[which] + (long long)layer * g.s_layer;
  __nv_bfloat16* dst = g.dst[which] + ((long long)layer * g.max_selected * g.C + (long long)i * g.C) * g.H * g.D;
  const int nvec = max(0, o_hi - o_lo) * vpt;
  if (g.s_h == g.D && g.s_l == (long long)g.H * g.D) {
    // tokens are contiguous in the source as they are in the compact cache: a plain copy of one range,
    // four vectors per thread and round, all loads issued before the first store
    const uint4* sp = reinterpret_cast<const uint4*>(src + (long long)(c * g.C + o_lo) * g.s_l);
    uint4* dp = reinterpret_cast<uint4*>(dst + (long long)o_lo * g.H * g.D);
    for (int v0 = threadIdx.x; v0 < nvec; v0 += 4 * blockDim.x) {
      uint4 x[4];
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (v0 + q * (int)blockDim.x < nvec) x[q] = __ldg(sp + v0 + q * blockDim.x);
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (v0 + q * (int)blockDim.x < nvec) dp[v0 + q * blockDim.x] = x[q];
    }
    return;
  }
  // strided source: four vectors per thread and round, all loads issued before the first store
  for (int v0 = threadIdx.x; v0 < nvec; v0 += 4 * blockDim.x) {
    uint4 x[4];
    long long off[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int v = v0 + q * blockDim.x;
      if (v < nvec) {
        const int o = o_lo + v / vpt;
        const int w = v - (v / vpt) * vpt;
        const int hh = w / vpr, dv = w - hh * vpr;
        x[q] = *reinterpret_cast<const uint4*>(src + (long long)(c * g.C + o) * g.s_l + (long long)hh * g.s_h + dv * 8);
        off[q] = ((long long)o * g.H + hh) * g.D + dv * 8;
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (v0 + q * blockDim.x < nvec) *reinterpret_cast<uint4*>(dst + off[q]) = x[q];
  }
}

__global__ void __launch_bounds__(256) gather_kernel(const __grid_constant__ GatherArgs g) {
  const int i = blockIdx.x / g.sub;                  // which selected chunk
  const int part = blockIdx.x - i * g.sub;           // which slice of its tokens
  const int layer = blockIdx.y;
  const int which = blockIdx.z;                      // 0 = K, 1 = V
  sm100::pdl_launch_dependents();
  sm100::pdl_wait();                                 // idx and n_selected are complete
  int nsel = *g.n_selected;
  nsel = max(0, min(nsel, g.max_selected));
  if (blockIdx.x == 0 && layer == 0 && which == 0 && threadIdx.x == 0) {
    int ntok = 0;
    if (nsel > 0) {
      const int last = g.idx[nsel - 1];
      if (last >= 0 && last < g.NC) ntok = (nsel - 1) * g.C + min(g.C, g.L - last * g.C);
    }
    *g.n_tokens_out = ntok;
  }
  if (i >= nsel) return;
  const int c = g.idx[i];
  if (c < 0 || c >= g.NC) {
    if (threadIdx.x == 0 && part == 0) spx_raise(g.status, SPECEXT_ERR_INVALID_ARG);
    return;
  }
  gather_part(g, i, c, part, layer, which);
}

// Copies the kept chunks in segments of 64 16-byte vectors, dealt to the warps of the grid; a warp has four segments (eight
// loads a lane) in flight.  Where a segment lies is worked out once for the warp: per vector, the integer divisions took
// longer than the copy.
__device__ __forceinline__ void gather_segments(const GatherArgs& g, const int32_t* s_idx, int keff) {
  const int vpr = g.D / 8, vpt = g.H * vpr;                        // vectors per head row, token
  const unsigned long long vpc = (unsigned long long)g.C * vpt;    // per chunk of the compact cache
  // segments per chunk, which may be longer than the prefix (the vectors that exist in a layer fit 32 bits: 64 GB)
  const uint32_t spc = ((uint32_t)min(g.C, g.L) * (uint32_t)vpt + 63) / 64;
  const uint32_t n_seg = 2u * g.n_layers * keff * spc;
  const bool contiguous = g.s_h == g.D && g.s_l == (long long)g.H * g.D;
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t n_warps = gridDim.x * (blockDim.x / 32);
  // warps of different blocks next to each other in the line, so that a short line keeps every SM busy
  const uint32_t first = (threadIdx.x / 32) * gridDim.x + blockIdx.x;
  for (uint32_t s0 = first; s0 < n_seg; s0 += 4 * n_warps) {
    uint4 x[4][2];
    uint4* dst[4];
    uint32_t lim[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint32_t s = s0 + q * n_warps;
      lim[q] = 0;
      if (s < n_seg) {
        const uint32_t chunk = s / spc, w0 = (s - chunk * spc) * 64;
        const uint32_t part = chunk / (uint32_t)keff, i = chunk - part * keff;
        const uint32_t which = part / (uint32_t)g.n_layers, layer = part - which * g.n_layers;
        const int c = s_idx[i];
        // vectors of the chunk from here on
        if (c >= 0 && c < g.NC) {
          const uint32_t total = (uint32_t)min(g.C, g.L - c * g.C) * (uint32_t)vpt;
          lim[q] = total - min(total, w0);
        }
        const __nv_bfloat16* base = g.src[which] + (long long)layer * g.s_layer + (long long)c * g.C * g.s_l;
        const uint32_t row = layer * g.max_selected + i;             // (at most 65535 layers x 1024 chunks)
        dst[q] = reinterpret_cast<uint4*>(g.dst[which]) + row * vpc + w0 + lane;
        if (contiguous) {
          const uint4* src = reinterpret_cast<const uint4*>(base) + w0 + lane;
#pragma unroll
          for (int e = 0; e < 2; ++e)
            if (lane + 32 * e < lim[q]) x[q][e] = __ldg(src + 32 * e);
        } else {
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const uint32_t w = w0 + lane + 32 * e, o = w / (uint32_t)vpt;
            const int r = (int)(w - o * vpt), h = r / vpr;
            if (lane + 32 * e < lim[q])
              x[q][e] = __ldg(reinterpret_cast<const uint4*>(base + (long long)o * g.s_l + (long long)h * g.s_h + (r - h * vpr) * 8));
          }
        }
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int e = 0; e < 2; ++e)
        if (lane + 32 * e < lim[q]) dst[q][32 * e] = x[q][e];
  }
}

// SelectChunks and UpdateDraftCache in one launch: every block repeats the (deterministic) selection in its own shared
// memory and then copies its share of the kept chunks, so no block waits for another; block 0 also writes idx,
// n_selected and n_tokens.  At most two blocks per SM: with one the call alone is 1.0 us shorter (the
// selections of two blocks share an SM's pipes), but behind a verification call, with the draft cache in DRAM, 0.4 to 1.1 us
// longer (4K: 23.9 against 23.3 us for call and retrieval; 8K, two-layer draft: 42.2 against 41.1).
template <int IPT>
__global__ void __launch_bounds__(kSelThreads) select_gather_kernel(const __grid_constant__ GatherArgs g) {
  __shared__ __align__(16) SelectSmem<kSelThreads> sm;
  __shared__ int32_t s_idx[kFusedMaxK];
  sm100::pdl_launch_dependents();
  const int keff = min(g.k, g.NC);
  // (the selection fills all of them; should a caller rewrite the scores meanwhile and a key be read twice, one left over is
  // skipped by the copy instead of becoming an address)
  for (int j = threadIdx.x; j < keff; j += kSelThreads) s_idx[j] = -1;
  const SelShape sh = {g.NC, g.L, g.C, g.n_sink, g.n_recent};
  sm100::pdl_wait();                                 // the scores are complete
  select_block<kSelThreads, IPT>(sm, g.score, sh, keff, s_idx);
  __syncthreads();
  gather_segments(g, s_idx, keff);
  if (blockIdx.x == 0) {
    for (int j = threadIdx.x; j < keff; j += kSelThreads) g.idx_out[j] = s_idx[j];
    if (threadIdx.x == 0) {
      *g.n_selected_out = keff;
      const int last = s_idx[keff - 1];
      *g.n_tokens_out = (keff - 1) * g.C + min(g.C, g.L - last * g.C);
    }
  }
}

cudaError_t launch_pdl(const void* kernel, dim3 grid, dim3 block, void** args, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = 0;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelExC(&cfg, kernel, args);
}

void fill_gather_args(GatherArgs& g, const void* dK, const void* dV, int n_layers, int H, int D, int L, int C,
                      long long s_layer, long long s_l, long long s_h, int max_selected, void* K_out, void* V_out,
                      int32_t* n_tokens_out, int32_t* status) {
  g.src[0] = static_cast<const __nv_bfloat16*>(dK);
  g.src[1] = static_cast<const __nv_bfloat16*>(dV);
  g.dst[0] = static_cast<__nv_bfloat16*>(K_out);
  g.dst[1] = static_cast<__nv_bfloat16*>(V_out);
  g.n_tokens_out = n_tokens_out;
  g.status = status;
  g.n_layers = n_layers; g.H = H; g.D = D; g.L = L; g.C = C;
  g.NC = (L + C - 1) / C;
  g.max_selected = max_selected;
  // aim for ~16 KB per CTA
  const long long chunk_bytes = (long long)C * H * D * 2;
  int sub = (int)((chunk_bytes + 16383) / 16384);
  sub = max(1, min(sub, C));
  g.sub = sub;
  g.s_layer = s_layer; g.s_l = s_l; g.s_h = s_h;
  g.idx = nullptr; g.n_selected = nullptr;
  g.score = nullptr; g.idx_out = nullptr; g.n_selected_out = nullptr; g.k = 0; g.n_sink = 0; g.n_recent = 0;
}

}  // namespace

cudaError_t spx_launch_select(const float* score_row, int NC, int L, int C, int k, int n_sink, int n_recent,
                              int32_t* idx, int32_t* n_selected, cudaStream_t st) {
  SelShape sh = {NC, L, C, n_sink, n_recent};
  void* args[] = {&score_row, &sh, &k, &idx, &n_selected};
  // The fewest keys a thread that hold NC: one block, whose time is its threads' chain of keys.  1024 threads with 16 keys
  // between the two largest classes: 8193 to 10000 chunks took 40 us with 64 keys, more than the 28 to 31 of the form before.
  const void* kernel = NC <= 512     ? reinterpret_cast<const void*>(select_kernel<512, 1>)
                       : NC <= 2048  ? reinterpret_cast<const void*>(select_kernel<512, 4>)
                       : NC <= 8192  ? reinterpret_cast<const void*>(select_kernel<512, 16>)
                       : NC <= 16384 ? reinterpret_cast<const void*>(select_kernel<1024, 16>)
                                     : reinterpret_cast<const void*>(select_kernel<1024, 64>);
  return launch_pdl(kernel, dim3(1), dim3(NC <= 8192 ? 512 : 1024), args, st);
}

cudaError_t spx_launch_gather(const void* dK, const void* dV, int n_layers, int H, int D, int L, int C,
                              long long s_layer, long long s_l, long long s_h, const int32_t* idx,
                              const int32_t* n_selected, int max_selected, void* K_out, void* V_out,
                              int32_t* n_tokens_out, int32_t* status, cudaStream_t st) {
  GatherArgs g;
  fill_gather_args(g, dK, dV, n_layers, H, D, L, C, s_layer, s_l, s_h, max_selected, K_out, V_out, n_tokens_out,
                   status);
  g.idx = idx;
  g.n_selected = n_selected;
  void* args[] = {&g};
  return launch_pdl(reinterpret_cast<const void*>(gather_kernel), dim3(max_selected * g.sub, n_layers, 2), dim3(256),
                    args, st);
}

// True when SelectChunks + UpdateDraftCache of this size run as one launch.
bool spx_select_gather_fusable(int NC, int k) { return NC >= 1 && NC <= kFusedMaxChunks && k <= kFusedMaxK; }

cudaError_t spx_launch_select_gather(const float* score_row, int k, int n_sink, int n_recent, const void* dK,
                                     const void* dV, int n_layers,
                                     int H, int D, int L, int C, long long s_layer, long long s_l, long long s_h,
                                     int32_t* idx, int32_t* n_selected, void* K_out, void* V_out,
                                     int32_t* n_tokens_out, int n_sm, int32_t* status, cudaStream_t st) {
  GatherArgs g;
  fill_gather_args(g, dK, dV, n_layers, H, D, L, C, s_layer, s_l, s_h, k, K_out, V_out, n_tokens_out, status);
  g.score = score_row;
  g.idx_out = idx;
  g.n_selected_out = n_selected;
  g.k = k;
  g.n_sink = n_sink;
  g.n_recent = n_recent;
  void* args[] = {&g};
  const int keff = k < g.NC ? k : g.NC;
  const long long segments = 2ll * n_layers * keff * (((long long)(C < L ? C : L) * H * (D / 8) + 63) / 64);
  const long long blocks = (segments + kSelThreads / 32 - 1) / (kSelThreads / 32);
  const void* kernel = g.NC <= kSelThreads       ? reinterpret_cast<const void*>(select_gather_kernel<1>)
                       : g.NC <= 4 * kSelThreads ? reinterpret_cast<const void*>(select_gather_kernel<4>)
                       : g.NC <= 8 * kSelThreads ? reinterpret_cast<const void*>(select_gather_kernel<8>)
                                                 : reinterpret_cast<const void*>(select_gather_kernel<16>);
  return launch_pdl(kernel, dim3((unsigned)(blocks < 2 * n_sm ? blocks : 2 * n_sm)), dim3(kSelThreads), args, st);
}
