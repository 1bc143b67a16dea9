// Host side of the C ABI: argument checks, work decomposition, workspace layout and launches.
#include <atomic>
#include <cmath>
#include <cstring>

#include "common.cuh"

cudaError_t spx_launch_select(const float* score_row, int NC, int L, int C, int k, int n_sink, int n_recent,
                              int32_t* idx, int32_t* n_selected, cudaStream_t st);
cudaError_t spx_launch_gather(const void* dK, const void* dV, int n_layers, int H, int D, int L, int C,
                              long long s_layer, long long s_l, long long s_h, const int32_t* idx,
                              const int32_t* n_selected, int max_selected, void* K_out, void* V_out,
                              int32_t* n_tokens_out, int32_t* status, cudaStream_t st);
cudaError_t spx_launch_prefill(const void* Q, const void* K, const void* V, void* O, float* lse, int L, int Hq, int Hkv,
                               float scale2, long long q_st, long long q_sh, long long kv_sl, long long kv_sh,
                               long long o_st, long long o_sh, int n_sm, int32_t* status, cudaStream_t st);
bool spx_select_gather_fusable(int NC, int k);
cudaError_t spx_launch_select_gather(const float* score_row, int k, int n_sink, int n_recent, const void* dK,
                                     const void* dV, int n_layers,
                                     int H, int D, int L, int C, long long s_layer, long long s_l, long long s_h,
                                     int32_t* idx, int32_t* n_selected, void* K_out, void* V_out,
                                     int32_t* n_tokens_out, int n_sm, int32_t* status, cudaStream_t st);

// Scratch of the entry point that takes no workspace.  Part of the library image: resident on every
// device that loads the library until the process exits.  Device code may name it directly; host
// code must go through cudaGetSymbolAddress (see specext_verify_attn_static_scratch).
static __device__ __align__(256) unsigned char g_static_scratch[SPECEXT_STATIC_SCRATCH_BYTES];

namespace {

constexpr int kMaxDevices = kSpxMaxDevices;
std::atomic<void*> g_static_scratch_addr[kMaxDevices];

std::atomic<long long> g_launches{0};

// Kernel choice and split granularity.  The product library has one choice per shape; the test library
// (SPECEXT_TESTING) can override it so that the tests reach the other kernels and coarser splits.
#ifdef SPECEXT_TESTING
std::atomic<int> g_attn_kernel{0};       // 0 = default, 1 = CUDA-core kernel, 2 = one-CTA kernel, 3 = paired kernel
std::atomic<int> g_min_units{1};         // lower bound on key tiles per worker
int tuning_kernel() { return g_attn_kernel.load(); }
int tuning_min_units() { return g_min_units.load() < 1 ? 1 : g_min_units.load(); }
#else
constexpr int tuning_kernel() { return 0; }
constexpr int tuning_min_units() { return 1; }
#endif

// Multiprocessor count of the current device (looked up once per device).
int sm_count() {
  static std::atomic<int> cached[kMaxDevices];
  int dev = -1, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) {
    (void)cudaGetLastError();
    return 148;                           // B200; used only when no device is present (size queries)
  }
  if (dev < kMaxDevices && (n = cached[dev].load()) > 0) return n;
  if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) {
    (void)cudaGetLastError();
    return 148;
  }
  if (dev < kMaxDevices) cached[dev].store(n);
  return n;
}

bool is_pow2(int x) { return x > 0 && (x & (x - 1)) == 0; }
bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Row blocks, workers and workspace of one kernel (plan.kernel); cluster > 0: its workers merge in clusters of that size.
int lay_out(AttnPlan* plan, int kernel, int row_block, int cluster) {
  AttnPlan& p = *plan;
  p.kernel = kernel;
  p.cluster = cluster;
  p.RB = row_block;
  p.n_rblk = (p.rows + p.RB - 1) / p.RB;
  p.NP = p.Hkv * p.n_rblk;
  const long long U = (long long)p.NP * p.UPP;
  if (U > (1ll << 30)) return SPECEXT_ERR_UNSUPPORTED;
  p.U = (int)U;
  const int min_units = tuning_min_units();
  if (cluster > 0) {
    p.cpp = cluster;
    p.n_cta = p.NP * p.cpp;
    p.q = p.UPP / p.cpp;
    p.rem = p.UPP % p.cpp;
    p.max_segs = p.cpp;
  } else if (p.kernel == 3) {
    // one worker = a cluster of two CTAs; every problem gets the same number of workers when possible
    const int n_workers = sm_count() / 2 > 0 ? sm_count() / 2 : 1;
    if (p.NP <= n_workers) {
      int cpp = n_workers / p.NP;
      if (cpp > p.UPP / min_units) cpp = p.UPP / min_units;
      if (cpp < 1) cpp = 1;
      p.cpp = cpp;
      p.n_cta = p.NP * cpp;
      p.q = p.UPP / cpp;
      p.rem = p.UPP % cpp;
      p.max_segs = cpp;
    } else {
      p.cpp = 0;
      p.n_cta = n_workers;
      p.q = p.U / p.n_cta;
      p.rem = p.U % p.n_cta;
      p.max_segs = (p.UPP + p.q - 1) / p.q + 1;
    }
  } else {
    int n_cta = p.U / min_units;
    if (n_cta < 1) n_cta = 1;
    if (n_cta > sm_count()) n_cta = sm_count();
    p.cpp = 0;
    p.n_cta = n_cta;
    p.q = p.U / n_cta;
    p.rem = p.U % n_cta;
    p.max_segs = (p.UPP + p.q - 1) / p.q + 1;
  }
  if (p.max_segs > p.n_cta) p.max_segs = p.n_cta;
  // Rows of Q a CTA of the one-CTA kernel keeps.  Its MMAs read 128 rows whatever there are, and what lies behind Q is K: at
  // the power limit, where long passes run, multiplying it costs more than the stage of the K ring that 128 rows of Q (zeros
  // behind the last) take up.  us per pass, one by one, 64 / 128 rows kept: 60 rows of 32 KV heads, two layers at 8K (16 tiles a
  // CTA) 73.9 / 72.8, at 16K 122.9 / 120.6; of 8 KV heads, 4 rows, two layers at 32K (13 tiles) 71.9 / 70.4, 32 rows at 48K
  // 97.7 / 95.0, 64 rows at 32K 77.5 / 75.3, one layer of 64 rows at 128K (55 tiles) 120.2 / 119.0; one row of 32 KV heads at 16K
  // and 40K the same.  Below the line: 4 rows of 8 KV heads at 16K (7 tiles) the same, short calls up to 1 % longer with 128.
  // (The cleared rows of P in verify.cu are the other half: without them 60 rows of 32 KV heads, four layers, take 134.8 instead
  // of 133.3 at 8K and 229.0 instead of 225.9 at 16K, 64 rows of 8 at 128K 119.7 instead of 118.5, 16 rows and fewer the same.)
  p.q_rows = 128;
  if (p.kernel == 2 && p.D == 128) {
    if (p.cluster > 0 && p.rows <= kSpxClusterRowsBySmem) p.q_rows = 32;       // (the exchange needs the room, see Layout)
    else if (p.rows <= 64 && p.U / p.n_cta < 12) p.q_rows = 64;
  }
  p.n_slots = p.cluster > 0 ? p.n_cta : p.n_cta + p.NP - 1;
  long long off = 0;
  p.off_part_o = off; off += (long long)p.n_slots * p.D * p.RB;
  p.off_part_m = off; off += (long long)p.n_slots * p.RB;
  p.off_part_l = off; off += (long long)p.n_slots * p.RB;
  if (p.want_score) {
    p.off_mass = off; off += (long long)p.NP * p.TPH * p.RB * p.CPT;
    p.off_mref = off; off += (long long)p.NP * p.TPH * p.RB;
  }
  p.total_floats = off;
  return SPECEXT_OK;
}

// Size of the cluster whose CTAs share the key tiles of a problem and merge among themselves, or 0 for workers that leave
// partial results to the merge kernel.  dev_len: the prefix length is on the device (a draft call).
int cluster_size(const AttnPlan& p, bool pair, bool dev_len) {
  const long long np = (long long)p.Hkv * ((p.rows + 127) / 128);
  int dev = -1, size = 0;
  if (np > sm_count() / 2) return 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    (void)cudaGetLastError();
    return 0;
  }
  // the largest clusters of which one per problem is resident at once (above the portable size of 8 where that pays: 40 rows
  // on 1K 7.8 -> 7.5 us, 120 rows at 8K 16.0 -> 14.8; up to 32 rows, which merge through shared memory, 0.2 slower)
  for (int s = p.rows > kSpxClusterRowsBySmem ? 16 : 8; s >= 2 && size == 0; --s)
    if (s <= p.UPP && np * s <= sm_count() && np <= spx_verify_max_clusters(dev, s)) size = s;
  if (size == 0) return 0;
  // A prefix of one tile gives clusters of two, which merge half of the rows' columns each: above 64 rows longer than the
  // merge kernel takes, unless the problems are many.  us per call, before clusters / split / cluster, 100 tokens: 60 nodes
  // 9.4 / 9.2 / 9.6, 100 nodes of 16 query / 2 KV heads 9.0 / 9.2 / 9.9, of 32 KV heads 12.4 / 10.0 / 10.5; but 60 nodes of
  // 32 KV heads (60 rows) 10.5 / 9.0 / 8.9, 100 nodes of 64 query / 8 KV heads (56 problems) 14.5 / 12.6 / 11.5, of 64 KV
  // heads 17.1 / 12.2 / 11.0.  (Between them 40 problems take 1.08 of the split form's time, 50 0.95.  Draft calls stay: their
  // split form is longer, see below.)
  if (p.UPP == 2 && p.D == 128 && p.rows > 64 && np <= 40 && !dev_len) return 0;
  const int tiles = (p.UPP + size - 1) / size;
  int split;
  if (pair) {
    const long long np2 = (long long)p.Hkv * ((p.rows + 255) / 256), workers = sm_count() / 2;
    split = (int)(np2 <= workers ? (p.UPP + workers / np2 - 1) / (workers / np2) : (np2 * p.UPP + workers - 1) / workers);
  } else {
    split = (int)((np * p.UPP + sm_count() - 1) / sm_count());
  }
  // (A draft call is laid out for its capacity: with half of it filled the first CTAs of a cluster have most of the tiles.
  // 100 nodes of 64 KV heads in a cache of 16384: full 128 before clusters / 100 split / 93, with 8229 tokens 74 / 80 / 83;
  // 60 nodes in a cache of 2048: full 14.1 / 14.2 / 11.0, with 1061 13.6 / 13.6 / 14.2.  Sharing the tiles that exist evenly
  // costs every full call 0.2 to 0.4 us.)
  // What merging in the cluster saves (3 to 4 us with the second launch) against the tiles it adds; the pairs, whose CTAs
  // fetch half of every K/V tile, win again when the tiles are many.  us per call, split / cluster, replayed (32 query / 8 KV
  // heads unless said; launched one by one the cluster form gains another 0.5):
  //   60 nodes: 1K 10.9 / 9.9, 2K 11.6 / 10.7 (3 tiles against 2), 3K 12.5 / 13.1 (4 against 3), 4K 13.4 / 13.6 (5 against 4)
  //   60 nodes, 64 query heads: 1K 13.4 / 11.5, 2K 13.2 / 13.1 (5 against 5), 4K 16.3 / 16.9 (9; one by one 17.5 / 17.2)
  //   60 nodes, 32 KV heads: 1K 13.5 / 10.7, 8K 29.5 / 26.6 (17 against 15), 32K 91.3 / 88.9 (65 against 56)
  //   1 node: 2K 10.8 / 8.0, 8K 15.8 / 14.8 (9 against 4), 16K 19.3 / 22.5 (17 against 7)
  //   12 x 64 heads: 4K 11.7 / 9.3 (5 against 3);  60 nodes, 32 x 64 query / 8 KV heads, 16K: 22.7 / 24.5 (19 against 14)
  // Against the pairs the gain is used up at six tiles (7 against 7, 100 nodes at 3K 14.6 / 15.0, scored 17.9 / 18.4), unless
  //   the pairs have more tiles (80 nodes at 8K 22.2 / 20.7, 17 against 13: blocks of 256 rows pad 320 to 512) or
  //   their merge takes a second wave of blocks (256 threads: 32 query / 4 KV heads, 80 nodes at 5K 17.1 / 14.9, scored
  //   20.5 / 18.2; 512 threads: 64 query / 8 KV heads, 80 nodes at 5K 22.2 / 21.6, scored 26.8 / 25.9), which two segments a
  //   row make up for sooner (100 nodes at 2K 18.0 / 17.6 with 9 tiles, 3K 21.0 / 21.2 with 13);
  //   a draft call goes there (the pairs' form with the length on the device is another 2 us longer: 60 nodes of 64 query
  //   heads in a cache of 4096 19.1 / 17.0 with 9 tiles, 100 nodes of 16 / 2 heads in 16384 24.6 / 21.6 with 15);
  //   without scores also a cluster of more than 8 CTAs (100 nodes of 16 query / 2 KV heads at 8K 15.8 / 15.1 with 8 tiles,
  //   scored 19.5 / 20.3).
  int limit = 0;
  if (pair) {
    const int np2 = p.Hkv * ((p.rows + 255) / 256), per = sm_count() / 2 / np2;      // (np2 <= np <= half of the SMs)
    const bool second_wave = 8 * np2 * (per > 4 ? 2 : 1) > sm_count();
    limit = dev_len || tiles < split || (second_wave && per > 2) ? 16 : second_wave || (!p.want_score && size > 8) ? 11 : 6;
    if (p.want_score && p.C < 32) limit = 16;                                         // (see below)
  }
  int most = pair ? (tiles <= limit ? (split > 3 ? split : 3) : 0)
                  : split + (p.D == 64 ? 3 : split > 30 ? split / 6 : 5);
  // Chunks of fewer than 32 keys make a tile cost more than twice as much (a running sum and a store per chunk), so that extra
  // tiles outweigh the launch they save.  Chunks of 16, before clusters / split / cluster: 60 nodes at 2K 24.0 / 22.0 / 26.1
  // (3 tiles against 2), 32 x 64 query / 8 KV heads at 8K 52.0 / 47.0 / 58.7 (11 against 8), one node of 16 query / 2 KV heads
  // at 4K 25.8 / 21.1 / 29.9 (5 against 1); but 100 nodes at 1K 30.3 / 28.3 / 26.4 (3 against 3), 32 KV heads of 60 nodes at
  // 6K 124 / 67.4 / 65.3 (12 against 11), 12 x 64 heads of 100 nodes at 4K 37.9 / 30.6 / 25.2 (4 against 3).
  if (p.want_score && p.C < 32) {
    int most_small;
    if (pair) most_small = tiles <= (p.C == 16 ? 12 : 5) ? split : 0;    // 4 keys: 7 against 7 0.3 to 9 % slower, 12 1 to 11 %
    else most_small = tiles <= 4 && (size > 8 || split >= 3) ? 4 : p.D == 64 ? split : split * 6 / 5;
    if (most_small < 2 && p.C >= 4) most_small = 2;      // (a key or two: 60 nodes at 1K 35.4 before, 43.2 in clusters)
    if (most > most_small) most = most_small;
  }
  if (tiles > most) return 0;
  while (size > 2 && (p.UPP + size - 2) / (size - 1) == tiles) --size;     // no more CTAs than the tile count needs
  return size;
}

// (The workspace is that of the split form whatever dev_len is: the clusters' is never larger.)
int build_plan(const specext_attn_desc* d, AttnPlan* out, bool dev_len = false) {
  if (!d) return SPECEXT_ERR_INVALID_ARG;
  if (d->n_q_heads < 1 || d->n_kv_heads < 1 || d->n_q_heads % d->n_kv_heads != 0) return SPECEXT_ERR_INVALID_ARG;
  if (d->prefix_len < 0 || d->prefix_len > (1 << 24)) return SPECEXT_ERR_INVALID_ARG;
  if (d->n_tree < 1 || d->n_tree > kSpxMaxTree) return SPECEXT_ERR_UNSUPPORTED;
  if (d->head_dim != 64 && d->head_dim != 128) return SPECEXT_ERR_UNSUPPORTED;
  if (!is_pow2(d->chunk_size) || d->chunk_size > 128) return SPECEXT_ERR_UNSUPPORTED;
  const int G = d->n_q_heads / d->n_kv_heads;
  if (!is_pow2(G) || G > 64) return SPECEXT_ERR_UNSUPPORTED;
  if (!(d->softmax_scale >= 0.f) || !std::isfinite(d->softmax_scale)) return SPECEXT_ERR_INVALID_ARG;
  const long long strides[8] = {d->q_stride_t, d->q_stride_h, d->kv_stride_l, d->kv_stride_h,
                                d->tkv_stride_t, d->tkv_stride_h, d->o_stride_t, d->o_stride_h};
  for (long long s : strides)
    if (s < d->head_dim || (s & 7) != 0) return SPECEXT_ERR_INVALID_ARG;

  AttnPlan p;
  std::memset(&p, 0, sizeof(p));
  p.Hq = d->n_q_heads; p.Hkv = d->n_kv_heads; p.G = G; p.D = d->head_dim;
  p.L = d->prefix_len; p.T = d->n_tree; p.C = d->chunk_size;
  p.rows = G * p.T;
  p.TPH = (p.L + SPX_TILE_KEYS - 1) / SPX_TILE_KEYS;
  p.UPP = p.TPH + 1;
  p.CPT = SPX_TILE_KEYS / p.C;
  p.NC = (p.L + p.C - 1) / p.C;
  p.want_score = d->want_chunk_score != 0;
  const float scale = d->softmax_scale > 0.f ? d->softmax_scale : 1.0f / std::sqrt((float)p.D);
  p.scale2 = scale * 1.44269504088896340736f;
  // Kernel: pairs of CTAs on 256-row blocks for head_dim 128 and more than 128 stacked rows; otherwise one CTA on
  // 128-row blocks (want != 0 only in the test library).
  const int want = tuning_kernel();
  const bool pair = p.D == 128 && p.rows > 128 && want != 2;
  int rc = lay_out(&p, want == 1 ? 1 : (pair ? 3 : 2), pair ? 256 : 128, 0);
  if (rc != SPECEXT_OK) return rc;
  const int size = want == 0 && tuning_min_units() == 1 ? cluster_size(p, pair, dev_len) : 0;
  if (size > 0) {
    // (the workspace keeps its size: it does not depend on what clusters the device holds)
    const long long split_floats = p.total_floats;
    rc = lay_out(&p, 2, 128, size);
    if (rc != SPECEXT_OK) return rc;
    if (p.total_floats < split_floats) p.total_floats = split_floats;
  }
  *out = p;
  return SPECEXT_OK;
}

int check_gather_args(const void* draft_K, const void* draft_V, int32_t n_layers, int32_t n_kv_heads,
                      int32_t head_dim, int32_t prefix_len, int32_t chunk_size, int64_t stride_layer,
                      int64_t stride_l, int64_t stride_h, int32_t max_selected, const void* K_out,
                      const void* V_out, const int32_t* n_tokens_out) {
  if (!draft_K || !draft_V || !K_out || !V_out || !n_tokens_out) return SPECEXT_ERR_INVALID_ARG;
  if (n_layers < 1 || n_layers > 65535 || n_kv_heads < 1 || head_dim < 8 || (head_dim & 7) != 0 ||
      prefix_len < 0 || chunk_size < 1 || max_selected < 1)
    return SPECEXT_ERR_INVALID_ARG;
  if (stride_h < head_dim || (stride_h & 7) || stride_l < head_dim || (stride_l & 7) || (stride_layer & 7) ||
      stride_layer < 0)
    return SPECEXT_ERR_INVALID_ARG;
  if (!aligned16(draft_K) || !aligned16(draft_V) || !aligned16(K_out) || !aligned16(V_out))
    return SPECEXT_ERR_INVALID_ARG;
  if ((long long)max_selected * chunk_size > (1ll << 28)) return SPECEXT_ERR_UNSUPPORTED;
  return SPECEXT_OK;
}

}  // namespace

extern "C" {

size_t specext_verify_attn_workspace(const specext_attn_desc* desc) {
  AttnPlan p;
  if (build_plan(desc, &p) != SPECEXT_OK) return 0;
  return (size_t)p.total_floats * sizeof(float);
}

}  // extern "C"

namespace {

// Checks, plan and launches shared by specext_verify_attn (prefix_len_dev == null) and
// specext_draft_attn (the prefix length is read on the device, desc->prefix_len is its upper bound).
int run_attn(const specext_attn_desc* desc, const void* Q, const void* K_prefix, const void* V_prefix,
             const void* K_tree, const void* V_tree, const int32_t* parent, const int32_t* prefix_len_dev,
             void* O, float* lse, float* chunk_score, void* workspace, size_t workspace_bytes,
             int32_t* device_status, void* cuda_stream) {
  AttnArgs a;
  const int rc = build_plan(desc, &a.plan, prefix_len_dev != nullptr);
  if (rc != SPECEXT_OK) return rc;
  const AttnPlan& p = a.plan;
  if (prefix_len_dev && (p.want_score || p.kernel == 1 || (reinterpret_cast<uintptr_t>(prefix_len_dev) & 3u) != 0))
    return p.want_score ? SPECEXT_ERR_INVALID_ARG : (p.kernel == 1 ? SPECEXT_ERR_UNSUPPORTED : SPECEXT_ERR_INVALID_ARG);
  a.L_dev = prefix_len_dev;
  if (!Q || !K_tree || !V_tree || !parent || !O || !lse || !workspace) return SPECEXT_ERR_INVALID_ARG;
  if (p.L > 0 && (!K_prefix || !V_prefix)) return SPECEXT_ERR_INVALID_ARG;
  if (p.want_score && p.NC > 0 && !chunk_score) return SPECEXT_ERR_INVALID_ARG;
  if (!aligned16(Q) || !aligned16(K_prefix) || !aligned16(V_prefix) || !aligned16(K_tree) ||
      !aligned16(V_tree) || !aligned16(O) || (reinterpret_cast<uintptr_t>(workspace) & 255u) != 0 ||
      (reinterpret_cast<uintptr_t>(lse) & 3u) != 0 || (reinterpret_cast<uintptr_t>(parent) & 3u) != 0)
    return SPECEXT_ERR_INVALID_ARG;
  if (workspace_bytes < (size_t)p.total_floats * sizeof(float)) return SPECEXT_ERR_WORKSPACE;

  a.Q = static_cast<const __nv_bfloat16*>(Q);
  a.Kp = static_cast<const __nv_bfloat16*>(K_prefix);
  a.Vp = static_cast<const __nv_bfloat16*>(V_prefix);
  a.Kt = static_cast<const __nv_bfloat16*>(K_tree);
  a.Vt = static_cast<const __nv_bfloat16*>(V_tree);
  a.parent = parent;
  a.O = static_cast<__nv_bfloat16*>(O);
  a.lse = lse;
  a.chunk_score = chunk_score;
  a.ws = static_cast<float*>(workspace);
  a.status = device_status;
  a.q_st = desc->q_stride_t; a.q_sh = desc->q_stride_h;
  a.kv_sl = desc->kv_stride_l; a.kv_sh = desc->kv_stride_h;
  a.tkv_st = desc->tkv_stride_t; a.tkv_sh = desc->tkv_stride_h;
  a.o_st = desc->o_stride_t; a.o_sh = desc->o_stride_h;

  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  int n = 0;
  cudaError_t e;
#ifdef SPECEXT_TESTING
  if (p.kernel == 1) e = spx_launch_attn_simt(a, st, &n); else
#endif
  e = p.kernel == 3 ? spx_launch_attn_tc2(a, st, &n) : spx_launch_verify(a, st, &n);
  if (e == cudaSuccess) e = spx_launch_merge(a, st, &n);
  g_launches.fetch_add(n);
  if (e != cudaSuccess) {
    (void)cudaGetLastError();
    return SPECEXT_ERR_CUDA;
  }
  return SPECEXT_OK;
}

}  // namespace

extern "C" {

int specext_verify_attn(const specext_attn_desc* desc, const void* Q, const void* K_prefix,
                        const void* V_prefix, const void* K_tree, const void* V_tree,
                        const int32_t* parent, void* O, float* lse, float* chunk_score,
                        void* workspace, size_t workspace_bytes, int32_t* device_status,
                        void* cuda_stream) {
  return run_attn(desc, Q, K_prefix, V_prefix, K_tree, V_tree, parent, nullptr, O, lse, chunk_score, workspace,
                  workspace_bytes, device_status, cuda_stream);
}

int specext_draft_attn(const specext_attn_desc* desc, const void* Q, const void* K_cache,
                       const void* V_cache, const int32_t* n_tokens, const void* K_tree,
                       const void* V_tree, const int32_t* parent, void* O, float* lse, void* workspace,
                       size_t workspace_bytes, int32_t* device_status, void* cuda_stream) {
  if (!n_tokens) return SPECEXT_ERR_INVALID_ARG;
  return run_attn(desc, Q, K_cache, V_cache, K_tree, V_tree, parent, n_tokens, O, lse, nullptr, workspace,
                  workspace_bytes, device_status, cuda_stream);
}

int specext_prefill_attn(const specext_attn_desc* desc, const void* Q, const void* K, const void* V, void* O,
                         float* lse, int32_t* device_status, void* cuda_stream) {
  if (!desc || !Q || !K || !V || !O || !lse) return SPECEXT_ERR_INVALID_ARG;
  if (desc->n_q_heads < 1 || desc->n_kv_heads < 1 || desc->n_q_heads % desc->n_kv_heads != 0)
    return SPECEXT_ERR_INVALID_ARG;
  if (desc->prefix_len < 1 || desc->prefix_len > (1 << 24)) return SPECEXT_ERR_INVALID_ARG;
  if (!(desc->softmax_scale >= 0.f) || !std::isfinite(desc->softmax_scale)) return SPECEXT_ERR_INVALID_ARG;
  const int G = desc->n_q_heads / desc->n_kv_heads;
  if (desc->head_dim != 128 || !is_pow2(G) || G > 256) return SPECEXT_ERR_UNSUPPORTED;
  const long long strides[6] = {desc->q_stride_t, desc->q_stride_h, desc->kv_stride_l, desc->kv_stride_h,
                                desc->o_stride_t, desc->o_stride_h};
  for (long long s : strides)
    if (s < desc->head_dim || (s & 7) != 0) return SPECEXT_ERR_INVALID_ARG;
  if (!aligned16(Q) || !aligned16(K) || !aligned16(V) || !aligned16(O) || (reinterpret_cast<uintptr_t>(lse) & 3u) != 0)
    return SPECEXT_ERR_INVALID_ARG;
  const float scale = desc->softmax_scale > 0.f ? desc->softmax_scale : 1.0f / std::sqrt((float)desc->head_dim);
  const cudaError_t e = spx_launch_prefill(Q, K, V, O, lse, desc->prefix_len, desc->n_q_heads, desc->n_kv_heads,
                                           scale * 1.44269504088896340736f, desc->q_stride_t, desc->q_stride_h,
                                           desc->kv_stride_l, desc->kv_stride_h, desc->o_stride_t, desc->o_stride_h,
                                           sm_count(), device_status, static_cast<cudaStream_t>(cuda_stream));
  g_launches.fetch_add(1);
  if (e != cudaSuccess) {
    (void)cudaGetLastError();
    return SPECEXT_ERR_CUDA;
  }
  return SPECEXT_OK;
}

int specext_verify_attn_static_scratch(const specext_attn_desc* desc, const void* Q,
                                       const void* K_prefix, const void* V_prefix,
                                       const void* K_tree, const void* V_tree,
                                       const int32_t* parent, void* O, float* lse,
                                       float* chunk_score, int32_t* device_status,
                                       void* cuda_stream) {
  // Reject a bad descriptor, or a shape that does not fit, before touching the device.
  AttnPlan plan;
  const int rc = build_plan(desc, &plan);
  if (rc != SPECEXT_OK) return rc;
  if ((size_t)plan.total_floats * sizeof(float) > SPECEXT_STATIC_SCRATCH_BYTES) return SPECEXT_ERR_WORKSPACE;
  // g_static_scratch names a host-side handle of the device array, not a device address: the address
  // valid on the current device comes from cudaGetSymbolAddress, looked up once per device.
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    (void)cudaGetLastError();
    return SPECEXT_ERR_CUDA;
  }
  void* scratch = g_static_scratch_addr[dev].load();
  if (!scratch) {
    if (cudaGetSymbolAddress(&scratch, g_static_scratch) != cudaSuccess || !scratch) {
      (void)cudaGetLastError();
      return SPECEXT_ERR_CUDA;
    }
    g_static_scratch_addr[dev].store(scratch);
  }
  return specext_verify_attn(desc, Q, K_prefix, V_prefix, K_tree, V_tree, parent, O, lse, chunk_score, scratch,
                             SPECEXT_STATIC_SCRATCH_BYTES, device_status, cuda_stream);
}

int specext_select_chunks(const float* chunk_score, int32_t n_tree, int32_t n_chunks, int32_t row,
                          int32_t prefix_len, int32_t chunk_size, int32_t k, int32_t n_sink_chunks,
                          int32_t n_recent_chunks, int32_t* idx, int32_t* n_selected, int32_t* device_status,
                          void* cuda_stream) {
  (void)device_status;
  if (!idx || !n_selected) return SPECEXT_ERR_INVALID_ARG;
  if (n_tree < 1 || row < 0 || row >= n_tree || k < 1 || chunk_size < 1 || prefix_len < 0 || n_sink_chunks < 0 ||
      n_recent_chunks < 0)
    return SPECEXT_ERR_INVALID_ARG;
  const long long nc = ((long long)prefix_len + chunk_size - 1) / chunk_size;
  if (nc != n_chunks) return SPECEXT_ERR_INVALID_ARG;
  if (n_chunks > 65536) return SPECEXT_ERR_UNSUPPORTED;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  cudaError_t e;
  if (n_chunks == 0) {
    e = cudaMemsetAsync(n_selected, 0, sizeof(int32_t), st);
  } else {
    if (!chunk_score) return SPECEXT_ERR_INVALID_ARG;
    e = spx_launch_select(chunk_score + (long long)row * n_chunks, n_chunks, prefix_len, chunk_size, k,
                          n_sink_chunks, n_recent_chunks, idx, n_selected, st);
    g_launches.fetch_add(1);
  }
  if (e != cudaSuccess) {
    (void)cudaGetLastError();
    return SPECEXT_ERR_CUDA;
  }
  return SPECEXT_OK;
}

int specext_gather_kv(const void* draft_K, const void* draft_V, int32_t n_layers,
                      int32_t n_kv_heads, int32_t head_dim, int32_t prefix_len, int32_t chunk_size,
                      int64_t stride_layer, int64_t stride_l, int64_t stride_h, const int32_t* idx,
                      const int32_t* n_selected, int32_t max_selected, void* K_out, void* V_out,
                      int32_t* n_tokens_out, int32_t* device_status, void* cuda_stream) {
  if (!idx || !n_selected) return SPECEXT_ERR_INVALID_ARG;
  const int rc = check_gather_args(draft_K, draft_V, n_layers, n_kv_heads, head_dim, prefix_len, chunk_size,
                                   stride_layer, stride_l, stride_h, max_selected, K_out, V_out, n_tokens_out);
  if (rc != SPECEXT_OK) return rc;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  cudaError_t e = spx_launch_gather(draft_K, draft_V, n_layers, n_kv_heads, head_dim, prefix_len, chunk_size,
                                    stride_layer, stride_l, stride_h, idx, n_selected, max_selected, K_out,
                                    V_out, n_tokens_out, device_status, st);
  g_launches.fetch_add(1);
  if (e != cudaSuccess) {
    (void)cudaGetLastError();
    return SPECEXT_ERR_CUDA;
  }
  return SPECEXT_OK;
}

int specext_select_gather(const float* chunk_score, int32_t n_tree, int32_t n_chunks, int32_t row,
                          int32_t prefix_len, int32_t chunk_size, int32_t k, int32_t n_sink_chunks,
                          int32_t n_recent_chunks, const void* draft_K,
                          const void* draft_V, int32_t n_layers, int32_t n_kv_heads, int32_t head_dim,
                          int64_t stride_layer, int64_t stride_l, int64_t stride_h, int32_t* idx,
                          int32_t* n_selected, void* K_out, void* V_out, int32_t* n_tokens_out,
                          int32_t* device_status, void* cuda_stream) {
  const long long nc = chunk_size >= 1 && prefix_len >= 0 ? ((long long)prefix_len + chunk_size - 1) / chunk_size : -1;
  const bool fuse = nc == n_chunks && n_tree >= 1 && row >= 0 && row < n_tree && k >= 1 && chunk_score &&
                    n_sink_chunks >= 0 && n_recent_chunks >= 0 && spx_select_gather_fusable(n_chunks, k);
  if (!fuse) {
    // sizes the single launch is not built for, and every invalid argument, take the two calls
    const int rc = specext_select_chunks(chunk_score, n_tree, n_chunks, row, prefix_len, chunk_size, k,
                                         n_sink_chunks, n_recent_chunks, idx, n_selected, device_status, cuda_stream);
    if (rc != SPECEXT_OK) return rc;
    return specext_gather_kv(draft_K, draft_V, n_layers, n_kv_heads, head_dim, prefix_len, chunk_size, stride_layer,
                             stride_l, stride_h, idx, n_selected, k, K_out, V_out, n_tokens_out, device_status,
                             cuda_stream);
  }
  if (!idx || !n_selected) return SPECEXT_ERR_INVALID_ARG;
  const int rc = check_gather_args(draft_K, draft_V, n_layers, n_kv_heads, head_dim, prefix_len, chunk_size,
                                   stride_layer, stride_l, stride_h, k, K_out, V_out, n_tokens_out);
  if (rc != SPECEXT_OK) return rc;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  const cudaError_t e = spx_launch_select_gather(chunk_score + (long long)row * n_chunks, k, n_sink_chunks,
                                                 n_recent_chunks, draft_K, draft_V,
                                                 n_layers, n_kv_heads, head_dim, prefix_len, chunk_size,
                                                 stride_layer, stride_l, stride_h, idx, n_selected, K_out, V_out,
                                                 n_tokens_out, sm_count(), device_status, st);
  g_launches.fetch_add(1);
  if (e != cudaSuccess) {
    (void)cudaGetLastError();
    return SPECEXT_ERR_CUDA;
  }
  return SPECEXT_OK;
}

int specext_read_status(const int32_t* device_status, void* cuda_stream) {
  if (!device_status) return -SPECEXT_ERR_INVALID_ARG;
  int32_t h = 0;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  if (cudaMemcpyAsync(&h, device_status, sizeof(h), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess) {
    (void)cudaGetLastError();
    return -SPECEXT_ERR_CUDA;
  }
  return h;
}

const char* specext_status_string(int status) {
  switch (status) {
    case SPECEXT_OK: return "ok";
    case SPECEXT_ERR_INVALID_ARG: return "invalid argument";
    case SPECEXT_ERR_UNSUPPORTED: return "unsupported shape";
    case SPECEXT_ERR_WORKSPACE: return "workspace too small";
    case SPECEXT_ERR_BAD_TREE: return "parent[] is not a topologically ordered forest";
    case SPECEXT_ERR_TIMEOUT: return "bounded device wait expired";
    case SPECEXT_ERR_CUDA: return "CUDA call failed";
    default: return "unknown status";
  }
}

int64_t specext_launch_count(void) { return g_launches.load(); }


#ifdef SPECEXT_TESTING
// Test library only: forces an attention kernel / a lower bound on key tiles per worker for every
// later call in the process (see testing.h).
int specext_test_set_tuning(int32_t attn_kernel, int32_t min_tiles_per_cta) {
  if (attn_kernel < 0 || attn_kernel > 3 || min_tiles_per_cta < 0) return SPECEXT_ERR_INVALID_ARG;
  g_attn_kernel.store(attn_kernel);
  if (min_tiles_per_cta > 0) g_min_units.store(min_tiles_per_cta);
  return SPECEXT_OK;
}

// Test library only: the form that a call with this descriptor takes (see testing.h).
int specext_test_plan(const specext_attn_desc* desc, int32_t length_on_device, int32_t* out) {
  AttnPlan p;
  const int rc = build_plan(desc, &p, length_on_device != 0);
  if (rc != SPECEXT_OK) return rc;
  out[0] = p.kernel;
  out[1] = p.cluster;
  out[2] = p.q_rows;
  out[3] = p.U / p.n_cta;
  return SPECEXT_OK;
}
#endif

}  // extern "C"
