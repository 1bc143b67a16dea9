"""The one-CTA verification kernel at the edges of its row blocks and segments, and prefill with many query heads per KV
head, against the oracle (tolerances of test_gpu_parity: bf16 inputs and probabilities, fp32 sums)."""
import pytest

from tests.test_gpu_parity import check_attn, make_hp
from tests.test_gpu_prefill import _compare, _inputs, _run
from tests.testing_lib import tuned
from workloads import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Hq,Hkv,D,T,L", [
    (2, 2, 128, 63, 300),      # 64-row form of Q, one row short
    (2, 2, 128, 64, 256),      # 64-row form, full
    (2, 2, 128, 65, 129),      # 128-row form, tree of more than 64 nodes
    (2, 2, 128, 128, 127),     # 128-row form, full
    (8, 2, 128, 8, 1),         # 32 rows: one warp works, one key
    (4, 1, 64, 33, 640),       # head_dim 64: a second row block with 4 rows
    (4, 1, 64, 128, 131),      # head_dim 64: four row blocks
    (256, 256, 128, 3, 40),    # more problems than CTAs: several segments per worker, each of one tile or two
    (160, 160, 64, 5, 515),    # the same with head_dim 64 and segments of an odd and an even number of tiles
    # clusters that merge among themselves: 2 to 8 CTAs, rows dealt (up to 32) and columns dealt (more), uneven deals
    (2, 2, 128, 1, 100), (32, 8, 128, 1, 500), (32, 8, 128, 8, 700), (32, 8, 128, 9, 700), (8, 8, 128, 7, 900),
    (12, 12, 64, 32, 900), (12, 12, 64, 33, 4096), (32, 32, 128, 100, 300), (32, 8, 128, 60, 130), (32, 8, 128, 60, 2048),
    (64, 8, 128, 60, 1000), (32, 8, 128, 127, 513),
    (32, 8, 128, 10, 1012), (32, 8, 128, 30, 1300), (16, 4, 128, 32, 2000), (8, 2, 64, 40, 2048),    # more than 8 CTAs
])
def test_one_cta_row_blocks(cuda_device, Hq, Hkv, D, T, L):
    w = synth.Workload("rows", Hq, Hkv, D, L, T, 32, 4, "uniform", "needle", seed=Hq + T + L)
    check_attn(make_hp(w, cuda_device), synth.make_layer(w), synth.make_tree(w), L, 32)


@pytest.mark.parametrize("Hq,Hkv,D,T,L", [
    (12, 12, 128, 31, 600), (12, 12, 128, 32, 600), (12, 12, 64, 32, 600),     # 6 CTAs: 36 parts, all the room there is
    (4, 4, 128, 29, 800), (8, 1, 128, 4, 900), (2, 1, 64, 16, 250),            # 8, 5 and 3 CTAs: 32, 35 and 33 parts
    (4, 4, 128, 32, 700),                                                      # 7 CTAs, 35 parts
])
def test_parts_in_shared_memory(cuda_device, Hq, Hkv, D, T, L):
    """Clusters of few rows write their parts into each other's shared memory: as many parts as it has room for."""
    w = synth.Workload("parts", Hq, Hkv, D, L, T, 32, 4, "uniform", "needle", seed=Hq + T + L)
    check_attn(make_hp(w, cuda_device), synth.make_layer(w), synth.make_tree(w), L, 32)


@pytest.mark.parametrize("G", [64, 128, 256])
def test_prefill_wide_groups(cuda_device, G):
    """Blocks of 4, 2 and 1 tokens: more problems than clusters, and (G = 256) one token's heads on two CTAs."""
    L = 131
    Q, K, V = _inputs(L, G, 1, seed=G)
    O, lse = _run(cuda_device, Q, K, V)
    _compare(O, lse, Q, K, V, [0, 1, 2, 3, 4, 63, 64, 126, 127, 128, 129, 130], f"prefill-small-G{G}")


@pytest.mark.parametrize("Hq,Hkv,D,T,L,C", [
    (8, 2, 128, 128, 9500, 4),      # groups of 8 chunks: two row blocks, 32 chunks in a tile, a ragged last one
    (8, 8, 64, 3, 6400, 1),         # 128 chunks in a tile
])
def test_chunk_scores_in_groups_of_eight(cuda_device, Hq, Hkv, D, T, L, C):
    w = synth.Workload("score8", Hq, Hkv, D, L, T, C, 4, "uniform", "needle", seed=T + C)
    check_attn(make_hp(w, cuda_device), synth.make_layer(w), synth.make_tree(w), L, C)


@pytest.mark.parametrize("C", [8, 16, 64, 128])
@pytest.mark.parametrize("kernel,Hq,Hkv,D,T,L", [
    (0, 2, 2, 128, 64, 700),       # one cluster per problem
    (2, 2, 2, 128, 64, 700),       # workers that leave partial results
    (2, 8, 2, 128, 60, 1000),      # two row blocks of the one-CTA kernel
    (0, 160, 160, 64, 5, 515),     # several segments per worker
    (0, 32, 8, 128, 60, 3001),     # paired kernel
])
def test_chunk_sums_of_every_class(cuda_device, kernel, Hq, Hkv, D, T, L, C):
    """Chunks of fewer than 32 keys, of 64 and of 128, whose sums the kernels store in three ways."""
    w = synth.Workload("chunks", Hq, Hkv, D, L, T, C, 4, "uniform", "needle", seed=C + L)
    with tuned(kernel, 0):
        check_attn(make_hp(w, cuda_device), synth.make_layer(w), synth.make_tree(w), L, C)


@pytest.mark.parametrize("Hq,Hkv,D,T,L,C", [
    (32, 8, 128, 60, 4096, 64), (32, 8, 128, 60, 4700, 128),     # pairs; 37 tiles x 4 groups of 64 rows: all the blocks there are
    (32, 8, 128, 60, 4737, 32),                                  # one tile more: a launch of its own
    (32, 8, 128, 37, 4000, 32),                                  # 148 rows: two and a third groups
    (32, 8, 128, 1, 16383, 32),                                  # one-CTA kernel, fewer rows than a group
    (16, 4, 128, 8, 16000, 32),                                  # one head a thread, 43 segments, blocks without a merge
    (24, 6, 128, 8, 9000, 64),                                   # two heads for two of the four slices
    (48, 3, 128, 16, 126, 128),                                  # no head for the last slice
    (16, 2, 64, 3, 16000, 128), (32, 1, 128, 2, 14000, 32),      # more than 48 segments: a launch of their own
])
def test_chunk_scores_beside_the_merge(cuda_device, Hq, Hkv, D, T, L, C):
    w = synth.Workload("beside", Hq, Hkv, D, L, T, C, 4, "uniform", "needle", seed=T + C)
    check_attn(make_hp(w, cuda_device), synth.make_layer(w), synth.make_tree(w), L, C)
