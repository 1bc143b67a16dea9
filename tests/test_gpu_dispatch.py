"""Which form a call takes, seen by the kernels it launches: one whose clusters merge by themselves is one launch, one that
leaves partial results two, and the chunk scores are one more, unless they are added up beside the merge (chunks of 32 keys and
more on up to 148 tiles of 64 rows).  On the B200 (clusters of up to 16 of its CTAs)."""
import pytest
import torch

from paper_2505_20776_b200 import api

pytestmark = pytest.mark.gpu


def launches(dev, Hq, Hkv, D, T, L, C=32, scored=False, n_tokens=None):
    """Kernels launched by one call on zeros; n_tokens: the device-side length of a draft call."""
    z = lambda *s: torch.zeros(*s, dtype=torch.bfloat16, device=dev)
    Q, K, Kt, O = z(T, Hq, D), z(max(L, 1), Hkv, D), z(T, Hkv, D), z(T, Hq, D)
    lse = torch.zeros(Hq, T, device=dev)
    score = torch.zeros(T, -(-L // C), device=dev) if scored else None
    parent = torch.full((T,), -1, dtype=torch.int32, device=dev)
    status = torch.zeros(1, dtype=torch.int32, device=dev)
    d = api.make_attn_desc(Q, K, Kt, O, L, C, 0.0, scored)
    ws = torch.empty(api.specext_verify_attn_workspace(d), dtype=torch.uint8, device=dev)
    before = api.specext_launch_count()
    if n_tokens is None:
        api.specext_verify_attn(d, Q, K, K, Kt, Kt, parent, O, lse, score, ws, status)
    else:
        n = torch.tensor([n_tokens], dtype=torch.int32, device=dev)
        api.specext_draft_attn(d, Q, K, K, n, Kt, Kt, parent, O, lse, ws, status)
    after = api.specext_launch_count()
    assert api.specext_read_status(status) == 0
    return after - before


@pytest.mark.parametrize("Hq,Hkv,D,T,L,C,want", [
    (32, 8, 128, 60, 2048, 16, 3),      # clusters of 6: 3 tiles instead of 2
    (32, 8, 128, 60, 2048, 32, 2),      # which is fine for larger chunks
    (32, 8, 64, 60, 8192, 4, 3), (32, 8, 64, 60, 8192, 64, 2),          # 11 tiles instead of 8
    (16, 2, 128, 1, 4096, 16, 3), (16, 2, 128, 1, 4096, 128, 2),        # 5 instead of 1
    (32, 8, 128, 100, 1000, 16, 2),     # 3 instead of 3
    (32, 8, 128, 100, 2048, 4, 2), (32, 8, 128, 100, 3000, 4, 3),       # 5, 7
    (32, 32, 128, 60, 6000, 16, 2),     # 12 instead of 11
    (12, 12, 64, 100, 4096, 16, 2),     # 4 instead of 3
    (32, 32, 128, 60, 200, 1, 2),       # one tile
    (32, 8, 128, 60, 1000, 1, 3), (32, 8, 128, 60, 1000, 4, 2),         # 2 instead of 1
])
def test_small_chunks_stay_on_the_split_path(cuda_device, Hq, Hkv, D, T, L, C, want):
    assert launches(cuda_device, Hq, Hkv, D, T, L, C, scored=True) == want


@pytest.mark.parametrize("Hq,Hkv,T,L,scored,want", [
    (64, 8, 60, 2048, False, 1), (64, 8, 60, 3000, False, 2),        # 5 and 7 tiles in clusters of 4
    (64, 8, 60, 2048, True, 2), (64, 8, 60, 4096, True, 3),
    (64, 8, 100, 2048, False, 1), (64, 8, 100, 2048, True, 2),       # 9 tiles, 32 blocks of 256 rows
    (16, 2, 100, 8192, False, 1), (16, 2, 100, 8192, True, 3),       # 8 tiles in clusters of 9
    (64, 8, 100, 3000, False, 2), (64, 8, 80, 4096, True, 2),        # 13 tiles; 11, 24 blocks
    (32, 8, 80, 8192, True, 2),                                      # 13 tiles against 17
    (32, 4, 80, 6000, True, 2),                                      # 8 tiles, 12 blocks of 256 rows and 6 segments to merge
])
def test_many_tiles_go_to_the_pairs(cuda_device, Hq, Hkv, T, L, scored, want):
    assert launches(cuda_device, Hq, Hkv, 128, T, L, 32, scored) == want


@pytest.mark.parametrize("Hq,Hkv,D,T,L,want", [
    (32, 8, 128, 60, 100, 2), (32, 8, 128, 60, 129, 1),      # one tile and the tree, two and the tree
    (32, 8, 128, 16, 128, 1), (32, 8, 128, 17, 128, 2),      # 64 and 68 rows
    (64, 64, 128, 100, 100, 1), (12, 12, 64, 100, 100, 1),   # many problems, head_dim 64
])
def test_prefix_of_one_tile(cuda_device, Hq, Hkv, D, T, L, want):
    assert launches(cuda_device, Hq, Hkv, D, T, L) == want


@pytest.mark.parametrize("Hq,Hkv,T,cap", [(64, 8, 60, 4096), (32, 8, 100, 4096), (16, 2, 100, 16384), (32, 8, 60, 128)])
def test_draft_calls_stay_in_clusters(cuda_device, Hq, Hkv, T, cap):
    """Shapes that verification takes to the pairs; the workspace is the same for both."""
    assert launches(cuda_device, Hq, Hkv, 128, T, cap) == 2
    assert launches(cuda_device, Hq, Hkv, 128, T, cap, n_tokens=cap) == 1
