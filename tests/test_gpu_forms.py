"""Forms that a rule on sizes chooses: that the sizes meant to reach a form do, and its results against the oracle (tolerances of
test_gpu_parity).  On the B200 (clusters of up to 16 of its CTAs)."""
import numpy as np
import pytest
import torch

from tests.test_gpu_dispatch import launches
from tests.test_gpu_draft_attn import DraftSide, _oracle
from tests.test_gpu_parity import LSE_ATOL, O_ATOL, check_attn, make_hp
from tests.testing_lib import plan
from tests.util import f64
from workloads import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Hq,Hkv,T,L,cluster,q_rows,tiles", [
    (32, 32, 60, 5500, 4, 64, 11), (32, 32, 60, 6000, 4, 128, 12), (32, 32, 60, 8201, 4, 128, 16),     # clusters
    (32, 32, 30, 8201, 4, 32, 16),                                           # up to 32 rows: the exchange needs the room
    (128, 128, 3, 1500, 0, 64, 11), (128, 128, 3, 2000, 0, 128, 14),         # workers across problems, few rows
    (160, 160, 64, 1600, 0, 128, 15),                                        # as many rows as the smaller form has
])
def test_rows_of_q(cuda_device, Hq, Hkv, T, L, cluster, q_rows, tiles):
    """Up to 64 rows: 128 rows of Q (zeros behind the last) from 12 tiles per CTA on."""
    assert plan(Hq, Hkv, 128, T, L) == (2, cluster, q_rows, tiles)
    w = synth.Workload("q-rows", Hq, Hkv, 128, L, T, 32, 4, "uniform", "needle", seed=T + L)
    check_attn(make_hp(w, cuda_device), synth.make_layer(w), synth.make_tree(w), L, 32, want_score=False)


@pytest.mark.parametrize("Hq,Hkv,T,cap,cluster", [(32, 32, 40, 8192, 4), (128, 128, 3, 2048, 0)])
def test_rows_of_q_with_a_length_on_the_device(cuda_device, Hq, Hkv, T, cap, cluster):
    dev = cuda_device
    form = plan(Hq, Hkv, 128, T, cap, length_on_device=True)
    assert form[:3] == (2, cluster, 128) and form[3] >= 12
    w = synth.Workload("q-rows-draft", Hq, Hkv, 128, cap, T, 32, 1, "uniform", "normal", seed=T + cap)
    cpu, parent = synth.make_layer(w), synth.make_tree(w)
    t, par = {k: v.to(dev) for k, v in cpu.items()}, torch.from_numpy(parent).to(dev)
    side = DraftSide(Hq, Hkv, 128, T, cap, dev)
    for n in (cap // 3 + 5, cap - 61, cap):
        K, V = t["K_prefix"].clone(), t["V_prefix"].clone()
        K[n:] = V[n:] = float("nan")
        side.n_tokens.fill_(n)
        side.run(t, par, K, V)
        assert side.hp.read_status() == 0
        side.hp.check()
        O, lse, _ = _oracle(cpu, cpu["K_prefix"], cpu["V_prefix"], n, parent)
        assert np.abs(f64(side.hp.O) - O).max() <= O_ATOL and np.abs(f64(side.hp.lse) - lse).max() <= LSE_ATOL, f"n_tokens={n}"


# The sizes of test_gpu_row_blocks.py, whose results are compared there.
@pytest.mark.parametrize("Hq,Hkv,D,T,L,cluster", [
    (12, 12, 128, 31, 600, 6), (12, 12, 128, 32, 600, 6), (12, 12, 64, 32, 600, 6),
    (4, 4, 128, 29, 800, 8), (8, 1, 128, 4, 900, 5), (2, 1, 64, 16, 250, 3), (4, 4, 128, 32, 700, 7),
])
def test_clusters_that_exchange_through_shared_memory(cuda_device, Hq, Hkv, D, T, L, cluster):
    assert T * Hq // Hkv <= 32
    assert plan(Hq, Hkv, D, T, L)[:2] == (2, cluster)
    assert launches(cuda_device, Hq, Hkv, D, T, L) == 1


@pytest.mark.parametrize("Hq,Hkv,D,T,L,C,want", [
    (32, 8, 128, 60, 4096, 64, 2), (32, 8, 128, 60, 4700, 128, 2), (32, 8, 128, 60, 4737, 32, 3), (32, 8, 128, 37, 4000, 32, 2),
    (32, 8, 128, 1, 16383, 32, 2), (16, 4, 128, 8, 16000, 32, 2), (32, 8, 128, 43, 78, 32, 2), (24, 6, 128, 8, 9000, 64, 2),
    (48, 3, 128, 16, 126, 128, 2),
    # a launch of their own: chunks of fewer than 32 keys, more than 8 KV heads, more than 48 segments
    (32, 8, 128, 60, 4096, 16, 3), (48, 12, 128, 43, 78, 32, 3), (12, 12, 64, 9, 15607, 32, 3),
    (16, 4, 128, 8, 18000, 32, 3), (16, 2, 64, 3, 16000, 128, 3), (32, 1, 128, 2, 14000, 32, 3),
])
def test_scores_beside_the_merge(cuda_device, Hq, Hkv, D, T, L, C, want):
    assert plan(Hq, Hkv, D, T, L, C, scored=True)[1] == 0
    assert launches(cuda_device, Hq, Hkv, D, T, L, C, scored=True) == want
