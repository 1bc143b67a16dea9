"""Short calls back to back on one workspace, inputs changing from call to call, in a CUDA graph: a call's set-up overlaps the
end of the one before it, whose clusters may still be exchanging partial results (through shared memory, or through the
workspace), and must not disturb it."""
import numpy as np
import pytest
import torch

from paper_2505_20776_b200 import api
from tests.test_gpu_dispatch import launches
from tests.test_gpu_parity import LSE_ATOL, O_ATOL, SCORE_RTOL, oracle_layer, to_dev
from tests.util import f64
from workloads import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Hq,Hkv,D,T,L,want", [
    (32, 8, 128, 8, 700, 1),         # 32 rows: exchange through shared memory
    (12, 12, 64, 8, 1024, 1),        # the same with head_dim 64
    (32, 8, 128, 60, 1003, 1),       # through L2, clusters of up to 8
    (32, 8, 128, 10, 1012, 1),       # through L2, larger clusters
    (32, 8, 128, 60, 100, 2),        # two launches on a prefix of one tile
])
def test_short_calls_share_a_workspace(cuda_device, Hq, Hkv, D, T, L, want):
    dev = cuda_device
    assert launches(dev, Hq, Hkv, D, T, L) == want
    w = synth.Workload("overlap", Hq, Hkv, D, L, T, 32, 4, "uniform", "normal", seed=L + T)
    parent = synth.make_tree(w)
    par = torch.from_numpy(parent).to(dev)
    cpu = [synth.make_layer(w, layer=i) for i in range(6)]
    layers = [to_dev(t, dev) for t in cpu]
    outs = [torch.zeros(T, Hq, D, dtype=torch.bfloat16, device=dev) for _ in layers]
    lses = [torch.zeros(Hq, T, dtype=torch.float32, device=dev) for _ in layers]
    status = torch.zeros(1, dtype=torch.int32, device=dev)
    d = api.make_attn_desc(layers[0]["Q"], layers[0]["K_prefix"], layers[0]["K_tree"], outs[0], L, 32)
    ws = torch.zeros(api.specext_verify_attn_workspace(d), dtype=torch.uint8, device=dev)

    def call(i):
        t = layers[i]
        api.specext_verify_attn(d, t["Q"], t["K_prefix"], t["V_prefix"], t["K_tree"], t["V_tree"], par, outs[i], lses[i],
                                None, ws, status)

    alone = []
    for i in range(len(layers)):
        call(i)
        torch.cuda.synchronize()
        alone.append((outs[i].clone(), lses[i].clone()))
        O_ref, lse_ref, _ = oracle_layer(cpu[i], parent, L, 32, None)
        assert np.abs(f64(outs[i]) - O_ref).max() <= O_ATOL
        assert np.abs(f64(lses[i]) - lse_ref).max() <= LSE_ATOL
    s = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(s):
        with torch.cuda.graph(g, stream=s):
            for _ in range(4):
                for i in range(len(layers)):
                    call(i)
        for _ in range(10):
            for x in outs + lses:
                x.zero_()
            ws.fill_(0xFF)                       # NaN: what a call has not written itself shows
            for _ in range(5):
                g.replay()
            s.synchronize()
            for i, (O, lse) in enumerate(alone):
                assert torch.equal(outs[i], O) and torch.equal(lses[i], lse)
    assert int(status.item()) == 0


@pytest.mark.parametrize("Hq,Hkv,T,L,want", [
    (32, 8, 60, 4096, 2),            # pairs, scores beside the merge
    (32, 8, 1, 16383, 2),            # workers of one CTA, scores beside the merge
    (32, 8, 60, 4737, 3),            # scores by a launch of their own
    (32, 8, 60, 1003, 2),            # clusters, scores by a launch of their own
])
def test_scored_calls_share_a_workspace(cuda_device, Hq, Hkv, T, L, want):
    dev = cuda_device
    assert launches(dev, Hq, Hkv, 128, T, L, scored=True) == want
    w = synth.Workload("overlap-scored", Hq, Hkv, 128, L, T, 32, 4, "uniform", "needle", seed=L + T)
    parent = synth.make_tree(w)
    par = torch.from_numpy(parent).to(dev)
    cpu = [synth.make_layer(w, layer=i) for i in range(4)]
    layers = [to_dev(t, dev) for t in cpu]
    outs = [torch.zeros(T, Hq, 128, dtype=torch.bfloat16, device=dev) for _ in layers]
    lses = [torch.zeros(Hq, T, dtype=torch.float32, device=dev) for _ in layers]
    scores = [torch.zeros(T, -(-L // 32), dtype=torch.float32, device=dev) for _ in layers]
    status = torch.zeros(1, dtype=torch.int32, device=dev)
    d = api.make_attn_desc(layers[0]["Q"], layers[0]["K_prefix"], layers[0]["K_tree"], outs[0], L, 32, 0.0, True)
    ws = torch.zeros(api.specext_verify_attn_workspace(d), dtype=torch.uint8, device=dev)

    def call(i):
        t = layers[i]
        api.specext_verify_attn(d, t["Q"], t["K_prefix"], t["V_prefix"], t["K_tree"], t["V_tree"], par, outs[i], lses[i],
                                scores[i], ws, status)

    alone = []
    for i in range(len(layers)):
        call(i)
        torch.cuda.synchronize()
        alone.append((outs[i].clone(), lses[i].clone(), scores[i].clone()))
        O_ref, lse_ref, score_ref = oracle_layer(cpu[i], parent, L, 32, None)
        assert np.abs(f64(outs[i]) - O_ref).max() <= O_ATOL
        assert np.abs(f64(lses[i]) - lse_ref).max() <= LSE_ATOL
        assert (np.abs(f64(scores[i]) - score_ref) / np.maximum(score_ref, 1e-30)).max() <= SCORE_RTOL
    s = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(s):
        with torch.cuda.graph(g, stream=s):
            for _ in range(4):
                for i in range(len(layers)):
                    call(i)
        for _ in range(10):
            for x in outs + lses + scores:
                x.zero_()
            ws.fill_(0xFF)                       # NaN: what a call has not written itself shows
            for _ in range(5):
                g.replay()
            s.synchronize()
            for i, (O, lse, score) in enumerate(alone):
                assert torch.equal(outs[i], O) and torch.equal(lses[i], lse) and torch.equal(scores[i], score)
    assert int(status.item()) == 0
