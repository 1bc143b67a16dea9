"""Calls from several threads at once, each on a stream of its own with buffers of its own, the first calls of the process
among them: results equal, bit for bit, those of one thread."""
import threading

import pytest
import torch

from paper_2505_20776_b200.hotpath import HotPath
from workloads import synth

pytestmark = pytest.mark.gpu

SHAPES = [(32, 8, 128, 60, 3100), (32, 8, 128, 60, 700), (32, 8, 128, 10, 1012), (12, 12, 64, 8, 900)]   # pairs; clusters


def _steps(hp, t, parent, L, dK, dV):
    for _ in range(5):
        hp.verify_attn(t, parent, L, True)
        hp.select_gather(1, L, dK, dV)
    return [x.clone() for x in (hp.O, hp.lse, hp.chunk_score(L), hp.idx, hp.K_compact)]


def test_threads_on_streams_of_their_own(cuda_device):
    dev = cuda_device
    work = []
    for i, (Hq, Hkv, D, T, L) in enumerate(SHAPES):
        w = synth.Workload("threads", Hq, Hkv, D, L, T, 32, 4, "uniform", "normal", seed=40 + i)
        dK, dV = synth.make_draft_kv(w)
        work.append((w, {k: v.to(dev) for k, v in synth.make_layer(w).items()}, torch.from_numpy(synth.make_tree(w)).to(dev),
                     dK.to(dev), dV.to(dev)))
    make = lambda w: HotPath(w.n_q_heads, w.n_kv_heads, w.head_dim, w.n_tree, 32, 4, w.prefix_len, device=dev)
    hps = [make(w[0]) for w in work]
    torch.cuda.synchronize()
    got, errors = [None] * len(work), []

    def run(i):
        try:
            w, t, parent, dK, dV = work[i]
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                got[i] = _steps(hps[i], t, parent, w.prefix_len, dK, dV)
            s.synchronize()
        except Exception as e:                       # reported below: an exception of a thread does not fail the test by itself
            errors.append(e)

    threads = [threading.Thread(target=run, args=(i,)) for i in range(len(work))]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert not errors, errors
    for i, (w, t, parent, dK, dV) in enumerate(work):
        hp = make(w)
        want = _steps(hp, t, parent, w.prefix_len, dK, dV)
        torch.cuda.synchronize()
        assert hp.read_status() == 0 and hps[i].read_status() == 0
        for a, b in zip(got[i], want):
            assert torch.equal(a, b)
