"""Calls behind a kernel that lets its dependents be set up at once and then runs for longer than the library's bounded waits last:
the waits begin when that kernel has completed, and what it writes at its end is what the call reads."""
import numpy as np
import pytest
import torch

from paper_2505_20776_b200 import api
from tests.test_gpu_dispatch import launches
from tests.test_gpu_parity import LSE_ATOL, O_ATOL, SCORE_RTOL, make_hp, oracle_layer, to_dev
from tests.test_gpu_prefill import _compare, _inputs
from tests.testing_lib import load_testing_lib
from tests.util import f64
from workloads import synth

pytestmark = pytest.mark.gpu


def slow_then(dst, value):
    """Queues the slow kernel on the current stream; *dst becomes `value` at its end."""
    lib = load_testing_lib()
    cycles = lib.specext_test_wait_limit() * 6 // 5
    assert lib.specext_test_slow_kernel(cycles, dst.data_ptr(), value, torch.cuda.current_stream().cuda_stream) == 0


@pytest.mark.parametrize("Hq,Hkv,D,T,L,scored,want", [
    (32, 8, 128, 8, 700, False, 1),          # clusters: exchange through shared memory,
    (32, 8, 128, 60, 1003, False, 1),        # through L2,
    (32, 8, 128, 10, 1012, False, 1),        # through L2 with more than 8 CTAs
    (32, 8, 128, 1, 16383, True, 2),         # workers of one CTA, merge and chunk scores
    (32, 8, 128, 60, 4096, True, 2),         # pairs
])
def test_verification(cuda_device, Hq, Hkv, D, T, L, scored, want):
    dev = cuda_device
    assert launches(dev, Hq, Hkv, D, T, L, scored=scored) == want
    w = synth.Workload("slow", Hq, Hkv, D, L, T, 32, 4, "uniform", "needle", seed=T + L)
    cpu, parent = synth.make_layer(w), synth.make_tree(w)
    hp, t, par = make_hp(w, dev), to_dev(cpu, dev), torch.from_numpy(parent).to(dev)
    hp.verify_attn(t, par, L, scored)
    assert hp.read_status() == 0
    for x in (hp.O, hp.lse):
        x.fill_(float("nan"))
    par[0] = 5                                # no tree: an entry that a call must not see
    torch.cuda.synchronize()
    slow_then(par, int(parent[0]))
    hp.verify_attn(t, par, L, scored)
    assert hp.read_status() == 0
    O, lse, score = oracle_layer(cpu, parent, L, 32, None)
    assert np.abs(f64(hp.O) - O).max() <= O_ATOL
    assert np.abs(f64(hp.lse) - lse).max() <= LSE_ATOL
    if scored:
        assert (np.abs(f64(hp.chunk_score(L)) - score) / np.maximum(score, 1e-30)).max() <= SCORE_RTOL


@pytest.mark.parametrize("Hq,Hkv,T,cap,before,n", [
    (32, 8, 10, 1024, 1024, 500), (32, 8, 60, 8192, 8192, 3000),
    (32, 8, 10, 1024, 0, 1000), (32, 8, 10, 8192, 100, 8192), (32, 8, 10, 8192, 8192, 0),     # what the call may look at early
])
def test_draft(cuda_device, Hq, Hkv, T, cap, before, n):
    dev = cuda_device
    w = synth.Workload("slow-draft", Hq, Hkv, 128, cap, T, 32, 1, "uniform", "normal", seed=T + n)
    cpu, parent = synth.make_layer(w), synth.make_tree(w)
    hp, t, par = make_hp(w, dev), to_dev(cpu, dev), torch.from_numpy(parent).to(dev)
    d = api.make_attn_desc(t["Q"], t["K_prefix"], t["K_tree"], hp.O, cap, 32, 0.0, False)
    ws = torch.empty(api.specext_verify_attn_workspace(d), dtype=torch.uint8, device=dev)
    length = torch.full((1,), before, dtype=torch.int32, device=dev)
    for k in range(2):
        if k == 1:
            hp.O.fill_(float("nan"))
            torch.cuda.synchronize()
            slow_then(length, n)
        api.specext_draft_attn(d, t["Q"], t["K_prefix"], t["V_prefix"], length, t["K_tree"], t["V_tree"], par, hp.O, hp.lse, ws,
                               hp.status)
        assert hp.read_status() == 0
    cut = dict(cpu, K_prefix=cpu["K_prefix"][:n], V_prefix=cpu["V_prefix"][:n])
    O, lse, _ = oracle_layer(cut, parent, n, 32, None)
    # Without a prefix O is a mean of a few values up to 4 and not of hundreds: rounding O to bf16 gives up to 2^-8 |O|, rounding
    # the probabilities up to 2^-8 |V|, together more than O_ATOL.
    atol = O_ATOL if n > 0 else 2.0 ** -8 * (np.abs(O).max() + float(cpu["V_tree"].abs().max()))
    assert np.abs(f64(hp.O) - O).max() <= atol
    assert np.abs(f64(hp.lse) - lse).max() <= LSE_ATOL


def test_prefill(cuda_device):
    dev = cuda_device
    L = 700
    Q, K, V = _inputs(L, 8, 2, seed=9)
    q, k, v = Q.to(dev), K.to(dev), V.to(dev)
    O, lse = torch.empty_like(q), torch.empty(8, L, device=dev)
    status, at_end = torch.zeros(1, dtype=torch.int32, device=dev), torch.zeros(1, dtype=torch.int32, device=dev)
    for i in range(2):
        if i == 1:
            O.fill_(float("nan"))
            torch.cuda.synchronize()
            slow_then(at_end, 1)
        api.specext_prefill_attn(q, k, v, O, lse, status)
        assert api.specext_read_status(status) == 0
    assert int(at_end.item()) == 1
    _compare(O, lse, Q, K, V, [0, 1, 127, 128, 129, 511, 512, 698, 699], "prefill-after-slow-kernel")
