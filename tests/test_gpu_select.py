"""specext_select_gather at the edges of its chunk-count classes, exact against the oracle."""
import numpy as np
import pytest
import torch

from oracle import specext_oracle as orc
from paper_2505_20776_b200 import api
from tests.guards import GuardedAlloc
from tests.util import bf16_bits

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,C,k", [(511, 1, 7), (512, 1, 512), (513, 1, 512), (2048, 1, 1), (2049, 1, 1024), (4096, 1, 64),
                                   (4097, 1, 33), (8192, 1, 1000), (8193, 1, 40), (65536, 1, 300), (20001, 3, 50)])
@pytest.mark.parametrize("ties", [False, True])
def test_select_gather_chunk_counts(cuda_device, L, C, k, ties):
    """Chunk counts around what a thread holds (1, 4, 8, 16, 64 keys), with all keys distinct and with few distinct values
    (ties at the k-th key): indices, count and copied cache are exact.  Strided draft cache, two layers."""
    dev = cuda_device
    NC = -(-L // C)
    rng = np.random.default_rng(L + k)
    row = rng.integers(0, 5, NC).astype(np.float32) if ties else rng.permutation(NC).astype(np.float32) + 1
    scores = torch.from_numpy(np.stack([np.zeros(NC, np.float32), row])).to(dev)
    g = GuardedAlloc(dev)
    idx, ns, nt = (g.alloc((n,), torch.int32).fill_(-1) for n in (k, 1, 1))
    status = g.alloc((1,), torch.int32).zero_()
    big = torch.arange(2 * L * 3 * 16, dtype=torch.int32, device=dev).to(torch.int16).view(torch.bfloat16).view(2, L, 3, 16)
    dK, dV = big[:, :, 1:, :8], big[:, :, :2, 8:]                 # 2 heads x 8 of wider rows
    K, V = (g.alloc((2, k * C, 2, 8), torch.bfloat16).zero_() for _ in range(2))
    api.specext_select_gather(scores, 1, L, C, k, dK, dV, idx, ns, K, V, nt, status)
    assert api.specext_read_status(status) == 0
    g.check()
    want = orc.select_chunks(row, L, C, k, key_dtype=np.float32)
    assert int(ns.item()) == len(want)
    np.testing.assert_array_equal(idx[:len(want)].cpu().numpy(), want)
    for out, src in ((K, dK), (V, dV)):
        ref, _, n = orc.gather_kv(bf16_bits(src), bf16_bits(src), want, L, C)
        assert int(nt.item()) == n
        np.testing.assert_array_equal(bf16_bits(out)[:, :n], ref)


def test_chunk_size_far_beyond_the_prefix(cuda_device):
    """One chunk of 2^24 tokens, 2^32 vectors of 16 bytes in the compact cache's layout, of which 100 tokens exist: they are
    copied (only valid tokens are written, so the buffers hold just these; the binding would ask for the whole layout)."""
    dev, L, C, H, D = cuda_device, 100, 1 << 24, 16, 128
    dK, dV = (torch.randn(1, L, H, D, device=dev).to(torch.bfloat16) for _ in range(2))
    g = GuardedAlloc(dev)
    idx, ns, nt = (g.alloc((1,), torch.int32).fill_(-1) for _ in range(3))
    status = g.alloc((1,), torch.int32).zero_()
    K, V = (g.alloc((L, H, D), torch.bfloat16).zero_() for _ in range(2))
    scores = torch.ones(1, 1, device=dev)
    torch.cuda.synchronize()
    rc = api.lib().specext_select_gather(scores.data_ptr(), 1, 1, 0, L, C, 1, 0, 0, dK.data_ptr(), dV.data_ptr(), 1, H, D,
                                         L * H * D, H * D, D, idx.data_ptr(), ns.data_ptr(), K.data_ptr(), V.data_ptr(),
                                         nt.data_ptr(), status.data_ptr(), torch.cuda.current_stream().cuda_stream)
    assert rc == 0 and api.specext_read_status(status) == 0
    g.check()
    assert [int(x.item()) for x in (idx, ns, nt)] == [0, 1, L]
    assert torch.equal(K, dK[0]) and torch.equal(V, dV[0])


@pytest.mark.parametrize("L,k", [(16384, 900), (16385, 900), (16000, 16000)])
@pytest.mark.parametrize("ties", [False, True])
def test_select_gather_sixteen_keys_a_thread_of_1024(cuda_device, L, k, ties):
    """Both sides of the line between 16 and 64 keys per thread, and every chunk kept."""
    test_select_gather_chunk_counts(cuda_device, L, 1, k, ties)
