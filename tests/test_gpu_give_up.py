"""A role that gives up lets its CTA end only when copies that are on their way into shared memory have landed."""
import pytest
import torch

from tests.testing_lib import load_testing_lib

pytestmark = pytest.mark.gpu


def test_copies_land_before_the_cta_ends(cuda_device):
    L = load_testing_lib()
    src = torch.zeros(16384, dtype=torch.uint8, device=cuda_device)
    out = torch.zeros(2, dtype=torch.int64, device=cuda_device)
    assert L.specext_test_settle(src.data_ptr(), out.data_ptr(), torch.cuda.current_stream().cuda_stream) == 0
    cycles, landed = out.tolist()
    assert cycles >= L.specext_test_settle_cycles() and landed == 1
