"""Calls that run at the same time on streams of their own and share an array."""
from __future__ import annotations

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2503_08217_gb300 import binding, build
    build.build()
    binding.load()


@pytest.mark.parametrize("n", [4_000_001, 5])
def test_disjoint_records_of_one_life_array(n):
    """Two RECORD calls with masks that share no Gaussian: each updates its own
    and writes no other, so neither's update can be lost."""
    from paper_2503_08217_gb300 import binding
    words = (n + 31) // 32
    masks = [torch.full((words,), m, dtype=torch.int32, device="cuda") for m in (0x55555555, -0x55555556)]
    times = [0.25, -0.5]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    want = np.empty((n, 2), np.float32)
    want[0::2], want[1::2] = times[0], times[1]          # the empty life (1, -1) extended to one time
    for _ in range(10):
        life = torch.tensor([1.0, -1.0], device="cuda").repeat(n, 1).contiguous()
        torch.cuda.synchronize()
        for stream, mask, t in zip(streams, masks, times):
            binding.update_visibility(n, t, mask, life, None, binding.VIS_RECORD, stream)
        torch.cuda.synchronize()
        np.testing.assert_array_equal(life.cpu().numpy(), want)
