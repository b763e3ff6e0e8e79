"""Device blocks of the library: they go back when the last tensor of a closed handle is gone."""
import gc

import numpy as np
import pytest
import torch

from oracle import CU, D

pytestmark = pytest.mark.gpu

comet = pytest.importorskip("paper_2102_05187_b200")
from gpu_util import dev  # noqa: E402


@pytest.fixture(autouse=True)
def _need_gpu(cuda_device):
    yield


def _entries(n, dims, seed):
    rng = np.random.default_rng(seed)
    cell = rng.permutation(int(np.prod(dims)))[:n]
    return [c.astype(np.int32) for c in np.unravel_index(cell, dims)], rng.uniform(-1, 1, n)


@pytest.mark.parametrize("attr", [(D, CU), (CU, CU)])
@pytest.mark.parametrize("use", ["tensor", "view"])
def test_a_closed_handle_gives_its_blocks_back_with_the_last_tensor(use, attr):
    coords, val = _entries(50_000, (300, 400), 1)
    coords, val = [dev(c) for c in coords], dev(val)
    gc.collect()
    torch.cuda.synchronize()
    before = torch.cuda.memory_allocated()
    handle = comet.Handle()
    T = comet.pack(coords, val, (300, 400), (0, 1), attr, handle=handle)
    want = T.val.clone()
    view = T.val if use == "view" else None
    handle.close()
    del T, handle
    gc.collect()
    if use == "view":                                        # the values live as long as someone can read them
        assert torch.equal(view, want)
    del view, want
    gc.collect()
    assert torch.cuda.memory_allocated() == before
