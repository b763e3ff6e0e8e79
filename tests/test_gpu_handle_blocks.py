"""Device blocks of the library: they go back when the last tensor of a closed handle is gone, and a call for which the
allocator has no room for padded copies takes the shapes that need none."""
import ctypes
import gc

import numpy as np
import pytest
import torch

import oracle
from oracle import CN, CU, D, S

pytestmark = pytest.mark.gpu

comet = pytest.importorskip("paper_2102_05187_b200")
from paper_2102_05187_b200 import binding  # noqa: E402
from gpu_util import assert_close, dev  # noqa: E402


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


class _LimitedHandle:
    """A library handle whose allocator refuses blocks beyond a limit."""

    def __init__(self, limit):
        self.lib, self.blocks, self.refused = comet.load_library(), {}, 0

        def alloc(_ctx, nbytes, _stream):
            if nbytes > limit:
                self.refused += 1
                return None
            t = torch.empty(max(nbytes, 1), dtype=torch.uint8, device="cuda")
            self.blocks[t.data_ptr()] = t
            return t.data_ptr()

        def free(_ctx, ptr, _stream):
            self.blocks.pop(ptr, None)

        self._calls = binding._ALLOC_FN(alloc), binding._FREE_FN(free)
        self._allocator = binding.AllocatorStruct(*self._calls, None)
        self._h = ctypes.c_void_p()
        assert self.lib.comet_create(ctypes.byref(self._h), ctypes.byref(self._allocator)) == 0

    check = comet.Handle.check


@pytest.mark.parametrize("R", [3, 131])
def test_no_room_for_padded_copies(R):
    handle = _LimitedHandle((4 if R == 3 else 8) << 20)
    rows, cols, n = 5000, 200_000 if R == 3 else 12_000, 420_000
    rng = np.random.default_rng(R)
    cell = np.unique(rng.integers(0, rows * cols, n + 2000))[:n]
    r, c = (cell // cols).astype(np.int32), (cell % cols).astype(np.int32)
    v, B = rng.uniform(-1, 1, n), rng.uniform(-1, 1, (cols, R))

    def upload(pk):
        up = lambda a: dev(a, torch.int32) if a.size else None  # noqa: E731
        return comet.SpTensor.from_arrays(pk.dims, pk.mode_order, pk.attr, [up(p) for p in pk.pos], [up(x) for x in pk.crd],
                                          dev(pk.val), handle=handle)

    want, norm = oracle.spmm([r, c], v, (rows, cols), B)
    A = upload(oracle.pack([r, c], v, (rows, cols), (0, 1), (D, CU)))
    assert_close(comet.spmm(A, dev(B)), want, norm)
    refused, handle.refused = handle.refused, 0
    dims = (rows, 20, cols // 20) if R == 131 else (rows, cols // 2, cols // 2)
    coords = [r, (c % dims[1]).astype(np.int32), (c // dims[1]).astype(np.int32)]
    F = [None] + [rng.uniform(-1, 1, (d, R)) for d in dims[1:]]
    want, norm = oracle.mttkrp(coords, v, dims, 0, F)
    for attr in [(CN, S, S), (CU, CU, CU)]:
        X = upload(oracle.pack(coords, v, dims, (0, 1, 2), attr))
        assert_close(comet.mttkrp(X, 0, [None, dev(F[1]), dev(F[2])]), want, norm)
    assert (refused or handle.refused) if R == 131 else (refused and handle.refused), "the limit was not met"
    handle.lib.comet_destroy(handle._h)


def test_no_room_for_the_carries_of_short_tiles():
    """Workers of one lane (rows of B of 16 bytes) take tiles of 16 entries; with no room for their carries, long ones."""
    handle = _LimitedHandle(2 << 20)
    rows, cols, n = 100_000, 1000, 2_000_000
    rng = np.random.default_rng(2)
    cell = np.unique(rng.integers(0, rows * cols, n + 50_000))[:n]
    r, c = (cell // cols).astype(np.int32), (cell % cols).astype(np.int32)
    v, B = rng.uniform(-1, 1, n), rng.uniform(-1, 1, (cols, 2))
    want, norm = oracle.spmm([r, c], v, (rows, cols), B)
    pk = oracle.pack([r, c], v, (rows, cols), (0, 1), (D, CU))
    A = comet.SpTensor.from_arrays(pk.dims, pk.mode_order, pk.attr, [dev(p, torch.int32) for p in pk.pos],
                                   [None, dev(pk.crd[1], torch.int32)], dev(pk.val), handle=handle)
    assert_close(comet.spmm(A, dev(B)), want, norm)
    assert handle.refused == 1, "the limit was not met"
    handle.lib.comet_destroy(handle._h)
