"""comet_pack of larger inputs where the allocator has little room: whatever the splits by sampled keys or the result next to
their records are refused, the radix sort's 24 bytes per entry are enough, and no block stays behind."""
import ctypes as C
import functools

import numpy as np
import pytest
import torch

import oracle
import synth
from oracle import D, CU, CN, S

pytestmark = pytest.mark.gpu

comet = pytest.importorskip("paper_2102_05187_b200")
from paper_2102_05187_b200 import binding  # noqa: E402
from gpu_util import assert_equal_arrays  # noqa: E402

MATRIX, TENSOR = (1009, 997), (101, 103, 97)
CASES = [((D, CU), MATRIX), ((CU, CU), MATRIX), ((CN, S), MATRIX), ((CU, CU, CU), TENSOR), ((CN, S, S), TENSOR), ((D, CU, CU), TENSOR)]
N = 610_000                                                  # more than the cooperative launch of small inputs takes


class _Handle(comet.Handle):
    """A handle whose allocator counts the bytes in use, and refuses requests by number or beyond a limit of bytes in use."""

    def __init__(self):
        super().__init__()
        self.calls, self.used, self.most, self.limit, self.refuse = 0, 0, 0, None, ()
        sizes, inner_alloc, inner_free = {}, self._alloc_cb, self._free_cb

        def alloc(ctx, nbytes, stream):
            n, self.calls = self.calls, self.calls + 1
            if n in self.refuse or (self.limit is not None and self.used + nbytes > self.limit):
                return None
            ptr = inner_alloc(ctx, nbytes, stream)
            sizes[ptr] = nbytes
            self.used += nbytes
            self.most = max(self.most, self.used)
            return ptr

        def free(ctx, ptr, stream):
            self.used -= sizes.pop(ptr)
            inner_free(ctx, ptr, stream)

        self._callbacks = binding._ALLOC_FN(alloc), binding._FREE_FN(free)
        self._own = binding.AllocatorStruct(*self._callbacks, None)
        self.lib.comet_destroy(self._h)
        self._h = C.c_void_p()
        assert self.lib.comet_create(C.byref(self._h), C.byref(self._own)) == 0

    def arm(self, refuse=(), limit=None):
        self.refuse, self.limit, self.calls, self.most = refuse, limit, 0, 0


@pytest.fixture(autouse=True)
def _need_gpu(cuda_device):
    yield


@functools.lru_cache
def _entries(dims):
    coords, val = synth.random_coo(dims, N, 3)
    if len(dims) == 2:
        val = val.to(torch.float32)
    return [c.cuda() for c in coords], val.cuda(), [c.numpy() for c in coords], val.double().numpy()


@functools.lru_cache
def _packed(attr, dims):
    _, _, coords, val = _entries(dims)
    return oracle.pack(coords, val, dims, tuple(range(len(dims))), attr)


def _pack(handle, attr, dims, monkeypatch, split="1"):
    monkeypatch.setenv("COMET_PACK_SPLIT", split)
    coords, val, _, _ = _entries(dims)
    T = comet.pack(coords, val, dims, tuple(range(len(dims))), attr, handle)
    want = _packed(attr, dims)
    for level in range(len(dims)):
        assert_equal_arrays(T.pos(level), want.pos[level], f"pos{level}")
        assert_equal_arrays(T.crd(level), want.crd[level], f"crd{level}")
    assert np.array_equal(T.val.double().cpu().numpy(), want.val)
    held = handle.used                                       # the tensor's own arrays
    T.free()
    assert handle.used == 0, "blocks stayed behind"
    return held


@pytest.mark.parametrize("attr,dims", CASES)
def test_a_refused_request_is_no_failure(attr, dims, monkeypatch):
    h = _Handle()
    h.arm()
    _pack(h, attr, dims, monkeypatch)
    for k in range(h.calls):                                 # the records, their tables, each array of the result
        h.arm(refuse=(k,))
        _pack(h, attr, dims, monkeypatch)


@pytest.mark.parametrize("attr,dims", CASES)
def test_what_the_radix_sort_needs_is_enough(attr, dims, monkeypatch):
    h = _Handle()
    h.arm()
    _pack(h, attr, dims, monkeypatch, split="0")
    least = h.most
    h.arm()
    held = _pack(h, attr, dims, monkeypatch)
    most = h.most
    assert least < most
    for limit in [least, most - held, most - held + 4096, most - 256, most - 1, most]:
        h.arm(limit=max(limit, least))
        _pack(h, attr, dims, monkeypatch)


@pytest.mark.parametrize("attr,dims", CASES)
def test_less_than_that_is_reported_and_leaves_nothing_behind(attr, dims, monkeypatch):
    h = _Handle()
    h.arm()
    _pack(h, attr, dims, monkeypatch, split="0")
    least, calls = h.most, h.calls
    for limit in [0, 4096, least // 2, least - 1]:
        h.arm(limit=limit)
        with pytest.raises(comet.CometError) as e:
            _pack(h, attr, dims, monkeypatch)
        assert e.value.status == -6 and h.used == 0
    for k in range(1, calls + 6):                            # from some request on, all of them
        h.arm(refuse=range(k, 1000))
        try:
            _pack(h, attr, dims, monkeypatch)
        except comet.CometError as e:
            assert e.status == -6
        assert h.used == 0
    h.arm()
    _pack(h, attr, dims, monkeypatch)
