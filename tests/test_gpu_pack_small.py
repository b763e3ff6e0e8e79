"""Packing of small inputs in one launch: sizes around a CTA's tile, around the limits between tile sizes and around the
size from which the general path takes over, every order and attribute tuple, one to eight digits, and the error cases."""
import numpy as np
import pytest
import torch

import oracle
import synth
from oracle import D, CU, CN, S

pytestmark = pytest.mark.gpu

comet = pytest.importorskip("paper_2102_05187_b200")
from gpu_util import assert_equal_arrays  # noqa: E402

GRID = 148 * 512                                             # entries per item of a thread over the whole chip
FORMATS = {2: [(D, CU), (CU, CU), (CN, S)], 3: [(CU, CU, CU), (CN, S, S), (D, CU, CU)], 4: [(CU, CU, CU, CU), (CN, S, S, S)]}


@pytest.fixture(autouse=True)
def _need_gpu(cuda_device):
    yield


def _check(coords, val, dims, mode_order, attr):
    T = comet.pack([torch.as_tensor(c).cuda() for c in coords], torch.as_tensor(val).cuda(), dims, mode_order, attr)
    want = oracle.pack(coords, val.astype(np.float64), dims, mode_order, attr)
    for level in range(len(dims)):
        assert_equal_arrays(T.pos(level), want.pos[level], f"pos{level}")
        assert_equal_arrays(T.crd(level), want.crd[level], f"crd{level}")
    assert np.array_equal(T.val.cpu().numpy().astype(np.float64), want.val)


@pytest.mark.parametrize("n", [1, 2, 33, 1023, 1024, 1025, 5000, 2 * GRID, 2 * GRID + 1, 4 * GRID, 8 * GRID + 1, 16 * GRID, 16 * GRID + 1])
@pytest.mark.parametrize("order", [2, 3, 4])
def test_sizes(n, order):
    dims = {2: (3001, 4099), 3: (257, 300, 191), 4: (67, 61, 59, 64)}[order]
    coords, val = synth.random_coo(dims, n, n + order)
    coords, val = [c.numpy() for c in coords], val.numpy()
    if order % 2:
        val = val.astype(np.float32)
    modes = tuple(reversed(range(order)))
    for attr in FORMATS[order] if n < GRID else FORMATS[order][:1]:
        _check(coords, val, dims, modes, attr)


@pytest.mark.parametrize("dims", [(1, 200), (1, 1 << 20), (1 << 12, 1 << 12), ((1 << 31) - 2, 1 << 30)])
def test_digits(dims):
    """One to eight digits; a coordinate pair of the highest numbers."""
    rng = np.random.default_rng(5)
    cells = np.unique(rng.integers(0, dims[0], 700) * dims[1] + rng.integers(0, dims[1], 700))
    cells = np.append(np.setdiff1d(cells, [dims[0] * dims[1] - 1]), dims[0] * dims[1] - 1)
    rng.shuffle(cells)
    coords = [(cells // dims[1]).astype(np.int32), (cells % dims[1]).astype(np.int32)]
    _check(coords, rng.uniform(-1, 1, cells.size), dims, (0, 1), (CU, CU))


@pytest.mark.parametrize("n", [3000, 2 * GRID + 7])
@pytest.mark.parametrize("attr", [(CU, CU, CU), (CN, S, S)])
def test_errors_are_reported_and_leave_the_handle_usable(n, attr):
    dims = (300, 200, 250)
    coords, val = synth.random_coo(dims, n, 9)
    for make, status in [(lambda c: c[0].__setitem__(n - 1, 300), -3), (lambda c: c[1].__setitem__(0, -1), -3),
                         (lambda c: [x.__setitem__(5, int(x[n - 2])) for x in c], -4)]:
        bad = [c.clone() for c in coords]
        make(bad)
        with pytest.raises(comet.CometError) as e:
            comet.pack([c.cuda() for c in bad], val.cuda(), dims, (0, 1, 2), attr)
        assert e.value.status == status
    _check([c.numpy() for c in coords], val.numpy(), dims, (0, 1, 2), attr)


@pytest.mark.parametrize("n", [1, 2047, 2049, 100_003])
@pytest.mark.parametrize("order", [2, 3, 4])
def test_general_path_where_the_launch_is_refused(n, order, monkeypatch):
    """A context with fewer SMs than the device refuses the cooperative launch: the general path packs the same."""
    dims = {2: (3001, 4099), 3: (257, 300, 191), 4: (67, 61, 59, 64)}[order]
    coords, val = synth.random_coo(dims, n, n + order)
    coords, val = [c.numpy() for c in coords], val.numpy()
    handle = comet.default_handle()

    def launches():
        before = handle.kernel_launches()
        for attr in FORMATS[order]:
            _check(coords, val, dims, tuple(range(order)), attr)
        return handle.kernel_launches() - before

    one = launches()
    monkeypatch.setenv("COMET_PACK_SMALL", "0")
    assert launches() > one, "the one launch was taken all the same"
