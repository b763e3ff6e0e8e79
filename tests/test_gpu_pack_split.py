"""Packing by sampled splits: sizes around a tile, around one and several buckets and around the sizes from which it is taken,
every order, attribute tuple and value type, key ranges with clusters, arrays off the 16-byte grid, the error cases and an
input that its regions cannot hold."""
import numpy as np
import pytest
import torch

import oracle
import synth
from oracle import D, CU, CN, S

pytestmark = pytest.mark.gpu

comet = pytest.importorskip("paper_2102_05187_b200")
from gpu_util import assert_equal_arrays  # noqa: E402

FORMATS = {2: [(D, CU), (CU, CU), (CN, S)], 3: [(CU, CU, CU), (CN, S, S), (D, CU, CU)], 4: [(CU, CU, CU, CU), (CN, S, S, S)]}


@pytest.fixture(autouse=True)
def _force(cuda_device, monkeypatch):
    monkeypatch.setenv("COMET_PACK_SMALL", "0")
    monkeypatch.setenv("COMET_PACK_SPLIT", "1")
    yield


def _check(coords, val, dims, mode_order, attr, shift=0):
    """shift: the arrays start that many elements behind a 16-byte boundary."""
    def dev(a):
        t = torch.as_tensor(a)
        room = torch.empty(t.numel() + shift, dtype=t.dtype, device="cuda")
        room[shift:] = t
        return room[shift:]

    T = comet.pack([dev(c) for c in coords], dev(val), dims, mode_order, attr)
    want = oracle.pack(coords, val.astype(np.float64), dims, mode_order, attr)
    for level in range(len(dims)):
        assert_equal_arrays(T.pos(level), want.pos[level], f"pos{level}")
        assert_equal_arrays(T.crd(level), want.crd[level], f"crd{level}")
    assert np.array_equal(T.val.cpu().numpy().astype(np.float64), want.val)


@pytest.mark.parametrize("n", [1, 2, 31, 1400, 1401, 4095, 4096, 4097, 44_801, 200_003])
@pytest.mark.parametrize("order", [2, 3, 4])
def test_sizes(n, order):
    dims = {2: (3001, 4099), 3: (257, 300, 191), 4: (67, 61, 59, 64)}[order]
    coords, val = synth.random_coo(dims, n, n + order)
    coords, val = [c.numpy() for c in coords], val.numpy()
    if n % 2:
        val = val.astype(np.float32)
    for attr in FORMATS[order]:
        _check(coords, val, dims, tuple(reversed(range(order))), attr, shift=n % 3)


@pytest.mark.parametrize("n", [606_208, 606_209, 2_000_003])
def test_sizes_where_it_is_taken(n, monkeypatch):
    monkeypatch.delenv("COMET_PACK_SMALL")
    monkeypatch.delenv("COMET_PACK_SPLIT")
    coords, val = synth.random_coo((9001, 7001), n, n)
    coords, val = [c.numpy() for c in coords], val.numpy()
    for attr in FORMATS[2]:
        _check(coords, val, (9001, 7001), (0, 1), attr)


@pytest.mark.parametrize("sort", [False, True])
@pytest.mark.parametrize("kind", ["one row", "rows far apart", "one full bucket of columns", "powers of two", "high bits"])
def test_key_ranges(kind, sort):
    rng = np.random.default_rng(7)
    rows, cols = (1 << 31) - 2, 1 << 30
    if kind == "one row":
        cells = [(12345, np.unique(rng.integers(0, cols, 60_000)))]
    elif kind == "rows far apart":                 # each a run of neighbouring columns
        cells = [(r, 1000 * i + np.arange(500 + i)) for i, r in enumerate(np.unique(rng.integers(0, rows, 90)))]
    elif kind == "one full bucket of columns":
        cells = [(r, np.arange(4096)) for r in range(9)] + [(rows - 1, np.arange(7))]
    elif kind == "powers of two":                  # gaps that grow: nothing near an even spread between two samples
        cells = [(1 << a, np.unique(np.concatenate([1 << np.arange(30), 3 * (1 << np.arange(28))]))) for a in range(30)] * 1
    else:
        cells = [(rows - 1 - i, cols - 1 - np.arange(1500) * (i + 1)) for i in range(25)]
    i = np.concatenate([np.full(len(c), r) for r, c in cells]).astype(np.int32)
    j = np.concatenate([c for _, c in cells]).astype(np.int32)
    order = np.lexsort((j, i)) if sort else rng.permutation(i.size)
    val = rng.uniform(-1, 1, i.size)
    for attr in [(CU, CU), (CN, S)]:
        _check([i[order], j[order]], val, (rows, cols), (0, 1), attr)


def test_empty_rows_of_csr():
    """Rows without entries in front, behind, inside and between the buckets."""
    rng = np.random.default_rng(3)
    rows = np.sort(rng.choice(np.arange(50, 99_000), 400, replace=False))
    i = np.repeat(rows, 20).astype(np.int32)
    j = np.tile(np.arange(20) * 7, rows.size).astype(np.int32)
    o = rng.permutation(i.size)
    _check([i[o], j[o]], rng.uniform(-1, 1, i.size), (100_000, 200), (0, 1), (D, CU))


@pytest.mark.parametrize("n", [5000, 300_000])
@pytest.mark.parametrize("attr", [(CU, CU, CU), (CN, S, S)])
def test_errors_are_reported_and_leave_the_handle_usable(n, attr):
    dims = (300, 200, 250)
    coords, val = synth.random_coo(dims, n, 9)
    for make, status in [(lambda c: c[0].__setitem__(n - 1, 300), -3), (lambda c: c[1].__setitem__(0, -1), -3),
                         (lambda c: [x.__setitem__(5, int(x[n - 2])) for x in c], -4),
                         (lambda c: [x.fill_(3) for x in c], -4)]:
        bad = [c.clone() for c in coords]
        make(bad)
        with pytest.raises(comet.CometError) as e:
            comet.pack([c.cuda() for c in bad], val.cuda(), dims, (0, 1, 2), attr)
        assert e.value.status == status
    _check([c.numpy() for c in coords], val.numpy(), dims, (0, 1, 2), attr)


@pytest.mark.parametrize("rows", [1000, 1024])
def test_errors_of_a_csr_matrix(rows):
    """A row beyond the matrix whose number still fits the bits of a row (or does not), and equal cells."""
    coords, val = synth.random_coo((rows, 5000), 40_000, 4)
    for at, row in [(0, rows), (39_999, 1023 if rows < 1024 else 2047), (7, -1)]:
        bad = [c.clone() for c in coords]
        bad[0][at] = row
        with pytest.raises(comet.CometError) as e:
            comet.pack([c.cuda() for c in bad], val.cuda(), (rows, 5000), (0, 1), (D, CU))
        assert e.value.status == -3
    bad = [c.clone() for c in coords]
    for c in bad:
        c[100] = c[39_000]
    with pytest.raises(comet.CometError) as e:
        comet.pack([c.cuda() for c in bad], val.cuda(), (rows, 5000), (0, 1), (D, CU))
    assert e.value.status == -4
    _check([c.numpy() for c in coords], val.numpy(), (rows, 5000), (0, 1), (D, CU))


@pytest.mark.parametrize("attr", FORMATS[2])
def test_input_whose_samples_mislead(attr):
    """The entries that are sampled have the highest keys: all others fall into the first bucket, whose region is too small
    for them, and the radix sort packs the tensor."""
    n = 40_000
    x = np.arange(32 * 32, dtype=np.uint32)        # the sample positions (pack_split.cu: sample_hash)
    x ^= x >> np.uint32(16)
    x *= np.uint32(0x7FEB352D)
    x ^= x >> np.uint32(15)
    x *= np.uint32(0x846CA68B)
    x ^= x >> np.uint32(16)
    at = np.unique((x.astype(np.uint64) * np.uint64(n)) >> np.uint64(32)).astype(np.int64)
    rng = np.random.default_rng(1)
    cells = np.sort(rng.choice(900 * 1000, n, replace=False))
    rest = np.setdiff1d(np.arange(n), at)
    key = np.empty(n, dtype=np.int64)
    key[at] = rng.permutation(cells[n - at.size:])
    key[rest] = rng.permutation(cells[:n - at.size])
    handle = comet.default_handle()
    before = handle.kernel_launches()
    _check([(key // 1000).astype(np.int32), (key % 1000).astype(np.int32)], rng.uniform(-1, 1, n), (900, 1000), (0, 1), attr)
    assert handle.kernel_launches() - before > 12, "the radix sort was expected to follow"


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_many_coarse_buckets(dtype, monkeypatch):
    """512 coarse buckets: the first split writes its runs record by record, not as bulk copies. Cells: multiples of an odd number
    modulo 2^36, which are distinct and in no order."""
    monkeypatch.delenv("COMET_PACK_SMALL")
    monkeypatch.delenv("COMET_PACK_SPLIT")
    n, rows = 46_300_007, 1 << 18
    key = torch.arange(n, dtype=torch.int64, device="cuda") * (0x9E3779B97F4A7C15 - (1 << 64)) & ((1 << 36) - 1)
    val = (torch.arange(n, dtype=torch.int64, device="cuda") % 16_777_213).to(dtype)
    A = comet.pack([(key >> 18).to(torch.int32), (key & (rows - 1)).to(torch.int32)], val, (rows, rows), (0, 1), (D, CU))
    key, order = torch.sort(key)
    assert torch.equal(A.crd(1), (key & (rows - 1)).to(torch.int32))
    assert torch.equal(A.pos(1)[1:], torch.cumsum(torch.bincount(key >> 18, minlength=rows), 0).to(torch.int32)) and int(A.pos(1)[0]) == 0
    assert torch.equal(A.val, val[order])
