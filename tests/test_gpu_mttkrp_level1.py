"""MTTKRP, output mode stored at level 1 of a CSF tensor: widths around the half-warp, warp and 64-column limits, rows that
are not aligned, tiles of 32 entries (one chunk, one mask word) up to 1,024, fibers of an entry or two (a worker per eight
fibers) and long ones, and tensors that hold fibers and slices without entries."""
import numpy as np
import pytest
import torch

import oracle
from oracle import CU

pytestmark = pytest.mark.gpu

comet = pytest.importorskip("paper_2102_05187_b200")
from gpu_util import assert_close, dev, upload_packed  # noqa: E402


@pytest.fixture(autouse=True)
def _need_gpu(cuda_device):
    yield


def _tensor(n, seed):
    rng = np.random.default_rng(seed)
    dims = (37, 41, 53)
    cell = rng.permutation(dims[0] * dims[1] * dims[2])[:n]
    coords = [(cell // (41 * 53)).astype(np.int32), (cell // 53 % 41).astype(np.int32), (cell % 53).astype(np.int32)]
    return dims, coords, rng.uniform(-1, 1, n), rng


@pytest.mark.parametrize("n", [1, 31, 33, 1024, 30000])
@pytest.mark.parametrize("R", [1, 2, 15, 17, 32, 33, 65, 128])
@pytest.mark.parametrize("tile", [None, "8"])
def test_widths(n, R, tile, monkeypatch):
    if tile:
        monkeypatch.setenv("COMET_TILE_ITEMS", tile)
    dims, coords, v, rng = _tensor(n, R)
    F = [rng.uniform(-1, 1, (d, R)) for d in dims]
    want, norm = oracle.mttkrp(coords, v, dims, 1, F)
    X = upload_packed(oracle.pack(coords, v, dims, (0, 1, 2), (CU, CU, CU)))
    wide = [torch.zeros(d, R + 1, dtype=torch.float64, device="cuda") for d in dims]      # an odd leading dimension
    for w, f in zip(wide, F):
        w[:, :R] = dev(f)
    assert_close(comet.mttkrp(X, 1, [w[:, :R] for w in wide]), want, norm)


@pytest.mark.parametrize("R", [5, 32])
def test_fibers_and_slices_without_entries(R):
    # slices 0 (fibers of 2 and 0 entries), 1 (no fiber), 2 (one empty fiber), 3 (0, 3 and 0 entries), 4 (1 entry)
    pos1, crd0 = [0, 2, 2, 3, 6, 7], [0, 2, 3, 5, 6]
    pos2, crd1 = [0, 2, 2, 2, 2, 5, 5, 6], [1, 4, 2, 0, 3, 4, 1]
    crd2, v = [0, 3, 1, 2, 4, 0], np.arange(1.0, 7.0)
    rng = np.random.default_rng(R)
    dims = (7, 5, 5)
    F = [rng.uniform(-1, 1, (d, R)) for d in dims]
    i32 = lambda x: dev(np.array(x), torch.int32)  # noqa: E731
    X = comet.SpTensor.from_arrays(dims, (0, 1, 2), (CU, CU, CU), [i32([0, 5]), i32(pos1), i32(pos2)],
                                   [i32(crd0), i32(crd1), i32(crd2)], dev(v))
    comet.validate(X)
    entries = [(0, 1, 0), (0, 1, 3), (5, 3, 1), (5, 3, 2), (5, 3, 4), (6, 1, 0)]
    want = np.zeros((5, R))
    for (i, j, k), x in zip(entries, v):
        want[j] += x * F[0][i] * F[2][k]
    got = comet.mttkrp(X, 1, [dev(f) for f in F]).cpu().numpy()
    assert np.all(np.abs(got - want) <= 1e-12 * np.abs(v).sum())


def _check(i, j, k, v, dims, X, R, dtype, seed):
    """Against plain numpy sums (a caller-built tensor may hold fibers and slices without entries)."""
    rng = np.random.default_rng(seed)
    F = [rng.uniform(-1, 1, (d, R)).astype(dtype) for d in dims]
    terms = v.astype(np.float64)[:, None] * F[0].astype(np.float64)[i] * F[2].astype(np.float64)[k]
    want, norm = np.zeros((dims[1], R)), np.zeros((dims[1], R))
    np.add.at(want, j, terms)
    np.add.at(norm, j, np.abs(terms))
    wide = [dev(np.pad(f, ((0, 0), (0, 1)))) for f in F]     # an odd leading dimension: not the walker of the aligned widths
    got = comet.mttkrp(X, 1, [w[:, :R] for w in wide]).double().cpu().numpy()
    tol = 1e-12 if dtype == np.float64 else 2.0 ** -23       # fp32: sums in double, one rounding
    assert np.all(np.abs(got - want) <= tol * norm)


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
@pytest.mark.parametrize("tile", ["32", "64", "96", "1024"])
@pytest.mark.parametrize("R", [1, 5, 16, 32, 33, 70])
def test_tiles_fibers_and_slices_without_entries(tile, R, dtype, monkeypatch):
    """Several tiles of several chunks: fibers of 0 to 90 entries, slices of no, one and many fibers, runs of empty ones at the
    start, at the end and on tile boundaries."""
    monkeypatch.setenv("COMET_TILE_ITEMS", tile)
    rng = np.random.default_rng(int(tile) + R)
    dims = (400, 90, 100)
    per_slice = rng.choice([0, 1, 2, 7, 40], 200)
    per_slice[[0, 1, -1]] = 0
    fibers = int(per_slice.sum())
    lengths = rng.choice([0, 0, 1, 3, 32, 90], fibers)
    lengths[[0, 1, 2, -1, -2]] = 0
    for b in range(int(tile), int(lengths.sum()) // 2, 4 * int(tile)):   # a fiber that ends on a tile boundary, empty ones behind
        f = int(np.searchsorted(np.cumsum(lengths), b))
        lengths[f] -= int(np.cumsum(lengths)[f]) - b
        lengths[f + 1:f + 3] = 0
    crd0 = np.sort(rng.permutation(dims[0])[:200])
    crd1 = np.concatenate([np.sort(rng.permutation(dims[1])[:n]) for n in per_slice])
    crd2 = np.concatenate([np.sort(rng.permutation(dims[2])[:n]) for n in lengths])
    v = rng.uniform(-1, 1, crd2.size).astype(dtype)
    i32 = lambda x: dev(np.asarray(x).astype(np.int32))  # noqa: E731
    ptr = lambda n: np.concatenate([[0], np.cumsum(n)])  # noqa: E731
    X = comet.SpTensor.from_arrays(dims, (0, 1, 2), (CU, CU, CU), [i32([0, 200]), i32(ptr(per_slice)), i32(ptr(lengths))],
                                   [i32(crd0), i32(crd1), i32(crd2)], dev(v))
    comet.validate(X)
    fiber = np.repeat(np.arange(fibers), lengths)
    _check(np.repeat(crd0, per_slice)[fiber], crd1[fiber], crd2, v, dims, X, R, dtype, R)


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
@pytest.mark.parametrize("R", [1, 3, 4, 5, 17, 129])
@pytest.mark.parametrize("n", [3, 9000, 149_999, 150_001])
def test_short_fibers(n, R, dtype):
    """Fibers of an entry or two, on both sides of the size up to which they have a worker per eight fibers."""
    rng = np.random.default_rng(n + R)
    dims = (2000, 1500, 300)
    cell = np.unique(rng.integers(0, dims[0] * dims[1] * dims[2], n + 50))
    cell = np.sort(rng.permutation(cell)[:n])
    i, j, k = (x.astype(np.int32) for x in np.unravel_index(cell, dims))
    v = rng.uniform(-1, 1, n).astype(dtype)
    X = comet.pack([dev(i), dev(j), dev(k)], dev(v), dims, (0, 1, 2), (CU, CU, CU))
    _check(i, j, k, v, dims, X, R, dtype, R)


def test_as_many_entries_as_there_may_be():
    """2^31 - 2 entries: the look-ahead behind the last tile passes 2^31."""
    n = 2 ** 31 - 2
    free, _ = torch.cuda.mem_get_info()
    if free < 40 << 30:
        pytest.skip("needs 40 GB of device memory")
    ends = [0, 2 ** 29, 2 ** 30 + 5, 3 * 2 ** 29, n]                       # four fibers in two slices
    longest = max(b - a for a, b in zip(ends, ends[1:]))
    crd2 = torch.empty(n, dtype=torch.int32, device="cuda")
    for a, b in zip(ends, ends[1:]):
        torch.arange(b - a, dtype=torch.int32, device="cuda", out=crd2[a:b])
    i32 = lambda x: dev(np.array(x), torch.int32)  # noqa: E731
    X = comet.SpTensor.from_arrays((2, 3, longest), (0, 1, 2), (CU, CU, CU), [i32([0, 2]), i32([0, 2, 4]), i32(ends)],
                                   [i32([0, 1]), i32([0, 2, 1, 2]), crd2], torch.ones(n, device="cuda"))
    F = [torch.tensor([[1.0], [-2.0]], device="cuda"), None, torch.ones(longest, 1, device="cuda")]
    got = comet.mttkrp(X, 1, F).double().cpu()
    want = torch.tensor([[ends[1]], [-2.0 * (ends[3] - ends[2])], [ends[2] - ends[1] - 2.0 * (ends[4] - ends[3])]], dtype=torch.float64)
    assert torch.equal(got, want.float().double())           # sums of ones are exact in double
