"""The carry fix-up: segments that span from one tile to thousands of them, with run lengths around the number of tiles up to
which threads follow a run (12 to 104, by width; a whole CTA adds longer ones) and around the multiples of 1,024 tiles at which
long runs are cut in large problems. Small tiles are forced, so that small inputs reach every case."""
import numpy as np
import pytest
import torch

import oracle
from oracle import D, CU, CN, S

pytestmark = pytest.mark.gpu

comet = pytest.importorskip("paper_2102_05187_b200")
from gpu_util import assert_close, dev, upload_packed  # noqa: E402

TILE = 8                                                     # items per tile: a row of 8 k entries spans about k tiles


@pytest.fixture(autouse=True)
def _need_gpu(cuda_device, monkeypatch):
    monkeypatch.setenv("COMET_TILE_ITEMS", str(TILE))
    yield


@pytest.mark.parametrize("lengths", [[3, 8 * 10, 0, 8 * 11, 1, 8 * 12 + 5, 8 * 13, 2, 8 * 14, 8 * 20],
                                     [1, 8 * 700, 0, 8 * 64 - 3, 2, 8 * 1030, 8 * 3000]])
@pytest.mark.parametrize("R", [1, 5, 16, 100])
def test_spmm_runs(lengths, R):
    rng = np.random.default_rng(len(lengths) * 100 + R)
    cols = max(lengths) + 3
    r = np.repeat(np.arange(len(lengths)), lengths).astype(np.int32)
    c = np.concatenate([rng.permutation(cols)[:n] for n in lengths]).astype(np.int32)
    v, B = rng.uniform(-1, 1, r.size), rng.uniform(-1, 1, (cols, R))
    want, norm = oracle.spmm([r, c], v, (len(lengths), cols), B)
    A = upload_packed(oracle.pack([r, c], v, (len(lengths), cols), (0, 1), (D, CU)))
    first = comet.spmm(A, dev(B))
    assert_close(first, want, norm)
    assert torch.equal(first, comet.spmm(A, dev(B))), "not reproducible"


def _rows_of_runs(runs):
    """Row lengths so that the run of carries of each (head, tiles) pair starts in tile `head` and takes `tiles` tiles: an
    entry and the end of a row are an item each, a tile holds TILE of them."""
    lengths, at = [], 0                                      # items so far
    for head, tiles in runs:
        assert at <= TILE * head
        while at % TILE:                                     # rows without entries up to a tile boundary
            lengths.append(0)
            at += 1
        while at < TILE * head:                              # rows that end with their tile
            lengths.append(TILE - 1)
            at += TILE
        lengths += [2, TILE * (head + tiles) + 2 - (at + 3)]  # ends 2 items into the tile behind the run
        at = TILE * (head + tiles) + 3
    return lengths + [TILE - 1] * 700


@pytest.mark.parametrize("R,limit", [(1, 104), (4, 100), (5, 36), (16, 36), (24, 28), (100, 12)])
def test_runs_at_the_limits(R, limit):
    """Runs of `limit` tiles and one less and more, heads as many tiles in front of a multiple of 1,024, and runs that go on
    127, 128 and 129 tiles behind one (cut from 129 tiles on), alone and over several multiples."""
    at = {"short": [(5, limit - 1), (5 + limit, limit), (10 + 2 * limit, limit + 1)],
          "cut": [(1024 - limit + d, limit - d + 128 + e) for d in (-1, 0, 1) for e in (-1, 0, 1)]}
    for k, (head, tiles) in enumerate([(1024, 128), (1024, 1152), (1024, 1153), (1000, 2600), (1023, 1)] + at["cut"]):
        runs = at["short"] + [(head, tiles), (head + tiles + 1, 3), (4096 - limit, limit + 2)]
        lengths = _rows_of_runs(runs)
        rng = np.random.default_rng(100 * R + k)
        cols = max(lengths) + 3
        r = np.repeat(np.arange(len(lengths)), lengths).astype(np.int32)
        c = np.concatenate([(rng.integers(cols) + np.arange(n)) % cols for n in lengths if n]).astype(np.int32)
        order = np.lexsort((c, r))
        r, c = r[order], c[order]
        v, B = rng.uniform(-1, 1, r.size), rng.uniform(-1, 1, (cols, R))
        want, norm = oracle.spmm([r, c], v, (len(lengths), cols), B)
        ptr = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)
        A = comet.SpTensor.from_arrays((len(lengths), cols), (0, 1), (D, CU), [None, dev(ptr)], [None, dev(c)], dev(v))
        first = comet.spmm(A, dev(B))
        assert_close(first, want, norm, what=f"run of {tiles} tiles from tile {head}")
        assert torch.equal(first, comet.spmm(A, dev(B))), "not reproducible"


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
@pytest.mark.parametrize("kernel", ["stream", "stream2", "resident"])
def test_vector_runs(kernel, dtype, monkeypatch):
    """The form of the fix-up for vector results: runs below, at and beyond the length where the CTA takes over (104 tiles)."""
    span = 128
    monkeypatch.setenv("COMET_SEG_DOT_KERNEL", kernel)
    monkeypatch.setenv("COMET_STREAM_SPAN", str(span))
    rng = np.random.default_rng(7)
    lengths = [span * t + d for t in (7, 8, 9, 103, 104, 105, 106, 200) for d in (0, 1)] + [1, 0, 3]
    cols = max(lengths) + 3
    r = np.repeat(np.arange(len(lengths)), lengths).astype(np.int32)
    c = np.concatenate([rng.permutation(cols)[:n] for n in lengths]).astype(np.int32)
    v, x = rng.uniform(-1, 1, r.size).astype(dtype), rng.uniform(-1, 1, cols).astype(dtype)
    want, norm = oracle.spmv([r, c], v.astype(np.float64), (len(lengths), cols), x.astype(np.float64))
    ptr = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)
    A = comet.SpTensor.from_arrays((len(lengths), cols), (0, 1), (D, CU), [None, dev(ptr)], [None, dev(c)], dev(v))
    first = comet.spmv(A, dev(x))
    # fp32: a row is rounded when it is stored and once more when its carries are added (2 x 2^-24 of at most norm each)
    assert_close(first.double(), want, norm, 1e-12 if dtype == np.float64 else 1.01 * 2.0 ** -23)
    assert torch.equal(first, comet.spmv(A, dev(x))), "not reproducible"


@pytest.mark.parametrize("attr", [(CU, CU, CU), (CN, S, S)])
@pytest.mark.parametrize("R,n", [(4, 17000), (33, 180000), (128, 60000)])
def test_mttkrp_heavy_slice(attr, R, n):
    """A slice with most of the entries among slices of one entry, of about 20 tiles and of about 1,024; long runs are cut."""
    rng = np.random.default_rng(R)
    dims = (12, 811, 399)
    cell = rng.permutation(dims[1] * dims[2])[:n]
    i = np.full(n, 4)
    i[:8] = [0, 1, 2, 3, 5, 6, 7, 8]
    i[8:8 + 160] = 9
    i[200:200 + 8200] = 10
    coords = [i.astype(np.int32), (cell // dims[2]).astype(np.int32), (cell % dims[2]).astype(np.int32)]
    v = rng.uniform(-1, 1, n)
    F = [None] + [rng.uniform(-1, 1, (d, R)) for d in dims[1:]]
    want, norm = oracle.mttkrp(coords, v, dims, 0, F)
    X = upload_packed(oracle.pack(coords, v, dims, (0, 1, 2), attr))
    assert_close(comet.mttkrp(X, 0, [None, dev(F[1]), dev(F[2])]), want, norm)
