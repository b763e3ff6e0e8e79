"""MTTKRP, output mode stored at level 1 of a CSF tensor: widths around the half-warp, warp and 64-column limits, rows that
are not aligned, tiles of 32 entries and longer ones, and tensors that hold fibers and slices without entries."""
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
