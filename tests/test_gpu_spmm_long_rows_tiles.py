"""The general rows beside the long rows of comet_spmm: tiles that end anywhere in a chunk of staged entries, both types."""
import numpy as np
import pytest
import torch

import oracle
import synth
from oracle import D, CU

pytestmark = pytest.mark.gpu

comet = pytest.importorskip("paper_2102_05187_b200")
from gpu_util import assert_close, dev, upload_packed  # noqa: E402


@pytest.mark.parametrize("tile", [8, 9, 15, 16, 17, 23, 24, 25, 33, 40])
@pytest.mark.parametrize("R,dtype", [(32, "f64"), (64, "f64"), (128, "f64"), (64, "f32"), (128, "f32")])
def test_tiles(tile, R, dtype, cuda_device, monkeypatch):
    for name, value in [("LONG_MIN_NNZ", 1), ("LONG_MIN_B_MB", 0), ("LONG_ROW", 48), ("LONG_TILE", 32), ("PIECE", 8), ("BLOCKS", 4),
                        ("LONG_CTAS", 2)]:
        monkeypatch.setenv("COMET_SPMM_" + name, str(value))
    monkeypatch.setenv("COMET_TILE_ITEMS", str(tile))
    rng = np.random.default_rng(tile)
    lengths = rng.integers(0, 30, 257)
    lengths[[0, 100, 256]] = [200, 61, 90]
    cols = 300
    i = np.repeat(np.arange(lengths.size), lengths).astype(np.int32)
    j = np.concatenate([np.sort(rng.choice(cols, n, replace=False)) for n in lengths]).astype(np.int32)
    val = rng.uniform(-1, 1, i.size)
    B = synth.random_dense((cols, R), 5).numpy()
    if dtype == "f32":
        val, B = val.astype(np.float32).astype(np.float64), B.astype(np.float32).astype(np.float64)
    want, norm = oracle.spmm([i, j], val, (lengths.size, cols), B)
    pk = oracle.pack([i, j], val, (lengths.size, cols), (0, 1), (D, CU))
    t = torch.float32 if dtype == "f32" else torch.float64
    A = upload_packed(pk) if dtype == "f64" else comet.SpTensor.from_arrays(
        pk.dims, pk.mode_order, pk.attr, [dev(p, torch.int32) if p.size else None for p in pk.pos],
        [dev(c, torch.int32) if c.size else None for c in pk.crd], dev(pk.val, t))
    C = torch.full((lengths.size, R), float("nan"), dtype=t, device="cuda")
    before = A.handle.kernel_launches()
    comet.spmm(A, dev(B, t), C)
    assert A.handle.kernel_launches() - before == 5           # the long-row path ran
    # fp32: sums in double, rounded when stored and once more where a carry or a long row's parts are added
    assert_close(C, want, norm, tol=1e-12 if dtype == "f64" else 3 * 2.0 ** -24, what="spmm")
