"""Tiles by whole waves of resident workers: sizes at which the number of waves, or the rule, changes, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import synth
from oracle import D, CU, CN, S

pytestmark = pytest.mark.gpu

comet = pytest.importorskip("paper_2102_05187_b200")
from gpu_util import assert_close, dev, upload_packed  # noqa: E402

SLOTS = 148 * 4                                              # resident CTAs of the kernels with four to an SM


@pytest.fixture(autouse=True)
def _need_gpu(cuda_device):
    yield


@pytest.mark.parametrize("R,workers", [(16, 32), (128, 8)])    # 8 lanes a worker; 32 lanes with two pieces, two CTAs to an SM
@pytest.mark.parametrize("items", [7, 8, 24, 48, 49])
@pytest.mark.parametrize("off", [-1, 0, 1])
def test_spmm(R, workers, items, off):
    total = SLOTS * workers * items // (2 if R == 128 else 1) + off
    rows = 2003
    n = total - rows                                         # the merge list holds a marker per row
    rng = np.random.default_rng(items)
    cols = 1 + 2 * n // rows
    cells = np.sort(rng.choice(rows * cols, n, replace=False))
    c = [(cells // cols).astype(np.int32), (cells % cols).astype(np.int32)]
    val = rng.uniform(-1, 1, n)
    B = synth.random_dense((cols, R), 5).numpy()
    want, norm = oracle.spmm(c, val, (rows, cols), B)
    A = upload_packed(oracle.pack(c, val, (rows, cols), (0, 1), (D, CU)))
    C = torch.full((rows, R), float("nan"), dtype=torch.float64, device="cuda")
    comet.spmm(A, dev(B), C)
    assert_close(C, want, norm, what="spmm")


@pytest.mark.parametrize("items", [31, 32, 128, 129])         # 128 = four chunks: from there on tiles are whole chunks
@pytest.mark.parametrize("off", [-1, 1])
def test_mttkrp_coo(items, off):
    dims, R = (301, 97, 211), 32
    coords, val = synth.random_coo(dims, SLOTS * 16 * items + off, 3)
    c, v = [x.numpy() for x in coords], val.numpy()
    F = [None] + [synth.random_dense((d, R), 4 + i).numpy() for i, d in enumerate(dims[1:])]
    want, norm = oracle.mttkrp(c, v, dims, 0, F)
    A = upload_packed(oracle.pack(c, v, dims, (0, 1, 2), (CN, S, S)))
    assert_close(comet.mttkrp(A, 0, [None] + [dev(f) for f in F[1:]]), want, norm, what="mttkrp")
