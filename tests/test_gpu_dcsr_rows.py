"""SpMM of a DCSR matrix: every row of C is written, the empty ones by CTAs of the gather launch (blocks of 1,024 rows) or by a
clear of C before it; empty rows in front, behind, in between and nowhere, whole pieces and scalar tails, rows apart in C."""
import numpy as np
import pytest
import torch

import oracle
import synth
from oracle import CU

pytestmark = pytest.mark.gpu

comet = pytest.importorskip("paper_2102_05187_b200")
from gpu_util import assert_close, dev, upload_packed  # noqa: E402


def _stored(kind, rows, rng):
    if kind == "all":
        return np.arange(rows)
    if kind == "ends":                                       # the first and the last row only
        return np.array([0, rows - 1])
    if kind == "middle":                                     # long gaps at both ends
        return np.arange(rows // 3, rows // 3 + 40)
    if kind == "one missing":
        return np.setdiff1d(np.arange(rows), [min(1024, rows - 1)])
    return np.sort(rng.choice(rows, rows * 2 // 3, replace=False))


@pytest.mark.parametrize("kind", ["all", "ends", "middle", "one missing", "two thirds"])
@pytest.mark.parametrize("rows", [1023, 1024, 1025, 5000])
@pytest.mark.parametrize("R,pad,dtype", [(1, 0, "f64"), (8, 0, "f32"), (16, 0, "f64"), (25, 3, "f64"), (31, 0, "f32"), (128, 4, "f64"), (200, 0, "f32")])
def test_rows(kind, rows, R, pad, dtype, cuda_device):
    rng = np.random.default_rng(rows + R)
    stored = _stored(kind, rows, rng)
    cols, per = 300, 3
    i = np.repeat(stored, per).astype(np.int32)
    j = np.sort(rng.permuted(np.tile(np.arange(cols), (stored.size, 1)), axis=1)[:, :per], axis=1).reshape(-1).astype(np.int32)
    val = rng.uniform(-1, 1, i.size)
    B = synth.random_dense((cols, R), 5).numpy()
    t = torch.float32 if dtype == "f32" else torch.float64
    if dtype == "f32":
        val, B = val.astype(np.float32).astype(np.float64), B.astype(np.float32).astype(np.float64)
    want, norm = oracle.spmm([i, j], val, (rows, cols), B)
    pk = oracle.pack([i, j], val, (rows, cols), (0, 1), (CU, CU))
    A = upload_packed(pk) if dtype == "f64" else comet.SpTensor.from_arrays(
        pk.dims, pk.mode_order, pk.attr, [dev(p, torch.int32) if p.size else None for p in pk.pos],
        [dev(c, torch.int32) if c.size else None for c in pk.crd], dev(pk.val, t))
    room = torch.full((rows, R + pad), float("nan"), dtype=t, device="cuda")
    C = room[:, :R]
    comet.spmm(A, dev(B, t), C)
    assert_close(C, want, norm, tol=1e-12 if dtype == "f64" else 3 * 2.0 ** -24, what=kind)
    assert torch.isnan(room[:, R:]).all(), "the padding between the rows of C was written"


def test_cleared_c(cuda_device):
    """Narrow rows, twice as many and more as are stored: C is cleared first."""
    rows, cols, R = 700_001, 400, 4
    rng = np.random.default_rng(2)
    stored = np.sort(rng.choice(rows, 90_000, replace=False))
    i, j = stored.astype(np.int32), rng.integers(0, cols, stored.size).astype(np.int32)
    val = rng.uniform(-1, 1, i.size)
    B = synth.random_dense((cols, R), 5).numpy()
    want, norm = oracle.spmm([i, j], val, (rows, cols), B)
    A = upload_packed(oracle.pack([i, j], val, (rows, cols), (0, 1), (CU, CU)))
    C = torch.full((rows, R), float("nan"), dtype=torch.float64, device="cuda")
    comet.spmm(A, dev(B), C)
    assert_close(C, want, norm, what="cleared")


@pytest.mark.parametrize("rows,stored,R", [(700_001, 90_000, 2), (700_001, 100_000, 19), (3_200_003, 2_100_000, 2)])
def test_cleared_where_gaps_are_many_and_rows_narrow(rows, stored, R, cuda_device):
    """The rules by which C is cleared first: narrow rows of which few are stored, few stored rows in a large C, 16-byte rows."""
    cols = 400
    rng = np.random.default_rng(rows)
    i = np.sort(rng.choice(rows, stored, replace=False)).astype(np.int32)
    j = rng.integers(0, cols, stored).astype(np.int32)
    val = rng.uniform(-1, 1, stored)
    B = synth.random_dense((cols, R), 5).numpy()
    want, norm = oracle.spmm([i, j], val, (rows, cols), B)
    A = upload_packed(oracle.pack([i, j], val, (rows, cols), (0, 1), (CU, CU)))
    C = torch.full((rows, R), float("nan"), dtype=torch.float64, device="cuda")
    comet.spmm(A, dev(B), C)
    assert_close(C, want, norm, what="cleared")
