"""Dense operands whose rows are no whole number of 16-byte pieces, or a number of pieces that is no power of two: every
width around the shapes' limits, odd leading dimensions, operands that start off a 16-byte boundary, outputs inside wider
buffers, operands with far more rows than the matrix has entries (no padded copy), and tiny inputs of one lane per row."""
import numpy as np
import pytest
import torch

import oracle
from oracle import D, CU, CN, S

pytestmark = pytest.mark.gpu

comet = pytest.importorskip("paper_2102_05187_b200")
from gpu_util import assert_close, dev, upload_packed  # noqa: E402

WIDTHS = [1, 2, 3, 4, 5, 7, 9, 12, 16, 17, 18, 31, 33, 34, 63, 65, 66, 100, 127, 129, 131]


@pytest.fixture(autouse=True)
def _need_gpu(cuda_device):
    yield


def _operand(a, lead, offset, dtype):
    """The array inside a wider buffer: leading dimension grown by `lead`, start moved by `offset` elements."""
    rows, R = a.shape
    buf = torch.full((rows * (R + lead) + offset,), float("nan"), dtype=dtype, device="cuda")
    view = buf[offset:].view(rows, R + lead)[:, :R]
    view.copy_(dev(a))
    return view


def _as(T, dtype):
    """The caller-built tensor with values of another type."""
    return comet.SpTensor.from_arrays(T.dims, T.mode_order, T.attr, [T.pos(l) if T.c.pos_len[l] else None for l in range(T.order)],
                                      [T.crd(l) if T.c.crd_len[l] else None for l in range(T.order)], T.val.to(dtype))


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("R", WIDTHS)
@pytest.mark.parametrize("lead,offset", [(0, 0), (1, 0), (4, 1)])
def test_spmm_and_root_mttkrp(R, lead, offset, dtype):
    rng = np.random.default_rng(R * 10 + lead)
    f = lambda a: a.astype(np.float32).astype(np.float64) if dtype == torch.float32 else a  # noqa: E731
    tol = 1e-12 if dtype == torch.float64 else 3 * 2.0 ** -24         # one rounding on the store, one more with a carry
    rows, cols, n = 90, 70, 2500
    cell = rng.permutation(rows * cols)[:n]
    cell = cell[(cell // cols) % 9 != 4]                               # some rows without entries
    r, c = (cell // cols).astype(np.int32), (cell % cols).astype(np.int32)
    v, B = f(rng.uniform(-1, 1, r.size)), f(rng.uniform(-1, 1, (cols, R)))
    want, norm = oracle.spmm([r, c], v, (rows, cols), B)
    out = torch.full((rows, R + 3), 7.0, dtype=dtype, device="cuda")
    for attr in [(D, CU), (CU, CU)]:
        A = _as(upload_packed(oracle.pack([r, c], v, (rows, cols), (0, 1), attr)), dtype)
        assert_close(comet.spmm(A, _operand(B, lead, offset, dtype)), want, norm, tol)
        comet.spmm(A, _operand(B, lead, offset, dtype), out[:, 1:R + 1])
        assert_close(out[:, 1:R + 1], want, norm, tol)
        assert (out[:, 0] == 7).all() and (out[:, R + 1:] == 7).all(), "columns beside the output were written"
    dims = (rows, 9, 8)
    coords = [r, (c % 9).astype(np.int32), (c // 9).astype(np.int32)]
    F = [None] + [f(rng.uniform(-1, 1, (d, R))) for d in dims[1:]]
    want, norm = oracle.mttkrp(coords, v, dims, 0, F)
    for attr in [(CU, CU, CU), (CN, S, S)]:
        X = _as(upload_packed(oracle.pack(coords, v, dims, (0, 1, 2), attr)), dtype)
        got = comet.mttkrp(X, 0, [None] + [_operand(x, lead, offset, dtype) for x in F[1:]])
        assert_close(got, want, norm, tol if dtype == torch.float64 else 2 * tol)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("R", [1, 3, 5, 9, 25, 33, 65, 67, 131])
def test_padded_copies(R, dtype):
    """Enough entries for the operands to be padded: rows that are no whole pieces, an odd leading dimension."""
    rng = np.random.default_rng(R)
    f = lambda a: a.astype(np.float32).astype(np.float64) if dtype == torch.float32 else a  # noqa: E731
    tol = 1e-12 if dtype == torch.float64 else 3 * 2.0 ** -24
    rows, cols, n = 700, 300, 110_000
    cell = rng.permutation(rows * cols)[:n]
    r, c = (cell // cols).astype(np.int32), (cell % cols).astype(np.int32)
    v, B = f(rng.uniform(-1, 1, n)), f(rng.uniform(-1, 1, (cols, R)))
    want, norm = oracle.spmm([r, c], v, (rows, cols), B)
    for attr in [(D, CU), (CU, CU)]:
        A = _as(upload_packed(oracle.pack([r, c], v, (rows, cols), (0, 1), attr)), dtype)
        assert_close(comet.spmm(A, _operand(B, 1, 1, dtype)), want, norm, tol)
    dims = (rows, 20, 15)
    coords = [r, (c % 20).astype(np.int32), (c // 20).astype(np.int32)]
    F = [None] + [f(rng.uniform(-1, 1, (d, R))) for d in dims[1:]]
    want, norm = oracle.mttkrp(coords, v, dims, 0, F)
    for attr in [(CU, CU, CU), (CN, S, S)]:
        X = _as(upload_packed(oracle.pack(coords, v, dims, (0, 1, 2), attr)), dtype)
        got = comet.mttkrp(X, 0, [None] + [_operand(x, 1, 1, dtype) for x in F[1:]])
        assert_close(got, want, norm, tol if dtype == torch.float64 else 2 * tol)


@pytest.mark.parametrize("R", [1, 2, 5, 50, 130])
def test_few_entries_many_operand_rows(R):
    rng = np.random.default_rng(R)
    r, c = np.arange(40, dtype=np.int32), rng.permutation(5000)[:40].astype(np.int32)
    v, B = rng.uniform(-1, 1, 40), rng.uniform(-1, 1, (5000, R))
    want, norm = oracle.spmm([r, c], v, (40, 5000), B)
    A = upload_packed(oracle.pack([r, c], v, (40, 5000), (0, 1), (D, CU)))
    assert_close(comet.spmm(A, _operand(B, 1, 0, torch.float64)), want, norm)
