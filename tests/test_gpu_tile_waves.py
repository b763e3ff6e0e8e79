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


def _tensor(total, dims, fibers, seed):
    """3-order coordinates sorted by storage order: `fibers` fibers that hold total - fibers entries, so that the merge list of a
    kernel that has a marker per fiber holds `total` items."""
    n = total - fibers
    rng = np.random.default_rng(seed)
    f = np.sort(rng.choice(dims[0] * dims[1], fibers, replace=False))
    cells = np.arange(fibers) * dims[2]                      # an entry in every fiber, the others anywhere
    more = np.setdiff1d(rng.choice(fibers * dims[2], n + fibers, replace=False), cells)
    cells = np.sort(np.concatenate([cells, rng.permutation(more)[:n - fibers]]))
    assert cells.size == n
    row = f[cells // dims[2]]
    return [(row // dims[1]).astype(np.int32), (row % dims[1]).astype(np.int32), (cells % dims[2]).astype(np.int32)], rng.uniform(-1, 1, n)


# Lanes a worker: one (three CTAs to an SM; tiles of 16 beyond 20), two, eight (two CTAs to an SM below 24 items in a full wave, three
# below 64; three waves beyond 192 where fibers are long on average).
@pytest.mark.parametrize("R,workers,ctas,items", [(2, 256, 3, 11), (2, 256, 3, 12), (2, 256, 3, 20), (2, 256, 3, 21), (4, 128, 4, 23), (4, 128, 4, 24),
                                                  (16, 32, 4, 7), (16, 32, 4, 23), (16, 32, 4, 24), (16, 32, 4, 63), (16, 32, 4, 64), (16, 32, 4, 192)])
@pytest.mark.parametrize("off", [0, 1])
def test_ttm(R, workers, ctas, items, off):
    total, dims = 148 * ctas * workers * items + off, (97, 89, 4003)
    c, v = _tensor(total, dims, total // 40 if total < 320_000 else 8001, items)
    U = synth.random_dense((dims[2], R), 5).numpy()
    _, want, norm = oracle.ttm(c, v, dims, 2, U)
    A = upload_packed(oracle.pack(c, v, dims, (0, 1, 2), (CU, CU, CU)))
    assert_close(comet.ttm(A, 2, dev(U)).val.reshape(want.shape), want, norm, what="ttm")


@pytest.mark.parametrize("R,dtype,workers", [(25, "f64", 16), (25, "f32", 32), (37, "f64", 8)])      # copies of B, the last lane masked
@pytest.mark.parametrize("items", [48, 49])
@pytest.mark.parametrize("off", [-1, 1])
def test_spmm_ragged(R, dtype, workers, items, off):
    items = items * 32 // workers                             # enough entries for the ragged shapes: 250,000 and more
    rows, t = 2003, torch.float32 if dtype == "f32" else torch.float64
    n = SLOTS * workers * items + off - rows
    rng = np.random.default_rng(items)
    cols = 1 + 2 * n // rows
    cells = np.sort(rng.choice(rows * cols, n, replace=False))
    c = [(cells // cols).astype(np.int32), (cells % cols).astype(np.int32)]
    val, B = rng.uniform(-1, 1, n).astype(np.float32).astype(np.float64), synth.random_dense((cols, R), 5).numpy().astype(np.float32).astype(np.float64)
    want, norm = oracle.spmm(c, val, (rows, cols), B)
    pk = oracle.pack(c, val, (rows, cols), (0, 1), (D, CU))
    A = comet.SpTensor.from_arrays(pk.dims, pk.mode_order, pk.attr, [dev(p, torch.int32) for p in pk.pos],
                                   [None, dev(pk.crd[1], torch.int32)], dev(pk.val, t))
    # fp32: sums in double, rounded when stored and once more where a carry is added
    assert_close(comet.spmm(A, dev(B, t)), want, norm, tol=1e-12 if dtype == "f64" else 3 * 2.0 ** -24, what="spmm")


@pytest.mark.parametrize("off", [0, 1])                       # one full wave of the longest tiles; two waves of half as long ones
def test_spmm_second_wave(off):
    rows, R = 2003, 128
    n = 148 * 2 * 8 * 1024 + off - rows                       # 32 lanes with two pieces: two CTAs of eight workers to an SM
    rng = np.random.default_rng(off)
    cols = 1 + 2 * n // rows
    cells = np.sort(rng.choice(rows * cols, n, replace=False))
    c = [(cells // cols).astype(np.int32), (cells % cols).astype(np.int32)]
    val, B = rng.uniform(-1, 1, n), synth.random_dense((cols, R), 5).numpy()
    want, norm = oracle.spmm(c, val, (rows, cols), B)
    A = upload_packed(oracle.pack(c, val, (rows, cols), (0, 1), (D, CU)))
    assert_close(comet.spmm(A, dev(B)), want, norm, what="spmm")


# Lanes a worker: one (a CTA to an SM, four waves), two (three CTAs to an SM), 16, and 32 with two pieces.
@pytest.mark.parametrize("R,workers,ctas,items", [(2, 256, 4, 31), (2, 256, 4, 33), (4, 128, 3, 23), (4, 128, 3, 33), (32, 16, 4, 35),
                                                  (32, 16, 4, 36), (32, 16, 4, 64), (64, 8, 4, 23), (64, 8, 4, 24), (128, 8, 2, 33), (128, 8, 2, 49)])
@pytest.mark.parametrize("off", [0, 1])
def test_mttkrp_csf(R, workers, ctas, items, off):
    total, dims = 148 * ctas * workers * items + off, (97, 89, 4003)
    c, v = _tensor(total, dims, min(8001, total // 10), items)
    F = [None] + [synth.random_dense((d, R), 4 + i).numpy() for i, d in enumerate(dims[1:])]
    want, norm = oracle.mttkrp(c, v, dims, 0, F)
    A = upload_packed(oracle.pack(c, v, dims, (0, 1, 2), (CU, CU, CU)))
    assert_close(comet.mttkrp(A, 0, [None] + [dev(f) for f in F[1:]]), want, norm, what="mttkrp")


# One lane (two CTAs to an SM, two waves beyond 32 items), two, 16 (whole chunks in many waves only), 32 with two pieces whole (one CTA)
# and ragged (two).
@pytest.mark.parametrize("R,workers,ctas,items", [(2, 256, 2, 11), (2, 256, 2, 12), (2, 256, 2, 33), (4, 128, 4, 23), (4, 128, 4, 24), (32, 16, 4, 47),
                                                  (32, 16, 4, 48), (32, 16, 4, 129), (128, 8, 1, 31), (128, 8, 1, 33), (100, 8, 2, 23), (100, 8, 2, 24)])
def test_mttkrp_coo_widths(R, workers, ctas, items):
    dims = (301, 97, 211)
    coords, val = synth.random_coo(dims, 148 * ctas * workers * items + 1, 3)
    c, v = [x.numpy() for x in coords], val.numpy()
    F = [None] + [synth.random_dense((d, R), 4 + i).numpy() for i, d in enumerate(dims[1:])]
    want, norm = oracle.mttkrp(c, v, dims, 0, F)
    A = upload_packed(oracle.pack(c, v, dims, (0, 1, 2), (CN, S, S)))
    assert_close(comet.mttkrp(A, 0, [None] + [dev(f) for f in F[1:]]), want, norm, what="mttkrp")


@pytest.mark.parametrize("items", [192, 193])                 # whole warps; beyond 192 three waves of the row adds of long fibers
def test_mttkrp_level1(items):
    total, dims, R = SLOTS * 8 * items, (97, 89, 4003), 64
    c, v = _tensor(total, dims, 8001, items)
    F = [synth.random_dense((d, R), 4 + i).numpy() for i, d in enumerate(dims)]
    want, norm = oracle.mttkrp(c, v, dims, 1, F)
    A = upload_packed(oracle.pack(c, v, dims, (0, 1, 2), (CU, CU, CU)))
    assert_close(comet.mttkrp(A, 1, [dev(f) for f in F]), want, norm, what="mttkrp")


@pytest.mark.parametrize("form", ["coo", "csf"])
@pytest.mark.parametrize("off", [0, 1])
def test_mttkrp_second_wave(form, off):
    dims, R = (97, 89, 4003), 64                              # whole warps, four CTAs to an SM, tiles of at most 512
    total, fibers = SLOTS * 8 * 512 + off, 8001
    c, v = _tensor(total if form == "csf" else total + fibers, dims, fibers, off)
    F = [None] + [synth.random_dense((d, R), 4 + i).numpy() for i, d in enumerate(dims[1:])]
    want, norm = oracle.mttkrp(c, v, dims, 0, F)
    A = upload_packed(oracle.pack(c, v, dims, (0, 1, 2), (CU, CU, CU) if form == "csf" else (CN, S, S)))
    assert_close(comet.mttkrp(A, 0, [None] + [dev(f) for f in F[1:]]), want, norm, what="mttkrp")
