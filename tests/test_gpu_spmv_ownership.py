"""SpMV / TTV of small inputs: rows around the length up to which one tile takes a row whole (64 entries), straddling many
tiles at every offset, with empty rows between them, with and without any carry left, in one tile and in thousands."""
import numpy as np
import pytest
import torch

import oracle
from oracle import D, CU

pytestmark = pytest.mark.gpu

comet = pytest.importorskip("paper_2102_05187_b200")
from gpu_util import assert_close, dev, upload_packed  # noqa: E402


@pytest.fixture(autouse=True)
def _need_gpu(cuda_device, monkeypatch):
    monkeypatch.delenv("COMET_SEG_DOT_KERNEL", raising=False)
    yield


@pytest.mark.parametrize("pattern", [[64], [63, 0, 65], [1, 64, 0, 0, 64], [65], [576], [575, 1, 0, 577], [64, 5000, 64, 0], [40000]])
@pytest.mark.parametrize("rows", [1, 7, 400, 3000])
@pytest.mark.parametrize("attr", [(D, CU), (CU, CU)])
def test_row_lengths(pattern, rows, attr):
    lengths = (pattern * rows)[:rows]
    while sum(lengths) > 900_000:
        lengths = lengths[: len(lengths) // 2]
    rng = np.random.default_rng(rows)
    cols = 41_000
    r = np.repeat(np.arange(len(lengths)), lengths).astype(np.int32)
    c = np.concatenate([(np.arange(n) * 3 + 7 * i) % cols for i, n in enumerate(lengths)]).astype(np.int32)
    order = np.lexsort((c, r))
    r, c = r[order], c[order]
    v, x = rng.uniform(-1, 1, r.size), rng.uniform(-1, 1, cols)
    want, norm = oracle.spmv([r, c], v, (len(lengths), cols), x)
    A = upload_packed(oracle.pack([r, c], v, (len(lengths), cols), (0, 1), attr))
    first = comet.spmv(A, dev(x))
    assert_close(first, want, norm)
    for _ in range(3):                                       # the counters of the last CTA are back at zero
        assert torch.equal(first, comet.spmv(A, dev(x)))
