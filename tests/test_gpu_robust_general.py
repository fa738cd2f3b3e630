"""Median and MAD of long rows that the one-pass kernel hands to the general
selection, shared by the blocks of a row's cluster: rows that its sample shows to be
unsuited (two far-apart modes, wide rows), rows whose sample misleads it (the sampled
places differ from the rest) and periodic rows, exact against the CPU oracle for every
number of blocks per row."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _misleading(nout, rng):
    """A 16-byte aligned row whose sampled pieces are noise around 0 and whose other values lie around 900."""
    row = np.rint(900 + 100 * rng.normal(size=nout)).astype(np.int64)
    n4 = nout // 4
    step = n4 // 1024
    piece = np.arange(1024, dtype=np.uint64)
    at = piece * np.uint64(step) + (((piece * np.uint64(2654435761)) & np.uint64(0xFFFFFFFF)) * np.uint64(step) >> np.uint64(32))
    for k in range(4):
        row[4 * at.astype(np.int64) + k] = np.rint(100 * rng.normal(size=1024))
    return row


def _rows(nout, seed):
    rng = np.random.default_rng(seed)
    n = rng.normal(size=nout)
    t = np.arange(nout)
    return np.stack([
        _misleading(nout, rng), np.rint(300 * n) + 20000 * rng.integers(0, 2, nout), np.rint(2e4 * n) + 2_000_000,
        t % 64 * 100, t % 4096, np.rint(300 * n) + 5000 * t // nout, rng.integers(0, 4000, nout),
        np.where(rng.random(nout) < 0.49, -2_000_000_000, 2_000_000_000) + np.rint(5 * n), np.rint(1200 * n) + 30000,
        np.where(rng.random(nout) < 0.3, 0, np.rint(1000 + 30 * n)), np.full(nout, -3), np.rint(0.7 * n),
    ]).astype(np.int32)


# the first row of a plane is the aligned one; blocks per row: 1, 2, 4, 8 (by length and by rows), 1 (many rows)
@pytest.mark.parametrize("nout,repeat", [(16384, 1), (32768, 1), (65540, 1), (131075, 1), (40000, 60), (70004, 30), (40001, 110)])
def test_general_selection_shared(nout, repeat):
    from paper_2511_02328_gb300 import _lib
    base = _rows(nout, nout)
    Y = np.tile(base, (repeat, 1))
    y = torch.from_numpy(Y).cuda()
    ndm = Y.shape[0]
    p = _lib.af_plan(16, 1000.0, 1500.0, 1e-3, np.zeros(ndm))
    r = torch.full((ndm, 2), -5, dtype=torch.int64, device="cuda")
    for _ in range(2):
        _lib.af_rowstats_robust(p, y.data_ptr(), nout, r.data_ptr())
    torch.cuda.synchronize()
    med, mad = oracle.row_robust(base)
    got = r.cpu().numpy()
    assert np.array_equal(got[:, 0], np.tile(med, repeat))
    assert np.array_equal(got[:, 1], np.tile(mad, repeat))
    _lib.af_plan_destroy(p)
