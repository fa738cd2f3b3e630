"""Median and MAD of long rows (the one-pass kernel): exact against the CPU
oracle for every number of blocks per row, row lengths off 16-byte
boundaries, and distributions that the sample's windows hold (noise, heavy
tails, a few distinct values) and that they do not (bimodal, sorted, spans of
the whole int32 range), where the row takes the general selection."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _rows(nout, seed):
    rng = np.random.default_rng(seed)
    n = rng.normal(0.0, 1.0, nout)
    i32 = np.iinfo(np.int32)
    alt = np.where(np.arange(nout) % 2 == 0, 100, 900)
    return np.stack([
        np.rint(524288 + 768 * n), np.rint(30000 * n), np.rint(3 * n), np.rint(0.4 * n), np.full(nout, 7),
        np.rint(1000 * rng.standard_cauchy(nout)).clip(-2 ** 30, 2 ** 30),
        np.sort(np.rint(5000 * n)), alt, np.where(rng.random(nout) < 0.5001, -40000, 50000) + np.rint(10 * n),
        rng.integers(i32.min, i32.max, nout, endpoint=True), i32.max - np.abs(np.rint(50 * n)),
        i32.min + np.abs(np.rint(50 * n)), np.rint(200 * n) + np.where(rng.random(nout) < 0.01, 100000, 0),
        np.rint(2e6 * n),
    ]).astype(np.int64).clip(i32.min, i32.max).astype(np.int32)


@pytest.mark.parametrize("nout,repeat", [(16383, 1), (16384, 1), (16385, 3), (32771, 1), (70001, 1), (200003, 1),
                                         (33001, 90), (17002, 30)])
def test_long_rows_exact(nout, repeat):
    from paper_2511_02328_gb300 import _lib
    base = _rows(nout, nout)
    Y = np.tile(base, (repeat, 1))
    y = torch.from_numpy(Y).cuda()
    ndm = Y.shape[0]
    p = _lib.af_plan(16, 1000.0, 1500.0, 1e-3, np.zeros(ndm))
    r = torch.full((ndm, 2), -5, dtype=torch.int64, device="cuda")
    _lib.af_rowstats_robust(p, y.data_ptr(), nout, r.data_ptr())
    torch.cuda.synchronize()
    med, mad = oracle.row_robust(base)
    got = r.cpu().numpy()
    assert np.array_equal(got[:, 0], np.tile(med, repeat))
    assert np.array_equal(got[:, 1], np.tile(mad, repeat))
    _lib.af_plan_destroy(p)
