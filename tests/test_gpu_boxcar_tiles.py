"""The boxcar kernel at the edges of its tiles: rows of every misalignment
(odd row lengths), lengths around one and two tiles, width lists that are not
whole groups of three or multiples of four, the widest windows (both tile
sizes), and window sums of 2^31 and above, on the float and the integer path,
against the CPU oracle.  S/N tolerance: the project's bound 1e-5 max(|snr|, 1);
the best width where it is unique by more than that."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

W = 6144  # prefix words of a tile for widths up to 1024


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("nout,widths,nchan", [
    (1, [1], 4), (2, [1, 2], 4), (7, [1, 3, 5, 7], 4), (129, [1, 2, 3, 4, 5, 6, 7], 4),
    (W - 5, [1, 2, 5], 256), (W - 4, [1, 3, 4, 9], 256), (W - 1, [1], 256), (W, [1], 256), (W + 1, [1, 1023], 256),
    (2 * (W - 256) - 3, [1, 2, 4, 8, 16, 32, 64, 128, 256], 4096),
    (2 * (W - 256) + 1, [2, 6, 30, 255], 4096), (3 * W + 2, [1, 7, 1024], 256),
    (12288 - 1025, [1, 2, 1025], 64), (20011, [1, 63, 1025, 4097, 8192], 64),
    (9001, list(range(1, 33)), 64),
    (9002, [1, 5, 600], 16384), (15003, [4, 1101, 2050], 4200),
])
def test_boxcar_tiles(nout, widths, nchan):
    from paper_2511_02328_gb300 import _lib
    rng = np.random.default_rng(nout)
    ndm = 5
    mean, sd = 128.0 * nchan, 12.0 * np.sqrt(nchan)
    Y = np.clip(np.rint(rng.normal(mean, sd, (ndm, nout))), 0, 255 * nchan).astype(np.int32)
    Y[1, nout // 2:] = 255 * nchan                      # half a row at full scale: the integer path
    Y[2] = 77                                           # constant row
    Y[3, nout // 3] = 0
    y = torch.from_numpy(Y).cuda()
    snr = torch.full((ndm, nout), 7.0, dtype=torch.float32, device="cuda")
    bw = torch.full((ndm, nout), 99, dtype=torch.uint8, device="cuda")
    _lib.af_boxcar_snr_noalloc(y.data_ptr(), ndm, nout, nchan, widths, snr.data_ptr(), bw.data_ptr())
    torch.cuda.synchronize()
    got, gbw = snr.cpu().numpy().astype(np.float64), bw.cpu().numpy()
    ref, rbw = oracle.boxcar_snr(Y, widths)
    rbw = np.where(rbw < 0, 255, rbw)
    fin = np.isfinite(ref)
    assert np.array_equal(fin, np.isfinite(got))
    assert np.all(np.abs(got - ref)[fin] <= 1e-5 * np.maximum(np.abs(ref[fin]), 1.0))
    # a different best width is accepted only where its own S/N is within the tolerance of the best
    S = Y.astype(np.int64).sum(1)
    P = np.concatenate([np.zeros((ndm, 1), np.int64), np.cumsum(Y.astype(np.int64), axis=1)], axis=1)
    sigma = np.sqrt(((Y - S[:, None] / nout) ** 2).mean(1))
    for d, t in zip(*np.nonzero(gbw != rbw)):
        assert gbw[d, t] < len(widths) and rbw[d, t] < len(widths) and sigma[d] > 0
        w = widths[gbw[d, t]]
        v = (nout * (P[d, t + w] - P[d, t]) - w * S[d]) / (nout * sigma[d] * np.sqrt(w))
        assert abs(v - ref[d, t]) <= 1e-5 * max(abs(ref[d, t]), 1.0)
