"""Boxcar S/N on either side of the line between the tile sizes: small and large
planes, row lengths at the edges of both, widths up to the largest of the small
tile and past it, and the reference's best widths, against the CPU oracle."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-5


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


# 2048-word tiles give 2048 - w outputs (in fours), 6144-word tiles 6144 - w; 4 tiles per SM of the larger are the line
@pytest.mark.parametrize("ndm,nout,widths", [
    (1, 1, [1]), (3, 2047, [1]), (3, 2048, [1, 2]), (2, 2049, [1, 4]), (5, 2016, [1, 2, 4, 8, 16, 32]), (5, 2017, [1, 32]),
    (2, 1536, [512]), (2, 1537, [1, 511, 512]), (2, 4000, [3, 513]), (1, 70001, list(range(1, 33))),
    (608, 300, [1, 3, 7]), (609, 301, [1, 3, 7]), (304, 6145, [1, 64]), (305, 6145, [1, 64]), (900, 2100, [5, 512]),
])
@pytest.mark.parametrize("nchan", [64, 30000])
def test_tile_sizes(ndm, nout, widths, nchan):
    from paper_2511_02328_gb300.search import Plan
    rng = np.random.default_rng(ndm + nout + nchan)
    y = np.rint(127.5 * nchan + 74 * nchan ** 0.5 * rng.normal(size=(ndm, nout))).astype(np.int32)
    y[:, nout // 2] += int(600 * nchan ** 0.5)
    if widths[-1] * 255 * nchan >= 2 ** 32:
        pytest.skip("windows past exact 32-bit sums")
    p = Plan(nchan, 1000.0, 1500.0, 1e-4, np.zeros(ndm))
    snr, bw = p.boxcar_snr(torch.from_numpy(y).cuda(), widths)
    torch.cuda.synchronize()
    ref, ref_w = oracle.boxcar_snr(y, widths)
    got, fin = snr.cpu().numpy().astype(np.float64), np.isfinite(ref)
    assert np.array_equal(np.isfinite(got), fin)
    err = np.abs(got[fin] - ref[fin]) / np.maximum(1.0, np.abs(ref[fin]))
    assert err.size == 0 or float(err.max()) <= TOL
    # the best width is the reference's, or one whose S/N ties with it within the tolerance
    other = bw.cpu().numpy() != ref_w
    assert np.count_nonzero(other & fin) <= 1e-4 * other.size + 1
    p.close()
