"""Area gridding pixel by pixel and by columns, on either side of the lines between
them: small and large images, pixels of about one sample and of many, ragged last
slices, planes of 8-bit sums and of any int32 values, exact against the oracle."""
import numpy as np
import pytest

from oracle import grid

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("M,ndm,ns,nout", [(2, 3, 3, 3001), (2, 61, 40, 1000), (3, 64, 4000, 8001), (16, 17, 17, 1700), (31, 95, 3100, 3500),
                                           (64, 65, 1536, 3200), (64, 65, 1537, 3200), (64, 257, 1600, 1600), (100, 101, 101, 2424),
                                           (128, 129, 129, 2600), (128, 300, 3072, 3073), (200, 601, 3700, 3701), (255, 256, 257, 1029),
                                           (256, 1537, 1200, 1301), (257, 258, 7000, 7001), (300, 2000, 420, 900)])
@pytest.mark.parametrize("kind", ["sums", "any", "edge"])
def test_pixels_and_columns(M, ndm, ns, nout, kind):
    from paper_2511_02328_gb300 import _lib
    rng = np.random.default_rng(M + ndm + ns)
    if kind == "sums":
        y = rng.integers(0, 1 << 20, (ndm, nout))
    elif kind == "any":
        y = rng.integers(-2 ** 31, 2 ** 31, (ndm, nout))
    else:  # a column of largest values among small ones: int32 column sums do for most blocks, not for all
        y = rng.integers(0, 50, (ndm, nout))
        y[:, nout // 3] = 2 ** 31 - 1
    y = y.astype(np.int32)
    S = -(-nout // ns)
    d = torch.from_numpy(y).cuda()
    out = torch.full((S, M, M), 99, dtype=torch.uint8, device="cuda")
    work = torch.empty(2 * S, dtype=torch.int64, device="cuda")
    _lib.af_grid(d.data_ptr(), ndm, nout, ns, M, out.data_ptr(), work.data_ptr())
    torch.cuda.synchronize()
    got = out.cpu().numpy()
    area = [s for s in range(S) if min(ns, nout - s * ns) > M]
    assert area
    for s in area[:30] + area[-2:]:
        assert np.array_equal(got[s], grid.grid_slice(y[:, s * ns:(s + 1) * ns], M=M)[0]), s
