"""DM-time gridding at the edges of its kernels' blocks: area slices wider than
one shared-memory run, image sizes around a block's 256 columns, full-range
values (normalisation beyond 54 bits); Lanczos images around the 64 x 64 tile,
one output row per block (very tall slices), single rows and columns.  The
area path bit-exact, the Lanczos path by the tie rule of test_gpu_grid.py."""
import numpy as np
import pytest

from oracle import grid
from test_gpu_grid import _gpu_grid, _lanczos_close

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("ndm,nout,ns,M,big", [
    (3, 20011, 20011, 2, False), (5, 30000, 14999, 2, False), (258, 1000, 400, 257, False),
    (300, 3000, 1000, 255, False), (300, 2049, 1024, 256, False), (600, 2100, 700, 513, False),
    (300, 20000, 20000, 64, True), (7, 50, 9, 4, True),
])
def test_area_blocks(ndm, nout, ns, M, big):
    rng = np.random.default_rng(ndm + nout)
    i32 = np.iinfo(np.int32)
    Y = rng.integers(i32.min if big else 0, i32.max if big else 1 << 20, (ndm, nout), dtype=np.int32, endpoint=True)
    if big:
        Y[: ndm // 2, : nout // 2] = i32.max
        Y[ndm // 2:, nout // 2:] = i32.min
    got = _gpu_grid(Y, ns, M)
    for s in range(got.shape[0]):
        X = Y[:, s * ns:(s + 1) * ns]
        if X.shape[1] > M:
            assert np.array_equal(got[s], grid.grid_slice(X, M=M)[0]), s
        else:
            _lanczos_close(got[s], X, M)


@pytest.mark.parametrize("ndm,nout,ns,M", [
    (1, 1, 1, 2), (1, 300, 150, 64), (50, 1400, 700, 512), (130, 130, 60, 65), (2000, 30, 10, 16), (12001, 12, 6, 64),
    (64, 200, 100, 63), (169, 999, 333, 128),
])
def test_lanczos_tiles(ndm, nout, ns, M):
    rng = np.random.default_rng(ndm * 7 + nout)
    Y = rng.integers(0, 5000, (ndm, nout), dtype=np.int32)
    got = _gpu_grid(Y, ns, M)
    for s in range(got.shape[0]):
        X = Y[:, s * ns:(s + 1) * ns]
        if ndm > M and X.shape[1] > M:
            assert np.array_equal(got[s], grid.grid_slice(X, M=M)[0]), s
        else:
            _lanczos_close(got[s], X, M)
