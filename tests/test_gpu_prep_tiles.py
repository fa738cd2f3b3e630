"""Zero-DM tiles and the downsampling kernels at the sizes where they change
form, bit-exact against the CPU oracle: channel counts at the edges of a
block's and a cluster's share, row lengths around a 16-byte piece and a
128-sample tile, inputs and outputs off a 16-byte boundary, in place; every
bin length with its own kernel and others, ragged last bins."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _at(a, off):
    """A copy of the uint8 array `a` on the GPU that starts `off` bytes past a 16-byte boundary."""
    buf = torch.full((a.size + off + 64,), 201, dtype=torch.uint8, device="cuda")
    view = buf[off:off + a.size]
    view.copy_(torch.from_numpy(a.reshape(-1)))
    return buf, view


@pytest.mark.parametrize("nchan,nsamp,off_in,off_out", [
    (1, 1, 0, 0), (1, 128, 0, 0), (3, 15, 0, 0), (4, 16, 1, 3), (63, 17, 0, 0), (64, 127, 5, 0), (65, 129, 0, 7),
    (512, 256, 0, 0), (513, 144, 0, 0), (1024, 131, 0, 0), (1025, 640, 0, 0), (2049, 1000, 0, 0), (4096, 384, 0, 0),
    (4096, 77, 3, 3), (4095, 272, 0, 0), (4097, 512, 0, 0), (4097, 130, 0, 0), (300, 2048, 16, 8), (300, 1999, 0, 0),
])
@pytest.mark.parametrize("in_place", [False, True])
def test_zerodm_tiles(nchan, nsamp, off_in, off_out, in_place):
    from paper_2511_02328_gb300 import _lib
    rng = np.random.default_rng(nchan * 4099 + nsamp)
    x = rng.integers(0, 256, (nchan, nsamp), dtype=np.uint8)
    x[:, : nsamp // 3] = 255
    x[: nchan // 2, nsamp // 2:] = 0
    buf, d = _at(x, off_in)
    obuf, o = (buf, d) if in_place else _at(np.zeros_like(x), off_out)
    _lib.af_zerodm(d.data_ptr(), nchan, nsamp, o.data_ptr())
    torch.cuda.synchronize()
    assert np.array_equal(o.cpu().numpy().reshape(nchan, nsamp), oracle.zerodm(x))
    off = off_in if in_place else off_out                    # nothing outside the output is written
    assert torch.all(obuf[:off] == 201) and torch.all(obuf[off + x.size:] == 201)


@pytest.mark.parametrize("D", [1, 2, 3, 4, 5, 8, 10, 16, 31, 32, 64, 300, 16384, 16385, 32768])
@pytest.mark.parametrize("nchan,nsamp,off", [(1, 1, 0), (3, 64, 0), (5, 4096 + 16, 0), (2, 65536 + 48, 0),
                                             (3, 32769, 0), (4, 5003, 3), (2, 40000, 16), (3, 131072, 0)])
def test_downsample_kernels(D, nchan, nsamp, off):
    from paper_2511_02328_gb300 import _lib
    rng = np.random.default_rng(D * 131 + nsamp)
    x = rng.integers(0, 256, (nchan, nsamp), dtype=np.uint8)
    x[0] = 255
    x[-1, : nsamp // 2] = rng.integers(0, 3, nsamp // 2)
    _, d = _at(x, off)
    nout = (nsamp + D - 1) // D
    obuf, o = _at(np.zeros((nchan, nout), dtype=np.uint8), off % 4)
    _lib.af_downsample(d.data_ptr(), nchan, nsamp, D, o.data_ptr())
    torch.cuda.synchronize()
    assert np.array_equal(o.cpu().numpy().reshape(nchan, nout), oracle.downsample_sqlaw(x, D))
    assert torch.all(obuf[:off % 4] == 201) and torch.all(obuf[off % 4 + nchan * nout:] == 201)
