"""Zero-DM filter on either side of the line between the tile kernel and the
kernels that read twice: few channels by row lengths around it, rows of whole
16-byte pieces that are no multiple of a block, rows at any byte address, in place
and not, bit-exact; and long rows of few channels in a time that goes with their
bytes."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("nchan,nsamp", [(1, 65535), (1, 65536), (1, 65552), (1, 4095), (1, 4096), (3, 12287), (3, 12288), (7, 70000),
                                         (17, 65520), (17, 65536 + 496), (17, 69631), (17, 69632), (71, 65536), (72, 65536),
                                         (159, 4096 * 159 - 1), (159, 4096 * 159), (4097, 1040), (4100, 513)])
@pytest.mark.parametrize("offset", [0, 5])
@pytest.mark.parametrize("in_place", [False, True])
def test_zerodm_lines(nchan, nsamp, offset, in_place):
    from paper_2511_02328_gb300 import _lib
    if nchan > 158 and offset == 0 and in_place:
        pytest.skip("the largest once per address")
    X = np.random.default_rng(nchan + nsamp).integers(0, 256, (nchan, nsamp), dtype=np.uint8)
    buf = torch.zeros(X.size + 64, dtype=torch.uint8, device="cuda")
    buf[offset:offset + X.size] = torch.from_numpy(X.reshape(-1)).cuda()
    out = buf if in_place else torch.full_like(buf, 77)
    _lib.af_zerodm(buf.data_ptr() + offset, nchan, nsamp, out.data_ptr() + offset)
    torch.cuda.synchronize()
    got = out.cpu().numpy()
    assert np.array_equal(got[offset:offset + X.size].reshape(nchan, nsamp), oracle.zerodm(X))
    rest = np.concatenate([got[:offset], got[offset + X.size:]])
    assert np.all(rest == (0 if in_place else 77))  # nothing written outside the rows


@pytest.mark.parametrize("nchan", [1, 4, 16])
@pytest.mark.parametrize("offset", [0, 3])
def test_long_rows_of_few_channels(nchan, offset):
    """At most 16 times a copy of the same bytes (measured: 3 to 6; a tile of 128 samples a block: 26 to 110 for one channel)."""
    from paper_2511_02328_gb300 import _lib
    nsamp = 1 << 24
    x = torch.randint(0, 256, (nchan * nsamp + 16,), dtype=torch.uint8, device="cuda")
    z = torch.empty_like(x)

    def us(fn):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        fn()
        best = 1e9
        for _ in range(5):
            a.record()
            for _ in range(4):
                fn()
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b) / 4 * 1e3)
        return best
    copy = us(lambda: z.copy_(x))
    own = us(lambda: _lib.af_zerodm(x.data_ptr() + offset, nchan, nsamp, z.data_ptr() + offset))
    print("%d channels + %d: %.1f us, copy %.1f us" % (nchan, offset, own, copy))
    assert own < 16 * copy
