"""Cut-outs of inputs at every byte address (words across the input's ends) and of
candidate lists around the lengths up to which they are taken widest first,
bit-exact against the oracle."""
import numpy as np
import pytest

import oracle
from oracle import cutout

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BAND, TSAMP = (1300.0, 1500.0), 2e-4


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _cutouts(X, dms, cands, offset=0):
    from paper_2511_02328_gb300 import _lib
    from paper_2511_02328_gb300.search import Plan
    nchan, nsamp = X.shape
    D = oracle.delay_table(nchan, *BAND, TSAMP, dms)
    Y = oracle.dedisperse(X, D)
    p = Plan(nchan, *BAND, TSAMP, dms)
    buf = torch.zeros(X.size + 16, dtype=torch.uint8, device="cuda")
    buf[offset:offset + X.size] = torch.from_numpy(X.reshape(-1)).cuda()
    plane = torch.from_numpy(Y).cuda()
    a = np.zeros(len(cands), dtype=_lib.CAND_DTYPE)
    for i, (d, t, w) in enumerate(cands):
        a[i] = (d, t, w, 0.0, t)
    cd = torch.from_numpy(a.view(np.uint8)).cuda()
    out = torch.empty((len(cands), 64, 64, 2), dtype=torch.bfloat16, device="cuda")
    _lib.af_cutouts(p.handle, buf.data_ptr() + offset, nsamp, plane.data_ptr(), plane.shape[1], cd.data_ptr(), len(cands),
                    out.data_ptr())
    torch.cuda.synchronize()
    p.close()
    return out.float().cpu().numpy().transpose(0, 3, 1, 2), D, Y


@pytest.mark.parametrize("nchan,nsamp", [(64, 2001), (320, 1503)])
@pytest.mark.parametrize("offset", [0, 1, 2, 3, 7])
def test_input_addresses(nchan, nsamp, offset):
    X = np.random.default_rng(nsamp + offset).integers(1, 256, (nchan, nsamp), dtype=np.uint8)
    dms = np.arange(9.0)
    nout = nsamp - int(oracle.delay_table(nchan, *BAND, TSAMP, dms).max())
    cands = [(d, t, w) for d, w in ((0, 1), (8, 2), (4, 9), (8, 40), (0, 256)) for t in (0, 1, 2, 31, nout // 2, nout - 33, nout - 1)]
    got, D, Y = _cutouts(X, dms, cands, offset)
    assert np.array_equal(got, cutout.cutouts(X, D, Y, cands))


@pytest.mark.parametrize("nchan,n", [(64, 8), (64, 9), (64, 31), (64, 33), (64, 511), (64, 512), (64, 513), (512, 1023),
                                     (512, 1024), (512, 1025)])
def test_list_lengths(nchan, n):
    """Every candidate of the list is cut out, in its own place, whatever order they are taken in."""
    rng = np.random.default_rng(n)
    X = rng.integers(0, 256, (nchan, 700), dtype=np.uint8)
    dms = np.arange(4.0)
    # few different candidates, so that the oracle's part stays short; widths of every order of magnitude, 0 among them
    some = [(int(d), int(t), int(w)) for d, t, w in zip(rng.integers(0, 4, 24), rng.integers(0, 600, 24),
                                                        [0, 1, 2, 3, 4, 7, 8, 15, 16, 31, 33, 64] * 2)]
    pick = rng.integers(0, 24, n) if n % 2 else np.sort(rng.integers(0, 24, n))
    got, D, Y = _cutouts(X, dms, [some[i] for i in pick])
    ref = cutout.cutouts(X, D, Y, some)
    assert np.array_equal(got, ref[pick])
