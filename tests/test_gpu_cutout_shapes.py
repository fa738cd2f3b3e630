"""Cut-outs bit-exact against the oracle where the kernel's paths change: more
than 256 channels per frequency-time row, channel counts that leave a short last
group of loads, rows that start at every byte offset, bins too wide for 32-bit
sums, windows that leave the plane on either side, and more candidates than are
sorted by width."""
import numpy as np
import pytest

import oracle
from oracle import cutout

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _run(nchan, nsamp, dms, cands, pick=None):
    from paper_2511_02328_gb300 import _lib
    from paper_2511_02328_gb300.search import Plan
    f_lo, f_hi, tsamp = 1300.0, 1500.0, 2e-4
    X = np.random.default_rng(nchan + nsamp).integers(0, 256, (nchan, nsamp), dtype=np.uint8)
    D = oracle.delay_table(nchan, f_lo, f_hi, tsamp, dms)
    Y = oracle.dedisperse(X, D)
    p = Plan(nchan, f_lo, f_hi, tsamp, dms)
    xd = torch.from_numpy(X).cuda()
    plane = p.dedisperse(xd)
    a = np.zeros(len(cands), dtype=_lib.CAND_DTYPE)
    for i, (d, t, w) in enumerate(cands):
        a[i] = (d, t, w, 0.0, t)
    cd = torch.from_numpy(a.view(np.uint8)).cuda()
    out = torch.empty((len(cands), 64, 64, 2), dtype=torch.bfloat16, device="cuda")
    _lib.af_cutouts(p.handle, xd.data_ptr(), nsamp, plane.data_ptr(), plane.shape[1], cd.data_ptr(), len(cands),
                    out.data_ptr())
    torch.cuda.synchronize()
    got = out.float().cpu().numpy().transpose(0, 3, 1, 2)
    at = range(len(cands)) if pick is None else pick
    ref = cutout.cutouts(X, D, Y, [cands[i] for i in at])
    assert np.array_equal(got[list(at)], ref)
    p.close()


@pytest.mark.parametrize("nchan,nsamp", [(64, 4001), (320, 3003), (384, 2002), (19200, 1100)])
def test_shapes(nchan, nsamp):
    cands = [(5, 1, 1), (0, nsamp // 2, 2), (11, nsamp // 3, 7), (7, nsamp // 2, 16), (2, 400, 33), (11, 3, 64),
             (6, nsamp - 200, 129), (3, 500, 256), (9, 700, 5000), (4, 10, 300)]
    _run(nchan, nsamp, np.arange(12.0), cands)


def test_more_candidates_than_are_sorted():
    rng = np.random.default_rng(2)
    cands = [(int(d), int(t), int(w)) for d, t, w in zip(rng.integers(0, 8, 4099), rng.integers(0, 1500, 4099),
                                                         2 ** rng.integers(0, 6, 4099))]
    _run(64, 1800, np.arange(8.0), cands, pick=[0, 1, 77, 2048, 4095, 4096, 4098])
