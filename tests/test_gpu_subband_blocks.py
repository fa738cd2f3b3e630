"""Two-stage subband dedispersion over several time blocks, cut where stage 1
fills whole waves, with 16-bit and 32-bit partial sums: plane and row sums
bit-exact against the CPU oracle."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


# nchan, nsamp, dms, n0, nsub, block_len; bright = all samples 255 (largest sums)
CASES = [
    (96, 41003, np.arange(0.0, 280.0, 1.0), 2, 3, 12001, False),   # 10 row blocks, odd block length
    (520, 17001, np.arange(0.0, 60.0, 0.5), 1, 2, 5000, True),     # 260 channels per subband: 32-bit sums
    (514, 9001, np.arange(0.0, 30.0, 1.0), 1, 2, 4100, True),      # 257 per subband: 65535, the 16-bit limit
    (64, 9002, np.arange(0.0, 15.0, 1.0), 1, 64, 0, False),        # one channel per subband, 15 rows
]


@pytest.mark.parametrize("nchan,nsamp,dms,n0,nsub,block_len,bright", CASES)
def test_time_blocks(nchan, nsamp, dms, n0, nsub, block_len, bright):
    from paper_2511_02328_gb300.search import Plan
    f_lo, f_hi, tsamp = 1000.0, 1500.0, 98.304e-6
    rng = np.random.default_rng(nchan + nsamp)
    X = np.full((nchan, nsamp), 255, np.uint8) if bright else \
        rng.integers(0, 256, size=(nchan, nsamp), dtype=np.uint8)
    tab = oracle.subband_tables(nchan, f_lo, f_hi, tsamp, dms, n0, nsub, 1)
    ref = oracle.subband_dedisperse(X, tab)
    S, Q = oracle.rowstats(ref)
    p = Plan(nchan, f_lo, f_hi, tsamp, dms, subband=dict(n0=n0, nsub=nsub, fs_mode=1, block_len=block_len))
    stats = torch.empty((p.ndm, 2), dtype=torch.int64, device="cuda")
    Y = p.dedisperse(torch.from_numpy(X).cuda(), stats=stats).cpu().numpy()
    st = stats.cpu().numpy()
    assert np.array_equal(Y, ref)
    assert np.array_equal(st[:, 0], S) and np.array_equal(st[:, 1], Q)
    p.close()
