"""The fused inference kernel with two, four and eight blocks per image (the
choice follows the batch size): an image's logits do not depend on the batch
it is in, bit for bit, and are the oracle's within the project's logit
tolerance (1e-2)."""
import numpy as np
import pytest

from oracle import cnn, cutout

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _forward(m, x, n, with_logits=True):
    from paper_2511_02328_gb300 import _lib
    logits = torch.full((n, 2), 9.0, dtype=torch.float32, device="cuda")
    prob = torch.full((n,), 9.0, dtype=torch.float32, device="cuda")
    _lib.af_model_forward(m, x.data_ptr(), n, logits.data_ptr() if with_logits else 0, prob.data_ptr())
    torch.cuda.synchronize()
    return logits.cpu().numpy(), prob.cpu().numpy()


def test_fused_batches_agree_and_match_oracle():
    from paper_2511_02328_gb300 import _lib
    rng = np.random.default_rng(23)
    p = cnn.init_params(9)
    for l in range(3):
        p["b%d" % l] = rng.normal(0, 0.05, p["b%d" % l].shape).astype(np.float32)
    n = 255
    x = cutout.bf16_round(rng.uniform(0, 1, (n, 64, 64, 2)).astype(np.float32))
    x[0] = 0.0
    x[1, 0] = x[1, -1] = x[1, :, 0] = x[1, :, -1] = 1.0     # bright border: the halo rows and columns
    xd = torch.from_numpy(x).cuda().to(torch.bfloat16).contiguous()
    m = _lib.af_model_create(n, 1)
    _lib.af_model_set_params(m, np.concatenate([p[k].reshape(-1) for k in ("w0", "b0", "w1", "b1", "w2", "b2", "fw",
                                                                            "fb")]).astype(np.float32))
    logits, prob = _forward(m, xd, n)
    for k in (1, 2, 18, 19, 20, 37, 38, 39, 76, 77, 153):
        lg, pr = _forward(m, xd, k)
        assert np.array_equal(lg, logits[:k]) and np.array_equal(pr, prob[:k]), k
        lg, pr = _forward(m, xd[n - k:].contiguous(), k)
        assert np.array_equal(lg, logits[n - k:]) and np.array_equal(pr, prob[n - k:]), k
    _, pr = _forward(m, xd, 5, with_logits=False)
    assert np.array_equal(pr, prob[:5])
    k = 6
    ref = cnn.forward(p, x[:k], bf16=True)[0]
    assert np.max(np.abs(logits[:k] - ref)) <= 1e-2 * max(1.0, np.abs(ref).max())
    _lib.af_model_destroy(m)
