"""Gradients of batches that repeat a smaller one a power of two times: the
loss and every gradient are the smaller batch's up to the order of fp32
additions (scaling by a power of two changes no rounding), over the head's
partial passes, one and several tiles per block, and blocks that add their
sums together.  And parameters packed by an inference call serve a backward
pass that packs only what is missing."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# additions of up to 2^13 products per fp32 accumulator in another order, and
# of one partial sum per block: errors of about sqrt(2^13) 2^-24 = 5e-6 of the
# tensor's norm where the terms' signs are mixed
TOL = 2e-5


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _grads(m, x, y):
    from paper_2511_02328_gb300 import _lib
    loss = torch.empty(1, dtype=torch.float32, device="cuda")
    _lib.af_model_backward(m, x.data_ptr(), y.data_ptr(), x.shape[0], loss.data_ptr())
    torch.cuda.synchronize()
    return float(loss.item()), np.asarray(_lib.af_model_get_grads(m), dtype=np.float64)


def _batch(n, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.rand((n, 64, 64, 2), device="cuda", generator=g).to(torch.bfloat16)
    return x, torch.randint(0, 2, (n,), device="cuda", generator=g, dtype=torch.int32)


# the parameters' layout: weights and biases of three layers, the head's weights and biases
CUTS = np.cumsum([288, 16, 4608, 32, 18432, 64, 128])


@pytest.mark.parametrize("n,rep", [(1, 4), (3, 512), (5, 256), (613, 2)])
def test_repeated_batch(n, rep):
    from paper_2511_02328_gb300 import _lib
    m = _lib.af_model_create(n * rep, 7)
    x, y = _batch(n, n)
    l0, g0 = _grads(m, x, y)
    l1, g1 = _grads(m, x.repeat(rep, 1, 1, 1), y.repeat(rep))
    assert abs(l0 - l1) <= TOL * max(1.0, abs(l0))
    for a, b in zip(np.split(g0, CUTS), np.split(g1, CUTS)):
        assert np.linalg.norm(a - b) <= TOL * np.linalg.norm(a)
    _lib.af_model_destroy(m)


def test_backward_after_inference_packed_the_weights():
    from paper_2511_02328_gb300 import _lib
    x, y = _batch(300, 5)  # the layered inference path, which packs the forward weights
    a, b = (_lib.af_model_create(300, 3) for _ in range(2))
    logits = torch.empty((300, 2), dtype=torch.float32, device="cuda")
    _lib.af_model_forward(a, x.data_ptr(), 300, logits.data_ptr(), 0)
    (la, ga), (lb, gb) = _grads(a, x, y), _grads(b, x, y)
    assert abs(la - lb) <= TOL * max(1.0, abs(la)) and np.linalg.norm(ga - gb) <= TOL * np.linalg.norm(ga)
    (lc, gc) = _grads(a, x, y)  # nothing left to pack
    assert abs(la - lc) <= TOL * max(1.0, abs(la)) and np.linalg.norm(ga - gc) <= TOL * np.linalg.norm(ga)
    for m in (a, b):
        _lib.af_model_destroy(m)
