"""The surrogate's use of streams and memory: its uploads stay on its own stream,
and its calls fit where one member's arrays fit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    from paper_2604_09243_gb300 import build

    build.build()
    import paper_2604_09243_gb300 as G

    return G


def _samples(n, seed):
    rng = np.random.default_rng(seed)
    x = np.stack([rng.uniform(0, 360, n), rng.uniform(-30, 30, n), np.exp(rng.uniform(np.log(1e9), np.log(12e9), n))], 1)
    return x, rng.normal(0, 1, (n, 4))


def test_creation_uses_its_own_stream_alone(G):
    """Parameters, Fourier matrices and Adam moments reach the device on the object's (non-blocking) stream: with the
    default stream busy for a second or so the object is ready before that has ended, and trains to the same bits."""
    torch = pytest.importorskip("torch")
    net = dict(n_members=2, width=128, depth=2, n_fourier=128, fourier_sigma=2.0, seed=5)
    x, y = _samples(512, 1)
    ref = G.Surrogate(0, **net)
    ref.train(x, y, epochs=2, batch=256)
    torch.zeros(1, device="cuda")
    torch.cuda.synchronize()
    busy = torch.cuda.Event()
    torch.cuda._sleep(2_000_000_000)
    busy.record()
    s = G.Surrogate(0, **net)
    early = not busy.query()
    torch.cuda.synchronize()
    s.train(x, y, epochs=2, batch=256)
    assert early
    for e in range(2):
        assert np.array_equal(s.params(e), ref.params(e)) and np.array_equal(s.fourier(e), ref.fourier(e))
    s.close()
    ref.close()


def _fill(torch, leave):
    """Tensors that take the GPU's free memory but for `leave` bytes."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    return torch.empty(free - leave, dtype=torch.uint8, device="cuda")


def test_training_fits_where_the_whole_ensemble_does_not(G):
    """With 300 MB free the workspace of all four members (282 MB) fits only without the call's own arrays (48 MB while
    the inputs are read, 96 MB in all): fewer members train together, to the same bits."""
    torch = pytest.importorskip("torch")
    net = dict(n_members=4, width=512, depth=2, n_fourier=128, fourier_sigma=2.0, seed=7)
    x, y = _samples(2_000_000, 2)
    ref = G.Surrogate(0, **net)
    ref.train(x, y, epochs=1, batch=8192)
    want = [ref.params(e) for e in range(4)]
    ref.close()
    s = G.Surrogate(0, **net)
    hold = _fill(torch, 300 << 20)
    try:
        s.train(x, y, epochs=1, batch=8192)
    finally:
        del hold
        torch.cuda.empty_cache()
    for e in range(4):
        assert np.array_equal(s.params(e), want[e])
    s.close()


@pytest.mark.parametrize("net,n,leave", [(dict(n_members=4, width=512, depth=2, n_fourier=128), 2_000_000, 300 << 20),
                                         (dict(n_members=4, width=128, depth=1, n_fourier=8192), 300_000, 1200 << 20)])
def test_prediction_fits_where_its_usual_batches_do_not(G, net, n, leave):
    """A batch of 65,536 points of the wide network (0.6 GB of activations) does not fit into what is free, nor would
    one sized by a narrow network's activations alone (17 GB of Fourier features): smaller ones give the same bits."""
    torch = pytest.importorskip("torch")
    x, y = _samples(n, 3)
    s = G.Surrogate(0, fourier_sigma=2.0, seed=8, **net)
    s.train(x[:256], y[:256], epochs=1, batch=256)
    want = s.predict(x)
    s.close()
    s = G.Surrogate(0, fourier_sigma=2.0, seed=8, **net)
    s.train(x[:256], y[:256], epochs=1, batch=256)
    hold = _fill(torch, leave)
    try:
        got = s.predict(x)
    finally:
        del hold
        torch.cuda.empty_cache()
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
    s.close()


def test_arrays_kept_between_calls_hold_nothing_over(G):
    """Calls of every kind and of falling and rising sizes on one object, some of them with arrays of more than the 64 MB
    that are kept, give the bits of the same training on an object that makes no other calls."""
    net = dict(n_members=2, width=128, depth=1, n_fourier=128, fourier_sigma=2.0, seed=11)
    x, y = _samples(40_000, 4)
    big = np.tile(x, (75, 1))  # 3,000,000 points: 72 MB of inputs, 96 MB of predictions
    a, b = G.Surrogate(0, **net), G.Surrogate(0, **net)
    a.train(x, y, epochs=1, batch=1024)
    all_big = a.predict(big)
    a.grads(x[:256], y[:256])
    a.train(x[:5000], y[:5000], epochs=3, batch=512)
    small = a.predict(x[:700])
    a.train(x, y, epochs=2, batch=2048)
    b.train(x, y, epochs=1, batch=1024)
    one = b.predict(x)
    b.train(x[:5000], y[:5000], epochs=3, batch=512)
    two = b.predict(x[:700])
    b.train(x, y, epochs=2, batch=2048)
    for k in range(2):
        assert np.array_equal(all_big[k], np.concatenate([one[k]] * 75))
        assert np.array_equal(small[k], two[k])
    for e in range(2):
        assert np.array_equal(a.params(e), b.params(e))
    a.close()
    b.close()
