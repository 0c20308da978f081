"""Training of the surrogate (mdeos_surrogate_train, mdeos_surrogate_grads): what its fused
kernels and staged segments must keep, beside the comparisons with the oracle."""
import numpy as np
import pytest

from oracle import surrogate as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def m():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2508_06012_gb300 as m
    m.build()
    return m


@pytest.fixture(scope="module")
def h(m):
    h = m.mdeos_create()
    yield h
    m.mdeos_destroy(h)


IDENTITY = np.array([0.0, 0.0, 1.0, 1.0, 0.0, 0.0, 1.0, 1.0])


def _inputs(n, seed):
    rng = np.random.default_rng(seed)
    return np.stack([rng.uniform(-1.0, 1.0, n), rng.uniform(-1.0, 1.0, n)], axis=1)


@pytest.mark.parametrize("n", [100, 700])
def test_an_overflowing_loss_is_infinite(m, h, n):
    """Errors whose square exceeds FP32 make the sum of squares +inf (not NaN), wherever
    their samples lie and however many other tiles follow."""
    x = _inputs(n, n)
    for at in (0, n // 2, n - 1):
        y = np.zeros((n, 2))
        y[at, 1] = 1e30
        with m.Surrogate(h, 2, n, seed=3) as sg:
            sg.set_params(S.init_params(2, 2).astype(np.float32), IDENTITY)
            g, loss = sg.grads(x, y)
            assert np.isfinite(g).all() and loss == np.inf
            assert sg.train(x, y, epochs=1, batch=n, lr=1e-6, seed=1, set_norm=False)[0] == np.inf


def test_predict_allocates_no_device_memory(m, h):
    """The first predict of a surrogate, and one larger than any before it, take no memory:
    its staging comes with the surrogate (here 4 MB, so an allocation would show)."""
    import torch
    n = 1 << 16
    x = _inputs(n, 1)
    with m.Surrogate(h, 4, n, seed=1) as warm:   # the kernels' own first-use memory
        warm.predict(x)
    with m.Surrogate(h, 4, n, seed=1) as sg:
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        small = sg.predict(x[:100])
        assert torch.cuda.mem_get_info()[0] == free
        full = sg.predict(x)
        assert torch.cuda.mem_get_info()[0] == free
    assert np.array_equal(small[0], full[0][:100]) and np.array_equal(small[1], full[1][:100])


def test_predict_in_pieces_of_its_staging(m, h):
    """More queries than the staging holds, a ragged last piece: the answers of the same
    queries asked in another order of pieces."""
    n = 2 * 5000 + 777
    x = _inputs(n, 2)
    with m.Surrogate(h, 3, 5000, seed=1) as sg:
        mean, sd, pm = sg.predict(x, per_model=True)
        m2, s2, p2 = sg.predict(x[::-1], per_model=True)
    assert np.array_equal(mean, m2[::-1]) and np.array_equal(sd, s2[::-1])
    assert np.array_equal(pm, p2[:, ::-1])


def test_training_allocates_no_device_memory(m, h):
    """The first training call of a surrogate takes no memory: its segments (2 MB each here, so
    an allocation would show) come with the surrogate."""
    import torch
    batch = 1 << 17
    x = _inputs(2 * batch, 1)
    y = np.stack([x[:, 0] * x[:, 1], x[:, 1]], axis=1)
    with m.Surrogate(h, 1, batch, seed=1) as warm:   # the kernels' own first-use memory
        warm.train(x, y, epochs=1, batch=batch, set_norm=False)
    with m.Surrogate(h, 1, batch, seed=1) as sg:
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        sg.train(x[:200], y[:200], epochs=1, batch=100, set_norm=False)
        assert torch.cuda.mem_get_info()[0] == free
        sg.train(x, y, epochs=1, batch=batch, set_norm=False)
        assert torch.cuda.mem_get_info()[0] == free
