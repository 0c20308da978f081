"""Training of the surrogate (mdeos_surrogate_train, mdeos_surrogate_grads): what its fused
kernels and staged segments must keep, beside the comparisons with the oracle."""
import ctypes
import subprocess

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


# pieces of max_batch, of the staging's 32768, one query more, an odd number of pieces
@pytest.mark.parametrize("n,max_batch", [(2 * 5000 + 777, 5000), (32768, 1 << 18),
                                         (32769, 1 << 18), (5 * 32768 - 1, 1 << 18),
                                         (3 * 20000 + 1, 20000)])
def test_predict_in_pieces(m, h, n, max_batch):
    """The answers do not depend on the pieces and the way a call's arrays take: the same
    queries in reverse, and a few of them alone."""
    x = _inputs(n, 2)
    with m.Surrogate(h, 3, max_batch, seed=1) as sg:
        mean, sd, pm = sg.predict(x, per_model=True)
        m2, s2, p2 = sg.predict(x[::-1], per_model=True)
        m3, s3 = sg.predict(x[-50:])
    assert np.array_equal(mean, m2[::-1]) and np.array_equal(sd, s2[::-1])
    assert np.array_equal(pm, p2[:, ::-1])
    assert np.array_equal(mean[-50:], m3) and np.array_equal(sd[-50:], s3)


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


ORDER_SOURCE = """
#include <algorithm>
#include <cstdint>
#include <random>
#include <vector>
// the sample order of each epoch of a training call: one generator, one permutation
extern "C" void order(uint64_t seed, int n, int epochs, int* out) {
  std::mt19937_64 rng(seed);
  std::vector<int> perm(n);
  for (int i = 0; i < n; ++i) perm[i] = i;
  for (int e = 0; e < epochs; ++e) {
    std::shuffle(perm.begin(), perm.end(), rng);
    std::copy(perm.begin(), perm.end(), out + (size_t)e * n);
  }
}
"""


@pytest.fixture(scope="module")
def order(tmp_path_factory):
    d = tmp_path_factory.mktemp("order")
    (d / "order.cpp").write_text(ORDER_SOURCE)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-o", str(d / "order.so"),
                    str(d / "order.cpp")], check=True)
    f = ctypes.CDLL(str(d / "order.so")).order
    f.argtypes = [ctypes.c_uint64, ctypes.c_int, ctypes.c_int, ctypes.c_void_p]
    f.restype = None

    def get(seed, n, epochs=1):
        out = np.zeros((epochs, n), dtype=np.int32)
        f(seed, n, epochs, out.ctypes.data_as(ctypes.c_void_p))
        return out
    return get


# one batch, a full segment, one more, two segments and one, a ragged third; whole segments
# of one large batch; a remainder of samples that no batch holds
@pytest.mark.parametrize("batch,nb,extra,epochs", [(64, 1, 0, 1), (64, 16, 0, 1), (64, 17, 5, 1),
                                                   (64, 33, 0, 2), (64, 37, 63, 2), (129, 20, 1, 1),
                                                   (40000, 3, 7, 1)])
def test_an_epoch_equals_its_batches_one_call_at_a_time(m, h, order, batch, nb, extra, epochs):
    """Parameters and losses of a training call, bit for bit, against the same batches in the
    same order, each a call of its own on the same Adam state."""
    n = batch * nb + extra
    x = _inputs(n, n)
    y = np.stack([x[:, 0] * x[:, 1], np.sin(3.0 * x[:, 1])], axis=1)
    norm = np.array([0.1, -0.2, 0.7, 0.6, 0.05, 0.1, 0.4, 0.8])
    inside = order(77, batch)[0]   # the order in which a call of one batch takes its rows
    with m.Surrogate(h, 2, batch, seed=4) as a, m.Surrogate(h, 2, batch, seed=4) as b:
        a.set_params(None, norm)
        b.set_params(None, norm)
        la = a.train(x, y, epochs=epochs, batch=batch, lr=1e-3, seed=8, set_norm=False)
        lb = []
        for perm in order(8, n, epochs):
            lsum = 0.0
            for k in range(nb):
                rows = np.empty(batch, dtype=np.int64)
                rows[inside] = perm[k * batch:(k + 1) * batch]
                lsum += b.train(x[rows], y[rows], epochs=1, batch=batch, lr=1e-3, seed=77,
                                set_norm=False)[0]
            lb.append(lsum / nb)
        pa, pb = a.get_params()[0], b.get_params()[0]
        assert pa.tobytes() == pb.tobytes() and list(la) == lb
        # and the comparison sees a batch that is not the same
        b.train(x[rows][::-1], y[rows], epochs=1, batch=batch, lr=1e-3, seed=77, set_norm=False)
        a.train(x[rows], y[rows], epochs=1, batch=batch, lr=1e-3, seed=77, set_norm=False)
        assert a.get_params()[0].tobytes() != b.get_params()[0].tobytes()


@pytest.mark.parametrize("n", [1, 2, 63, 65, 127, 128, 129, 192, 193, 257, 640, 1025, 4203])
def test_every_sample_of_a_ragged_batch_reaches_every_gradient(m, h, n):
    """All targets but one are the network's own outputs, so the gradient is one sample's
    alone: per parameter block it is the oracle's, wherever the sample lies.  A sample lost
    from a block leaves it zero, one counted twice doubles it.

    Bound: the oracle takes the same bfloat16 roundings, and a value that rounds the other
    way moves by 2^-8 of itself; 2e-2 allows five such steps in every element of a block.
    The other samples' errors, at most 2^-20 each against 5, add n 2^-20 / 5 < 1e-3."""
    x = _inputs(n, n)
    p = S.init_params(9, 1)
    d = S.unpack(p[0])
    rng = np.random.default_rng(n)
    for name in ("b1", "b2", "b3", "b4"):
        d[name] = 0.1 * rng.standard_normal(d[name].shape)
    p = S.pack(d)[None].astype(np.float32).astype(np.float64)
    edges = [0, 1, 62, 63, 64, 65, 127, 128, 191, 192, 255, 256, n // 2, n - 66, n - 65, n - 2, n - 1]
    with m.Surrogate(h, 1, n, seed=1) as sg:
        sg.set_params(p.astype(np.float32), IDENTITY)
        y = sg.predict(x, per_model=True)[2][0].astype(np.float64)
        g0, _ = sg.grads(x, y)
        assert np.abs(g0).max() <= 1e-5   # nothing but those rounding errors
        for at in sorted({k for k in edges if 0 <= k < n}):
            t = y.copy()
            t[at] += [5.0, -3.0]
            g, loss = sg.grads(x, t)
            # the oracle on that sample alone, with the batch's error signal d / n
            out = S.forward(p[0], x[at:at + 1])[0]
            _, ref = S.loss_and_grad(p[0], x[at:at + 1], out + np.array([5.0, -3.0]) / n)
            got, want = S.unpack(g[0]), S.unpack(ref)
            for name, _ in S.SHAPES:
                err = np.linalg.norm(got[name] - want[name])
                assert err <= 2.1e-2 * np.linalg.norm(want[name]), (at, name)
            assert loss == pytest.approx((25.0 + 9.0) / (2 * n), rel=1e-5)


def test_launch_counts(m, h):
    """Kernels counted by mdeos_stats: a gradient is two, and a third where the batch's K is
    split (from four chunks of 64 samples on); a training step three; inference three on the
    fused path, eight on the layered one."""
    def count(f):
        before = m.mdeos_stats(h)["launches"]
        f()
        return m.mdeos_stats(h)["launches"] - before

    x = _inputs(640, 1)
    with m.Surrogate(h, 2, 640, seed=1) as sg:
        for n, k in ((1, 2), (192, 2), (193, 3), (640, 3)):
            assert count(lambda: sg.grads(x[:n], x[:n])) == k, n
        assert count(lambda: sg.train(x, x, epochs=2, batch=64, set_norm=False)) == 3 * 20
        assert count(lambda: sg.predict(x)) == 3
        sg.set_infer_path(1)
        assert count(lambda: sg.predict(x)) == 8


def test_both_halves_of_the_packed_tanh(m):
    """The tanh of the fused kernels takes two values at a time: each value in either half
    gives the same bits, beside whatever value, within 2e-6 of tanh."""
    import torch
    g = np.linspace(-12.0, 12.0, 100001)
    tiny = 10.0 ** np.linspace(-37, -1, 1001)
    edge = np.array([0.25, np.nextafter(np.float32(0.25), np.float32(0)), 43.9, 44.0, 88.0, 3e38,
                     np.inf, 0.0])
    x = np.concatenate([g, tiny, -tiny, edge, -edge]).astype(np.float32)
    rng = np.random.default_rng(1)

    def tanh(v):
        return m.mdeos_debug_tanh(torch.from_numpy(np.ascontiguousarray(v)).cuda()).cpu().numpy()

    y = tanh(x)
    ref = np.tanh(x.astype(np.float64))
    nz = np.abs(ref) > 1e-36
    assert (np.abs(y[nz] - ref[nz]) < 2e-6 * np.abs(ref[nz])).all()
    assert (np.signbit(y) == np.signbit(x)).all()
    assert tanh(x[1:]).tobytes() == y[1:].tobytes()      # every value in the other half
    p = rng.permutation(len(x))
    assert tanh(x[p]).tobytes() == y[p].tobytes()
    with_nan = np.repeat(x, 2)
    with_nan[0::4] = np.nan                               # a NaN beside either half
    with_nan[3::4] = np.nan
    yn = tanh(with_nan)
    keep = ~np.isnan(with_nan)
    assert np.isnan(yn[~keep]).all() and yn[keep].tobytes() == np.repeat(y, 2)[keep].tobytes()
