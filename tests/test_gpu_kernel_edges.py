"""Kernels at the sizes where their splits change: list builds at tile and ring edges, boxes
with a cell grid on thread-block clusters, hydro slabs at cluster-size edges, training batches
that are not whole tiles, inference at group-count edges."""
import numpy as np
import pytest

from oracle import hydro as H
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


def _box(n, rho, seed):
    """n atoms on a jittered FCC lattice in a float32 box (some pairs near every distance)."""
    rng = np.random.default_rng(seed)
    L = np.float32((n / rho) ** (1.0 / 3.0))
    nc = 1
    while 4 * nc ** 3 < n:
        nc += 1
    i = np.arange(n)
    c, b = i >> 2, i & 3
    x = np.stack([c % nc + 0.5 * np.isin(b, (1, 2)), c // nc % nc + 0.5 * np.isin(b, (1, 3)),
                  c // nc ** 2 + 0.5 * np.isin(b, (2, 3))], axis=1) * (float(L) / nc)
    x = (x + 0.08 * rng.standard_normal(x.shape)).astype(np.float32)
    return np.mod(x, L).astype(np.float32), float(L)


def _count_within(x, L, R):
    """Ordered pairs with minimum-image distance below R."""
    x = x.astype(np.float64)
    k = 0
    for i0 in range(0, len(x), 256):
        d = x[i0:i0 + 256, None, :] - x[None, :, :]
        d -= L * np.round(d / L)
        k += int(((d * d).sum(-1) < R * R).sum())
    return k - len(x)


# brute-force lists with four sub-lists (to 384 atoms) and one (to 768), then cells; atoms
# per thread 1, 2 and 4; counts at and around multiples of 32, of the turn of 8 candidates
@pytest.mark.parametrize("n,rho", [(131, 0.35), (257, 0.8), (383, 0.9), (384, 1.1), (385, 0.5),
                                   (500, 0.8), (767, 1.15), (768, 0.6), (769, 0.4), (1000, 0.8),
                                   (1024, 1.2), (1025, 0.9), (2049, 0.3), (4095, 1.2), (4096, 0.6)])
def test_list_holds_every_neighbour_once(m, n, rho):
    """The list's entry count is the number of ordered pairs within rc + skin (pairs within
    rounding of that distance may fall either way), and its forces match the sum over all
    pairs within FP32 rounding."""
    import torch
    x, L = _box(n, rho, n)
    skin = 0.3
    x4 = torch.zeros((n, 4), dtype=torch.float32, device="cuda")
    x4[:, :3] = torch.from_numpy(x).cuda()
    entries = int(m.mdeos_debug_force_bench(x4[None].contiguous(), L, skin, 1)[0, 1])
    eps = 4 * 2.0 ** -24 * L                      # rounding of a difference across a face
    assert _count_within(x, L, 2.5 + skin - eps) <= entries <= _count_within(x, L, 2.5 + skin + eps)
    f, ew, pairs = m.mdeos_debug_forces(x4, L, m.PATH_NLIST, skin=skin)
    assert _count_within(x, L, 2.5 - eps) <= pairs <= _count_within(x, L, 2.5 + eps)
    xd = torch.from_numpy(x).cuda().double()
    fr = torch.zeros_like(xd)
    mag = torch.zeros(n, device="cuda", dtype=torch.float64)
    for i0 in range(0, n, 512):
        d = xd[i0:i0 + 512, None, :] - xd[None, :, :]
        d -= L * torch.round(d / L)
        r2 = (d * d).sum(-1)
        on = (r2 < 6.25) & (r2 > 0)
        ir2 = torch.where(on, 1.0 / torch.where(on, r2, 1.0), 0.0)
        s6 = ir2 ** 3
        fac = 24.0 * s6 * (2.0 * s6 - 1.0) * ir2
        fr[i0:i0 + 512] = (fac[:, :, None] * d).sum(1)
        # |f| and |df/dr| L: the scales of the rounding of a term and of its difference
        mag[i0:i0 + 512] = (fac.abs() * r2.sqrt() + 24.0 * (26.0 * s6 + 7.0) * s6 * ir2 * L).sum(1)
    err = (f[:, :3].double() - fr).norm(dim=1)
    assert bool((err <= 16 * 2.0 ** -24 * mag + 1e-5 * fr.norm(dim=1)).all())


@pytest.mark.parametrize("n", [769, 1000, 1372, 2500, 4096])
def test_cell_boxes_on_clusters_equal_one_cta(m, n):
    reqs = [dict(rho=0.35 + 0.4 * k, e=m.e_from_temperature(1.2 + 0.3 * k, n), natoms=n - k,
                 steps_equil=40, steps_avg=40, seed=n + k) for k in range(2)]
    with m.Engine(max_cluster=1) as e:
        ref = e.evaluate(reqs)
    assert (ref["status"] == 0).all() and (ref["nlist_builds"] > 2).all()
    for c in (0, 2, 4, 8):
        with m.Engine(max_cluster=c) as e:
            assert e.evaluate(reqs).tobytes() == ref.tobytes(), c
    # a list overflow on a cluster, against the same on one CTA
    with m.Engine(nlist_capacity=16) as a, m.Engine(nlist_capacity=16, max_cluster=1) as b:
        ra, rb = a.evaluate(reqs), b.evaluate(reqs)
    assert (ra["nlist_retries"] > 0).all() and ra.tobytes() == rb.tobytes()


def test_mixed_small_batch_on_clusters(m):
    sizes = [108, 256, 500, 864, 4000]
    reqs = [dict(rho=0.7, e=m.e_from_temperature(1.5, n), natoms=n, steps_equil=30, steps_avg=30,
                 seed=9 + n, element_id=n) for n in sizes]
    cfg = dict(warm_slots=8, warm_atoms=4096)
    with m.Engine(**cfg) as a, m.Engine(max_cluster=1, **cfg) as b:
        for _ in range(2):   # cold, then warm
            ra, rb = a.evaluate(reqs), b.evaluate(reqs)
            assert (ra["status"] == 0).all() and ra.tobytes() == rb.tobytes()
        assert (ra["warm"] == 1).all()


# slabs of one CTA, cluster sizes 1 to 16 and their edges, more zones per CTA than threads,
# and a mesh whose slabs do not fit (the one-CTA kernel)
@pytest.mark.parametrize("nz", [1, 3, 63, 64, 65, 127, 1023, 1025, 20011, 40000])
def test_hydro_slabs_equal_the_oracle_bitwise(m, h, nz):
    o = H.shock_tube(nz, (1.0, 0.1, 1.0), (0.4, 0.0, 0.3), H.IdealGas(5.0 / 3.0))
    cfg = m.mdeos_hydro_config_default(nzones=nz, closure=m.CLOSURE_IDEAL_GAS)
    with m.Hydro(h, cfg, o.x, o.u, o.rho, o.e) as hy:
        for steps in (1, 6):
            hy.step(steps)
            for _ in range(steps):
                o.step()
            s = hy.state()
            for k in ("x", "u", "rho", "e", "P", "q"):
                assert np.array_equal(s[k], getattr(o, k)), (k, steps)
            assert s["t"] == o.t


@pytest.mark.parametrize("n", [1, 2, 63, 127, 128, 129, 257, 640, 4203])
def test_gradients_of_ragged_batches_match_oracle(m, h, n):
    """The bound of the 300-sample gradient test (bf16 roundings one ulp apart), for batches
    around the 128-sample tiles, the K chunks of 64, the split of K and its rings."""
    rng = np.random.default_rng(n)
    p = S.init_params(5, 2).astype(np.float32).astype(np.float64)
    norm = np.array([0.75, -1.0, 0.25, 2.0, 1.5, 1.2, 2.0, 0.6])
    x = np.stack([rng.uniform(0.3, 1.2, n), rng.uniform(-5.0, 3.0, n)], axis=1)
    y = np.stack([x[:, 0] * (x[:, 1] + 3.0), 0.5 * x[:, 1] + 2.0], axis=1)
    with m.Surrogate(h, 2, 4203, seed=1) as sg:
        sg.set_params(p, norm)
        g, loss = sg.grads(x, y)
        g2, _ = sg.grads(x, y)
    assert g.tobytes() == g2.tobytes()
    xn, yn = (x - norm[:2]) / norm[2:4], (y - norm[4:6]) / norm[6:8]
    ls = []
    for e in range(2):
        le, ge = S.loss_and_grad(p[e], xn, yn)
        ls.append(le)
        assert np.linalg.norm(g[e] - ge) <= 2e-2 * np.linalg.norm(ge)
    assert loss == pytest.approx(np.mean(ls), rel=2e-2 if n < 8 else 2e-3)


def test_training_segments_equal_single_steps(m, h):
    """An epoch of 37 batches (three segments, the last one short) equals the same batches
    trained one call at a time."""
    rng = np.random.default_rng(3)
    batch, nb = 64, 37
    x = np.stack([rng.uniform(0.3, 1.2, batch * nb), rng.uniform(-5.0, 3.0, batch * nb)], axis=1)
    y = np.stack([x[:, 0] ** 2, x[:, 1]], axis=1)
    norm = np.array([0.75, -1.0, 0.25, 2.0, 1.5, 1.2, 2.0, 0.6])
    with m.Surrogate(h, 2, batch, seed=4) as a, m.Surrogate(h, 2, batch, seed=4) as b:
        a.set_params(None, norm)
        b.set_params(None, norm)
        a.train(x, y, epochs=1, batch=batch, lr=1e-3, seed=8, set_norm=False)
        pa, _ = a.get_params()
        b.train(x, y, epochs=2, batch=batch, lr=1e-3, seed=8, set_norm=False)
        pb, _ = b.get_params()
        a.train(x, y, epochs=0, batch=batch, lr=1e-3, seed=8, set_norm=False)
        pc, _ = a.get_params()
    assert np.isfinite(pa).all() and not np.array_equal(pa, pb) and np.array_equal(pa, pc)


# one group per CTA, the switches to two and four groups, several tiles per group
@pytest.mark.parametrize("n", [1, 128, 129, 128 * 38, 128 * 38 + 1, 128 * 76 + 1, 128 * 152 + 77,
                               128 * 400 + 3])
def test_inference_groups_give_the_same_outputs(m, h, n):
    """A query's answer does not depend on how many are asked with it."""
    rng = np.random.default_rng(n)
    x = np.stack([rng.uniform(0.3, 1.2, n), rng.uniform(-5.0, 3.0, n)], axis=1)
    norm = np.array([0.75, -1.0, 0.25, 2.0, 1.5, 1.2, 2.0, 0.6])
    with m.Surrogate(h, 4, 1 << 16, seed=2) as big, m.Surrogate(h, 4, 128, seed=2) as one:
        big.set_params(None, norm)
        one.set_params(None, norm)
        mean, sd, pm = big.predict(x, per_model=True)
        k = np.unique(np.r_[0, n // 2, n - 1, rng.integers(0, n, 200)])
        mean1, sd1, pm1 = one.predict(x[k], per_model=True)
    assert np.isfinite(pm).all()
    assert np.array_equal(pm[:, k], pm1) and np.array_equal(mean[k], mean1)
    assert np.array_equal(sd[k], sd1)


def test_cluster_scratch_stays_within_the_budget(m):
    """A budget with room for one CTA's list scratch but not for a cluster's still takes the
    box (on one CTA), with the same answer."""
    q = [dict(rho=0.8, e=m.e_from_temperature(1.5, 4000), natoms=4000, steps_equil=20, steps_avg=20,
              seed=5)]
    budget = 4 << 20
    with m.Engine() as a, m.Engine(hbm_budget_bytes=budget) as b:
        ra, rb = a.evaluate(q), b.evaluate(q)
        assert m.mdeos_stats(a.h)["device_bytes"] > budget >= m.mdeos_stats(b.h)["device_bytes"]
        batch = m.mdeos_batch_create(b.h, q)
        assert m.mdeos_batch_info(batch)["ctas"] == 1
        m.mdeos_batch_destroy(batch)
    assert ra["status"][0] == 0 and ra.tobytes() == rb.tobytes()


@pytest.mark.parametrize("n", [4000, 16000])
def test_budget_halves_the_cluster_until_its_scratch_fits(m, n):
    """A budget with room for 4 (2, 1) list scratches of a box whose default is a cluster of
    8 plans 4 (2, 1) CTAs, not one."""
    q = [dict(rho=0.8, e=m.e_from_temperature(1.5, n), natoms=n, steps_equil=20, steps_avg=20,
              seed=5)]
    with m.Engine() as a:
        base = m.mdeos_stats(a.h)["device_bytes"]
        b = m.mdeos_batch_create(a.h, q)
        info = m.mdeos_batch_info(b)
        m.mdeos_batch_destroy(b)
    assert info["ctas"] == 8
    per = info["scratch_bytes"] // 8
    for ctas in (8, 4, 2, 1):
        # the tables of one request take far less than half a scratch
        with m.Engine(hbm_budget_bytes=base + ctas * per + per // 2) as a:
            b = m.mdeos_batch_create(a.h, q)
            got = m.mdeos_batch_info(b)["ctas"]
            m.mdeos_batch_destroy(b)
        assert got == ctas


def test_cluster_scratch_gives_way_to_later_calls(m):
    """After a box has run on a cluster of 8 whose list scratch fills the budget, a batch of
    many boxes (large tables) and a device-resident batch still get their room, and the box
    runs again with the same answer."""
    q = [dict(rho=0.8, e=m.e_from_temperature(1.5, 4000), natoms=4000, steps_equil=20, steps_avg=20,
              seed=5)]
    many = [dict(rho=0.3, e=m.e_from_temperature(1.5, 32), natoms=32, steps_equil=2, steps_avg=2,
                 seed=k) for k in range(4000)]
    with m.Engine() as a:
        base = m.mdeos_stats(a.h)["device_bytes"]
        ref = a.evaluate(q)
        per = (m.mdeos_stats(a.h)["device_bytes"] - base) // 8
        rmany = a.evaluate(many)
    with m.Engine(hbm_budget_bytes=base + 8 * per + per // 2) as a:
        assert a.evaluate(q).tobytes() == ref.tobytes()
        assert m.mdeos_stats(a.h)["device_bytes"] >= base + 8 * per
        assert a.evaluate(many).tobytes() == rmany.tobytes()
        assert a.evaluate(q).tobytes() == ref.tobytes()
        b = m.mdeos_batch_create(a.h, q + q)
        m.mdeos_batch_launch(b)
        assert m.mdeos_batch_results(b, 2)[:1].tobytes() == ref.tobytes()
        assert m.mdeos_stats(a.h)["device_bytes"] <= base + 8 * per + per // 2
        m.mdeos_batch_destroy(b)
        assert a.evaluate(q).tobytes() == ref.tobytes()
