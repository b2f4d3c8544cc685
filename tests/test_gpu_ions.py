"""The ion-list tile (kmc_ions.cu) against the oracle, bit for bit, at the sizes
where its shapes change: lanes per rail follow from the number of rails and of
ions, 32 rows of bits end at 32 entries a lane, and open rails grow, shrink and
have their entries dealt out again."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kmc():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2511_09413_gb300 import build, kmc as K
    build.build()
    K.load()
    torch.cuda.init()
    return K


def _dev(**kw):
    d = dict(R=48, L=100, Z=10, electrodes=0, d=1.0, dt=5e-7, T=300.0, Ea=0.40, nu=1e12,
             alpha=0.2, kappa=1.0, k_e=0.0, rho_e=0.0, seed=33, instance=2)
    d.update(kw)
    return d


def _check(K, dev, V, fill, chunks, Ea=None):
    occ0 = oracle.init_occupancy(dev, 1, fill=fill)
    sim = K.Sim(dev, V, 2, occ0=occ0, Ea_site=Ea)
    orc = oracle.OracleSim(dev, V, occ0, Ea)
    for c in chunks:
        sim.step_n(c)
    n = sum(chunks)
    Jo, Zo = orc.step_n(n)
    Jg, Zg = sim.traces()
    assert np.array_equal(Zg, Zo), "zone-count traces differ"
    assert np.array_equal(Jg, Jo), "current traces differ"
    assert np.array_equal(sim.occupancy(), orc.occ), "occupancy differs"
    assert np.array_equal(sim.rail_current(), orc.J_rail), "per-rail current differs"
    sim.close()


# (rails, sites): 4, 8, 16 and 32 lanes per rail, each at the last number of
# sites whose full rails fit 32 rows and one beyond, the fewest sites, and 64 rows
@pytest.mark.parametrize("R,L", [(49153, 8), (19201, 128), (19201, 129), (24001, 256), (24001, 257),
                                 (12289, 512), (12289, 513), (300, 1024), (300, 1025), (64, 2048)])
@pytest.mark.parametrize("electrodes", [0, 1])
@pytest.mark.parametrize("dt", [5e-7, 2e-8])
def test_shapes_of_the_lists(kmc, R, L, electrodes, dt):
    Z = min(L, 10 if R % 2 else 32)
    k = 1.0 / dt if electrodes else 0.0
    dev = _dev(R=R, L=L, Z=Z, electrodes=electrodes, k_e=k, rho_e=0.3, dt=dt)
    n = 7 if R * L > 1000000 else 40
    V = np.where(np.arange(n) % 6 < 3, 1.0, -0.5)
    _check(kmc, dev, V, 0.25, [n // 3, n - n // 3])


# either side of the lines between the occupancy words and the lists for few sites and
# zones on many rails
@pytest.mark.parametrize("R,L,Z", [(40001, 16, 2), (40001, 16, 3), (40001, 33, 2), (40001, 33, 3), (40001, 23, 8),
                                   (40001, 23, 9), (4001, 12, 3), (20001, 17, 2)])
@pytest.mark.parametrize("electrodes", [0, 1])
@pytest.mark.parametrize("dt", [5e-7, 2e-8])
def test_few_sites_on_many_rails(kmc, R, L, Z, electrodes, dt):
    dev = _dev(R=R, L=L, Z=Z, electrodes=electrodes, k_e=1.0 / dt if electrodes else 0.0, rho_e=0.3, dt=dt)
    _check(kmc, dev, np.where(np.arange(24) % 6 < 3, 1.0, -0.5), 0.3, [9, 15])


# per-site barriers where several rails share a warp (4, 8 and 16 lanes a rail), with
# and without classes of sites in the bounds' rows
@pytest.mark.parametrize("R,L", [(49153, 64), (19201, 100), (12289, 300), (6001, 500)])
@pytest.mark.parametrize("Z", [10, 32])
@pytest.mark.parametrize("electrodes", [0, 1])
@pytest.mark.parametrize("dt", [5e-7, 2e-8])
def test_per_site_barriers_on_few_lanes(kmc, R, L, Z, electrodes, dt):
    dev = _dev(R=R, L=L, Z=Z, electrodes=electrodes, k_e=1.0 / dt if electrodes else 0.0, rho_e=0.3, dt=dt)
    Ea = np.maximum(np.random.default_rng(L).normal(0.40, 0.02, (R, L)), 0.35)
    _check(kmc, dev, np.where(np.arange(20) % 6 < 3, 1.0, -0.5), 0.25, [5, 15], Ea)


# more than 32 entries a lane: CTAs of up to 20 warps, in one wave and in several,
# each with a last CTA that is not full
@pytest.mark.parametrize("R,L,fill", [(2500, 2048, 0.5), (5001, 1100, 0.25)])
@pytest.mark.parametrize("dt", [5e-7, 2e-8])
def test_wide_ctas(kmc, R, L, fill, dt):
    dev = _dev(R=R, L=L, Z=32, electrodes=1, k_e=1.0 / dt, rho_e=0.3, dt=dt)
    _check(kmc, dev, np.where(np.arange(9) % 6 < 3, 1.0, -0.5), fill, [4, 5])


# open rails that fill up from empty, drain from half full, and swap their ions
# at a high rate: entries come and go at both ends
@pytest.mark.parametrize("L", [8, 33, 64, 200])
@pytest.mark.parametrize("fill,rho", [(0.0, 0.95), (0.4, 0.0), (0.3, 0.5)])
@pytest.mark.parametrize("rule", [0, 1])
def test_open_rails_grow_and_shrink(kmc, L, fill, rho, rule):
    dev = _dev(R=70, L=L, Z=min(L, 7), electrodes=1, k_e=4e6, rho_e=rho, dt=2e-6, rule=rule)
    V = 2.0 * np.sin(np.arange(500) / 40.0)
    _check(kmc, dev, V, fill, [500])


# rare moves: four steps drawn at once, ions that move and exchanges in between,
# launches and voltage jumps that end inside the four.  kappa sets how many moves
# the decision bounds hold for (3: exchanges count as well; 300: none is left);
# barriers of a wide spread fill every class of sites
@pytest.mark.parametrize("L,Z", [(8, 8), (33, 1), (100, 10), (777, 32)])
@pytest.mark.parametrize("electrodes", [0, 1])
@pytest.mark.parametrize("kappa", [1.0, 3.0, 300.0])
@pytest.mark.parametrize("spread,rule", [(None, 0), (0.06, 0), (0.06, 1), (None, 1)])
def test_rare_moves(kmc, L, Z, electrodes, kappa, spread, rule):
    dev = _dev(R=45, L=L, Z=Z, electrodes=electrodes, k_e=2e7 if electrodes else 0.0, rho_e=0.4, dt=1e-8,
               kappa=kappa, rule=rule)
    Ea = None if spread is None else np.maximum(np.random.default_rng(L).normal(0.40, spread, (45, L)), 0.30)
    V = np.where(np.arange(603) % 150 < 71, 1.0, -0.5) + 1e-3 * np.sin(np.arange(603))
    _check(kmc, dev, V, 0.3, [1, 2, 3, 261, 336], Ea)


# a voltage that moves within a window, by 0.01 to 1 of the exponent in a step, with
# jumps beside it: wide bounds without the accept path, windows that end inside the
# steps drawn ahead
@pytest.mark.parametrize("L,Z", [(8, 8), (33, 1), (100, 10), (777, 32)])
@pytest.mark.parametrize("electrodes", [0, 1])
@pytest.mark.parametrize("dt", [5e-7, 1e-8])
@pytest.mark.parametrize("spread", [None, 0.03])
def test_fast_voltage(kmc, L, Z, electrodes, dt, spread):
    dev = _dev(R=45, L=L, Z=Z, electrodes=electrodes, k_e=0.2 / dt if electrodes else 0.0, rho_e=0.4, dt=dt)
    Ea = None if spread is None else np.maximum(np.random.default_rng(L).normal(0.40, spread, (45, L)), 0.36)
    n = np.arange(400)
    V = np.where(n % 97 < 50, 1.0, -1.0) * 0.02 * L * np.abs(np.sin(n / (3.0 + 20.0 * (n > 200))))
    _check(kmc, dev, V, 0.3, [7, 150, 243], Ea)


# rails that share a warp are taken in the order of their ion counts: empty, full
# and uneven ones, with places beyond the last rail, and a count per rail that must
# come back at the rail's own index
@pytest.mark.parametrize("R", [1023, 1024, 1025, 4099])
@pytest.mark.parametrize("electrodes", [0, 1])
@pytest.mark.parametrize("dt", [5e-7, 2e-8])
def test_uneven_rails(kmc, R, electrodes, dt):
    L = 75
    dev = _dev(R=R, L=L, electrodes=electrodes, k_e=1.0 / dt if electrodes else 0.0, rho_e=0.3, dt=dt)
    rng = np.random.default_rng(R)
    share = rng.choice([0.0, 0.02, 0.2, 0.5, 1.0], size=R, p=[0.1, 0.3, 0.4, 0.15, 0.05])
    occ0 = (rng.random((R, L)) < share[:, None]).astype(np.uint8)
    V = np.where(np.arange(40) % 6 < 3, 1.0, -0.5)
    sim = kmc.Sim(dev, V, 2, occ0=occ0)
    orc = oracle.OracleSim(dev, V, occ0, None)
    sim.step_n(40)
    Jo, Zo = orc.step_n(40)
    Jg, Zg = sim.traces()
    assert np.array_equal(Zg, Zo) and np.array_equal(Jg, Jo)
    assert np.array_equal(sim.occupancy(), orc.occ)
    assert np.array_equal(sim.rail_current(), orc.J_rail)
    sim.close()


# launches of a few steps run on the occupancy words, longer ones on the lists
@pytest.mark.parametrize("R,L,chunks", [(1200, 300, [1, 2, 3, 4, 17, 1]), (10001, 256, [1, 5, 1, 3]),
                                        (32768, 1024, [1, 16, 3])])
@pytest.mark.parametrize("electrodes", [0, 1])
@pytest.mark.parametrize("dt", [5e-7, 2e-8])
def test_launches_of_few_steps(kmc, R, L, chunks, electrodes, dt):
    dev = _dev(R=R, L=L, electrodes=electrodes, k_e=1.0 / dt if electrodes else 0.0, rho_e=0.3, dt=dt)
    _check(kmc, dev, np.where(np.arange(sum(chunks)) % 6 < 3, 1.0, -0.5), 0.25, chunks)


# long launches look at the rails first: ions in one block at an end, rails that are
# full or empty, random ones, and rails whose filling changes between two launches
@pytest.mark.parametrize("start", ["block", "uneven", "random", "filling"])
@pytest.mark.parametrize("dt", [5e-7, 1e-8])
def test_long_launches_choose_their_tile(kmc, start, dt):
    R, L, n = 16385, 512, 240
    open_ = start == "filling"
    dev = _dev(R=R, L=L, kappa=0.0 if start == "block" else 1.0, electrodes=int(open_), k_e=1.0 / dt, rho_e=1.0, dt=dt)
    occ0 = np.zeros((R, L), np.uint8)
    rng = np.random.default_rng(3)
    if start == "block":
        occ0[:, :200] = 1
    elif start == "uneven":
        occ0[: R // 2] = 1
    else:
        occ0[:] = rng.random((R, L)) < (0.5 if open_ else 0.3)
    V = np.full(2 * n, 10.0)
    sim = kmc.Sim(dev, V, 2, occ0=occ0)
    orc = oracle.OracleSim(dev, V, occ0, None)
    for _ in range(2):
        sim.step_n(n)
    Jo, Zo = orc.step_n(2 * n)
    Jg, Zg = sim.traces()
    assert np.array_equal(Zg, Zo) and np.array_equal(Jg, Jo)
    assert np.array_equal(sim.occupancy(), orc.occ)
    assert np.array_equal(sim.rail_current(), orc.J_rail)
    sim.close()


# a batch chooses its tiles from all rails together: the same devices alone
# and together give the same results, lists and words side by side
def test_batch_of_lists_and_words(kmc):
    devs, fills = [], []
    for i, (R, L, f, e) in enumerate([(30000, 40, 0.2, 0), (20000, 130, 0.3, 1), (9000, 300, 0.25, 0),
                                      (500, 1500, 0.2, 1), (3000, 100, 0.9, 0), (4000, 4, 0.4, 0),
                                      (200, 900, 0.1, 0)]):
        devs.append(_dev(R=R, L=L, Z=min(L, 10), electrodes=e, k_e=1e6 if e else 0.0, rho_e=f, instance=i))
        fills.append(f)
    V = np.where(np.arange(48) % 20 < 9, 0.8, 0.0)
    b = kmc.Batch(devs, [V] * len(devs), [1] * len(devs), fills=fills)
    b.set_launch(8, 16)
    b.step_n(40)
    for i, (d, f) in enumerate(zip(devs, fills)):
        s = kmc.Sim(d, V, 1, fill=f)
        s.step_n(40)
        for x, y in zip((*b.traces(i), b.occupancy(i), b.rail_current(i)),
                        (*s.traces(), s.occupancy(), s.rail_current())):
            assert np.array_equal(x, y)
        s.close()
    b.close()
