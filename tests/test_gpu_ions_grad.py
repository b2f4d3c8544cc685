"""The gradient pass on ion lists against the oracle's estimator, on 4, 8, 16 and
32 lanes per rail (which follow from the number of rails), at the edges of 32 and
64 rows of bits, with ragged rails and lanes without ions."""
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


# tolerances of tests/test_gpu_grad.py: the same FP64 sums in another order
@pytest.mark.parametrize("R,L,Z,fill", [(9601, 40, 7, 0.3), (9601, 253, 10, 0.2), (9601, 300, 10, 0.55),
                                        (5001, 130, 32, 0.25), (2403, 520, 10, 0.3), (40, 8, 3, 0.02),
                                        (40, 1040, 10, 0.6)])
@pytest.mark.parametrize("electrodes", [0, 1])
def test_gradient_on_lists(kmc, R, L, Z, fill, electrodes):
    dev = dict(R=R, L=L, Z=Z, electrodes=electrodes, d=1.0, dt=5e-7, T=300.0, Ea=0.40, nu=1e12, alpha=0.4,
               kappa=1.0, k_e=1e6 if electrodes else 0.0, rho_e=0.4 if electrodes else 0.0, seed=5, instance=1)
    n = 14 if R > 1000 else 120
    V = np.where(np.arange(n) % 10 < 6, 1.2, 0.0)
    rng = np.random.default_rng(R + L)
    wJ, wZ = rng.normal(size=n), rng.normal(size=(n, Z))
    sim = kmc.Sim(dev, V, 1, fill=fill)
    sim.step_n(n)
    occ0 = oracle.init_occupancy(dev, 1, fill=fill)
    for a, b in [(wJ, wZ), (None, wZ), (wJ, None)]:
        g, se = sim.grad(a, b)
        ref = oracle.lr_gradient(dev, V, occ0, n, wJ=a, wZ=b, fill=fill)
        scale = np.abs(ref["G"]).sum(axis=0)
        assert np.all(np.abs(g - ref["grad"]) <= 1e-11 * scale + 1e-10 * np.abs(ref["grad"]))
        np.testing.assert_allclose(se, ref["stderr"], rtol=1e-8)
    sim.close()


# either side of the lines between the occupancy words and the lists
@pytest.mark.parametrize("R,L,Z", [(5001, 100, 4), (5001, 100, 5), (20001, 30, 3), (20001, 30, 4), (40001, 60, 10)])
@pytest.mark.parametrize("electrodes", [0, 1])
def test_gradient_of_few_sites_on_many_rails(kmc, R, L, Z, electrodes):
    test_gradient_on_lists(kmc, R, L, Z, 0.2, electrodes)
