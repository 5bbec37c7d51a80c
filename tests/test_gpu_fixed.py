"""J/K of the classes with the fixed-point Eq. 1 assembly (s, p and d shells in more than one
lane per quartet) against the oracle: batches of one primitive quartet, batches that do not
divide the primitive quartets, and exponents over many binades (one scale per batch and table
entry must hold tight and diffuse primitives together)."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import paper_2407_09700_gb300 as pkg  # noqa: E402
from oracle import oracle  # noqa: E402
from workloads import custom_molecule, random_psd_density  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pkg.build()


# Every quartet is off by at most 2^-57 of a batch's largest product (2^-48 with products 2^9
# above the sum they cancel to) and FP64 sums of 1e4..1e5 of them by 1e-13 of the largest
# element, as are the oracle's: 1e-12 of it bounds both.
@pytest.mark.parametrize("depths,beta,spread", [
    ((1,), 2.5, 1.5),          # one primitive quartet per batch
    ((2, 3), 2.5, 3.0),        # ragged batches
    ((1, 7), 2.5, 1.2),        # up to 2 401 primitive quartets per quartet
    ((5, 4), 8.0, 2.0),        # exponents 0.12 .. 500
    ((3,), 40.0, 0.0),         # one centre, exponents 0.12 .. 200
])
def test_jk_fixed_point_classes(depths, beta, spread):
    rng = np.random.default_rng(len(depths) + int(10 * beta))
    coords = rng.uniform(-spread, spread, (2, 3)) if spread else np.zeros((1, 3))
    shells, k = [], 0
    for a in range(len(coords)):
        for l in (0, 1, 2):
            K = depths[k % len(depths)]
            k += 1
            shells.append((a, l, 0.12 * beta ** np.arange(K), rng.uniform(0.1, 1.0, K)))
    m = custom_molecule(coords, shells)
    m.D = random_psd_density(m.nbf, max(2, m.nbf // 3), rng, 2)
    plan = pkg.Plan(m, tau=0.0)
    J, K = plan.jk(torch.from_numpy(m.D).cuda())
    Jr, Kr, _ = oracle.jk(m, tau=0.0)
    for got, ref in ((J, Jr), (K, Kr)):
        assert np.abs(got.cpu().numpy() - ref).max() <= 1e-12 * np.abs(ref).max()
