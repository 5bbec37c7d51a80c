"""Rounding of the gradient's sums over the ranges of split quartets."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import paper_2407_09700_gb300 as pkg  # noqa: E402
from workloads import custom_molecule, random_psd_density  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pkg.build()


# The order of the atomic additions changes from call to call, so the spread of equal calls shows what they
# round away.  With quartets in one task each and one copy of the gradient it is up to 1.5e-15 on such
# molecules; ranges of split quartets must not leave more.
@pytest.mark.parametrize("seed", range(4))
def test_equal_calls_agree(seed):
    rng = np.random.default_rng(seed)
    coords = rng.uniform(-2, 2, (4, 3))
    shells = [(a, l, 0.2 * 2.5 ** np.arange(K), rng.uniform(0.1, 1.0, K))
              for a in range(4) for l, K in ((0, 6), (0, 3), (1, 3), (1, 1))]
    m = custom_molecule(coords, shells)
    D = torch.from_numpy(random_psd_density(m.nbf, m.nbf // 3, rng, 1)[0]).cuda()
    plan = pkg.Plan(m, tau=0.0)
    g = torch.stack([torch.stack(plan.jk_grad(D)) for _ in range(16)])
    mean = g.mean(0)
    for k in (0, 1):                            # gJ, gK
        assert max(float((x[k] - mean[k]).norm()) for x in g) <= 1.5e-15 * float(mean[k].norm())
