"""J/K of the classes that run in integer arithmetic against the oracle.

The classes with the fixed-point Eq. 1 assembly (s, p and d shells in more than one
lane per quartet): batches of one primitive quartet, batches that do not
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


def _check(m, tol=1e-12, plan=None):
    plan = plan or pkg.Plan(m, tau=0.0)
    J, K = plan.jk(torch.from_numpy(m.D).cuda())
    Jr, Kr, _ = oracle.jk(m, tau=0.0)
    for got, ref in ((J, Jr), (K, Kr)):
        assert np.abs(got.cpu().numpy() - ref).max() <= tol * np.abs(ref).max()


# The one-lane classes' integer scalars: one centre (P = Q, T = 0), the large-T limit (centres far
# apart: every T above the table), extents that shift the unit of P, exponents over eight decades,
# and an exponent outside the integers' range, which keeps FP64 kernels.  Tolerance as above.
@pytest.mark.parametrize("dist,exps", [
    (0.0, (0.2, 1.1)),
    (1.3, (0.15, 1.2, 40.0, 2e3, 5e7)),
    (45.0, (0.3, 6.0)),
    (900.0, (0.4,)),
    (1.1, (0.3, 2.0, 1e-31)),
])
def test_jk_integer_scalars(dist, exps):
    rng = np.random.default_rng(int(dist * 10) + len(exps))
    axis = np.array([0.48, -0.6, 0.64])
    shells = [(a, l, np.array(exps), rng.uniform(0.2, 1.0, len(exps))) for a in (0, 1) for l in (0, 1)]
    shells += [(0, 2, np.array(exps[:1]), np.ones(1)), (1, 3, np.array(exps[-1:]), np.ones(1))]
    m = custom_molecule(np.array([[0.1, 0.2, -0.3], axis * dist + [0.1, 0.2, -0.3]]), shells)
    m.D = random_psd_density(m.nbf, max(2, m.nbf // 3), rng, 1)
    _check(m)


def test_batch_with_a_plan_outside_the_integer_range():
    rng = np.random.default_rng(3)
    mols, plans = [], []
    for top in (4.0, 1e-31):
        m = custom_molecule(rng.uniform(-1, 1, (2, 3)), [(a, l, np.array([0.4, top]), np.array([0.7, 0.4]))
                                                         for a in (0, 1) for l in (0, 1)])
        m.D = random_psd_density(m.nbf, 2, rng, 1)
        mols.append(m)
        plans.append(pkg.Plan(m, tau=0.0))
    Js, Ks = pkg.Batch().jk(plans, [torch.from_numpy(m.D).cuda() for m in mols])
    for m, J, K in zip(mols, Js, Ks):
        Jr, Kr, _ = oracle.jk(m, tau=0.0)
        for got, ref in ((J, Jr), (K, Kr)):
            assert np.abs(got.cpu().numpy() - ref).max() <= 1e-12 * np.abs(ref).max()


def _uncontracted(coords, shells, D):
    """The molecule of the shells' primitives, and D (of s and p functions) in its functions."""
    prims, cols, n = [], [], 0
    for a, l, e, c in shells:
        S = (2.0 * np.sqrt(np.outer(e, e)) / np.add.outer(e, e)) ** (l + 1.5)
        w = c / np.sqrt(c @ S @ c)
        for comp in range(2 * l + 1):
            cols.append({n + k * (2 * l + 1) + comp: w[k] for k in range(len(e))})
        prims += [(a, l, e[k:k + 1], np.ones(1)) for k in range(len(e))]
        n += len(e) * (2 * l + 1)
    C = np.zeros((n, len(cols)))
    for j, col in enumerate(cols):
        for i, v in col.items():
            C[i, j] = v
    return custom_molecule(coords, prims), np.ascontiguousarray(C @ D @ C.T)


# Classes with quartets enough to fill the grid, a few of them deep (6^4 primitive quartets among
# quartets of one): the deep ones are split over primitive ranges, the shallow ones have ranges
# without a primitive.  ns s1 shells and np_ p1 shells around one s6 and one p6 shell; the
# tolerance as above, of the gradient as in its own tests.
@pytest.mark.parametrize("ns,np_", [(24, 13), (30, 2)])
def test_deep_quartets_in_a_full_grid(ns, np_):
    rng = np.random.default_rng(ns)
    coords = rng.uniform(-2, 2, (6, 3))
    one = lambda l, a: (a, l, rng.uniform(0.2, 2.0, 1), np.ones(1))  # noqa: E731
    shells = [one(0, i % 6) for i in range(ns)] + [one(1, i % 6) for i in range(np_)]
    deep = 0.15 * 4.0 ** np.arange(6)
    shells += [(1, 0, deep, rng.uniform(0.1, 0.6, 6)), (4, 1, deep, rng.uniform(0.1, 0.6, 6))]
    shells.sort(key=lambda s: s[0])
    m = custom_molecule(coords, shells)
    m.D = random_psd_density(m.nbf, 5, rng, 1)
    _check(m)
    # the gradient against that of the same density in the primitives as shells of their own, where
    # no quartet is deep
    got = pkg.Plan(m, tau=0.0).jk_grad(torch.from_numpy(m.D[0]).cuda())
    u, D = _uncontracted(coords, shells, m.D[0])
    for g, r in zip(got, pkg.Plan(u, tau=0.0).jk_grad(torch.from_numpy(D).cuda())):
        assert (g - r).abs().max() <= 1e-10 * max(1.0, float(r.abs().max()))
