"""Element-wise accuracy of the integer kernels at the ends of their range.

J, K and gradients of a molecule are dominated by its largest integrals, so the tests here look
at single elements whose values are known: shells far apart, where the repulsion of two
s functions is 1 / R."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import paper_2407_09700_gb300 as pkg  # noqa: E402
from workloads import custom_molecule  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pkg.build()


def _separated(zeta, R=8.0):
    """J of an s and a p shell at the origin in the field of an s function, and of a px s and a py s
    product, at (R, 0, 0): (ss|ss), (px s|ss), (px px|ss), (px s|px s), (py s|py s) and the values of their
    multipoles (T = zeta R^2 far above 40, so exponentially small terms are left out)."""
    one = np.ones(1)
    m = custom_molecule(np.array([[0.0, 0, 0], [R, 0, 0]]),
                        [(a, l, np.array([zeta]), one) for a in (0, 1) for l in (0, 1)])
    D = np.zeros((3, m.nbf, m.nbf))
    D[0, 4, 4] = 1.0
    D[1, 4, 5] = D[1, 5, 4] = D[2, 4, 6] = D[2, 6, 4] = 0.5
    J = pkg.Plan(m, tau=0.0).jk(torch.from_numpy(D).cuda())[0].cpu().numpy()
    mu, q = 0.5 / np.sqrt(zeta), 0.25 / zeta      # <s|x|px>; <px|x^2|px> - <px|y^2|px> is 2 q
    return (np.array([J[0, 0, 0], J[0, 0, 1], J[0, 1, 1], J[1, 0, 1], J[2, 0, 2]]),
            np.array([1 / R, mu / R ** 2, 1 / R + 2 * q / R ** 3, -2 * mu ** 2 / R ** 3, mu ** 2 / R ** 3]))


# Weights of the large-T limit carry 60 bits relative to 1 / sqrt(T) and everything else about 20
# FP64 roundings (normalisation, prefactors, J): 20 * 2^-53 = 2.2e-15.
@pytest.mark.parametrize("zeta", [1e2, 1e4, 1e6, 1e8, 1e10, 1e12, 1e16])
def test_repulsion_of_tight_shells(zeta):
    got, want = _separated(zeta)
    assert abs(got[0] / want[0] - 1) <= 4e-15
    assert abs(got[2] / want[2] - 1) <= 4e-15


# (ps|ss), a dipole's repulsion, is about 1 / sqrt(zeta R^2) of the pair's extent and (ps|ps) 1 / (zeta R^2): their C
# and the term of both sides are held in units of their own size, so the bound is that of the other
# elements, doubled for the second C.
@pytest.mark.parametrize("zeta", [10.0, 1e2, 1e3, 2e3, 1e4, 1e6, 1e8, 1e12])
def test_dipole_of_tight_shells(zeta):
    got, want = _separated(zeta)
    for k in (1, 3, 4):
        assert abs(got[k] / want[k] - 1) <= 8e-15


def _cluster(far, rng):
    """Three atoms with s, p and d shells near the origin and an s function at (far, 0, 0); the
    cluster's blocks of J and K and its gradients, of a density of its own."""
    coords = np.vstack([rng.uniform(-1.5, 1.5, (3, 3)), [[far, 0.0, 0.0]]])
    e = np.array([0.3, 1.9, 11.0])
    m = custom_molecule(coords, [(a, l, e, np.ones(3)) for a in range(3) for l in (0, 1, 2)] + [(3, 0, e[:1], e[:1])])
    C = rng.standard_normal((m.nbf - 1, 4)) / 5
    D = np.zeros((m.nbf, m.nbf))
    D[:-1, :-1] = C @ C.T
    D = torch.from_numpy(D).cuda()
    plan = pkg.Plan(m, tau=0.0)
    J, K = plan.jk(D)
    return [x.cpu().numpy()[:-1, :-1] for x in (J, K)] + [g.cpu().numpy()[:3] for g in plan.jk_grad(D)]


# A far atom leaves the cluster's values as they are; the bound is that of the sums' own roundings
# (about 1e4 atomic additions: sqrt(1e4) 2^-53 = 1.1e-14 of the largest element, 2e-15 in practice;
# gradients cancel to a quarter of their parts).
@pytest.mark.parametrize("far", [60.0, 300.0, 1e3, 1e5, 1e9, 1e15])
def test_cluster_with_an_atom_far_away(far):
    for got, ref, tol in zip(_cluster(far, np.random.default_rng(3)), _cluster(30.0, np.random.default_rng(3)),
                             (1.1e-14, 1.1e-14, 4.4e-14, 4.4e-14)):
        assert np.abs(got - ref).max() <= tol * np.abs(ref).max()


# FP32 launches (a threshold that takes every quartet): T = 1e40, where u would leave FP32's range, positions in
# coarse units, and the large-T limit; each block of the first atom in the field of the second's s
# function by its own size, FP32 sums to 1e-5.
@pytest.mark.parametrize("zeta,R", [(1e22, 1e9), (3.0, 1e7), (1e10, 8.0)])
def test_mixed_at_the_ends_of_fp32(zeta, R):
    got, ref = _mixed_and_fp64(zeta, R, R)
    s0, p0 = slice(0, 1), slice(1, 4)
    for rows, cols in ((s0, s0), (s0, p0), (p0, p0)):
        g, r = got[rows, cols], ref[rows, cols]
        assert (g - r).abs().max() <= 1e-5 * r.abs().max()


# Centres 1e-30 bohr apart, where the positions' unit would leave it: as for one centre.
def test_mixed_of_nearly_coincident_centres():
    got, ref = _mixed_and_fp64(1.0, 1e-30, 0.0)
    assert (got - ref).abs().max() <= 1e-5 * ref.abs().max()


def _mixed_and_fp64(zeta, R, R64):
    one, J = np.ones(1), []
    for r, opts in ((R, dict(precision=pkg.ERI_MIXED, mixed_thresh=1e300, mixed_min_tasks=0)), (R64, {})):
        m = custom_molecule(np.array([[0.0, 0, 0], [r, 0, 0]]),
                            [(a, l, np.array([zeta]), one) for a in (0, 1) for l in (0, 1)])
        D = np.zeros((m.nbf, m.nbf))
        D[-4, -4] = 1.0                           # the second atom's s function
        J.append(pkg.Plan(m, tau=0.0, **opts).jk(torch.from_numpy(D).cuda())[0])
    return J
