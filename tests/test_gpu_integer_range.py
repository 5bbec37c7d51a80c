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
    """J of an s and a p shell at the origin in the field of an s function at (R, 0, 0): (ss|ss),
    (px s|ss), (px px|ss) and the values of their multipoles (T = zeta R^2 far above 40, so
    exponentially small terms are left out)."""
    one = np.ones(1)
    m = custom_molecule(np.array([[0.0, 0, 0], [R, 0, 0]]),
                        [(0, 0, np.array([zeta]), one), (0, 1, np.array([zeta]), one), (1, 0, np.array([zeta]), one)])
    D = np.zeros((1, m.nbf, m.nbf))
    D[0, -1, -1] = 1.0
    J, _ = pkg.Plan(m, tau=0.0).jk(torch.from_numpy(D).cuda())
    J = J.cpu().numpy()[0]
    mu, q = 0.5 / np.sqrt(zeta), 0.25 / zeta      # <s|x|px>; <px|x^2|px> - <px|y^2|px> is 2 q
    return np.array([J[0, 0], J[0, 1], J[1, 1]]), np.array([1 / R, mu / R ** 2, 1 / R + 2 * q / R ** 3])


# Weights of the large-T limit carry 60 bits relative to 1 / sqrt(T) and everything else about 20
# FP64 roundings (normalisation, prefactors, J): 20 * 2^-53 = 2.2e-15.
@pytest.mark.parametrize("zeta", [1e2, 1e4, 1e6, 1e8, 1e10, 1e12, 1e16])
def test_repulsion_of_tight_shells(zeta):
    got, want = _separated(zeta)
    assert abs(got[0] / want[0] - 1) <= 4e-15
    assert abs(got[2] / want[2] - 1) <= 4e-15


# (ps|ss), a dipole's repulsion, is about 1 / sqrt(zeta R^2) of the unit its C is held in; a few units of
# 2^-60 leave 2^-57.6 sqrt(zeta R^2), 1.7e-15 at the largest zeta R^2 that the integers take (2^17, between
# 1e3 and 2e3 here), beside the roundings of the other elements: twice the sum of both.
@pytest.mark.parametrize("zeta", [1e2, 1e3, 2e3, 1e4, 1e6, 1e8, 1e12])
def test_dipole_of_tight_shells(zeta):
    got, want = _separated(zeta)
    assert abs(got[1] / want[1] - 1) <= 8e-15
