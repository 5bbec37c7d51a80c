"""Which kernel the FP64 launches of a class take at the ends of the integer kernels' ranges, by the
launch records, and J / K on both sides of each limit against the oracle."""

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


def _jk(m, **opts):
    """J, K of both densities and {class: kernel} of the FP64 launches."""
    plan = pkg.Plan(m, tau=0.0, **opts)
    plan.set_profiling(True)
    J, K = plan.jk(torch.from_numpy(m.D).cuda())
    kern = {(r["la"], r["lb"], r["lc"], r["ld"]): r["kernel"] for r in plan.launch_records() if not r["fp32"]}
    return J.cpu().numpy(), K.cpu().numpy(), kern


def _spd(d_exps, seed):
    """Two atoms with s, p and d shells, the d shells with the given exponents, and the shells."""
    rng = np.random.default_rng(seed)
    e = np.array([0.2, 1.1, 6.0])
    shells = [(a, l, e, rng.uniform(0.2, 1.0, 3)) for a in (0, 1) for l in (0, 1)]
    shells += [(a, 2, np.array(d_exps), rng.uniform(0.2, 1.0, len(d_exps))) for a in (0, 1)]
    shells.sort(key=lambda s: s[0])
    m = custom_molecule(rng.uniform(-1.2, 1.2, (2, 3)), shells)
    m.D = random_psd_density(m.nbf, m.nbf // 3, rng, 1)
    return m, shells


def _primitives(m, shells, D):
    """The molecule of the shells' primitives, D in its functions, and the contraction."""
    prims, cols, n = [], [], 0
    for a, l, e, c in shells:
        S = (2.0 * np.sqrt(np.outer(e, e)) / np.add.outer(e, e)) ** (l + 1.5)
        w, nc = c / np.sqrt(c @ S @ c), (l + 1) * (l + 2) // 2
        cols += [{n + k * nc + i: w[k] for k in range(len(e))} for i in range(nc)]
        prims += [(a, l, e[k:k + 1], np.ones(1)) for k in range(len(e))]
        n += len(e) * nc
    C = np.zeros((n, len(cols)))
    for j, col in enumerate(cols):
        for i, v in col.items():
            C[i, j] = v
    u = custom_molecule(m.coords, prims)
    u.D = np.ascontiguousarray(C @ D @ C.T)
    return u, C


# A (dd| pair spans 2 log2(largest / smallest exponent) binades: 13.3 and 19.9 are fixed point, 20.2 FP64; in a
# mixed plan, unsorted, 13.9 and 14.2.  The reference takes the primitives as shells of their own, where no scale
# is shared: against 128-bit sums the oracle is 1.2e-13 off here and FP64 sums 2.6e-14, the fixed-point sums
# 6.5e-15 at most (they claim FP64's accuracy or better), so both sides' within 2e-14 of the largest element.
# FP64 kernels: 1e-12, as elsewhere against the oracle.
@pytest.mark.parametrize("ratio,mixed,kernel", [(100.0, False, "fixed"), (1000.0, False, "fixed"), (1100.0, False, "class"),
                                                (124.0, True, "fixed"), (138.0, True, "class")])
def test_spread_of_a_shells_exponents(ratio, mixed, kernel):
    m, shells = _spd(0.12 * np.array([1.0, ratio ** 0.4, ratio]), int(ratio))
    # a mixed plan whose quartets all run FP64: its launches keep the primitives' order
    J, K, kern = _jk(m, **(dict(precision=pkg.ERI_MIXED, mixed_thresh=0.0, mixed_min_tasks=0) if mixed else {}))
    for c in ((2, 2, 1, 1), (2, 2, 2, 0), (2, 2, 2, 1), (2, 2, 2, 2)):
        assert kern[c] == kernel
    assert kern[2, 1, 2, 1] == "fixed"          # the (dp| pairs span fewer
    u, C = _primitives(m, shells, m.D)
    for got, ref in zip((J, K), _jk(u)):
        ref = C.T @ ref @ C
        assert np.abs(got - ref).max() <= (2e-14 if kernel == "fixed" else 1e-12) * np.abs(ref).max()


# The one-lane integer kernel: up to zeta |P - Q|^2 = 2^17 for (dp| and (fs| pairs, any for the others; positions in
# units of 2^-52 bohr, which a box above 128 bohr leaves; exponents within 1e-18 .. 1e18.
@pytest.mark.parametrize("zeta,R,ps,dp", [(1e3, 8.0, "small_fx", "small_fx"), (2e3, 8.0, "small_fx", "small"),
                                          (1.0, 120.0, "small_fx", "small_fx"), (1.0, 130.0, "small", "small"),
                                          (1e19, 1.0, "small", None)])
def test_range_of_the_integer_kernel(zeta, R, ps, dp):
    one = np.ones(1)
    m = custom_molecule(np.array([[0.0, 0, 0], [R, 0, 0]]),
                        [(a, l, np.array([zeta]), one) for a in (0, 1) for l in ((0, 1, 2) if dp else (0, 1))])
    m.D = random_psd_density(m.nbf, 3, np.random.default_rng(1), 2)
    J, K, kern = _jk(m)
    assert all(kern[c] == ps for c in ((0, 0, 0, 0), (1, 0, 0, 0), (1, 0, 1, 0)))
    if dp:
        assert kern[2, 0, 0, 0] == ps and kern[2, 1, 0, 0] == dp and kern[2, 1, 1, 0] == dp
    Jr, Kr, _ = oracle.jk(m, tau=0.0)
    for got, ref in ((J, Jr), (K, Kr)):
        assert np.abs(got - ref).max() <= 2e-14 * np.abs(ref).max()


# A contracted core s shell (exponents up to 2e4) beside an f shell counts as its diffuse primitives: the integer
# kernel serves it, and the dipole (px s| and (fxxx s| in the field of an s function 8 bohr away, where P = A is
# exact in the oracle too, are as close as those of single exponents.
def test_contracted_core_stays_in_integers():
    core = np.array([2e4, 3e3, 600.0, 150.0, 40.0, 10.0])
    one = np.ones(1)
    m = custom_molecule(np.array([[0.0, 0, 0], [8.0, 0, 0]]),
                        [(0, 0, core, np.array([0.002, 0.015, 0.07, 0.22, 0.47, 0.36])),
                         (0, 1, np.array([8.0, 2.0]), np.array([0.4, 0.7])), (0, 3, np.array([1.5]), one),
                         (1, 0, np.array([0.5]), one)])
    m.D = np.zeros((1, m.nbf, m.nbf))
    m.D[0, -1, -1] = 1.0
    J, _, kern = _jk(m)
    assert kern[3, 0, 0, 0] == "small_fx" and kern[3, 0, 1, 0] == "small_fx"
    Jr, _, _ = oracle.jk(m, tau=0.0)
    for at in ((0, 0), (0, 1), (1, 1), (0, 4)):
        assert abs(J[0][at] / Jr[0][at] - 1) <= 8e-15
