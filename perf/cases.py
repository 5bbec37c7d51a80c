"""What this framework is measured on: integral-direct J/K builds and gradients as its users run them.

A case is one call on one molecule (or one batch of molecules): the molecule recipe and its size,
the number of densities, the precision, which matrices are wanted and the entry point
(`variant` numbers molecules of one recipe and size).  The recipes are the repository's own
synthetic ones (jittered 1.8 A lattice, even-tempered shells):

  tiny    2s1p per atom, three primitives each, atoms in a box (a small molecule, latency bound)
  medium  3s2p1d per atom, contraction depths 1..6 (6-31G(d)-like, deeply contracted)
  scf     30 % heavy 3s2p1d / 70 % light 2s1p atoms, depths 6 3 1 | 3 1 | 1 and 3 1 | 1
  high_l  one s, p, d, f and g shell per atom, depths 1..3 (cc-pVTZ-like, extended to g)
"""

import math
import types

import numpy as np
import torch

import paper_2407_09700_gb300 as pkg

BOHR = 1.0 / 0.529177210903
TAU = 1e-12
GRAD, JK, J_ONLY, K_ONLY = "grad", "jk", "j", "k"


def _case(name, recipe, natm, what=JK, nD=1, mixed=False, entry="device", njobs=1, change=False, variant=0):
    return {"name": name, "recipe": recipe, "natm": natm, "what": what, "nD": nD, "mixed": mixed, "entry": entry,
            "njobs": njobs, "change": change, "variant": variant}


def listed():
    return [
        # the smallest call: one Fock build of a three-atom molecule, where launches and latency count
        _case("tiny", "tiny", 3),
        # alpha and beta densities of an open-shell small molecule (UHF)
        _case("medium_5_uhf", "medium", 5, nD=2),
        # the ordinary deeply contracted build, and the same in the mixed precision mode
        _case("medium_16", "medium", 16),
        _case("medium_13_mixed", "medium", 13, mixed=True),
        # one SCF iteration's build with mostly shallow shells, from host buffers to host buffers
        _case("scf_33_host", "scf", 33, entry="host"),
        # a later iteration of an incremental SCF in the mixed mode: J, K of a density change
        _case("scf_41_mixed_change", "scf", 41, mixed=True, change=True),
        # Coulomb alone, as a density functional without exact exchange asks for
        _case("scf_27_coulomb", "scf", 27, what=J_ONLY),
        # f and g shells: the largest classes
        _case("high_l_12", "high_l", 12),
        # a serving tick: several small molecules in one batched call
        _case("serve_batch_9", "scf", 11, mixed=True, entry="batch", njobs=9),
        # energy gradients: a geometry step of a small, a contracted and a high angular momentum molecule
        _case("scf_5_grad", "scf", 5, what=GRAD, variant=4),
        _case("medium_8_grad", "medium", 8, what=GRAD),
        _case("high_l_4_grad", "high_l", 4, what=GRAD),
    ]


# (recipe, what, entry, most atoms): the kinds of call, each over its whole range of sizes
_KINDS = [("medium", JK, "device", 16), ("scf", JK, "device", 41), ("scf", JK, "host", 33), ("high_l", JK, "device", 12),
          ("scf", JK, "batch", 12), ("scf", J_ONLY, "device", 33), ("scf", K_ONLY, "device", 27),
          ("medium", GRAD, "device", 8), ("scf", GRAD, "device", 16), ("high_l", GRAD, "device", 4)]


def draw(rng):
    recipe, what, entry, most = rng.choice(_KINDS)
    natm = int(round(math.exp(rng.uniform(math.log(2), math.log(most)))))
    nD = 1 if what == GRAD or natm > most // 2 else rng.choice([1, 1, 2, 3])
    c = _case("", recipe, natm, what, nD, what != GRAD and rng.random() < 0.4, entry,
              rng.randint(2, 12) if entry == "batch" else 1, what != GRAD and rng.random() < 0.25, rng.randrange(1, 1000))
    del c["name"]
    return c


# ---------------------------------------------------------------- molecules and densities

def _molecule(recipe, natm, kind, rng):
    """`kind` draws what the molecule is made of (elements, contraction depths), `rng` the rest."""
    if recipe == "tiny":
        while True:
            coords = rng.uniform(0.0, 3.0, (natm, 3))
            d = np.linalg.norm(coords[:, None] - coords[None], axis=-1) + 9.0 * np.eye(natm)
            if d.min() >= 0.9:
                break
    else:
        m = 1
        while m ** 3 < natm:
            m += 1
        sites = np.array([(i, j, k) for i in range(m) for j in range(m) for k in range(m)][:natm], dtype=np.float64)
        coords = sites * 1.8 + rng.uniform(-0.2, 0.2, (natm, 3))
    atom, ls, nprim, off, exps, coefs = [], [], [], [], [], []
    for a in range(natm):
        if recipe == "tiny":
            shells, beta = [(0, 3), (0, 3), (1, 3)], 3.0
        elif recipe == "medium":
            shells, beta = [(l, int(kind.integers(1, 7))) for l in (0, 0, 0, 1, 1, 2)], 2.5
        elif recipe == "scf":
            heavy = kind.uniform() < 0.3
            shells, beta = [(0, 6), (0, 3), (0, 1), (1, 3), (1, 1), (2, 1)] if heavy else [(0, 3), (0, 1), (1, 1)], 2.5
        else:
            shells, beta = [(l, int(kind.integers(1, 4))) for l in range(5)], 2.2
        for l, K in shells:
            a0 = 0.15 if recipe == "high_l" else rng.uniform(0.1, 0.3)
            atom.append(a)
            ls.append(l)
            nprim.append(K)
            off.append(len(exps))
            exps.extend(a0 * beta ** np.arange(K))
            coefs.extend(rng.uniform(0.1, 1.0, K))
    i32 = lambda v: np.asarray(v, dtype=np.int32)  # noqa: E731
    return types.SimpleNamespace(coords=coords * BOHR, shell_atom=i32(atom), shell_l=i32(ls), shell_nprim=i32(nprim),
                                 shell_off=i32(off), exps=np.asarray(exps), coefs=np.asarray(coefs),
                                 nbf=sum((l + 1) * (l + 2) // 2 for l in ls))


def _density(nbf, nD, change, rng):
    """Positive semidefinite densities of about a third of the functions occupied, or (change) the
    small symmetric difference of two of them."""
    out = []
    for _ in range(nD):
        C = rng.standard_normal((nbf, max(1, nbf // 3))) / math.sqrt(nbf)
        D = C @ C.T
        if change:
            C1 = C + 1e-3 / math.sqrt(nbf) * rng.standard_normal(C.shape)
            D = C1 @ C1.T - D
            D = 0.5 * (D + D.T)
        out.append(D)
    return np.stack(out)


def _jobs(case, seed):
    kind = np.random.default_rng([case["natm"], case["njobs"], case["variant"]])
    rng = np.random.default_rng([int(seed), case["natm"], case["njobs"], case["variant"]])
    jobs = []
    for _ in range(case["njobs"]):
        # the molecules of a batch differ in size, up to the case's
        natm = case["natm"] if case["njobs"] == 1 else int(kind.integers(max(1, case["natm"] // 2), case["natm"] + 1))
        mol = _molecule(case["recipe"], natm, kind, rng)
        jobs.append((mol, _density(mol.nbf, case["nD"], case["change"], rng)))
    return jobs


def prepare(case, seed):
    jobs = _jobs(case, seed)
    prec = pkg.ERI_MIXED if case["mixed"] else pkg.ERI_FP64
    state = {"case": case, "plans": [pkg.Plan(mol, tau=TAU, precision=prec) for mol, _ in jobs]}
    if case["entry"] == "host":
        state["D"] = [D for _, D in jobs]
    else:
        state["D"] = [torch.from_numpy(D).cuda() for _, D in jobs]
    if case["entry"] == "batch":
        state["batch"] = pkg.Batch()
    if case["what"] == GRAD:
        state["D"] = [D[0].contiguous() for D in state["D"]]
    return state


_WANT = {JK: pkg.ERI_WANT_J | pkg.ERI_WANT_K, J_ONLY: pkg.ERI_WANT_J, K_ONLY: pkg.ERI_WANT_K}


def run(state):
    case, plans, D = state["case"], state["plans"], state["D"]
    if case["what"] == GRAD:
        return plans[0].jk_grad(D[0])
    want = _WANT[case["what"]]
    if case["entry"] == "batch":
        return state["batch"].jk(plans, D, want=want)
    J, K = plans[0].jk_host(D[0], want=want) if case["entry"] == "host" else plans[0].jk(D[0], want=want)
    return [x for x, w in ((J, pkg.ERI_WANT_J), (K, pkg.ERI_WANT_K)) if want & w]


# ---------------------------------------------------------------- the work a pass cannot do without

def _ncart(l):
    return (l + 1) * (l + 2) // 2


def work(case):
    """Arithmetic of the Rys quadrature of every unique shell quartet of overlapping pairs (one multiply-add
    per root and contracted [e0|f0] value, 28 operations per root for roots and weights) and of
    its digestion; the matrices and the pair data once."""
    flops = bytes_ = 0.0
    grad = case["what"] == GRAD
    for mol, D in _jobs(case, 0):
        nsh = len(mol.shell_l)
        amin = np.array([mol.exps[o] for o in mol.shell_off])
        pairs = {}
        for i in range(nsh):
            for j in range(i + 1):
                ab = mol.coords[mol.shell_atom[i]] - mol.coords[mol.shell_atom[j]]
                if amin[i] * amin[j] / (amin[i] + amin[j]) * float(ab @ ab) > 28.0:
                    continue
                key = tuple(sorted((int(mol.shell_l[i]), int(mol.shell_l[j])), reverse=True))
                n, p = pairs.get(key, (0, 0))
                pairs[key] = (n + 1, p + int(mol.shell_nprim[i]) * int(mol.shell_nprim[j]))
        wants = {JK: 6, J_ONLY: 2, K_ONLY: 4, GRAD: 6}[case["what"]]
        for (la, lb), (n1, p1) in pairs.items():
            for (lc, ld), (n2, p2) in pairs.items():
                L = la + lb + lc + ld + (1 if grad else 0)
                ne = sum(_ncart(l) for l in range(la, la + lb + 1))
                nf = sum(_ncart(l) for l in range(lc, lc + ld + 1))
                nabcd = _ncart(la) * _ncart(lb) * _ncart(lc) * _ncart(ld)
                N = L // 2 + 1
                flops += 0.5 * p1 * p2 * N * (28 + 2 * ne * nf * (3 if grad else 1))
                flops += 0.5 * n1 * n2 * 2 * wants * nabcd * case["nD"]
        mats = 2 if case["what"] in (J_ONLY, K_ONLY) else 1 if grad else 3
        bytes_ += 8.0 * mats * D.size + 80.0 * sum(p for _, p in pairs.values()) + 64.0 * sum(n for n, _ in pairs.values())
    return {"bytes": bytes_, "flops": flops}


# ---------------------------------------------------------------- 64-bit values by plain torch

_GL_X, _GL_W = np.polynomial.legendre.leggauss(32)


def _cart(l):
    return [(x, y, l - x - y) for x in range(l, -1, -1) for y in range(l - x, -1, -1)]


def _normalised(mol):
    c = np.array(mol.coefs, dtype=np.float64)
    for l, K, o in zip(mol.shell_l, mol.shell_nprim, mol.shell_off):
        l, a = int(l), mol.exps[o:o + K]
        df = float(np.prod(np.arange(2 * l - 1, 0, -2))) if l else 1.0
        v = c[o:o + K] * (2 * a / math.pi) ** 0.75 * (4 * a) ** (0.5 * l) / math.sqrt(df)
        s = a[:, None] + a[None]
        c[o:o + K] = v / math.sqrt(float((np.outer(v, v) * df / (2 * s) ** l * (math.pi / s) ** 1.5).sum()))
    return c


def _pair_groups(mol, dev):
    """Canonical shell pairs (larger l first) by type, as index and primitive tensors."""
    c, l, o = _normalised(mol), mol.shell_l, mol.shell_off
    bf = np.concatenate([[0], np.cumsum([_ncart(int(x)) for x in l])])
    groups = {}
    for i in range(len(l)):
        for j in range(i + 1):
            a, b = (i, j) if l[i] >= l[j] else (j, i)
            g = groups.setdefault((int(l[a]), int(l[b])), {"at": [], "bf": [], "f": [], "sp": [], "al": [], "be": [], "cc": []})
            k = len(g["f"])
            g["at"].append((mol.shell_atom[a], mol.shell_atom[b]))
            g["bf"].append((bf[a], bf[b]))
            g["f"].append(1.0 if i == j else 2.0)
            ab = mol.coords[mol.shell_atom[a]] - mol.coords[mol.shell_atom[b]]
            for u in range(o[a], o[a] + mol.shell_nprim[a]):
                for v in range(o[b], o[b] + mol.shell_nprim[b]):
                    x, y = mol.exps[u], mol.exps[v]
                    if x * y / (x + y) * float(ab @ ab) < 69.0:  # the rest is below 1e-30
                        g["sp"].append(k)
                        g["al"].append(x)
                        g["be"].append(y)
                        g["cc"].append(c[u] * c[v])
    for g in groups.values():
        for key in ("f", "al", "be", "cc"):
            g[key] = torch.tensor(np.array(g[key]), dtype=torch.float64, device=dev)
        for key in ("at", "bf", "sp"):
            g[key] = torch.tensor(np.array(g[key]), dtype=torch.int64, device=dev)
    return groups


def _geometry(g, coords, p0, p1):
    """zeta, P - A, A - B, A and the prefactor of a range of a group's primitive pairs."""
    at = g["at"][g["sp"][p0:p1]]
    A, B = coords[at[:, 0]], coords[at[:, 1]]
    al, be = g["al"][p0:p1], g["be"][p0:p1]
    z = al + be
    AB = A - B
    E = g["cc"][p0:p1] * torch.exp(-al * be / z * (AB * AB).sum(1)) / z
    return z, -(be / z)[:, None] * AB, AB, A, E


def _axis_tables(x, Le, Lf, la, lb, lc, ld, C, Cp, B00, B10, B01, AB, CD):
    """{(a, b, c, d): 1D integral} of one axis by recurrence on (n, 0 | m, 0) and transfer to (a, b | c, d)."""
    t = {(0, 0): torch.ones_like(B00)}
    for n in range(Le):
        t[n + 1, 0] = C * t[n, 0] + (n * B10 * t[n - 1, 0] if n else 0.0)
    for m in range(Lf):
        for n in range(Le + 1):
            t[n, m + 1] = Cp * t[n, m] + (n * B00 * t[n - 1, m] if n else 0.0) + (m * B01 * t[n, m - 1] if m else 0.0)
    h = {(n, 0, m): t[n, m] for n in range(Le + 1) for m in range(Lf + 1)}
    for b in range(lb):
        for a in range(Le - b):
            for m in range(Lf + 1):
                h[a, b + 1, m] = h[a + 1, b, m] + AB * h[a, b, m]
    out = {}
    for a in range(la + 1):
        for b in range(lb + 1):
            k = {(m, 0): h[a, b, m] for m in range(Lf + 1)}
            for d in range(ld):
                for c in range(Lf - d):
                    k[c, d + 1] = k[c + 1, d] + CD * k[c, d]
            for c in range(lc + 1):
                for d in range(ld + 1):
                    out[a, b, c, d] = k[c, d]
    return out


def _block(gx, lx, gy, ly, coords, b0, b1, k0, k1):
    """Contributions of primitive pairs [b0, b1) x [k0, k1) to the blocks (ab|cd) of two groups'
    shell pairs, [pairs, pairs, n_a n_b, n_c n_d]: Gauss-Legendre quadrature over t in [0, 1] of the
    Gaussian transform of 1/r, cut where exp(-T t^2) is below 1e-18."""
    (la, lb), (lc, ld) = lx, ly
    z, PA, AB, A, Eb = _geometry(gx, coords, b0, b1)
    e, QC, CD, C, Ek = _geometry(gy, coords, k0, k1)
    dev = z.device
    node = torch.tensor(0.5 * (_GL_X + 1.0), device=dev)
    wt = torch.tensor(0.5 * _GL_W, device=dev)
    z2, e2 = z[:, None, None], e[None, :, None]
    s = z2 + e2
    PQ = (A + PA)[:, None] - (C + QC)[None]
    T = (z2 * e2 / s)[..., 0] * (PQ * PQ).sum(2)
    top = torch.clamp(6.4 / torch.sqrt(torch.clamp(T.detach(), min=1e-30)), max=1.0)[..., None]
    u = (top * node) ** 2
    w = top * wt * torch.exp(-T[..., None] * u) * (2.0 * math.pi ** 2.5 / torch.sqrt(s)) * Eb[:, None, None] * Ek[None, :, None]
    B00, B10, B01 = 0.5 * u / s, 0.5 / z2 * (1.0 - u * e2 / s), 0.5 / e2 * (1.0 - u * z2 / s)
    ax = []
    for x in range(3):
        d = PQ[:, :, x, None]
        ax.append(_axis_tables(x, la + lb, lc + ld, la, lb, lc, ld, PA[:, None, x, None] - u * e2 / s * d,
                               QC[None, :, x, None] + u * z2 / s * d, B00, B10, B01, AB[:, None, x, None], CD[None, :, x, None]))
    ab = [(a, b) for a in _cart(la) for b in _cart(lb)]
    cd = [(c, d) for c in _cart(lc) for d in _cart(ld)]
    zw = {k: v * w for k, v in ax[2].items()}
    xy = {}
    vals = []
    for a, b in ab:
        for c, d in cd:
            k = tuple((a[x], b[x], c[x], d[x]) for x in range(3))
            if k[:2] not in xy:
                xy[k[:2]] = ax[0][k[0]] * ax[1][k[1]]
            vals.append((xy[k[:2]] * zw[k[2]]).sum(-1))
    V = torch.stack(vals, -1)
    out = torch.zeros((len(gx["f"]), V.shape[1], V.shape[2]), dtype=torch.float64, device=dev).index_add(0, gx["sp"][b0:b1], V)
    out = torch.zeros((len(gx["f"]), len(gy["f"]), V.shape[2]), dtype=torch.float64, device=dev).index_add(1, gy["sp"][k0:k1], out)
    return out.reshape(len(gx["f"]), len(gy["f"]), len(ab), len(cd))


def _d_blocks(D, ga, ia, na, gb, ib, nb):
    """[pairs, pairs, n, m] blocks of D between shell ia of group ga's pairs and shell ib of gb's."""
    r = ga["bf"][:, ia, None] + torch.arange(na, device=D.device)
    c = gb["bf"][:, ib, None] + torch.arange(nb, device=D.device)
    return D[r[:, None, :, None], c[None, :, None, :]]


def _pair_blocks(D, g, n0, n1):
    r = g["bf"][:, 0, None] + torch.arange(n0, device=D.device)
    c = g["bf"][:, 1, None] + torch.arange(n1, device=D.device)
    return D[r[:, :, None], c[:, None, :]].reshape(len(g["f"]), n0 * n1)


def _energies(mol, coords, D, groups, grads_of):
    """Gradients of E_J = 1/2 sum (ab|cd) D_ab D_cd and E_K = -1/4 sum (ab|cd) D_ac D_bd with respect
    to `grads_of` (the coordinates or D), range of primitive pairs by range."""
    gJ, gK = torch.zeros_like(grads_of), torch.zeros_like(grads_of)
    keys = sorted(groups)
    for x in keys:
        for y in keys:
            if y > x:
                continue
            gx, gy = groups[x], groups[y]
            na, nb, nc, nd = (_ncart(v) for v in x + y)
            tables = (x[0] + 1) * (x[1] + 1) * (y[0] + 1) * (y[1] + 1)
            vals = 32 * (na * nb * nc * nd + 6 * tables + 20) * (3 if coords.requires_grad else 1)
            nx, ny = len(gx["sp"]), len(gy["sp"])
            step_k = max(1, min(ny, 1024))
            step_b = max(1, min(nx, int(1.2e9 / vals / step_k)))
            if step_b == 1:
                step_k = max(1, min(ny, int(1.2e9 / vals)))
            f = (1.0 if x == y else 2.0) * gx["f"][:, None] * gy["f"][None]
            V = 0.0
            for b0 in range(0, nx, step_b):
                for k0 in range(0, ny, step_k):
                    v = _block(gx, x, gy, y, coords, b0, min(nx, b0 + step_b), k0, min(ny, k0 + step_k))
                    if coords.requires_grad:
                        for g, e in zip((gJ, gK), _contract(v, D, f, gx, gy, na, nb, nc, nd)):
                            g += torch.autograd.grad(e, grads_of, retain_graph=g is gJ)[0]
                    else:
                        V = V + v
            if not coords.requires_grad:
                for g, e in zip((gJ, gK), _contract(V, D, f, gx, gy, na, nb, nc, nd)):
                    g += torch.autograd.grad(e, grads_of, retain_graph=g is gJ)[0]
    return gJ, gK


def _contract(V, D, f, gx, gy, na, nb, nc, nd):
    Dab, Dcd = _pair_blocks(D, gx, na, nb), _pair_blocks(D, gy, nc, nd)
    eJ = 0.5 * torch.einsum("pq,pqxy,px,qy->", f, V, Dab, Dcd)
    V6 = V.reshape(V.shape[0], V.shape[1], na, nb, nc, nd)
    Dac, Dbd = _d_blocks(D, gx, 0, na, gy, 0, nc), _d_blocks(D, gx, 1, nb, gy, 1, nd)
    Dad, Dbc = _d_blocks(D, gx, 0, na, gy, 1, nd), _d_blocks(D, gx, 1, nb, gy, 0, nc)
    k1 = torch.einsum("pqabcd,pqac,pqbd->pq", V6, Dac, Dbd)
    k2 = torch.einsum("pqabcd,pqad,pqbc->pq", V6, Dad, Dbc)
    return eJ, -0.125 * (f * (k1 + k2)).sum()


def _exact_cost(mol, grad):
    """Quadrature values of _block over all primitive pairs, about."""
    per = {}
    for i in range(len(mol.shell_l)):
        for j in range(i + 1):
            k = tuple(sorted((int(mol.shell_l[i]), int(mol.shell_l[j]))))
            per[k] = per.get(k, 0) + int(mol.shell_nprim[i]) * int(mol.shell_nprim[j])
    t = sum(p * math.prod(_ncart(l) for l in k) for k, p in per.items())
    return 32.0 * 0.5 * t * t * (8 if grad else 1)


def exact(case, seed):
    jobs = _jobs(case, seed)
    grad = case["what"] == GRAD
    if sum(_exact_cost(mol, grad) for mol, _ in jobs) * max(1, case["nD"] // 2) > 4e10:
        return None
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    Js, Ks = [], []
    for mol, D in jobs:
        groups = _pair_groups(mol, dev)
        Dt = torch.tensor(D, device=dev)
        coords = torch.tensor(mol.coords, device=dev)
        if grad:
            coords.requires_grad_(True)
            return _energies(mol, coords, Dt[0], groups, coords)
        J, K = [], []
        for Dx in Dt:
            Dx = Dx.clone().requires_grad_(True)
            gJ, gK = _energies(mol, coords, Dx, groups, Dx)
            J.append(0.5 * (gJ + gJ.T))
            K.append(-(gK + gK.T))
        Js.append(torch.stack(J))
        Ks.append(torch.stack(K))
    if case["entry"] == "batch":
        return Js, Ks
    return [v[0] for v, what in ((Js, (JK, J_ONLY)), (Ks, (JK, K_ONLY))) if case["what"] in what]
