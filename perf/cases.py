"""The work that users of this framework have it do, case by case.

A user holds a periodic cell, its basis and an SCF density, keeps one plan
per geometry and calls the build again and again: a J+K build per iteration
of a hybrid-functional SCF loop (with the reciprocal cache switched on while
the geometry stays), a J build alone for a semilocal functional, one build
per frame of a trajectory, FP64 builds to verify the mixed path, the
one-electron operators once per geometry, the energies once per iteration,
and small requests side by side through the request server.

The cells are those of ``synthcells``: the tiny cell, small skewed cells with
s, p and d shells, boxes of 1 to 64 water molecules at the density of the
64-molecule box, and diamond supercells with d shells.  A seed stands for one
frame: every atom is displaced by a Gaussian step of 0.02 bohr, and the
occupied orbitals are orthonormalised Gaussian vectors, so the density has
the rank and the norm of a closed-shell one.
"""
import math

import numpy as np
import torch

import synthcells as sc
from paper_2410_22278_gb300 import jk

PRECISION = {"fp64": jk.JK_FP64, "mixed": jk.JK_MIXED}
EDGE3 = 29.94  # cubic angstrom per water molecule (12.42^3 / 64)
SMALL = (1, 5, 8, 9)  # the small cells drawn: skewed (odd) or cubic (even), exponents of their own


def _case(name, kind, cell, size, precision="mixed", k=True, cache=False, variant=1, omega=0.0):
    return {"name": name, "kind": kind, "cell": cell, "size": size, "precision": precision, "k": k, "cache": cache,
            "variant": variant, "omega": omega}


def listed():
    return [
        # the smallest call: 8 basis functions, every step in FP64, where launches and latency count
        _case("tiny_fp64", "jk", "tiny", 2, "fp64"),
        # a small skewed (non-orthogonal) cell with s, p and d shells, every step in FP64
        _case("skew2_fp64", "jk", "small", 2, "fp64"),
        # an SCF iteration of a small molecular crystal: reciprocal data kept, latency counts
        _case("water5_scf", "jk", "water", 5, cache=True),
        # a verification build in FP64 of a small box
        _case("water6_fp64", "jk", "water", 6, "fp64"),
        # an SCF iteration of one conventional diamond cell (s, p and d shells)
        _case("diamond8_scf", "jk", "diamond", 1, cache=True),
        # the steady state of a hybrid SCF loop: geometry kept, a new density each iteration
        _case("water31_scf", "jk", "water", 31, cache=True),
        # the benchmark's box as one frame of a trajectory: every geometry is new, J and K
        _case("water64_frame", "jk", "water", 64),
        # the same box for a semilocal functional: J alone
        _case("water64_j", "jk", "water", 64, k=False),
        # a diamond supercell with d shells (704 basis functions), J and K
        _case("diamond64_mixed", "jk", "diamond", 2),
        # kinetic energy and nuclear attraction, once per geometry
        _case("water27_onee", "onee", "water", 27),
        # E_J and E_K of one iteration from matrices on the device
        _case("water64_energy", "energy", "water", 64),
        # four small requests side by side through the request server
        _case("serve_small", "serve", "water", 9),
    ]


def draw(rng):
    kind = rng.choice(["jk", "jk", "jk", "jk", "jk", "jk", "onee", "energy", "serve"])
    cell = rng.choice(["water", "water", "water", "small", "small", "diamond", "tiny"])
    precision = rng.choice(["mixed", "mixed", "mixed", "fp64"])
    if kind == "serve":
        cell, precision = "water", "mixed"
    size = {"tiny": 2, "small": rng.randint(1, 2), "diamond": rng.choice([1, 1, 2]),
            "water": int(round(math.exp(rng.uniform(0.0, math.log(63.0)))))}[cell]
    if kind == "serve":
        size = min(size, 12)
    if cell == "diamond" and kind == "jk":
        precision = "mixed"
    if kind == "jk" and precision == "fp64":  # FP64 is for small cells: its rate is 1/74 of FP32's here
        size = min(size, 7)
    k = kind != "jk" or rng.random() < 0.75
    cache = kind == "jk" and rng.random() < 0.5 and not (cell == "water" and size > 40)
    omega = {"tiny": round(rng.uniform(0.4, 0.6), 3), "small": round(rng.uniform(0.5, 0.8), 3),
             "diamond": round(rng.uniform(0.4, 0.6), 3), "water": round(rng.uniform(0.38, 0.45), 3)}[cell]
    c = _case("", kind, cell, size, precision, k, cache, rng.choice(SMALL), omega)
    del c["name"]
    return c


def _cell(case):
    size, omega = case["size"], case["omega"]
    if case["cell"] == "tiny":
        c = sc.tiny_cell()
    elif case["cell"] == "small":
        c = sc.small_random_cell(case["variant"], natom=size, lmax=2, skew=case["variant"] % 2 == 1)
    elif case["cell"] == "diamond":
        c = sc.diamond_cell(size)
    else:
        c = sc.water_cell(size, (EDGE3 * size) ** (1.0 / 3.0), n_occ=4 * size)
    if omega > 0:
        c.omega = omega
    return c


def _frame(case, seed):
    """The cell of one frame and its seeded orbital guess."""
    c = _cell(case)
    rng = np.random.default_rng([seed & 0x7FFFFFFF, 2410])
    step = 0.02 * rng.standard_normal(c.positions.shape)
    atom = {tuple(r): i for i, r in enumerate(c.positions)}
    for s in c.shells:
        s.center = s.center + step[atom[tuple(s.center)]]
    c.positions = c.positions + step
    return c, rng.standard_normal((c.nbf, c.n_occ)), rng


def _density(X, S):
    """D = 2 C C^T with C^T S C = 1, from the guess X."""
    X = torch.as_tensor(X, device=S.device)
    M = X.T @ S @ X
    Li = torch.linalg.cholesky(0.5 * (M + M.T))
    C = torch.linalg.solve_triangular(Li, X.T, upper=False)
    D = 2.0 * C.T @ C
    return 0.5 * (D + D.T).contiguous()


def _stream():
    return torch.cuda.current_stream().cuda_stream


def _plan_and_density(cell, X, precision):
    plan = jk.plan_from_cell(cell, precision=PRECISION[precision])
    S = torch.empty((cell.nbf, cell.nbf), dtype=torch.float64, device="cuda")
    plan.overlap(S.data_ptr(), _stream())
    return plan, _density(X, S)


def _matrices(rng, n):
    """Symmetric stand-ins for J and K on the device (the energies' inputs)."""
    A = torch.as_tensor(rng.standard_normal((n, n)), device="cuda")
    return (A @ A.T / n).contiguous(), (A + A.T).contiguous()


def prepare(case, seed):
    if case["kind"] == "serve":
        # four requests of different sizes with plans of their own, and one server with as many slots
        work = []
        for i in range(4):
            cell, X, _ = _frame(dict(case, size=max(1, case["size"] - 2 * i)), seed + 1000003 * i)
            plan, D = _plan_and_density(cell, X, case["precision"])
            work.append((plan, D, torch.empty_like(D), torch.empty_like(D)))
        torch.cuda.synchronize()
        return {"kind": "serve", "work": work, "server": jk.Server(device=0, hbm_budget_bytes=64 << 30, max_slots=4)}
    cell, X, rng = _frame(case, seed)
    plan, D = _plan_and_density(cell, X, case["precision"])
    s = {"kind": case["kind"], "plan": plan, "D": D, "J": torch.empty_like(D), "K": torch.empty_like(D), "want_k": case["k"]}
    if case["kind"] == "jk" and case["cache"]:
        plan.cache(1 << 38)
    if case["kind"] == "onee":
        s["Z"], s["xyz"] = sc.nuclear_charges(cell), cell.positions
    if case["kind"] == "energy":
        s["J"], s["K"] = _matrices(rng, cell.nbf)
    return s


def run(state):
    if state["kind"] == "serve":
        srv = state["server"]
        tickets = [srv.submit(p, D.data_ptr(), J.data_ptr(), K.data_ptr()) for p, D, J, K in state["work"]]
        for t in tickets:
            status, _ = srv.wait(t)
            if status != 0:
                raise RuntimeError("build status %d" % status)
        return [[J, K] for _, _, J, K in state["work"]]
    plan, D, J, K = state["plan"], state["D"], state["J"], state["K"]
    if state["kind"] == "onee":
        plan.one_electron(state["Z"], state["xyz"], J.data_ptr(), K.data_ptr(), _stream())
        return {"T": J, "V": K}
    if state["kind"] == "energy":
        ej, ek = plan.energy(D.data_ptr(), J.data_ptr(), K.data_ptr(), _stream())
        return {"EJ": ej, "EK": ek}
    plan.build(D.data_ptr(), J.data_ptr(), K.data_ptr() if state["want_k"] else 0, _stream())
    return {"J": J, "K": K} if state["want_k"] else {"J": J}


def work(case):
    """Matrices read and written once; of the flops the reciprocal part (structure factors of every local pair and G
    unless the user keeps them, the Coulomb contraction over one triangle, and the exchange in its low-rank form).  The
    real-space quartets come on top: their number is known only after the screening, so it is not in here."""
    if case["kind"] == "serve":
        parts = [work(dict(case, kind="jk", size=max(1, case["size"] - 2 * i))) for i in range(4)]
        return {key: sum(p[key] for p in parts) for key in ("bytes", "flops")}
    c = _cell(case)
    n, r = c.nbf, c.n_occ
    if case["kind"] == "energy":
        return {"bytes": 3 * 8.0 * n * n, "flops": 4.0 * n * n}
    _, _, local, _, n_g = jk.pair_counts(c.lattice, c.shells, c.omega, c.cutoffs)
    sfac = 20.0 * (local / 2) * n_g
    if case["kind"] == "onee":
        return {"bytes": 2 * 8.0 * n * n, "flops": sfac + 2.0 * n * n * n_g}
    flops = (0.0 if case["cache"] else sfac) + 4.0 * n * n * n_g + (6.0 * n * n * r * n_g if case["k"] else 0.0)
    return {"bytes": (3 if case["k"] else 2) * 8.0 * n * n, "flops": flops}


# ---- the same numbers on a plane-wave grid, in plain torch -------------------------------------------------------------
# The cells with modest exponents (tiny, small: at most 20) have smooth pair densities: their periodic Coulomb and exchange
# integrals without the K = 0 term are sums over the reciprocal lattice of a uniform grid, exact to rounding once the grid
# resolves the narrowest product.

def _cartesians(l):
    return [(x, y, l - x - y) for x in range(l, -1, -1) for y in range(l - x, -1, -1)]


def _grid(cell):
    """Basis functions on the grid, the Coulomb kernel and |G|^2 of its reciprocal lattice."""
    dev = "cuda"
    L = np.asarray(cell.lattice, dtype=np.float64)
    amax = max(float(s.exps.max()) for s in cell.shells)
    gm = math.sqrt(8.0 * amax * 36.0)
    ns = []
    for a in L:
        m = int(math.ceil(gm * np.linalg.norm(a) / math.pi))
        ns.append(m + (-m) % 4)
    f = [torch.arange(m, dtype=torch.float64, device=dev) / m for m in ns]
    F = torch.stack(torch.meshgrid(*f, indexing="ij"), dim=-1)
    lat = torch.as_tensor(L, device=dev)
    pts = F @ lat
    B = 2.0 * math.pi * np.linalg.inv(L).T
    k = [torch.fft.fftfreq(m, d=1.0 / m, dtype=torch.float64, device=dev) for m in ns]
    G = torch.stack(torch.meshgrid(*k, indexing="ij"), dim=-1) @ torch.as_tensor(B, device=dev)
    G2 = (G * G).sum(-1)
    kern = torch.where(G2 > 0, 4.0 * math.pi / G2.clamp_min(1e-300), torch.zeros_like(G2))
    heights = 1.0 / np.linalg.norm(np.linalg.inv(L), axis=0)
    chi = []
    for s in cell.shells:
        l, a = s.l, s.exps
        c = s.coefs * (2 * a / math.pi) ** 0.75 * (8 * a) ** (0.5 * l)
        self_overlap = np.sum(np.outer(s.coefs, s.coefs) * (2 * np.sqrt(np.outer(a, a)) / np.add.outer(a, a)) ** (l + 1.5))
        c = c / math.sqrt(self_overlap)
        radius = math.sqrt(44.0 / float(a.min()))
        reach = [int(math.ceil(radius / h)) + 1 for h in heights]
        base = np.floor(s.center @ np.linalg.inv(L))
        comps = _cartesians(l)
        val = [torch.zeros(tuple(ns), dtype=torch.float64, device=dev) for _ in comps]
        for i in range(-reach[0], reach[0] + 1):
            for j in range(-reach[1], reach[1] + 1):
                for m in range(-reach[2], reach[2] + 1):
                    ctr = s.center + (np.array([i, j, m]) - base) @ L
                    corner = np.array([[x, y, z] for x in (0, 1) for y in (0, 1) for z in (0, 1)]) @ L
                    mid = corner.mean(0)
                    if np.linalg.norm(ctr - mid) > radius + np.linalg.norm(corner - mid, axis=1).max():
                        continue
                    d = pts - torch.as_tensor(ctr, device=dev)
                    r2 = (d * d).sum(-1)
                    rad = sum(float(cc) * torch.exp(-float(aa) * r2) for cc, aa in zip(c, a))
                    for v, e in zip(val, comps):
                        t = rad
                        for ax in range(3):
                            if e[ax]:
                                t = t * d[..., ax] ** e[ax]
                        v += t
        for v, e in zip(val, comps):
            fac = math.sqrt(math.prod(math.factorial(x) / math.factorial(2 * x) for x in e))
            chi.append(v * fac)
    return torch.stack(chi), kern, G, G2, abs(float(np.linalg.det(L))) / math.prod(ns)


def exact(case, seed):
    if case["kind"] == "energy":
        cell, X, rng = _frame(case, seed)
        _, D = _plan_and_density(cell, X, case["precision"])
        J, K = _matrices(rng, cell.nbf)
        return {"EJ": float(0.5 * (D * J).sum()), "EK": float(-0.25 * (D * K).sum())}
    if case["cell"] not in ("tiny", "small") or case["kind"] == "serve":
        return None
    cell, X, _ = _frame(case, seed)
    chi, kern, G, G2, dv = _grid(cell)
    flat = chi.reshape(len(chi), -1)
    S = flat @ flat.T * dv

    def potential(rho):
        return torch.fft.ifftn(torch.fft.fftn(rho) * kern).real

    if case["kind"] == "onee":
        V = dv * chi[0].numel()
        F = torch.fft.fftn(chi, dim=(1, 2, 3)).reshape(len(chi), -1)
        T = 0.5 * (F.conj() * G2.reshape(-1)) @ F.T
        T = T.real * dv * dv / V
        rho = torch.zeros(kern.shape, dtype=torch.complex128, device=kern.device)
        for z, x in zip(sc.nuclear_charges(cell), cell.positions):
            rho += float(z) * torch.exp(-1j * (G @ torch.as_tensor(x, device=G.device)))
        v = torch.fft.ifftn(-rho * kern).real / dv
        return {"T": T, "V": (flat * v.reshape(-1)) @ flat.T * dv}
    D = _density(X, S)
    rho = torch.einsum("mx,mx->x", D @ flat, flat).reshape(kern.shape)
    J = (flat * potential(rho).reshape(-1)) @ flat.T * dv
    if not case["k"]:
        return {"J": J}
    w, U = torch.linalg.eigh(D)
    K = torch.zeros_like(J)
    for d, u in zip(w.tolist(), U.T):
        if abs(d) < 1e-13 * float(w.abs().max()):
            continue
        psi = (u @ flat).reshape(kern.shape)
        pot = torch.stack([potential(c * psi) for c in chi])
        K += d * ((pot * psi).reshape(len(chi), -1) @ flat.T) * dv
    return {"J": J, "K": 0.5 * (K + K.T)}
