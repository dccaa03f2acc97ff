"""Measured workloads of the library: what each case is, its inputs, one pass, and its 64-bit values.

A case is one call (or one group of calls) that a user of the library makes: building the screened
ACE operator, rebuilding it on a kept pair list, building many at once, applying it, and localising
orbitals before a build.  Inputs are synthetic orbitals of the shapes in workloads/generators.py,
made here on the GPU because they are made often: Gaussians at four centres per molecule, at liquid
water density or clustered in a mostly empty cell, symmetrically orthonormalised in FP64.
"""

import math

import numpy as np
import torch

import paper_2101_03155_gb300 as ace
from paper_2101_03155_gb300 import ace as abi

# volume per orbital of liquid water, four orbitals per molecule (32 molecules in an 18.63 bohr cube)
VOLUME_PER_ORBITAL = 18.63**3 / 128
# a screened water-like build keeps about this many pairs (i <= j) per orbital (threshold 1e-3)
PAIRS_PER_ORBITAL = 18.3


def _case(kind, n, grid, prec="mixed", system="water", rho_cut=1e-3, m=0, builds=""):
    return {"kind": kind, "n": n, "n1": grid[0], "n2": grid[1], "n3": grid[2], "prec": prec, "system": system,
            "rho_cut": rho_cut, "m": m, "builds": builds}


def listed():
    def named(name, case):
        return dict(case, name=name)

    return [
        # the plain method on a small periodic cell: every pair, 16 orbitals; launches and waits count
        named("build_16orb_32c_all_pairs", _case("build", 16, (32, 32, 32), rho_cut=0.0)),
        # a reuse step of a multiple-time-step run: the pair list of an earlier snapshot, odd axes
        named("pairs_24orb_45x48x50", _case("pairs", 24, (45, 48, 50))),
        # the usual construction step: 32 water molecules
        named("build_128orb_96c", _case("build", 128, (96, 96, 96))),
        # the largest box: 64 water molecules
        named("build_256orb_128c", _case("build", 256, (128, 128, 128))),
        # a QM region in a mostly empty orthorhombic cell, isolated-cell kernel
        named("build_isolated_112orb_160x144x128", _case("build", 112, (160, 144, 128), system="cluster")),
        # a grid that a plane-wave cut-off picks freely: axis lengths with no plane plan
        named("build_96orb_100x108x90", _case("build", 96, (100, 108, 90))),
        # independent replicas of uneven size in one call
        named("batch_6_uneven", _case("batch", 96, (108, 108, 108), builds="64:72 96:96 64:108 128:72 96:72 64:96")),
        # the plain double-precision form, used to check the mixed one
        named("build_fp64_64orb_72c", _case("build", 64, (72, 72, 72), prec="fp64")),
        # the double-precision form on a small grid with no plane plan, every pair
        named("build_fp64_12orb_40x45x48", _case("build", 12, (40, 45, 48), prec="fp64", rho_cut=0.0)),
        # the inner steps of a self-consistency cycle: the operator applied to all orbitals
        named("apply_128vec_128orb_96c", _case("apply", 128, (96, 96, 96), m=128)),
        # an iterative eigensolver's step: the operator applied to a few vectors
        named("apply_4vec_64orb_72c", _case("apply", 64, (72, 72, 72), m=4)),
        # localisation of canonical orbitals ahead of a build
        named("scdm_128orb_96c", _case("scdm", 128, (96, 96, 96))),
    ]


_AXES = [30, 32, 36, 40, 45, 48, 50, 54, 60, 64, 72, 75, 80, 81, 90, 96, 100, 108, 120, 125, 128]


def draw(rng):
    def axis_near(x):
        near = sorted(_AXES, key=lambda a: abs(math.log(a / x)))[:4]
        return rng.choice(near)

    kind = rng.choice(["build", "build", "build", "pairs", "batch", "fp64", "apply", "scdm"])
    if kind == "fp64":
        side = math.exp(rng.uniform(math.log(32), math.log(64)))
        n = 4 * rng.randint(2, 10)
        return _case("build", n, tuple(axis_near(side) for _ in range(3)), prec="fp64",
                     rho_cut=rng.choice([0.0, 1e-3]))
    side = math.exp(rng.uniform(math.log(32), math.log(112)))
    n = int(4 * round(math.exp(rng.uniform(math.log(4), math.log(36)))))
    grid = (axis_near(side),) * 3 if rng.random() < 0.4 else tuple(axis_near(side) for _ in range(3))
    if kind == "batch":
        k = rng.randint(2, 5)
        builds = " ".join("%d:%d" % (rng.choice([32, 64, 96]), rng.choice([48, 60, 72, 96])) for _ in range(k))
        return _case("batch", 64, (96, 96, 96), builds=builds)
    if kind == "apply":
        m = int(round(math.exp(rng.uniform(0.0, math.log(160)))))
        return _case("apply", n, grid, m=m)
    if kind == "build" and rng.random() < 0.25:
        return _case("build", n, grid, system="cluster")
    return _case(kind, n, grid)


# ---------------------------------------------------------------------------------------- inputs


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _builds(case):
    """(orbitals, grid) of every build of the case."""
    if case["kind"] == "batch":
        return [(int(n), (int(g),) * 3) for n, g in (b.split(":") for b in case["builds"].split())]
    return [(case["n"], (case["n1"], case["n2"], case["n3"]))]


def _cell(case, n, grid):
    """Cell sides (bohr) with the grid's aspect: liquid density, or a cluster in about eight times its volume."""
    volume = n * VOLUME_PER_ORBITAL * (6.8 if case["system"] == "cluster" else 1.0)
    h = (volume / (grid[0] * grid[1] * grid[2])) ** (1.0 / 3.0)
    return np.array([h * g for g in grid])


def _centres(case, n, cell, rng):
    """Centres of n orbitals: four per molecule, molecules kept apart by random sequential addition."""
    sites, tries, apart = [], 0, 4.4
    cluster = case["system"] == "cluster"
    radius = 0.9 * (3.0 * n * VOLUME_PER_ORBITAL / (4.0 * math.pi)) ** (1.0 / 3.0)
    while len(sites) < -(-n // 4):
        tries += 1
        if tries % 4000 == 0:
            apart *= 0.95
        if cluster:
            v = rng.uniform(-1.0, 1.0, 3)
            if v @ v > 1.0:
                continue
            p = 0.5 * cell + radius * v
            ok = all(np.sum((p - q) ** 2) >= (0.8 * apart) ** 2 for q in sites)
        else:
            p = rng.uniform(0.0, 1.0, 3) * cell
            ok = all(np.sum((p - q - cell * np.round((p - q) / cell)) ** 2) >= apart**2 for q in sites)
        if ok:
            sites.append(p)
    arms = np.array([[1, 1, 1], [1, -1, -1], [-1, 1, -1], [-1, -1, 1]]) / math.sqrt(3.0)
    out = []
    for s in sites:
        q, r = np.linalg.qr(rng.standard_normal((3, 3)))
        d = arms @ (q * np.sign(np.diag(r))).T
        out += [s + 0.9 * d[0], s + 0.9 * d[1], s + 0.6 * d[2], s + 0.6 * d[3]]
    return np.array(out[:n])


def _orbitals(case, n, grid, seed, moved=False):
    """Orthonormal orbitals (FP64, [n][N1][N2][N3]) and the lattice; ``moved``: the next snapshot, every
    centre 0.05 bohr away."""
    rng = np.random.default_rng(seed)
    cell = _cell(case, n, grid)
    c = _centres(case, n, cell, rng)
    spread = rng.uniform(0.8, 1.4, n)
    if moved:
        d = rng.standard_normal(c.shape)
        c = c + 0.05 * d / np.linalg.norm(d, axis=1, keepdims=True)
    dev = _device()
    axes, S = [], 1.0
    for k in range(3):  # a Gaussian over orthogonal axes, and its image sum, factorise
        x = np.arange(grid[k]) * (cell[k] / grid[k])
        t = x[None, :, None] - c[:, k, None, None] - cell[k] * np.arange(-1, 2)[None, None, :]
        g = np.exp(-(t**2) / (2.0 * spread[:, None, None] ** 2)).sum(-1)
        axes.append(torch.from_numpy(g).to(dev))
        S = S * (g @ g.T)
    S *= float(np.prod(cell)) / (grid[0] * grid[1] * grid[2])
    w, V = np.linalg.eigh(0.5 * (S + S.T))
    C = torch.from_numpy((V / np.sqrt(w)) @ V.T).to(dev)
    chi = axes[0][:, :, None, None] * axes[1][:, None, :, None] * axes[2][:, None, None, :]
    phi = (C @ chi.reshape(n, -1)).reshape((n,) + tuple(grid))
    return phi, np.diag(cell)


def _working(case, phi):
    return phi if case["prec"] == "fp64" else phi.float()


def _desc(case, n, grid, lattice):
    return ace.make_desc(grid, lattice, n, rho_cut=case["rho_cut"],
                         prec=abi.ACE_FP64 if case["prec"] == "fp64" else abi.ACE_MIXED,
                         coulomb=abi.ACE_COULOMB_TRUNCATED if case["system"] == "cluster" else 0)


def _rotation(n, seed):
    q, r = np.linalg.qr(np.random.default_rng(seed + 77).standard_normal((n, n)))
    return torch.from_numpy(q * np.sign(np.diag(r))).to(_device())


def _kept_pairs(phi, dV, rho_cut):
    """Pairs (i <= j) of the screen, in 64 bits."""
    n = phi.shape[0]
    a = phi.reshape(n, -1).double().abs()
    O = (dV * (a @ a.T)).cpu().numpy()
    keep = (O >= rho_cut) if rho_cut > 0 else np.ones((n, n), dtype=bool)
    np.fill_diagonal(keep, True)
    return np.argwhere(np.triu(keep)).astype(np.int32)


def _inputs(case, seed):
    """Of every build: descriptor, orbitals in the working type, and what else the call takes."""
    out = []
    for b, (n, grid) in enumerate(_builds(case)):
        phi, lattice = _orbitals(case, n, grid, seed * 64 + b)
        d = {"n": n, "grid": grid, "lattice": lattice, "desc": _desc(case, n, grid, lattice)}
        if case["kind"] == "pairs":
            d["pairs"] = _kept_pairs(phi, abs(np.linalg.det(lattice)) / phi[0].numel(), case["rho_cut"])
            phi, _ = _orbitals(case, n, grid, seed * 64 + b, moved=True)
        if case["kind"] == "scdm":
            phi = (_rotation(n, seed) @ phi.reshape(n, -1)).reshape(phi.shape)
        d["phi"] = _working(case, phi).contiguous()
        if case["kind"] == "apply":
            gen = torch.Generator(device=_device()).manual_seed(seed)
            psi = torch.randn((case["m"], n), generator=gen, device=_device(), dtype=torch.float64)
            noise = torch.randn((case["m"],) + tuple(grid), generator=gen, device=_device(), dtype=torch.float64)
            dV = abs(np.linalg.det(lattice)) / phi[0].numel()
            psi = (psi / math.sqrt(n) @ phi.reshape(n, -1)).reshape(noise.shape) + 0.1 * noise / math.sqrt(
                dV * phi[0].numel())
            d["psi"] = _working(case, psi).contiguous()
        out.append(d)
    return out


def prepare(case, seed):
    ins = _inputs(case, seed)
    state = {"case": case, "in": ins}
    if case["kind"] == "apply":
        d = ins[0]
        state["op"] = ace.ace_build(d["desc"], d["phi"], torch.cuda.current_stream())
        state["out"] = torch.empty_like(d["psi"])
    elif case["kind"] == "scdm":
        state["out"] = torch.empty_like(ins[0]["phi"])
    else:
        state["xi"] = [torch.empty_like(d["phi"]) for d in ins]
    return state


# ---------------------------------------------------------------------------------------- one pass


def _read(op, xi, stream):
    """The finished operator's vectors, energy and pair list (as the mask of kept pairs); the handle is given back."""
    abi.ace_get(op, abi.ACE_GET_XI, xi, stream)
    pairs = abi.get_numpy(op, abi.ACE_GET_PAIRS)
    kept = np.zeros((op.norb, op.norb), dtype=bool)
    kept[pairs[:, 0], pairs[:, 1]] = True
    out = {"xi": xi, "E_x": ace.exchange_energy(op), "kept": kept}
    op.close()
    return out


def run(state):
    kind, ins, stream = state["case"]["kind"], state["in"], torch.cuda.current_stream()
    d = ins[0]
    if kind == "build":
        return _read(ace.ace_build(d["desc"], d["phi"], stream), state["xi"][0], stream)
    if kind == "pairs":
        return _read(ace.ace_build_pairs(d["desc"], d["phi"], d["pairs"], stream), state["xi"][0], stream)
    if kind == "batch":
        ops = ace.ace_build_batched([x["desc"] for x in ins], [x["phi"] for x in ins], stream)
        return [_read(op, xi, stream) for op, xi in zip(ops, state["xi"])]
    if kind == "apply":
        return ace.ace_apply(state["op"], d["psi"], state["out"], stream)
    _, piv, U, _ = ace.ace_scdm(d["phi"], state["out"], abi.ACE_MIXED, stream)
    return {"phi": state["out"], "piv": piv, "U": U}


def work(case):
    """Bytes: orbitals (or vectors) in and results out.  Flops: per pair half a packed complex transform
    each way, the products around it and W; the contractions of the screen, M, xi and the application;
    the passes of the localisation.  Pairs of a screened build are estimated from its density."""
    size = 8 if case["prec"] == "fp64" else 4
    nbytes = flops = 0.0
    for n, grid in _builds(case):
        N = grid[0] * grid[1] * grid[2]
        if case["kind"] == "scdm":
            nbytes += 2.0 * size * n * N
            flops += 1.0 * n * n * N + 2.0 * n * n * N
            continue
        if case["kind"] == "apply":
            m = case["m"]
            nbytes += size * (n + 2.0 * m) * N
            flops += 4.0 * n * m * N
            continue
        every = n * (n + 1) / 2.0
        pairs = min(every, PAIRS_PER_ORBITAL * n) if case["rho_cut"] > 0 else every
        nbytes += 2.0 * size * n * N
        flops += pairs * N * (5.0 * math.log2(N) + 6.0)
        flops += N * (n * n * (1.0 if case["rho_cut"] > 0 and case["kind"] != "pairs" else 0.0) + 3.0 * n * n)
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------------------- 64 bits


def _kernel(case, grid, cell, dev):
    """4 pi / |G|^2 on the half box of a real transform, or its cut-off at the inscribed sphere's radius."""
    g2 = 0.0
    for k in range(3):
        m = np.fft.rfftfreq(grid[k]) if k == 2 else np.fft.fftfreq(grid[k])
        g = torch.from_numpy((2.0 * math.pi * grid[k] / cell[k] * m) ** 2).to(dev)
        g2 = g2 + g.reshape([-1 if a == k else 1 for a in range(3)])
    zero = g2 == 0
    q = torch.where(zero, torch.ones_like(g2), g2)
    if case["system"] == "cluster":
        rc = 0.5 * float(min(cell))
        return torch.where(zero, torch.full_like(g2, 2.0 * math.pi * rc * rc),
                           4.0 * math.pi * (1.0 - torch.cos(torch.sqrt(q) * rc)) / q)
    return torch.where(zero, torch.zeros_like(g2), 4.0 * math.pi / q)


def _exact_build(case, d):
    phi = d["phi"].double()
    n, grid, cell = d["n"], d["grid"], np.diag(d["lattice"])
    N = phi[0].numel()
    dV = float(np.prod(cell)) / N
    pairs = d["pairs"] if case["kind"] == "pairs" else _kept_pairs(d["phi"], dV, case["rho_cut"])
    K = _kernel(case, grid, cell, phi.device)
    W = torch.zeros_like(phi)
    most = max(1, int(4e7 // N))
    for i in range(n):
        js = pairs[pairs[:, 0] == i][:, 1]
        for c in range(0, len(js), most):
            j = torch.from_numpy(js[c:c + most].astype(np.int64)).to(phi.device)
            pj = phi[j]
            v = torch.fft.irfftn(torch.fft.rfftn(pj * phi[i], dim=(1, 2, 3)) * K, s=tuple(grid), dim=(1, 2, 3))
            W[i] += (v * pj).sum(0)
            other = j != i
            if bool(other.any()):
                W.index_add_(0, j[other], v[other] * phi[i])
    W = W.reshape(n, N)
    M = -dV * (phi.reshape(n, N) @ W.T)
    M = 0.5 * (M + M.T)
    L = torch.linalg.cholesky(-M)
    xi = torch.linalg.inv(L) @ W
    return xi, float(torch.trace(M)), dV


def exact(case, seed):
    ins = _inputs(case, seed)
    if case["kind"] == "scdm":
        psi = ins[0]["phi"].double().reshape(case["n"], -1)
        n = case["n"]
        left, piv, Q = (psi * psi).sum(0), [], torch.zeros((0, n), dtype=torch.float64, device=psi.device)
        for _ in range(n):
            c = int(torch.argmax(left))
            piv.append(c)
            u = psi[:, c]
            for _ in range(2):
                u = u - Q.T @ (Q @ u)
            u = u / torch.linalg.norm(u)
            Q = torch.cat([Q, u[None]])
            left = left - (u @ psi) ** 2
        M = psi[:, piv]
        w, V = torch.linalg.eigh(M.T @ M)
        U = M @ (V / torch.sqrt(w)) @ V.T
        return {"phi": (U.T @ psi).reshape(ins[0]["phi"].shape), "piv": None, "U": U}
    if case["kind"] == "apply":
        d = ins[0]
        xi, _, dV = _exact_build(case, d)
        psi = d["psi"].double().reshape(case["m"], -1)
        return (-dV * ((psi @ xi.T) @ xi)).reshape(d["psi"].shape)
    out = []
    for d in ins:
        xi, e, _ = _exact_build(case, d)
        out.append({"xi": xi.reshape(d["phi"].shape), "E_x": e, "kept": None})
    return out if case["kind"] == "batch" else out[0]
