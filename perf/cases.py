"""The work whose speed is measured: evaluations of the environment potential
through the package's public entry points.

A case is a dict of plain values.  `kind` names the entry point, the rest its
environment and sizes:

  graph      esp.Graph.launch: point cells, 1..128 positions, one replay per call
  eval       esp.Environment.eval, device tensors or host arrays
  walkers    esp.Environment.eval_walkers (potentials and walker energies)
  batch      esp.Batch.eval over systems of uneven size
  surrogate  esp.Surrogate.eval with a trained surrogate
  train      esp.Surrogate(...): label, train and validate, then predict

Environments (`env`):

  cells      the paper's shape: density cells (small point charges) and nuclei
  charges    nuclei and s-Gaussian charges in a 20 bohr cube about the QM sphere
  atoms      atoms on a jittered lattice with cc-pVDZ-shaped primitives (s, p and
             Cartesian d) and a density of on-site and neighbour products

Electron positions follow N(0, 2^2) bohr truncated to the 6 bohr QM sphere.
"""
import math

import numpy as np
import torch

from paper_1011_4687_gb300 import esp

QM_RADIUS = 6.0
CART = [(0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1),
        (2, 0, 0), (0, 2, 0), (0, 0, 2), (1, 1, 0), (1, 0, 1), (0, 1, 1)]
FIRST = np.array([0, 1, 4])   # first Cartesian component of a shell, by l
COUNT = np.array([1, 3, 6])   # number of its components

# Averages over the `atoms` environments per primitive product: operations of
# its multipole form (8 / 18 / 39 / 80 / 151 for total angular momentum 0..4)
# and bytes of centre, exponent and Hermite coefficients in 64 bits.
ATOM_OPS = 20.0
ATOM_BYTES = 66.0


def listed():
    return [
        # one Metropolis move of the paper's trimer: one position per call, replayed
        dict(name="cells move", kind="graph", env="cells", size=268782, n=1, precision="fp32c", host=False),
        # the electrons of one small walker, positions and potentials in host memory
        dict(name="cells host 16", kind="eval", env="cells", size=268782, n=16, precision="fp32c", host=True),
        # the few-position path at its upper end
        dict(name="cells 128", kind="eval", env="cells", size=268782, n=128, precision="fp32c", host=False),
        # single-electron moves in a Gaussian environment
        dict(name="atoms few 5", kind="eval", env="atoms", size=400, per_atom=240, n=5, precision="fp32c", host=False),
        # 100 walkers of 100 electrons in the small environment
        dict(name="charges walkers", kind="walkers", env="charges", size=2000, n=100, electrons=100,
             precision="fp32c", host=False),
        # an odd, mid-sized call from host memory
        dict(name="atoms host 1001", kind="eval", env="atoms", size=400, per_atom=240, n=1001, precision="fp32c",
             host=True),
        # a production step: many walkers of 32 electrons
        dict(name="atoms walkers", kind="walkers", env="atoms", size=800, per_atom=240, n=2048, electrons=32,
             precision="fp32c", host=False),
        # reference-accuracy energies of some walkers
        dict(name="atoms fp64", kind="walkers", env="atoms", size=400, per_atom=240, n=64, electrons=32,
             precision="fp64", host=False),
        # reference-accuracy potentials at a ragged number of positions
        dict(name="charges fp64 1999", kind="eval", env="charges", size=2000, n=1999, precision="fp64", host=False),
        # fragments of uneven size in one call
        dict(name="batch 12", kind="batch", env="atoms", size=120, per_atom=160, systems=12, n=4096,
             precision="fp32c", host=False),
        # a production step with the surrogate
        dict(name="surrogate", kind="surrogate", env="atoms", size=1200, per_atom=120, n=50000, precision="fp32c",
             host=False),
        # making a surrogate: forward and backward passes, labels, validation
        dict(name="train", kind="train", env="atoms", size=1200, per_atom=60, n=4096, samples=32768, epochs=4,
             precision="fp32c", host=False),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _atoms_size(rng, most=192000):
    """An atom count and products per atom: 2,000 products in all and more."""
    products, per_atom = _log(rng, 2000, most), _log(rng, 40, 480)
    return dict(size=max(8, products // per_atom), per_atom=per_atom)


def draw(rng):
    what = rng.choice(["graph", "eval cells", "few", "eval", "eval", "walkers", "walkers", "fp64", "fp64", "batch",
                       "surrogate", "train"])
    host = rng.random() < 0.3
    if what == "graph":
        return dict(kind="graph", env="cells", size=_log(rng, 5000, 268782), n=_log(rng, 1, 128), precision="fp32c",
                    host=False)
    if what == "eval cells":
        return dict(kind="eval", env="cells", size=_log(rng, 5000, 268782), n=_log(rng, 1, 600),
                    precision=rng.choice(["fp32c", "fp32c", "fp64"]), host=host)
    if what == "few":
        return dict(kind="eval", env="atoms", **_atoms_size(rng), n=rng.randint(1, 16),
                    precision=rng.choice(["fp32c", "fp64"]), host=host)
    env = rng.choice(["atoms", "atoms", "charges"])
    size = _atoms_size(rng) if env == "atoms" else dict(size=_log(rng, 200, 8000))
    if what == "eval":
        return dict(kind="eval", env=env, **size, n=_log(rng, 17, 60000), precision="fp32c", host=host)
    if what == "walkers":
        return dict(kind="walkers", env=env, **size, n=_log(rng, 2, 1000), electrons=rng.randint(8, 64),
                    precision="fp32c", host=host)
    if what == "fp64":
        if rng.random() < 0.5:
            return dict(kind="eval", env=env, **size, n=_log(rng, 17, 4000), precision="fp64", host=host)
        return dict(kind="walkers", env=env, **size, n=_log(rng, 1, 64), electrons=rng.randint(8, 64),
                    precision="fp64", host=host)
    if what == "batch":
        slow = rng.random() < 0.2
        return dict(kind="batch", env="atoms", **_atoms_size(rng, 20000), systems=rng.randint(2, 16),
                    n=_log(rng, 200, 1000 if slow else 6000), precision="fp64" if slow else "fp32c", host=False)
    if what == "surrogate":
        return dict(kind="surrogate", env="atoms", size=_log(rng, 600, 1400), per_atom=rng.randint(30, 120),
                    n=_log(rng, 2000, 100000), precision="fp32c", host=False)
    return dict(kind="train", env="atoms", size=_log(rng, 600, 1200), per_atom=rng.randint(20, 60),
                n=_log(rng, 1000, 4096), samples=_log(rng, 16384, 49152), epochs=rng.randint(1, 4),
                precision="fp32c", host=False)


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------
class Pairs:
    """Weighted primitive products in the layout esp.Environment takes."""

    def __init__(self, A, alpha, la, B, beta, lb, w):
        self.A, self.alpha, self.la = A, alpha, np.asarray(la, np.int32).reshape(-1, 3)
        self.B, self.beta, self.lb = B, beta, np.asarray(lb, np.int32).reshape(-1, 3)
        self.w = w

    def __len__(self):
        return int(self.alpha.shape[0])


def _no_pairs():
    z3, z = np.zeros((0, 3)), np.zeros(0)
    return Pairs(z3, z, z3, z3, z, z3, z)


def _positions(rng, n):
    out = np.empty((0, 3))
    while out.shape[0] < n:
        x = rng.normal(0.0, 2.0, size=(int((n - out.shape[0]) * 1.1) + 16, 3))
        out = np.concatenate([out, x[(x * x).sum(1) < QM_RADIUS ** 2]])
    return out[:n].copy()


def _outside(rng, n, half):
    out = np.empty((0, 3))
    while out.shape[0] < n:
        x = rng.uniform(-half, half, size=(2 * (n - out.shape[0]) + 16, 3))
        out = np.concatenate([out, x[(x * x).sum(1) >= QM_RADIUS ** 2]])
    return out[:n].copy()


def _cells(rng, size):
    R, Z = _outside(rng, 36, 10.0), rng.choice([1.0, 6.0, 7.0, 8.0], size=36)
    xyz, rho = _outside(rng, size, 10.0), np.abs(rng.normal(size=size))
    return np.concatenate([R, xyz]), np.concatenate([Z, -rho * (Z.sum() / rho.sum())]), _no_pairs()


def _charges(rng, size):
    k = max(1, size // 10)
    R, Z = _outside(rng, k, 10.0), rng.choice([1.0, 6.0, 7.0, 8.0], size=k)
    C = _outside(rng, size, 10.0)
    alpha = np.exp(rng.uniform(math.log(0.1), math.log(50.0), size=size))
    z = np.zeros((size, 3))
    return R, Z, Pairs(C, alpha / 2, z, C, alpha / 2, z, rng.normal(-1.0, 0.3, size=size) * (alpha / math.pi) ** 1.5)


def _norm(alpha, lmn):
    odd = np.array([1.0, 1.0, 3.0])
    return np.sqrt((2 * alpha / math.pi) ** 1.5 * (4 * alpha) ** lmn.sum(1) / odd[lmn].prod(1))


def _atoms(rng, size, per_atom):
    side = int(math.ceil((size * 1.15) ** (1 / 3))) + 1
    while True:
        g = (np.arange(side) - (side - 1) / 2) * 2.8
        sites = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
        sites = sites[(sites * sites).sum(1) >= QM_RADIUS ** 2]
        if sites.shape[0] >= size:
            break
        side += 1
    R = sites[np.sort(rng.choice(sites.shape[0], size=size, replace=False))] + rng.normal(0.0, 0.15, size=(size, 3))
    Z = rng.choice([1.0, 6.0, 7.0, 8.0], size=size)
    # shells: l and exponent; 9 s, 4 p and one d (hydrogen: 4 s and one p)
    heavy_e = np.concatenate([np.geomspace(0.1, 5000.0, 9), np.geomspace(0.1, 30.0, 4), [math.sqrt(0.45)]])
    heavy_l = np.array([0] * 9 + [1] * 4 + [2])
    light_e, light_l = np.concatenate([np.geomspace(0.1, 50.0, 4), [1.0]]), np.array([0] * 4 + [1])
    jitter = np.exp(rng.normal(0.0, 0.08, size=(size, 14)))

    def shell(atom, k):
        light = Z[atom] == 1.0
        kl = np.where(light, k % 5, k)
        e = np.where(light, light_e[kl % 5], heavy_e[kl]) * jitter[atom, kl]
        return e, np.where(light, light_l[kl % 5], heavy_l[kl])

    # products: a third on site, the others with one of the six nearest atoms
    d2 = ((R[:, None, :] - R[None, :, :]) ** 2).sum(-1)
    near = np.argsort(d2, axis=1)[:, 1:min(7, size)]
    n = size * per_atom
    a = np.repeat(np.arange(size), per_atom)
    b = np.where(rng.random(n) < 1 / 3, a, near[a, rng.integers(0, near.shape[1], size=n)] if near.size else a)
    ea, la = shell(a, rng.integers(0, 14, size=n))
    eb, lb = shell(b, rng.integers(0, 14, size=n))
    cart = np.array(CART)
    ca = cart[FIRST[la] + rng.integers(0, 1 << 20, size=n) % COUNT[la]]
    cb = cart[FIRST[lb] + rng.integers(0, 1 << 20, size=n) % COUNT[lb]]
    w = rng.normal(0.0, 0.3, size=n) * _norm(ea, ca) * _norm(eb, cb)
    keep = (ea * eb / (ea + eb) * d2[a, b] < 20.0)
    # the atoms' own electrons: on-site s products, partial charges of about 0.15 Z
    # per atom, the whole neutral
    part = rng.normal(1.0, 0.15, size=size)
    part *= Z.sum() / (part * Z).sum()
    a2 = np.repeat(np.arange(size), 3)
    e2 = np.tile([0.3, 2.0, 20.0], size) * np.exp(rng.normal(0.0, 0.08, size=3 * size))
    w2 = -(np.repeat(part * Z, 3) / 3) * (2 * e2 / math.pi) ** 1.5
    z = np.zeros((3 * size, 3), int)
    cat = np.concatenate
    return R, Z, Pairs(cat([R[a[keep]], R[a2]]), cat([ea[keep], e2]), cat([ca[keep], z]),
                       cat([R[b[keep]], R[a2]]), cat([eb[keep], e2]), cat([cb[keep], z]), cat([w[keep], w2]))


def _environment(rng, case, scale=1.0):
    size = max(8, int(case["size"] * scale))
    if case["env"] == "cells":
        return _cells(rng, size)
    if case["env"] == "charges":
        return _charges(rng, size)
    return _atoms(rng, size, case["per_atom"])


def _inputs(case, seed):
    """[(nuclei, Z, pairs, positions)], one per system."""
    rng = np.random.default_rng([1011, seed])
    if case["kind"] == "batch":
        # sizes over a factor of eight, position counts independently so
        sizes = np.random.default_rng([1011, case["systems"], case["size"], case["n"]])
        f = np.exp(sizes.uniform(math.log(0.25), math.log(2.0), size=(case["systems"], 2)))
        f[0] = 1.0
        return [(*_environment(rng, case, f[s, 0]), _positions(rng, max(1, int(case["n"] * f[s, 1]))))
                for s in range(case["systems"])]
    return [(*_environment(rng, case), _positions(rng, case["n"] * case.get("electrons", 1)))]


def _config(case, seed):
    if case["kind"] == "train":
        return dict(n_train=case["samples"], n_valid=8192, epochs=case["epochs"], seed=1011 + seed)
    return dict(n_train=16384, n_valid=8192, epochs=1, seed=1011 + seed)


def prepare(case, seed):
    systems = _inputs(case, seed)
    envs = [esp.Environment(R, Z, pairs, precision=case["precision"]) for R, Z, pairs, _ in systems]
    pos = [p if case["host"] else torch.from_numpy(p).cuda() for *_, p in systems]
    state = dict(case=case, seed=seed, envs=envs, pos=pos)
    if case["kind"] == "graph":
        out = torch.empty(case["n"], dtype=torch.float64, device="cuda")
        state["graph"] = esp.Graph(envs[0], pos[0], out)
    elif case["kind"] == "batch":
        state["batch"] = esp.Batch(envs)
    elif case["kind"] == "surrogate":
        state["surrogate"] = esp.Surrogate(envs[0], **_config(case, seed))
    return state


def run(state):
    case, env, pos = state["case"], state["envs"][0], state["pos"][0]
    kind = case["kind"]
    if kind == "graph":
        return state["graph"].launch()
    if kind == "eval":
        return env.eval(pos)
    if kind == "walkers":
        V, E = env.eval_walkers(pos, case["n"], case["electrons"])
        return {"V": V, "E": E}
    if kind == "batch":
        return state["batch"].eval(state["pos"])
    if kind == "surrogate":
        V, _ = state["surrogate"].eval(pos)
        return V
    with esp.Surrogate(env, **_config(case, state["seed"])) as sur:
        V = sur.predict(pos)
        weights, _, _ = sur.debug_step(np.zeros((1, 3)), np.zeros(1, np.float32))
    return {"V": V, "weights": weights}


# ----------------------------------------------------------------------------
# what a pass cannot do without
# ----------------------------------------------------------------------------
def work(case):
    mean = (2.0 - 0.25) / math.log(8.0)  # of the batch's size factors
    systems, scale = (case["systems"], mean) if case["kind"] == "batch" else (1, 1.0)
    positions = case["n"] * case.get("electrons", 1) * scale
    if case["env"] == "cells":
        ops, nbytes = 8.0 * (case["size"] + 36), 32.0 * (case["size"] + 36)
    elif case["env"] == "charges":
        ops, nbytes = 8.0 * 1.1 * case["size"], (40.0 + 3.2) * case["size"]
    else:
        entries = case["size"] * scale * (0.55 * case["per_atom"] + 10.0)
        ops, nbytes = ATOM_OPS * entries, ATOM_BYTES * entries
    if case["kind"] == "train":
        points = case["samples"] + 8192 + 58000  # labels and one validation point per voxel
        step = 6.0 * 213760 * case["samples"] * case["epochs"]
        return dict(bytes=nbytes + 32.0 * points, flops=ops * (points + positions) + step)
    if case["kind"] == "surrogate":
        # near tiles are summed, the network and the expansion give the rest
        return dict(bytes=nbytes + 32.0 * positions, flops=(0.35 * ops + 427520.0) * positions)
    return dict(bytes=systems * (nbytes + 32.0 * positions), flops=systems * ops * positions)


# ----------------------------------------------------------------------------
# the same potentials in 64 bits with torch
# ----------------------------------------------------------------------------
def _boys(L, T):
    """F_0..F_L(T): incomplete gamma (T < 45) or its limit, then downward recursion."""
    a = L + 0.5
    F = math.gamma(a) / 2 * T.clamp_min(1e-30) ** -a
    low = (T < 45.0).nonzero(as_tuple=True)
    if low[0].numel():
        t = T[low]
        tiny = t < 1e-3
        series = 1 / (2 * L + 1) - t / (2 * L + 3) + t * t / (4 * L + 10) - t ** 3 / (12 * L + 42) \
            + t ** 4 / (48 * L + 216)
        F[low] = torch.where(tiny, series, F[low] * torch.special.gammainc(torch.full_like(t, a), t))
    out, e = [F], torch.exp(-T)
    for n in range(L - 1, -1, -1):
        out.append((2 * T * out[-1] + e) / (2 * n + 1))
    return out[::-1]


def _hermite(pairs):
    """Centre, exponent, Hermite coefficients {tuv: [n]} and total l of every product."""
    dev = dict(device="cuda", dtype=torch.float64)
    A, B = torch.tensor(pairs.A, **dev), torch.tensor(pairs.B, **dev)
    alpha, beta, w = (torch.tensor(v, **dev) for v in (pairs.alpha, pairs.beta, pairs.w))
    la, lb = torch.tensor(pairs.la, device="cuda").long(), torch.tensor(pairs.lb, device="cuda").long()
    p = alpha + beta
    P = (alpha[:, None] * A + beta[:, None] * B) / p[:, None]
    dims = []
    for d in range(3):
        XA, XB, X = P[:, d] - A[:, d], P[:, d] - B[:, d], A[:, d] - B[:, d]
        zero = torch.zeros_like(p)
        E = {(0, 0): [torch.exp(-alpha * beta / p * X * X)] + [zero] * 6}
        for i in range(3):
            for j in range(3):
                if (i, j) == (0, 0):
                    continue
                src, s = (E[i - 1, j], XA) if i else (E[i, j - 1], XB)
                E[i, j] = [(src[t - 1] / (2 * p) if t else zero) + s * src[t] + (t + 1) * src[t + 1]
                           for t in range(6)] + [zero]
        table = torch.stack([torch.stack(E[i, j][:5], 1) for i in range(3) for j in range(3)], 1)
        dims.append(table[torch.arange(len(pairs), device="cuda"), la[:, d] * 3 + lb[:, d]])
    D = {(t, u, v): w * dims[0][:, t] * dims[1][:, u] * dims[2][:, v]
         for t in range(5) for u in range(5 - t) for v in range(5 - t - u)}
    return P, p, D, (la + lb).sum(1)


def _gaussians(pairs, C, V):
    P, p, D, ltot = _hermite(pairs)
    for L in range(5):
        sel = (ltot == L).nonzero()[:, 0]
        for k0 in range(0, sel.numel(), 4096):
            k = sel[k0:k0 + 4096]
            Pk, pk = P[k], p[k]
            Dk = {q: (D[q][k] * 2 * math.pi / pk)[:, None] for q in D if sum(q) <= L}
            rows = max(1, 4_000_000 // k.numel())
            for i0 in range(0, C.shape[0], rows):
                X = Pk[:, None, :] - C[None, i0:i0 + rows, :]
                F = _boys(L, pk[:, None] * (X * X).sum(-1))
                R = {(0, 0, 0): [(-2 * pk[:, None]) ** n * F[n] for n in range(L + 1)]}
                for N in range(1, L + 1):
                    for q in [q for q in Dk if sum(q) == N]:
                        d = next(d for d in range(3) if q[d])
                        one = tuple(q[e] - (e == d) for e in range(3))
                        two = tuple(q[e] - 2 * (e == d) for e in range(3))
                        R[q] = [X[..., d] * R[one][n + 1] + ((q[d] - 1) * R[two][n + 1] if q[d] > 1 else 0.0)
                                for n in range(L + 1 - N)]
                V[i0:i0 + rows] += sum(Dk[q] * R[q][0] for q in Dk).sum(0)


def _potential(R, Z, pairs, pos):
    dev = dict(device="cuda", dtype=torch.float64)
    C, R, Z = torch.tensor(pos, **dev), torch.tensor(R, **dev), torch.tensor(Z, **dev)
    V = torch.zeros(C.shape[0], **dev)
    rows = max(1, 20_000_000 // max(1, R.shape[0]))
    for i0 in range(0, C.shape[0], rows):
        V[i0:i0 + rows] = (Z / (C[i0:i0 + rows, None, :] - R[None]).square().sum(-1).sqrt()).sum(1)
    if len(pairs):
        _gaussians(pairs, C, V)
    return V


def exact(case, seed):
    V = [_potential(*s) for s in _inputs(case, seed)]
    if case["kind"] == "walkers":
        return {"V": V[0], "E": -V[0].view(case["n"], case["electrons"]).sum(1)}
    if case["kind"] == "train":
        return {"V": V[0], "weights": None}
    return V if case["kind"] == "batch" else V[0]
