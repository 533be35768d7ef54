"""What a user of the sampler has it do, as cases to time and to compare.

One pass is one Markov step of a batch of chains (evolve by beta/2, measure
the cluster, collapse the environment and reset), through the public calls a
sampling program makes; the susceptibility and the sliced evolution of a
serving program are options of it.  Sizes are the repository's own: the small
workload and the benchmark ladder, the uneven and served mixes
(Lx 8-16, 2W 0-8, chi 64-256), and the ladders of the tests, with beta
shortened so that a pass stays within two seconds.

Outputs are the observables, the outcomes and log p of the step: what a
program keeps of it, and the whole updated state (a collapsed chain is its
outcomes).  The evolved tensors are not among them: they are defined only up
to the sign, or the rotation within a multiplet, of each bond index.
Binary64 chains return binary64.  The mixed forms work in binary32 and
resolve about 1e-6, so a program keeps their series in binary32, and that is
what a pass returns.  Mixed chains run at the cutoffs 1e-9 and 1e-10: at 1e-7 a
rounding that moves one kept count moves a sample by up to 1e-4, and two
binary32 results could not be told apart from two wrong ones.
"""
import math

import numpy as np
import torch

from paper_1910_09142_gb300 import binding as hm

_PREC = {"fp64": hm.HM_FP64, "mixed": hm.HM_MIXED, "mixed32": hm.HM_MIXED32}


def _case(name, Lx, two_W, beta, tau, chi_max, cutoff, precision, chains, schedule="plain", tick=0, mix=False,
          susceptibility=False, zx=True):
    return dict(name=name, Lx=Lx, two_W=two_W, beta=beta, tau=tau, chi_max=chi_max, cutoff=cutoff,
                precision=precision, chains=chains, schedule=schedule, tick=tick, mix=mix,
                susceptibility=susceptibility, zx=zx)


def listed():
    return [
        # the smallest call: one METTS chain of the tests' short ladder, binary64 (latency)
        _case("metts_one", 4, 0, 1.0, 0.1, 64, 1e-10, "fp64", 1),
        # a reference run: the small workload's ladder in binary64 at its bond cap, a few walkers
        _case("small_fp64", 4, 4, 0.8, 0.1, 64, 1e-7, "fp64", 4),
        # a mixed run of the same size: a few walkers of a short ladder
        _case("small_mixed", 4, 2, 0.6, 0.1, 256, 1e-10, "mixed", 8),
        # nearly pure purification: every column but one has its ancillas
        _case("ancilla_mixed", 5, 8, 0.2, 0.05, 256, 1e-10, "mixed", 16),
        # METTS limit on the benchmark's ladder: many environment sites, small bonds, a wide batch
        _case("metts_wide", 16, 0, 0.5, 0.05, 256, 1e-10, "mixed", 256),
        # binary64 production: one chain per SM on a middle ladder
        _case("ladder6_fp64", 6, 4, 0.5, 0.05, 96, 1e-7, "fp64", 152),
        # a wide mixed batch: two chains per SM
        _case("ladder6_mixed", 6, 4, 0.3, 0.05, 256, 1e-10, "mixed", 304),
        # odd sizes, one chain on most SMs, S^z collapses only, with the susceptibility (Eq. sus)
        _case("ladder7_sus", 7, 4, 0.3, 0.07, 199, 1e-9, "mixed", 131, zx=False, susceptibility=True),
        # fused schedule, binary32 decompositions, a wide cluster
        _case("ladder9_fused32", 9, 8, 0.3, 0.05, 256, 1e-9, "mixed32", 152, schedule="fused"),
        # a serving program: chains of several sizes advanced in slices of 64 ops
        _case("served_mix", 8, 4, 0.4, 0.05, 256, 1e-9, "mixed", 44, tick=64, mix=True),
        # the benchmark ladder and batch (Lx = 16, 2W = 8, chi = 256, 256 chains); beta and the
        # cutoff lowered together, so that the bonds are as wide and a pass is short
        _case("ladder16", 16, 8, 0.3, 0.05, 256, 1e-9, "mixed", 256),
    ]


def draw(rng):
    """A ladder, an option set and a batch from the same ranges."""
    precision = rng.choice(["fp64", "mixed", "mixed", "mixed32"])
    two_W = rng.choice([0, 2, 4, 4, 6, 8])
    Lx = rng.randint(max(3, two_W // 2 + 1), {0: 16, 2: 14, 4: 12, 6: 11, 8: 10}[two_W])
    top = {0: 1.0, 2: 0.5, 4: 0.4, 6: 0.35, 8: 0.3}[two_W]
    beta = round(math.exp(rng.uniform(math.log(0.15), math.log(top))), 3)
    lo, cutoff = (48, 1e-7) if precision == "fp64" else (180, rng.choice([1e-9, 1e-10]))
    chi = int(round(math.exp(rng.uniform(math.log(lo), math.log(256)))))
    chains = int(round(math.exp(rng.uniform(0.0, math.log(160 if precision == "fp64" else 320)))))
    c = _case("", Lx, two_W, beta, rng.choice([0.05, 0.07, 0.1]), chi, cutoff, precision, chains,
              schedule=rng.choice(["plain", "plain", "fused"]), tick=rng.choice([0, 0, 0, 64]),
              mix=rng.random() < 0.2, susceptibility=rng.random() < 0.15, zx=rng.random() < 0.8)
    del c["name"]
    return c


def _ladders(case):
    """(Lx, two_W, chi_max) of every chain: alike, or a mix around the case's sizes."""
    Lx, W, chi = case["Lx"], case["two_W"], case["chi_max"]
    if not case["mix"]:
        return [(Lx, W, chi)] * case["chains"]
    alt = [(Lx, W, chi), (max(4, Lx - 3), max(0, W - 2), chi), (max(4, Lx - 1), max(0, W - 2), chi * 3 // 4),
           (max(4, Lx // 2), min(W, 2), chi)]
    return [alt[i % len(alt)] for i in range(case["chains"])]


def prepare(case, seed):
    ps = [hm.params(Lx, W, beta=case["beta"], tau=case["tau"], chi_max=chi, cutoff=case["cutoff"],
                    precision=_PREC[case["precision"]], seed=seed, chain_id=i, basis_zx=case["zx"],
                    schedule=case["schedule"], susceptibility=case["susceptibility"])
          for i, (Lx, W, chi) in enumerate(_ladders(case))]
    ctx = hm.Context(sum(hm.query_memory(p) for p in ps) + (4 << 20))
    ids = [ctx.init_chain(p) for p in ps]
    # chains of one kind share the output arrays of a measurement
    groups = {}
    for i, p in enumerate(ps):
        groups.setdefault((hm.num_obs(p), hm.num_env(p)), []).append(ids[i])
    out = []
    for (n_obs, n_env), members in groups.items():
        n = len(members)
        out.append(dict(ids=members, obs=torch.empty(n, n_obs, dtype=torch.float64, device="cuda"),
                        env=torch.empty(n, n_env, dtype=torch.int8, device="cuda"),
                        logp=torch.empty(n, dtype=torch.float64, device="cuda")))
    return dict(case=case, ctx=ctx, ids=ids, groups=out)


def run(state):
    case, ctx, ids = state["case"], state["ctx"], state["ids"]
    if case["tick"]:
        left = ids
        while left:                                # a serving program's ticks
            done = ctx.evolve_partial(left, case["tick"])
            left = [c for c, d in zip(left, done) if not d]
    else:
        ctx.evolve(ids)
    keep = torch.float64 if case["precision"] == "fp64" else torch.float32
    result = []
    for g in state["groups"]:
        ctx.measure_device(g["ids"], g["obs"])
        r = {"obs": g["obs"].to(keep)}
        if case["susceptibility"]:
            r["chi"] = torch.from_numpy(ctx.susceptibility(g["ids"])).to(keep)
        ctx.collapse_device(g["ids"], g["env"], g["logp"])
        r["env"], r["logp"] = g["env"], g["logp"].to(keep)
        result.append(r)
    return result


def _power(case, Lx, two_W, c):
    """exp of a form in the sizes, fitted (within about 1.6x) on 56 cases of these ranges."""
    b = math.log(case["beta"])
    return math.exp(c[0] + c[1] * two_W + c[2] * b - c[3] * math.log10(case["cutoff"]) + c[4] * math.log(Lx) +
                    c[5] * two_W * b + c[6] * two_W * two_W)


def work(case):
    """Arithmetic of one pass: theta's charge blocks and one decomposition
    4 m^2 n + 8 m n^2 + 9 n^3 of each, as the library's own statistics count
    them (flops a split); bytes: the evolved tensors, written by the evolution and
    read by the measurement and the collapse, and the outputs.  Both follow the bond
    dimensions, which only the evolution itself knows: hence the fits."""
    flops = moved = 0.0
    for Lx, W, chi in _ladders(case):
        p = hm.params(Lx, W, beta=case["beta"], tau=case["tau"], chi_max=chi, cutoff=case["cutoff"],
                      schedule=case["schedule"])
        flops += len(hm.plan(p)) * _power(case, Lx, W, (4.74, 1.229, 2.124, 0.637, 0.777, -0.086, -0.087))
        moved += 2 * _power(case, Lx, W, (5.875, 0.784, 1.763, 0.478, 1.312, -0.082, -0.051))
        moved += 8 * (hm.num_obs(p) + 1) + hm.num_env(p)
    return {"bytes": moved, "flops": flops}


# ---- the same step in plain numpy, 64 bits, one chain at a time, no charge blocks ----

_SZ = np.diag([1.0, 0.0, -1.0])
_SP = math.sqrt(2.0) * np.eye(3, k=1)


def _sites_and_bonds(Lx, two_W):
    """Site kinds ('e' environment, 'c' cluster, 'a' ancilla) and the sorted
    bonds (i, j) of the ladder in column-major order, an ancilla after its site."""
    w = two_W // 2
    x0 = (Lx - w) // 2
    kinds, at = [], {}
    for x in range(Lx):
        for y in (0, 1):
            at[x, y] = len(kinds)
            kinds += ["c", "a"] if x0 <= x < x0 + w else ["e"]
    bonds = [(at[x, 0], at[x, 1]) for x in range(Lx)]
    bonds += [(at[x, y], at[x + 1, y]) for x in range(Lx - 1) for y in (0, 1)]
    cols = range(x0, x0 + w) if w else range(Lx)
    inside = {at[x, y] for x in cols for y in (0, 1)}
    bonds.sort()
    return kinds, bonds, inside


def _splits(bonds, steps):
    """The second-order sweep as two-site splits and centre moves:
    (left site, 'swap' | 'gate', centre after: 0 left / 1 right) or ('move', to)."""
    order = [(b, d) for _ in range(steps) for d in (1, -1) for b in (bonds if d > 0 else bonds[::-1])]
    out, centre = [], 0
    for n, ((i, j), d) in enumerate(order):
        start = i if d > 0 else j
        if centre != start:
            out.append(("move", start))
        if d > 0:
            part = [[k, "swap", 1] for k in range(i, j - 1)] + [[j - 1, "gate", 0]]
            part += [[k, "swap", 0] for k in range(j - 2, i - 1, -1)]
        else:
            part = [[k, "swap", 0] for k in range(j - 1, i, -1)] + [[i, "gate", 1]]
            part += [[k, "swap", 1] for k in range(i + 1, j)]
        (ni, nj), nd = order[n + 1] if n + 1 < len(order) else ((0, 0), 1)
        part[-1][2] = 0 if (ni if nd > 0 else nj) <= part[-1][0] else 1
        centre = part[-1][0] + part[-1][2]
        out += [tuple(x) for x in part]
    if centre:
        out.append(("move", 0))
    return out


def _fused(ops):
    """Runs of splits on one pair as one split: a list of (left site, letters, side) and moves;
    two swaps in a row cancel."""
    out = []                                       # [site, letters, side, centre before]
    centre = 0
    for op in ops:
        if op[0] == "move":
            out.append(["move", op[1]])
            centre = op[1]
            continue
        k, what, side = op
        if out and out[-1][0] == k:
            top = out[-1]
            top[1] = top[1] + [what]
            top[2] = side
            if top[1][-2:] == ["swap", "swap"]:
                top[1] = top[1][:-2]
            if not top[1]:
                out.pop()
                if top[3] != k + side:
                    out.append(["move", k + side])
        else:
            out.append([k, [what], side, centre])
        centre = k + side
    return [tuple(x[:3]) for x in out]


def _move(A, c, to):
    while c < to:
        q, r = np.linalg.qr(A[c].reshape(-1, A[c].shape[2]))
        A[c] = q.reshape(A[c].shape[0], 3, -1)
        A[c + 1] = np.tensordot(r, A[c + 1], 1)
        c += 1
    while c > to:
        q, r = np.linalg.qr(A[c].reshape(A[c].shape[0], -1).T)
        A[c] = q.T.reshape(-1, 3, A[c].shape[2])
        A[c - 1] = np.tensordot(A[c - 1], r.T, 1)
        c -= 1


def _split(A, k, gate, side, chi_max, cutoff):
    th = np.einsum("abst,lstr->labr", gate, np.tensordot(A[k], A[k + 1], 1))
    l, r = th.shape[0], th.shape[3]
    u, s, v = np.linalg.svd(th.reshape(3 * l, 3 * r), full_matrices=False)
    w = np.append(np.cumsum((s * s)[::-1])[::-1], 0.0)
    n = min(max(1, int(np.argmax(w <= cutoff * w[0]))), chi_max)
    while 1 < n < len(s) and s[n] >= s[n - 1] * (1 - 1e-8):
        n -= 1
    u, v, s = u[:, :n], v[:n], s[:n] / np.linalg.norm(s[:n])
    A[k] = (u if side else u * s).reshape(l, 3, n)
    A[k + 1] = (s[:, None] * v if side else v).reshape(n, 3, r)


def _through(E, a, op=None):
    x = np.tensordot(E, a, 1)                      # bra, s, ket
    if op is not None:
        x = np.einsum("st,btk->bsk", op, x)
    return np.tensordot(a, x, ((0, 1), (0, 1)))


def _philox(counter, key):
    m = 0xFFFFFFFF
    c, k = list(counter), list(key)
    for r in range(10):
        p, q = 0xD2511F53 * c[0], 0xCD9E8D57 * c[2]
        c = [(q >> 32) ^ c[1] ^ k[0], q & m, (p >> 32) ^ c[3] ^ k[1], p & m]
        k = [(k[0] + 0x9E3779B9) & m, (k[1] + 0xBB67AE85) & m]
    return ((c[0] >> 5) * 67108864 + (c[1] >> 6)) / 9007199254740992.0


def _draw3(p, u):
    return next((b for b, c in enumerate(np.cumsum(p)) if u < c), 2)


def _first_step(case, seed, chain, Lx, two_W, chi_max):
    """Observables, outcomes and log p of sample 0 (S^z collapse) of one chain."""
    kinds, bonds, inside = _sites_and_bonds(Lx, two_W)
    n_env = kinds.count("e")

    def uniform(n, e):
        return _philox((n & 0xFFFFFFFF, e, seed >> 32, 0), (seed & 0xFFFFFFFF, chain))
    env = [_draw3([1 / 3.0] * 3, uniform(-1, e)) for e in range(n_env)]
    A, e = [], 0
    for kind in kinds:
        if kind == "e":
            A.append(np.eye(3)[env[e]].reshape(1, 3, 1))
            e += 1
        else:
            A.append(np.eye(3).reshape(1, 3, 3) / math.sqrt(3.0) if kind == "c" else np.eye(3).reshape(3, 3, 1))
    steps = max(1, int(math.floor(case["beta"] / (2 * case["tau"]) + 0.5)))
    h = np.kron(_SZ, _SZ) + 0.5 * (np.kron(_SP, _SP.T) + np.kron(_SP.T, _SP))
    w, v = np.linalg.eigh(h)
    g = (v * np.exp(-0.25 * case["beta"] / steps * w)) @ v.T
    letters = {"gate": g, "swap": np.eye(9).reshape(3, 3, 9).transpose(1, 0, 2).reshape(9, 9)}
    ops = _splits(bonds, steps)
    ops = _fused(ops) if case["schedule"] == "fused" else [o if o[0] == "move" else (o[0], [o[1]], o[2]) for o in ops]
    centre = 0
    for op in ops:
        if op[0] == "move":
            _move(A, centre, op[1])
            centre = op[1]
            continue
        k, word, side = op
        gate = np.eye(9)
        for x in word:
            gate = letters[x] @ gate
        _split(A, k, gate.reshape(3, 3, 3, 3), side, chi_max, case["cutoff"])
        centre = k + side
    n = len(A)
    R = [np.ones((1, 1))]
    for a in A[::-1]:
        R.append(_through(R[-1], a.transpose(2, 1, 0)))
    R = R[::-1]                                    # R[k]: sites >= k
    L = [np.ones((1, 1))]
    for a in A:
        L.append(_through(L[-1], a))
    norm = R[0][0, 0]

    def pair(i, j, p, q):
        E = _through(L[i], A[i], p)
        for k in range(i + 1, j):
            E = _through(E, A[k])
        return np.sum(_through(E, A[j], q) * R[j + 1]) / norm
    obs = [0.0]
    for i, j in bonds:
        if i in inside and j in inside:
            zz = pair(i, j, _SZ, _SZ)
            ss = zz + 0.5 * (pair(i, j, _SP, _SP.T) + pair(i, j, _SP.T, _SP))
            obs += [ss, zz]
            obs[0] += ss
    rho, out, logp = np.ones((1, 1)), [], 0.0
    for k in range(n):
        if kinds[k] != "e":
            rho = _through(rho, A[k])
            continue
        by = [A[k][:, s].T @ rho @ A[k][:, s] for s in range(3)]
        p = np.array([np.trace(x) for x in by])
        p = p / p.sum()
        b = _draw3(p, uniform(0, len(out)))
        rho = by[b] / np.trace(by[b])
        out.append(b)
        logp += math.log(p[b])
    return obs, out, logp


def exact(case, seed):
    """One sample of every chain by the plain steps above; None where that
    would take long.  The outcomes are draws, not computed numbers."""
    if case["susceptibility"] or case["chains"] > 8 or case["Lx"] * case["beta"] > 6 or case["two_W"] > 4:
        return None
    result = {}
    for i, (Lx, W, chi) in enumerate(_ladders(case)):
        kinds, bonds, inside = _sites_and_bonds(Lx, W)
        key = (1 + 2 * sum(a in inside and b in inside for a, b in bonds), kinds.count("e"))
        result.setdefault(key, []).append(_first_step(case, seed, i, Lx, W, chi))
    return [{"obs": np.array([x[0] for x in g]), "env": None, "logp": np.array([x[2] for x in g])}
            for g in result.values()]
