"""What this library is used for, as cases that can be timed and checked.

A case is one pass of a user's program: decoding a batch of sampled syndromes
(``coset_logprob``, ``decode``, the host-buffer call), the generator picture of the loop
sector, the layer sweep on its own, and the gradient of the mean log-probability.  The
problems are the ones of the tests and the benchmark: the rotated surface code under
phenomenological noise, the point and the loop sector of the 3D surface code.

``exact`` is the decoding method itself in plain numpy FP64, written from its definition:
QR-reduced simple update of every two-site gate, boundary-MPS zip-up of the last 2D network;
the untruncated point sector is summed exactly over all boundary states.
"""
import math

import numpy as np
import torch

import paper_2310_10722_gb300 as td

FP64, FP32, TC = "fp64", "fp32", "tc"
_PRECISION = {FP64: td.TD_FP64, FP32: td.TD_FP32, TC: td.TD_TC}
_GIB = 1 << 30


def _case(name, kind, d, batch, chi, chi_mps, precision, rounds=0, p=0.03, call="logp"):
    c = {"kind": kind, "d": d, "rounds": rounds, "p": p, "batch": batch, "chi": chi, "chi_mps": chi_mps,
         "precision": precision, "call": call}
    return {"name": name, **c} if name else c


def listed():
    return [
        # one syndrome as it arrives, small enough for an untruncated contraction: latency
        _case("point d3 exact, 1 shot", "point", 3, 1, 8, 64, FP64, p=0.05),
        # the same network over the stored batch of an exact reference run
        _case("point d3 exact, 512 shots", "point", 3, 512, 8, 64, FP64, p=0.05),
        # a small code decoded online in short ragged batches; the program reads the decisions
        _case("rotated d5 decode, 37 shots", "rotated", 5, 37, 8, 8, TC, rounds=4, call="decode"),
        # offline decoding from host buffers with FP32 storage, copies included
        _case("rotated d5 host buffers, 300", "rotated", 5, 300, 8, 8, FP32, rounds=4, call="host"),
        # the benchmark's workload, a ragged batch of it
        _case("rotated d9, 1000 shots", "rotated", 9, 1000, 8, 8, TC, rounds=9),
        # the plain FP64 path at the benchmark's bond caps
        _case("rotated d9 FP64, 152 shots", "rotated", 9, 152, 8, 8, FP64, rounds=9),
        # a network built with the default options (FP64, chi 8, chi_mps 16)
        _case("rotated d7 defaults, 48 shots", "rotated", 7, 48, 8, 16, FP64, rounds=7),
        # the point sector near its threshold, one code size of a mixed batch
        _case("point d5 chi16, 152 shots", "point", 5, 152, 16, 8, TC, p=0.1),
        # the bond caps of the published point-sector runs
        _case("point d4 chi24 mps32, 8 shots", "point", 4, 8, 24, 32, TC, p=0.08),
        # the loop sector, decoded in the generator picture
        _case("loop d5, 64 shots", "loop", 5, 64, 8, 16, TC, p=0.2),
        # the layer sweep on its own: every gate's truncation, no final contraction
        _case("sweep rotated d9 chi16, 16", "rotated", 9, 16, 16, 16, TC, rounds=9, call="sweep"),
        # one step of a noise-model fit: log P and its gradient over all rates
        _case("gradient rotated d7, 152", "rotated", 7, 152, 8, 8, FP64, rounds=7, p=0.005, call="grad"),
    ]


def draw(rng):
    """A case of the same ranges: kind, size, caps, precision and batch drawn, the batch cut
    to what the largest listed cases cost."""
    while True:
        kind = rng.choice(["rotated", "rotated", "rotated", "point", "loop"])
        call, rounds = "logp", 0
        if kind == "rotated":
            d = rng.choice([3, 5, 5, 7, 7, 9])
            rounds = rng.randint(max(1, d // 2), d)
            call = rng.choice(["logp", "logp", "decode", "host", "sweep", "grad"])
            p = round(rng.uniform(0.02, 0.04), 4) if call != "grad" else round(rng.uniform(0.004, 0.008), 4)
            chi = rng.randint(4, 10) if call != "sweep" else rng.randint(6, 18)
            chi_mps = rng.randint(6, 18) if call != "grad" else 8
            precision = FP64 if call == "grad" else rng.choice([FP64, TC, TC])
        elif kind == "point":
            d = rng.choice([3, 4, 4, 5])
            p = round(rng.uniform(0.04, 0.1), 4)
            chi, chi_mps = rng.randint(6, 18), rng.randint(6, 20)
            precision = rng.choice([FP64, TC, TC])
        else:
            d, p = rng.choice([3, 4, 5]), round(rng.uniform(0.12, 0.22), 4)
            chi, chi_mps = rng.randint(4, 10), rng.randint(6, 18)
            precision = rng.choice([FP64, TC])
        batch = int(round(2.0 ** rng.uniform(0.0, 10.0)))
        c = _case("", kind, d, batch, chi, chi_mps, precision, rounds, p, call)
        while c["batch"] > 1 and _seconds(c) > 0.7:
            c["batch"] = max(1, int(c["batch"] * 0.7))
        if _seconds(c) <= 0.7:
            return c


# ---- the problems ---------------------------------------------------------------------------
class _Problem:
    """A layered problem: sites (x, y), `layers` layers, and mechanisms in order, each
    (detectors, flips the class, rate); detector t * S + s sits at site s of layer t."""

    def __init__(self, sites, layers):
        self.sites, self.layers, self.S = sites, layers, len(sites)
        self.mechs = []

    def add(self, dets, flips, p):
        self.mechs.append((tuple(dets), flips, p))

    def rates(self):
        return np.array([m[2] for m in self.mechs])

    def csr(self):
        rows = [[] for _ in range(self.S * self.layers)]
        for j, (dets, _, _) in enumerate(self.mechs):
            for i in dets:
                rows[i].append(j)
        return _rows_csr(rows)

    def xyt(self):
        return np.array([(x, y, t) for t in range(self.layers) for (x, y) in self.sites], dtype=np.int32)

    def gates(self, t):
        """(first site, second site, rate) of the layer's two-detector mechanisms, in the order in
        which they are applied: bonds along x from even then odd x, then along y."""
        out = []
        for dets, _, p in self.mechs:
            if len(dets) == 2 and dets[0] // self.S == t and dets[1] // self.S == t:
                a, b = sorted(i % self.S for i in dets)
                (x, y), (x2, y2) = self.sites[a], self.sites[b]
                colour = (x % 2) if y == y2 else 2 + (y % 2)
                out.append(((colour, y, x), a, b, p))
        return [g[1:] for g in sorted(out, key=lambda g: g[0])]


def _rows_csr(rows):
    ptr = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int32)
    return ptr, np.array([j for r in rows for j in r], dtype=np.int32)


def _rotated(d, rounds, p, q):
    """Rotated surface code: data flips before every round, measurement flips on all but the
    last; the class is the parity of the flips on qubit column 0."""
    checks = []
    for i in range(-1, d):
        for j in range(d - 1):
            inside = 0 <= i < d - 1
            if (i + j) % 2 == 0 and (inside or (i == -1 and j % 2 == 1) or i == d - 1):
                qubits = [(a, b) for a in (i, i + 1) for b in (j, j + 1) if 0 <= a < d and 0 <= b < d]
                checks.append((((i + j) // 2, (i - j + d - 1) // 2), qubits))
    checks.sort(key=lambda c: (c[0][1], c[0][0]))
    pr = _Problem([c[0] for c in checks], rounds + 1)
    of = {}
    for s, (_, qubits) in enumerate(checks):
        for qubit in qubits:
            of.setdefault(qubit, []).append(s)
    for t in range(rounds + 1):
        for i in range(d):
            for j in range(d):
                pr.add([t * pr.S + s for s in of[i, j]], int(j == 0), p)
        if t < rounds:
            for s in range(pr.S):
                pr.add([t * pr.S + s, (t + 1) * pr.S + s], 0, q)
    return pr


def _point(d, p):
    """Point sector of the 3D surface code: vertex checks on d x d x (d-1), one mechanism per
    edge; the class is the parity of the edges dangling below layer 0."""
    pr = _Problem([(x, y) for y in range(d) for x in range(d)], d - 1)
    for t in range(d - 1):
        base = t * d * d
        if t == 0:
            for s in range(d * d):
                pr.add([s], 1, p)
        for y in range(d):
            for x in range(d - 1):
                pr.add([base + y * d + x, base + y * d + x + 1], 0, p)
        for y in range(d - 1):
            for x in range(d):
                pr.add([base + y * d + x, base + (y + 1) * d + x], 0, p)
        for s in range(d * d):
            pr.add([base + s] + ([base + d * d + s] if t < d - 2 else []), 0, p)
    return pr


class _Loop:
    """Loop sector: flips on the edges of the point sector's lattice, seen by its plaquettes."""

    def __init__(self, d, p):
        self.point = _point(d, p)
        self.d, self.p = d, p
        n = d * d
        self.edges = [m[0] for m in self.point.mechs]
        self.below = list(range(n))                       # the edges dangling below layer 0
        two = {e: j for j, e in enumerate(self.edges) if len(e) == 2}
        top = [j for j, e in enumerate(self.edges) if len(e) == 1 and j >= n]
        # vertical edge entering (site, layer) from below; layer d - 1: dangling above
        self.vertical = [[self.below[s] if t == 0 else top[s] if t == d - 1 else two[(t - 1) * n + s, t * n + s]
                          for s in range(n)] for t in range(d)]
        checks = []
        for t in range(d - 1):
            for y in range(d - 1):
                for x in range(d - 1):
                    a = t * n + y * d + x
                    checks.append([two[a, a + 1], two[a + d, a + d + 1], two[a, a + d], two[a + 1, a + d + 1]])
        for t in range(d):                                  # squares standing on layer t - 1 and t
            for step, sx, sy in ((1, 1, 0), (d, 0, 1)):
                for y in range(d - sy):
                    for x in range(d - sx):
                        s = y * d + x
                        face = [self.vertical[t][s], self.vertical[t][s + step]]
                        face += [two[u * n + s, u * n + s + step] for u in (t - 1, t) if 0 <= u < d - 1]
                        checks.append(face)
        self.checks = [sorted(c) for c in checks]
        self.zbar = [self.vertical[t][0] for t in range(d)]


def _problem(c):
    if c["kind"] == "rotated":
        return _rotated(c["d"], c["rounds"], c["p"], c["p"])
    return _point(c["d"], c["p"]) if c["kind"] == "point" else _Loop(c["d"], c["p"])


def _columns(pr):
    """Rows of the check matrix as lists of mechanisms, and the rates."""
    if isinstance(pr, _Loop):
        return pr.checks, np.full(len(pr.edges), pr.p)
    ptr, idx = pr.csr()
    return [idx[ptr[i]:ptr[i + 1]].tolist() for i in range(len(ptr) - 1)], pr.rates()


def _syndromes(pr, batch, seed, rates=None):
    """Syndromes of `batch` independent error patterns, uint8 [batch, checks] on the host."""
    rows, p = _columns(pr)
    p = p if rates is None else rates
    rng = np.random.Generator(np.random.PCG64(seed))
    flips = rng.random((batch, len(p))) < p
    return np.stack([np.bitwise_xor.reduce(flips[:, r], axis=1) for r in rows], axis=1).astype(np.uint8)


def _fit_rates(pr, c, seed):
    """Rates of a noise-model fit: spread log-uniformly around the case's p."""
    rng = np.random.Generator(np.random.PCG64(seed + 1))
    return c["p"] * np.exp(rng.uniform(-1.0, 1.0, len(pr.mechs)))


def prepare(case, seed):
    pr, B = _problem(case), case["batch"]
    kw = dict(chi=case["chi"], chi_mps=case["chi_mps"], precision=_PRECISION[case["precision"]],
              mem_budget=40 * _GIB, max_wave=B)
    state = {"call": case["call"]}
    if case["kind"] == "loop":
        gens = np.array([list(e) + [-1] * (2 - len(e)) for e in pr.edges], dtype=np.int32)
        n = pr.d * pr.d
        xyt = np.array([(s % pr.d, s // pr.d, t) for t in range(pr.d - 1) for s in range(n)], dtype=np.int32)
        kw["max_wave"] = 2 * B                      # every shot is two sweeps
        state["net"] = td.GenNetwork(gens, np.full(len(pr.edges), pr.p), xyt, *_rows_csr(pr.checks), pr.below, pr.zbar, **kw)
        syn = _syndromes(pr, B, seed)
    else:
        rates = _fit_rates(pr, case, seed) if case["call"] == "grad" else pr.rates()
        flips = np.array([j for j, m in enumerate(pr.mechs) if m[1]], dtype=np.int32)
        state["net"] = td.Network(*pr.csr(), np.array([0, len(flips)], dtype=np.int32), flips, rates, pr.xyt(),
                                  n_mech=len(pr.mechs), **kw)
        syn = _syndromes(pr, B, seed, rates)
    if case["call"] == "host":
        state["syn"] = torch.from_numpy(syn).pin_memory()
        state["out"] = torch.empty((B, 2), dtype=torch.float64).pin_memory()
    else:
        state["syn"] = torch.from_numpy(syn).cuda()
    state["gates"] = state["net"].info()["n_gates"]
    return state


def run(state):
    net, syn, call = state["net"], state["syn"], state["call"]
    if call == "logp":
        return {"logp": net.coset_logprob(syn)}
    if call == "decode":
        decision, margin = net.decode(syn)
        return {"decision": decision, "margin": margin}
    if call == "host":
        return {"logp": net.coset_logprob_host(syn, out=state["out"])}
    if call == "sweep":
        weights, scales, _ = net.debug_sweep(syn, state["gates"])
        return {"weights": weights, "scales": scales}
    logP, grad = net.grad_logprob(syn)
    return {"logP": logP, "grad": grad}


# ---- work -----------------------------------------------------------------------------------
def _bonds(pr):
    """Bonds in the order of their site pairs, and each site's bonds as left, right, down, up."""
    pairs = sorted({g[:2] for t in range(pr.layers) for g in pr.gates(t)})
    at = {xy: s for s, xy in enumerate(pr.sites)}
    site = []
    for x, y in pr.sites:
        s = at[x, y]
        row = []
        for xy in ((x - 1, y), (x + 1, y), (x, y - 1), (x, y + 1)):
            key = tuple(sorted((s, at[xy]))) if xy in at else None
            row.append(pairs.index(key) if key in pairs else -1)
        site.append(row)
    return pairs, site


def _counters(pr, kind):
    """Sites that carry a class bit: those of class-flipping single mechanisms before the last
    layer (the point sector counts its class at the readout instead)."""
    return {m[0][0] % pr.S for m in pr.mechs if kind == "rotated" and m[1] and len(m[0]) == 1 and m[0][0] // pr.S < pr.layers - 1}


def _flops(c):
    """Multiply-adds (x 2) of one shot: (sweep, final contraction), every bond at min(chi, 2^gates):
    Gram, truncation core and update of every gate; zip-up products and the chi_mps leading
    singular pairs of every cut (one pass of products with its matrix and its transpose each for
    a QR-reduced cut)."""
    pr = _problem(c)
    lay = pr.point if isinstance(pr, _Loop) else pr
    chi, cm = c["chi"], c["chi_mps"]
    pairs, site = _bonds(lay)
    count = _counters(lay, c["kind"])
    dim = [1] * len(pairs)
    sweep = 0.0
    for t in range(lay.layers):
        for a, b, _ in lay.gates(t):
            bond = pairs.index((a, b))
            D, Dn = dim[bond], min(chi, 2 * dim[bond])
            for s in (a, b):
                rows = (2 if s in count else 1) * math.prod(dim[k] for k in site[s] if k >= 0 and k != bond)
                sweep += 2.0 * rows * 2 * D * (D + Dn)
            sweep += 22.0 * (2 * D) ** 3 / 2
            dim[bond] = Dn
    at = {xy: s for s, xy in enumerate(lay.sites)}
    nx, ny = max(x for x, _ in lay.sites) + 1, max(y for _, y in lay.sites) + 1
    left, right = [1] * nx, [1] * (nx - 1) + [2]
    final = 0.0
    for y in range(ny):
        J, nl, nr = 1, [], []
        for x in range(nx):
            s = at.get((x, y))
            L, R, D, U = [dim[k] if k >= 0 else 1 for k in site[s]] if s is not None else (1, 1, 1, 1)
            aL, aR = left[x], right[x]
            m, n = J * U, aR * R * 2
            final += 2.0 * J * L * 2 * D * aR * aL + 2.0 * m * n * L * D
            nl.append(J)
            if x < nx - 1 and y < ny - 1:
                k = min(cm, m, n)
                final += 2.0 * min(m, n) ** 2 * max(m, n) + 4.0 * m * n * k
                J = k
            elif x < nx - 1:
                J = m
            nr.append(J if x < nx - 1 else 2)
        left, right = nl, nr
    return sweep, final


def _passes(c):
    """Sweeps of one shot: two in the generator picture; the gradient walks its sweep back."""
    return 2.0 if c["kind"] == "loop" else 3.0 if c["call"] == "grad" else 1.0


def work(case):
    sweep, final = _flops(case)
    pr, B = _problem(case), case["batch"]
    rows, p = _columns(pr)
    lay = pr.point if isinstance(pr, _Loop) else pr
    out = 16.0 * B
    if case["call"] == "sweep":
        final, out = 0.0, 8.0 * B * (len(_bonds(lay)[0]) * (case["chi"] + 1) + lay.S + 1)
    elif case["call"] == "decode":
        out = 12.0 * B
    elif case["call"] == "grad":
        out = 8.0 * B + 8.0 * len(p)
    return {"bytes": float(len(rows) * B + 8 * len(p) + out), "flops": _passes(case) * B * (sweep + final)}


def _seconds(c):
    """A rough bound on the time of a pass, for draw(): one shot of a large network cannot be
    spread over the chip, and a batch shares it."""
    sweep, final = _flops(c)
    if c["call"] == "sweep":
        final = 0.0
    k = _passes(c)
    sharp = (14.0 if c["precision"] == FP64 else 5.0) * (1.0 + c["chi"] * c["chi_mps"] / 256.0)
    one = k * (sweep / 4e10 + sharp * final / 3.0e9)
    return max(one, one * c["batch"] / 152.0 + k * sweep * c["batch"] / 2.5e11)


# ---- the method in plain numpy --------------------------------------------------------------
_CUTOFF, _MULTIPLET = 1e-12, 1e-8


class _Impossible(Exception):
    pass


def _kept(s, most):
    """How many of the descending values s a truncation keeps: those above the cutoff, at most
    `most`; a cut inside a multiplet leaves the whole multiplet out."""
    if not s[0] > 0:
        raise _Impossible
    rank = int((s > _CUTOFF * s[0]).sum())
    k = min(rank, most)
    if k < rank:
        j = k
        while j and s[j - 1] - s[j] <= _MULTIPLET * s[0]:
            j -= 1
        k = j or k
    return k


class _Boundary:
    """A PEPS over the sites of one layer: tensors [phys, left, right, down, up] and a weight
    vector on every bond (Gamma-lambda form)."""

    def __init__(self, lay, phys, chi):
        self.chi, self.lay = chi, lay
        self.pairs, self.site = _bonds(lay)
        self.lam = [np.ones(1) for _ in self.pairs]
        self.T = []
        for P in phys:
            g = np.zeros((P, 1, 1, 1, 1))
            g[0] = 1.0
            self.T.append(g)
        self.log = 0.0

    def local(self, s, M):
        g = np.tensordot(M, self.T[s], (1, 0))
        top = np.abs(g).max()
        if not top > 0:
            raise _Impossible
        self.T[s], self.log = g / top, self.log + math.log(top)

    def weighted(self, s, skip, power=1.0):
        g = self.T[s]
        for axis, k in enumerate(self.site[s]):
            if k >= 0 and k != skip:
                w = self.lam[k]
                w = np.where(w > 0, np.where(w > 0, w, 1.0) ** power, 0.0)
                shape = [1] * 5
                shape[1 + axis] = -1
                g = g * w.reshape(shape)
        return g

    def gate(self, a, b, G):
        """Applies the two-site gate G[a', b', a, b] on the physical legs (on bit 0 where a site has
        a class bit too) and truncates the bond to chi under its environment."""
        k = self.pairs.index((a, b))
        half = []
        for s in (a, b):
            axis = 1 + self.site[s].index(k)
            g = np.moveaxis(self.weighted(s, k), (axis, 0), (3, 4))         # (other bonds, bond, phys)
            g = g.reshape(g.shape[:4] + (-1, 2))                            # phys = class bit x bit 0
            g = np.moveaxis(g, 4, 3)                                        # (others, class, bond, bit)
            rest = g.shape[:4]
            q, r = np.linalg.qr(g.reshape(-1, g.shape[4] * 2))
            half.append((s, axis, rest, q, r.reshape(-1, g.shape[4], 2)))
        ra, rb = half[0][4], half[1][4]
        th = np.einsum("idx,d,jdy,uvxy->iujv", ra, self.lam[k], rb, G, optimize=True)
        u, s, vt = np.linalg.svd(th.reshape(th.shape[0] * 2, -1), full_matrices=False)
        n = _kept(s, self.chi)
        self.lam[k], self.log = s[:n] / s[0], self.log + math.log(s[0])
        for (site, axis, rest, q, _), w in zip(half, (u[:, :n], vt[:n].T)):
            g = np.tensordot(q, w.reshape(-1, 2, n), (1, 0)).reshape(rest + (2, n))
            g = g.reshape(rest[:3] + (-1, n))                               # (others, phys, bond)
            self.T[site] = np.moveaxis(g, (4, 3), (axis, 0))
            self.T[site] = self.weighted(site, k, -1.0)

    def contract(self, readout, most):
        """log weights of the two classes: zip-up boundary MPS of at most `most` states per bond."""
        lay = self.lay
        at = {xy: s for s, xy in enumerate(lay.sites)}
        nx, ny = max(x for x, _ in lay.sites) + 1, max(y for _, y in lay.sites) + 1
        log = self.log
        mps = [np.ones((1, 1, 1)) for _ in range(nx)]
        mps[-1] = np.array([[[1.0, 0.0]]])
        for y in range(ny):
            carry, out = np.array([[[[1.0, 0.0]]]]), []                     # [new, old, bond, class]
            for x in range(nx):
                s = at.get((x, y))
                if s is None:
                    F = np.array([1.0, 0.0]).reshape(2, 1, 1, 1, 1)
                else:
                    F = np.tensordot(readout[s].T, self.weighted(s, -1, 0.5), (1, 0))
                t = np.einsum("jalp,adb->jlpdb", carry, mps[x])
                full = [np.einsum("jldb,lrdu->jubr", t[:, :, i], F[c]) for i, c in ((0, 0), (0, 1), (1, 0), (1, 1))]
                M = np.stack([full[0] + full[3], full[1] + full[2]], axis=-1)   # class = incoming + site's
                J, U, Bd, R, _ = M.shape
                if x == nx - 1:
                    o = np.zeros((J, U, 2))
                    for old in range(Bd):
                        for c in range(2):
                            o[:, :, old ^ c] += M[:, :, old, 0, c]
                    top = np.abs(o).max()
                    if not top > 0:
                        raise _Impossible
                    out.append(o / top)
                    log += math.log(top)
                elif y == ny - 1:
                    out.append(np.eye(J * U).reshape(J, U, J * U))
                    carry = M.reshape(J * U, Bd, R, 2)
                else:
                    u, sv, vt = np.linalg.svd(M.reshape(J * U, -1), full_matrices=False)
                    k = _kept(sv, most)
                    out.append(u[:, :k].reshape(J, U, k))
                    carry = (sv[:k, None] / sv[0] * vt[:k]).reshape(k, Bd, R, 2)
                    log += math.log(sv[0])
            mps = out
        v = np.ones(1)
        for A in mps:
            v = v @ A[:, 0]
        with np.errstate(divide="ignore"):
            return np.log(np.maximum(v, 0.0)) + log


def _flip_gate(p):
    G = np.zeros((2, 2, 2, 2))
    for x in range(2):
        for y in range(2):
            G[x, y, x, y] += 1.0 - p
            G[x ^ 1, y ^ 1, x, y] += p
    return G


class _Detector:
    """The detector picture of a _Problem: what every layer applies."""

    def __init__(self, pr, kind):
        self.pr = pr
        count = _counters(pr, kind)
        self.phys = [4 if s in count else 2 for s in range(pr.S)]
        self.offset = kind == "point"                       # class counted at the top plane
        last = pr.layers - 1
        self.K = [[np.eye(P) for P in self.phys] for _ in range(pr.layers)]
        out = [np.array([[1.0, 0.0], [0.0, 0.0]]) for _ in range(pr.S)]     # weight of [last bit][its class]
        up = [[None] * pr.S for _ in range(pr.layers)]
        for dets, flips, p in pr.mechs:
            s, t = dets[0] % pr.S, dets[0] // pr.S
            if len(dets) == 1:
                flips ^= int(self.offset)
                if t == last:
                    out[s] = (1 - p) * out[s] + p * out[s][::-1][:, ::-1 if flips else 1]
                else:
                    P = self.phys[s]
                    X = np.eye(P)[np.arange(P) ^ (1 | 2 * flips)]
                    self.K[t][s] = ((1 - p) * np.eye(P) + p * X) @ self.K[t][s]
            elif dets[1] // pr.S == t + 1:
                up[t][s] = np.array([1 - p, p])
        for t in range(1, pr.layers):
            for s in range(pr.S):
                self.K[t][s] = self.K[t][s] * np.tile(up[t - 1][s], self.phys[s] // 2)[None, :]
        self.readout = [np.array([[out[s][i & 1][c ^ (i >> 1)] for c in range(2)] for i in range(P)])
                        for s, P in enumerate(self.phys)]
        self.gates = [[(a, b, _flip_gate(p)) for a, b, p in pr.gates(t)] for t in range(pr.layers)]

    def sweep(self, m, chi):
        st = _Boundary(self.pr, self.phys, chi)
        for t in range(self.pr.layers):
            for s, P in enumerate(self.phys):
                st.local(s, self.K[t][s][np.arange(P) ^ int(m[t * self.pr.S + s])])
            for a, b, G in self.gates[t]:
                st.gate(a, b, G)
        return st

    def logp(self, m, chi, most):
        try:
            lp = self.sweep(m, chi).contract(self.readout, most)
        except _Impossible:
            return np.full(2, -np.inf)
        return lp[::-1] if self.offset and m.sum() % 2 else lp


def _representatives(pr, syn):
    """For every syndrome the error on the greedy column basis of the checks that gives it."""
    rows = np.zeros((len(pr.checks), len(pr.edges)), dtype=np.uint8)
    for i, c in enumerate(pr.checks):
        rows[i, c] = 1
    M = np.concatenate([rows, syn.T], axis=1)
    r, pivots = 0, []
    for j in range(len(pr.edges)):
        hit = np.flatnonzero(M[r:, j])
        if not len(hit):
            continue
        M[[r, r + hit[0]]] = M[[r + hit[0], r]]
        others = np.flatnonzero(M[:, j])
        M[others[others != r]] ^= M[r]
        pivots.append(j)
        r += 1
    reps = np.zeros((len(syn), len(pr.edges)), dtype=np.uint8)
    reps[:, pivots] = M[:r, len(pr.edges):].T
    return reps


def _loop_row(pr, r, chi, most):
    """log weight of the coset of the error r: the sum over all vertex bits."""
    lay, w = pr.point, np.array([1 - pr.p, pr.p])
    st = _Boundary(lay, [2] * lay.S, chi)
    bit = np.arange(2)
    by_pair = {e: j for j, e in enumerate(pr.edges) if len(e) == 2}
    try:
        for t in range(lay.layers):
            for s in range(lay.S):
                st.local(s, w[bit[:, None] ^ bit[None, :] ^ r[pr.vertical[t][s]]])
            for a, b, _ in lay.gates(t):
                j = by_pair[t * lay.S + a, t * lay.S + b]
                G = np.zeros((2, 2, 2, 2))
                for x in range(2):
                    for y in range(2):
                        G[x, y, x, y] = w[r[j] ^ x ^ y]
                st.gate(a, b, G)
        read = [np.stack([w[bit ^ r[pr.vertical[lay.layers][s]]], np.zeros(2)], axis=1) for s in range(lay.S)]
        return st.contract(read, most)[0]
    except _Impossible:
        return -np.inf


def _point_sums(pr, syn, p):
    """Exact class weights of a small point sector: a vector over the bits of one layer's
    vertical edges and the class, every mechanism applied to all of it at once."""
    S, d2 = pr.S, pr.layers
    out = np.empty((len(syn), 2))
    idx = np.arange(1 << S)
    parity = np.array([bin(i).count("1") for i in range(1 << S)])
    for b, m in enumerate(syn):
        v = np.zeros((2, 1 << S))
        v[0, 0] = 1.0
        for t in range(d2):
            flip = int(sum(int(m[t * S + s]) << s for s in range(S)))
            v = v[:, idx ^ flip]
            for dets, cls, q in pr.mechs:
                if all(i // S == t for i in dets) and not (len(dets) == 1 and not cls):
                    mask = sum(1 << (i % S) for i in dets)
                    w = v[:, idx ^ mask]
                    v = (1 - q) * v + q * (w[::-1] if cls else w)
            v = v * (p ** parity * (1 - p) ** (S - parity))[None, :]
        out[b] = np.log(v.sum(axis=1))
    return out


def exact(case, seed):
    if case["call"] == "grad":
        return None
    sweep, final = _flops(case)
    if case["call"] == "sweep":
        final = 0.0
    gates = case["d"] ** 2 * (case["rounds"] + 1.0 if case["kind"] == "rotated" else 2.0 * case["d"])
    if case["batch"] * _passes(case) * (3.5e-4 * gates + 1.5e-10 * sweep + 1e-9 * final) > 18.0:
        return None         # too long on a host
    pr, chi, most = _problem(case), case["chi"], case["chi_mps"]
    syn = _syndromes(pr, case["batch"], seed)
    if case["kind"] == "loop":
        logp = np.empty((len(syn), 2))
        for b, r in enumerate(_representatives(pr, syn)):
            cls = int(r[pr.zbar].sum() % 2)
            logp[b, cls] = _loop_row(pr, r, chi, most)
            r[pr.below] ^= 1
            logp[b, 1 - cls] = _loop_row(pr, r, chi, most)
        return {"logp": logp}
    if case["kind"] == "point" and case["d"] == 3 and chi >= 8 and most >= 64:
        return {"logp": _point_sums(pr, syn, case["p"])}
    net = _Detector(pr, case["kind"])
    if case["call"] == "sweep":
        weights = np.zeros((len(syn), len(_bonds(pr)[0]), chi))
        for b, m in enumerate(syn):
            try:
                for k, lam in enumerate(net.sweep(m, chi).lam):
                    weights[b, k, :len(lam)] = lam
            except _Impossible:
                return None
        return {"weights": weights, "scales": None}
    logp = np.array([net.logp(m, chi, most) for m in syn])
    if case["call"] == "decode":
        decision = (logp[:, 1] > logp[:, 0]).astype(np.int32)
        return {"decision": decision, "margin": np.abs(logp[:, 1] - logp[:, 0])}
    return {"logp": logp}
