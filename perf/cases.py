"""The workloads whose speed this library is judged by, each one pass through its public entry points.

A state is a chain as a simulation holds it: an MPS handle at working entanglement plus the flattened
gates of its schedule.  What a pass returns is the updated state in gauge-free form: the Schmidt values
of the updated bonds (the site blocks themselves carry an arbitrary phase per bond state, and rotations
inside degenerate ones), amplitudes of occupation patterns (each multiplies one block of every site),
the weight each truncation kept, energies, drawn patterns.  In the reduced-precision modes the
amplitudes carry the rounding of the blocks in that arbitrary basis, so there the Schmidt values and
kept weights, which come from Theta before the basis is chosen, are returned alone.
"""
import math

import numpy as np

import paper_2303_11409_gb300 as m

CUTOFF = 1e-10
PRECISION = {"fp64": m.MPS_FP64, "tf32": m.MPS_TF32, "bf16x3": m.MPS_BF16X3}


def listed():
    return [
        # one two-site update of a small chain: the shortest call there is, the latency of a single gate
        dict(name="gate2_xxz_L16_chi24", kind="gate2", model="xxz", L=16, chi=24, grow=24),
        # a Strang step of the XXZ chain (L=16, chi<=64): three layers of small sectors
        dict(name="step_xxz_L16_chi64", kind="step", model="xxz", L=16, chi=64, grow=40),
        # one tick of the serving loop: the next layer of a mix of small XXZ and Bose-Hubbard requests
        dict(name="tick_16_requests", kind="tick", requests=16, L=16, chi=64, grow=8),
        # a Strang step of a short Bose-Hubbard chain (d=5) at moderate chi
        dict(name="step_bh_L24_chi128", kind="step", model="bh", L=24, chi=128, grow=8),
        # a layer at odd sizes: odd length, ragged sectors
        dict(name="layer_bh_L33_chi333", kind="layer", model="bh", L=33, chi=333, grow=10, precision="fp64"),
        # the Bose-Hubbard chain at chi<=512 in FP64, a layer of a half-length chain
        dict(name="layer_bh_L32_chi512", kind="layer", model="bh", L=32, chi=512, grow=11, precision="fp64"),
        # boson sampling: a layer of random beam splitters on a chain half filled with single photons
        dict(name="layer_boson_L40_chi400", kind="boson", L=40, chi=400, grow=6),
        # chi=1024 with BF16x3 sector GEMMs, the middle updates of a layer
        dict(name="pair_bh_L16_chi1024_bf16x3", kind="middle", L=16, chi=1024, updates=3, precision="bf16x3"),
        # the benchmark's sector sizes (chi=2048, TF32 sector GEMMs): one middle update
        dict(name="gate2_bh_L16_chi2048_tf32", kind="middle", L=16, chi=2048, updates=1, precision="tf32"),
        # a two-site DMRG sweep of a short Bose-Hubbard chain
        dict(name="dmrg_bh_L10_chi96", kind="dmrg", L=10, chi=96, grow=6),
        # a two-site TDVP step of the same chain
        dict(name="tdvp_bh_L10_chi64", kind="tdvp", L=10, chi=64, grow=6),
        # occupation patterns drawn from an evolved chain, and their amplitudes
        dict(name="sample_boson_L32_chi128_n512", kind="sample", L=32, chi=128, shots=512, grow=6),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["gate2", "step", "step", "tick", "layer", "layer", "boson", "middle", "dmrg", "tdvp", "sample"])
    if kind in ("gate2", "step"):
        model = rng.choice(["xxz", "bh"])
        c = dict(kind=kind, model=model, L=rng.randint(10, 24), chi=_log(rng, 12, 140),
                 grow=40 if model == "xxz" else 8)
    elif kind == "tick":
        c = dict(kind=kind, requests=rng.randint(3, 20), L=2 * rng.randint(5, 12), chi=_log(rng, 16, 96), grow=8)
    elif kind == "layer":
        c = dict(kind=kind, model="bh", L=rng.randint(14, 34), chi=_log(rng, 96, 520), grow=10, precision="fp64")
    elif kind == "boson":
        c = dict(kind=kind, L=2 * rng.randint(8, 20), chi=_log(rng, 64, 400), grow=6)
    elif kind == "middle":
        c = dict(kind=kind, L=16, chi=_log(rng, 300, 1500), updates=1, precision=rng.choice(["tf32", "bf16x3", "fp64"]))
    elif kind in ("dmrg", "tdvp"):
        c = dict(kind=kind, L=rng.randint(6, 10), chi=_log(rng, 16, 96 if kind == "dmrg" else 64), grow=6)
    else:
        c = dict(kind=kind, L=2 * rng.randint(6, 16), chi=_log(rng, 24, 128), shots=_log(rng, 16, 512), grow=6)
    return c


# ---------------------------------------------------------------------------
# Chains and gates
# ---------------------------------------------------------------------------

def _local_dim(c):
    return 2 if c.get("model") == "xxz" else 5


def _particles(c):
    return c["L"] // 2 if c.get("model") == "xxz" or c["kind"] in ("boson", "sample") else c["L"]


def _occupations(c, rng):
    """Neel, one photon in each mode of the left half (boson sampling), or the Mott state with a few
    particles moved, which makes each seed another quench."""
    L = c["L"]
    if c.get("model") == "xxz":
        return [1 - s % 2 if s < 2 * (L // 2) else 0 for s in range(L)]
    if c["kind"] in ("boson", "sample"):
        return [1] * (L // 2) + [0] * (L - L // 2)
    occ = [1] * L
    for _ in range(max(1, L // 8)):
        a = int(rng.integers(L - 1))
        if occ[a] == 1 and occ[a + 1] == 1:
            occ[a], occ[a + 1] = (2, 0) if rng.random() < 0.5 else (0, 2)
    return occ


def _gates(c, rng, dt):
    """sites, factor -> flattened gates, for a seeded coupling."""
    if c.get("model") == "xxz":
        return m.tebd.GateTable("xxz", c["L"], 2, dt, delta=float(rng.uniform(0.2, 1.5)))
    return m.tebd.GateTable("bh", c["L"], 5, dt, J=1.0, U=float(rng.uniform(1.0, 4.0)))


def _splitters(sites, rng):
    return [m.models.flatten(m.models.beam_splitter_gate(math.asin(math.sqrt(rng.random())),
                                                         2 * math.pi * rng.random(), 5)) for _ in sites]


def _bricks(L, k):
    return list(range(k % 2, L - 1, 2))


def _patterns(occ, d, n, rng):
    """Patterns a few hops away from the initial one (those an evolved state has weight on)."""
    out = [list(occ)]
    while len(out) < n:
        p = list(occ)
        for _ in range(int(rng.integers(1, 5))):
            a = int(rng.integers(len(p) - 1))
            x, y = (a, a + 1) if rng.random() < 0.5 else (a + 1, a)
            if p[x] > 0 and p[y] < d - 1:
                p[x] -= 1
                p[y] += 1
        out.append(p)
    return np.array(out, np.int32)


def _strings(n, d):
    row = [1]
    for _ in range(n):
        row = [sum(row[q - i] for i in range(d) if 0 <= q - i < len(row)) for q in range(len(row) + d - 1)]
    return row


def _dims(L, d, N, b, chi):
    """Sector dimensions of a saturated bond: chi over its charges in proportion to what the shorter
    side can carry."""
    left, right = _strings(b, d), _strings(L - b, d)
    bound = {q: min(left[N - q], right[q]) for q in range(len(right)) if 0 <= N - q < len(left)}
    total = sum(bound.values())
    if total <= chi:
        return bound
    dims = {q: min(v, int(chi * v / total)) for q, v in bound.items()}
    return {q: v for q, v in dims.items() if v > 0}


def _saturated(psi, c, rng):
    """A synthetic saturated chain of the benchmark's kind: every bond full, Schmidt weights
    exp(-0.3 (ln k)^2) dealt to the sectors at random, complex normal blocks."""
    L, d, N, chi = c["L"], 5, c["L"], c["chi"]
    bonds = [_dims(L, d, N, b, chi) for b in range(L + 1)]
    for b in range(1, L):
        n = sum(bonds[b].values())
        w = np.exp(-0.3 * np.log(np.arange(1, n + 1)) ** 2)[rng.permutation(n)]
        w /= np.linalg.norm(w)
        lam, off = {}, 0
        for q in sorted(bonds[b]):
            lam[q] = np.sort(w[off:off + bonds[b][q]])[::-1].copy()
            off += bonds[b][q]
        psi.set_bond(b, lam)
    for s in range(L):
        blk = {}
        for l, Dl in bonds[s].items():
            for r, Dr in bonds[s + 1].items():
                if 0 <= l - r <= d - 1:
                    x = rng.standard_normal((2, Dl, Dr))
                    blk[(l, r)] = (x[0] + 1j * x[1]) / math.sqrt(2 * max(Dl, Dr))
        psi.set_site(s, blk)


def _evolved(c, occ, gates, rng, steps, chi, precision=m.MPS_FP64):
    """The product state grown to working entanglement by the case's own schedule."""
    psi = m.MPS(_local_dim(c), occ, chi, precision=precision)
    if c["kind"] in ("boson", "sample"):
        for k in range(steps):
            sites = _bricks(c["L"], k)
            psi.apply_layer(sites, _splitters(sites, rng), chi, CUTOFF)
    else:
        for _ in range(steps):
            m.tebd.trotter_step(psi, gates, chi, CUTOFF)
    return psi


def prepare(case, seed):
    c = dict(case)
    rng = np.random.Generator(np.random.PCG64(seed))
    kind, chi, L = c["kind"], c["chi"], c["L"]
    s = dict(case=c, k=0)
    if kind == "middle":
        s["psi"] = m.MPS(5, [1] * L, chi, precision=PRECISION[c["precision"]])
        _saturated(s["psi"], c, rng)
        gates = _gates(c, rng, 0.02)
        mid = L // 2 - 1
        s["sites"] = [[mid], [mid - 2, mid], [mid - 2, mid, mid + 2]][c["updates"] - 1]
        s["gates"] = [gates(x, 1.0) for x in s["sites"]]
        return s
    if kind == "tick":
        s["exec"] = m.Executor()
        s["jobs"] = []
        for j in range(c["requests"]):
            r = dict(kind="step", model="xxz" if j % 2 else "bh", L=L * (1 + (j // 2) % 2),
                     chi=max(8, chi // (1 + j % 3)))
            gates = _gates(r, rng, 0.05)
            psi = m.MPS(_local_dim(r), _occupations(r, rng), r["chi"])
            layers = [(x, f) for x, f in m.tebd.strang_layers(r["L"])]
            s["jobs"].append((psi, gates, layers, r["chi"]))
        for _ in range(3 * c["grow"]):
            _tick(s)
        return s
    occ = _occupations(c, rng)
    gates = None if kind in ("boson", "sample") else _gates(c, rng, 0.1)
    s["psi"] = _evolved(c, occ, gates, rng, c["grow"], chi, PRECISION[c.get("precision", "fp64")])
    s["patterns"] = _patterns(occ, _local_dim(c), 16, rng)
    if kind == "gate2":
        s["sites"] = [L // 2 - 1]
        s["gates"] = [gates(L // 2 - 1, 1.0)]
    elif kind in ("step", "layer"):
        s["gates"] = gates
    elif kind == "boson":
        s["bricks"] = [(x, _splitters(x, rng)) for x in (_bricks(L, k) for k in range(2))]
        s["k"] = c["grow"]
    elif kind in ("dmrg", "tdvp"):
        s["terms"] = m.models.chain_bond_terms("bh", L, 5, J=1.0, U=float(rng.uniform(1.0, 4.0)))
    else:
        s["uniforms"] = rng.random((c["shots"], L))
    return s


# ---------------------------------------------------------------------------
# Passes
# ---------------------------------------------------------------------------

def _spectra(bonds, chi):
    """The entanglement spectra of bonds, one row each: the Schmidt values of all charges, descending,
    zeros behind them up to chi."""
    out = np.zeros((len(bonds), chi))
    for k, bond in enumerate(bonds):
        v = np.sort(np.concatenate(list(bond.values())))[::-1]
        out[k, :len(v)] = v
    return out


def _tick(s):
    """The next layer of every request, merged into one executor call (as serve.Server does)."""
    items = []
    for psi, gates, layers, chi in s["jobs"]:
        sites, f = layers[s["k"] % 3]
        items += [(psi, x, gates(x, f), chi, CUTOFF) for x in sites]
    s["k"] += 1
    return s["exec"].apply(items)[0]


def run(s):
    c, kind = s["case"], s["case"]["kind"]
    if kind == "tick":
        err = _tick(s)
        return {"kept": 1.0 - err, "lam": _spectra([psi.bond(psi.L // 2) for psi, _, _, _ in s["jobs"]], c["chi"])}
    psi, chi, L = s["psi"], c["chi"], c["L"]
    if kind == "gate2":
        err = psi.apply_gate2(s["sites"][0], s["gates"][0], chi, CUTOFF)
        return {"kept": 1.0 - err, "lam": _spectra([psi.bond(s["sites"][0] + 1)], chi), "amp": psi.amplitudes(s["patterns"])}
    if kind == "step":
        err = m.tebd.trotter_step(psi, s["gates"], chi, CUTOFF)
        return {"kept": 1.0 - np.concatenate(err), "lam": _spectra([psi.bond(b) for b in range(1, L)], chi), "amp": psi.amplitudes(s["patterns"])}
    if kind in ("layer", "boson"):
        if kind == "layer":      # odd and even bonds in turn
            sites = _bricks(L, s["k"])
            gates = [s["gates"](x, 1.0) for x in sites]
        else:
            sites, gates = s["bricks"][s["k"] % 2]
        s["k"] += 1
        err = psi.apply_layer(sites, gates, chi, CUTOFF)
        return {"kept": 1.0 - err, "lam": _spectra([psi.bond(x + 1) for x in sites], chi), "amp": psi.amplitudes(s["patterns"])}
    if kind == "middle":
        err = psi.apply_layer(s["sites"], s["gates"], chi, CUTOFF)
        return {"kept": 1.0 - err, "lam": _spectra([psi.bond(x + 1) for x in s["sites"]], chi)}
    if kind == "dmrg":
        en = psi.dmrg(s["terms"], 1, chi, CUTOFF)
        return {"energies": en, "lam": _spectra([psi.bond(b) for b in range(1, L)], chi), "amp": np.abs(psi.amplitudes(s["patterns"]))}
    if kind == "tdvp":
        en = psi.tdvp(s["terms"], 1, 0.05, chi, CUTOFF)
        return {"energies": en, "lam": _spectra([psi.bond(b) for b in range(1, L)], chi), "amp": psi.amplitudes(s["patterns"])}
    drawn, prob = psi.sample(s["uniforms"])
    return {"patterns": drawn, "prob": prob, "amp": psi.amplitudes(drawn)}


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------

def _update_work(L, d, N, s, chi):
    """(bytes, flops) of one update at saturated bonds: both sites read and written, the products B B,
    the sector SVDs (values and right vectors, 4 (6 a b^2 + 20 b^3) real operations) and Theta Y."""
    l, mid, r = (_dims(L, d, N, b, chi) for b in (s, s + 1, s + 2))
    by = fl = 0.0
    for p, q in ((l, mid), (mid, r)):
        by += 32.0 * sum(a * b for x, a in p.items() for y, b in q.items() if 0 <= x - y < d)
    by += 16.0 * sum(mid.values())
    for x, a in l.items():
        for y, b in mid.items():
            if 0 <= x - y < d:
                fl += 8.0 * a * b * sum(e for z, e in r.items() if 0 <= y - z < d)
    for q in range(max(l) + 1):
        rows = sum(a for x, a in l.items() if 0 <= x - q < d)
        cols = sum(e for z, e in r.items() if 0 <= q - z < d)
        a, b = max(rows, cols), min(rows, cols)
        fl += 4.0 * (6.0 * a * b * b + 20.0 * b ** 3) + 8.0 * rows * cols * mid.get(q, 0)
    return by, fl


def work(case):
    c, kind, L, chi = case, case["kind"], case["L"], case["chi"]
    ups = []
    if kind == "tick":
        for j in range(c["requests"]):
            x = "xxz" if j % 2 else "bh"
            Lj, d = L * (1 + (j // 2) % 2), 2 if x == "xxz" else 5
            ups += [(Lj, d, Lj // 2 if d == 2 else Lj, s, max(8, chi // (1 + j % 3))) for s in _bricks(Lj, 0)]
    else:
        d, N = _local_dim(c), _particles(c)
        mid = L // 2 - 1
        sites = {"gate2": [mid], "step": _bricks(L, 0) * 2 + _bricks(L, 1), "layer": _bricks(L, 0),
                 "boson": _bricks(L, 0), "middle": [[mid], [mid - 2, mid], [mid - 2, mid, mid + 2]][c.get("updates", 1) - 1],
                 "dmrg": list(range(L - 1)) * 2, "tdvp": list(range(L - 1)) * 2, "sample": []}[kind]
        ups = [(L, d, N, s, chi) for s in sites]
    by = fl = 0.0
    for u in ups:
        b, f = _update_work(*u)
        by, fl = by + b, fl + f
    if kind in ("dmrg", "tdvp"):       # at least one effective-Hamiltonian product per local step
        terms = 4
        for (L_, d, N, s, x) in ups:
            l, r = _dims(L_, d, N, s, x), _dims(L_, d, N, s + 2, x)
            fl += 8.0 * (2 + 2 * terms) * sum(a * b * (a + b) for p, a in l.items() for q, b in r.items()
                                              if 0 <= p - q <= 2 * (d - 1))
    if kind == "sample":               # each shot multiplies its blocks from left to right, twice
        for s in range(L):
            l, r = _dims(L, 5, L // 2, s, chi), _dims(L, 5, L // 2, s + 1, chi)
            n = sum(a * b for x, a in l.items() for y, b in r.items() if 0 <= x - y < 5)
            by += 16.0 * n
            fl += 16.0 * c["shots"] * n / max(1, len(l))
        by += c["shots"] * (12.0 * L + 24.0)
    return {"bytes": by + 16.0 * L, "flops": fl + 16.0 * L}


# ---------------------------------------------------------------------------
# The same passes in plain numpy (64 bits)
# ---------------------------------------------------------------------------

class _Chain:
    """Right-canonical U(1) MPS: lam[b] = {charge: values}, site[s] = {(l, r): block}."""

    def __init__(self, psi):
        self.L, self.d = psi.L, psi.d
        self.lam = [psi.bond(b) for b in range(psi.L + 1)]
        self.site = [psi.site(x) for x in range(psi.L)]

    def update(self, s, gate, chi):
        d, A, B = self.d, self.site[s], self.site[s + 1]
        G, off = {}, 0
        for n in range(2 * d - 1):
            lo, k = max(0, n - d + 1), min(d - 1, n) - max(0, n - d + 1) + 1
            G[n] = (lo, np.asarray(gate)[off:off + k * k].reshape(k, k))
            off += k * k
        rows, cols = self.lam[s], self.lam[s + 2]
        T = {}
        for (l, q), a in A.items():
            for (q2, r), b in B.items():
                if q2 == q:
                    T.setdefault((l, r), []).append((q, a @ b))
        theta = {}
        for (l, r), parts in T.items():
            lo, g = G[l - r]
            for i in range(g.shape[0]):
                theta[(l - lo - i, l, r)] = sum(g[i, l - q - lo] * p for q, p in parts)
        split, every = {}, []
        for q in sorted({x[0] for x in theta}):
            ls, rs = [l for l in sorted(rows) if 0 <= l - q < d], [r for r in sorted(cols) if 0 <= q - r < d]
            M = np.concatenate([np.concatenate([theta.get((q, l, r), np.zeros((len(rows[l]), len(cols[r])))) for r in rs], 1)
                                for l in ls], 0)
            w = np.concatenate([rows[l] for l in ls])
            _, S, Vh = np.linalg.svd(w[:, None] * M, full_matrices=False)
            split[q] = (ls, rs, M, S, Vh)
            every += [(-v, q, j) for j, v in enumerate(S)]
        norm = math.sqrt(sum(v[0] ** 2 for v in every))
        kept = sorted(x for x in every if -x[0] > CUTOFF * norm)[:chi]
        count = {}
        for _, q, _ in kept:
            count[q] = count.get(q, 0) + 1
        nk = math.sqrt(sum(v[0] ** 2 for v in kept))
        self.lam[s + 1], self.site[s], self.site[s + 1] = {}, {}, {}
        for q in sorted(count):
            k, (ls, rs, M, S, Vh) = count[q], split[q]
            self.lam[s + 1][q] = S[:k] / nk
            X, at = M @ Vh[:k].conj().T / nk, 0
            for l in ls:
                self.site[s][(l, q)] = X[at:at + len(rows[l])]
                at += len(rows[l])
            at = 0
            for r in rs:
                self.site[s + 1][(q, r)] = Vh[:k, at:at + len(cols[r])]
                at += len(cols[r])
        n = len(kept)
        return sum(x[0] ** 2 for x in sorted(every)[n:]) / norm ** 2

    def amplitudes(self, patterns):
        out = []
        for p in patterns:
            q = int(sum(p))
            v = np.ones((1, 1), complex)
            for x, i in enumerate(p):
                b = self.site[x].get((q, q - int(i)))
                if b is None:
                    v = np.zeros((1, 1), complex)
                    break
                v = v @ b
                q -= int(i)
            out.append(v[0, 0] * 1.0)
        return np.array(out)


def exact(case, seed):
    c, kind = dict(case), case["kind"]
    if kind in ("dmrg", "tdvp") or (kind == "middle" and (c["precision"] != "fp64" or c["chi"] > 1100)):
        return None      # iterative solvers on the chain; reduced-precision products
    s = prepare(case, seed)
    if kind == "tick":
        chains = [_Chain(j[0]) for j in s["jobs"]]
        err = []
        for ch, (psi, gates, layers, chi) in zip(chains, s["jobs"]):
            sites, f = layers[s["k"] % 3]
            err += [ch.update(x, gates(x, f), chi) for x in sites]
        return {"kept": 1.0 - np.array(err), "lam": _spectra([ch.lam[ch.L // 2] for ch in chains], c["chi"])}
    psi, chi, L = s["psi"], c["chi"], c["L"]
    if kind == "sample":
        drawn, _ = psi.sample(s["uniforms"])
        amp = _Chain(psi).amplitudes(drawn)
        return {"patterns": None, "prob": None, "amp": amp}
    ch = _Chain(psi)
    if kind == "gate2":
        err = ch.update(s["sites"][0], s["gates"][0], chi)
        return {"kept": 1.0 - err, "lam": _spectra([ch.lam[s["sites"][0] + 1]], chi), "amp": ch.amplitudes(s["patterns"])}
    if kind == "step":
        err = np.array([ch.update(x, s["gates"](x, f), chi) for sites, f in m.tebd.strang_layers(L) for x in sites])
        return {"kept": 1.0 - err, "lam": _spectra([ch.lam[b] for b in range(1, L)], chi), "amp": ch.amplitudes(s["patterns"])}
    if kind == "middle":
        err = np.array([ch.update(x, g, chi) for x, g in zip(s["sites"], s["gates"])])
        return {"kept": 1.0 - err, "lam": _spectra([ch.lam[x + 1] for x in s["sites"]], chi)}
    sites = _bricks(L, s["k"])
    gates = [s["gates"](x, 1.0) for x in sites] if kind == "layer" else s["bricks"][s["k"] % 2][1]
    err = np.array([ch.update(x, g, chi) for x, g in zip(sites, gates)])
    return {"kept": 1.0 - err, "lam": _spectra([ch.lam[x + 1] for x in sites], chi), "amp": ch.amplitudes(s["patterns"])}
