"""Performance cases of the bipartite H|psi> engine: what its users run.

Every case goes through the package's public entry points (apply_H,
lanczos_ground, lanczos_gf, entanglement_spectrum, DenseOperator.apply,
batch_apply) on the repository's own workloads and on sizes around them.
``exact`` evaluates the same quantities with plain torch / numpy in FP64 from
the documented vector layout (blocks of side-A charge s in ascending order,
each row-major d_A x d_B, side states ascending in their side-local bit
strings).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2605_07621_gb300 as gb
from workloads import dense as wd
from workloads import lattices as wl


# --------------------------------------------------------------------------- the cases

def listed():
    return [
        # one small ring solved to its ground-state energy, 150 Lanczos steps:
        # 12,870 states, bound by launches and latency (sectors of a parameter scan)
        _spin("ground_heis16", 16, 1, 0.0, 8, "ground", mode="f64", steps=150),
        # H|psi> of a mid-size Hubbard ring (924 x 924): the inner call of a
        # user's own Krylov loop on a sector that stays in L2
        _hub("apply_hub12_f64", "ring", 12, 1, 4.0, 0.0, 0.0, 6, 6, "apply", dtype="f64"),
        # FP32 H|psi> on a 28-site frustrated torus, 40 M states, both sides 14 sites
        _spin("apply_j1j2_4x7_f32", 7, 4, 0.5, 14, "apply", dtype="f32"),
        # FP64 H|psi> with a coupling that is not dyadic (a scan over J2)
        _spin("apply_j1j2_4x7_j03_f64", 7, 4, 0.3, 14, "apply", dtype="f64"),
        # the headline: FP64 H|psi> on the 32-site torus at Sz = 0, 601 M states
        _spin("apply_j1j2_4x8_f64", 8, 4, 0.5, 16, "apply", dtype="f64"),
        # FP64 H|psi> of the 4 x 4 Hubbard torus at half filling, 166 M states, one block
        _hub("apply_hub4x4_f64", "torus", 4, 4, 8.0, 0.0, 0.0, 8, 8, "apply", dtype="f64"),
        # quantum impurity with 14 bath orbitals: irrational on-site energies,
        # 41 M states, rows with few matrix elements
        _hub("apply_qim15_f64", "impurity", 14, 1, 4.0, 0.0, 0.0, 8, 7, "apply", dtype="f64"),
        # time to E0 in mixed precision (FP32 Lanczos, FP64 refinement), 40 M states
        _spin("ground_j1j2_4x7_mixed", 7, 4, 0.5, 14, "ground", mode="mixed", steps=0),
        # dynamical correlations: G(omega) of a random state (finite-temperature
        # Lanczos sampling), two shifted sectors, 300 re-orthogonalised steps each
        _hub("gf_hub12", "ring", 12, 1, 4.0, 0.0, 0.0, 6, 6, "gf", n_iter=300, n_omega=2048, eta=1.0),
        # entanglement spectrum of a 28-site state across its cut, 15 blocks up to 3432 x 3432
        _spin("entangle_j1j2_4x7", 7, 4, 0.5, 14, "entangle"),
        # dense-block (DMRG-style) H|psi>, 21 sectors, total bond dimension 4000
        {"name": "dense_a095", "kind": "dense", "alpha": 0.95, "total": 4000, "nq": 21, "pairs": 2},
        # one batched H|psi> over 512 independent small Hubbard instances
        {"name": "batch_apply_512", "kind": "batch", "n": 512},
    ]


def draw(rng):
    what = rng.choice(["spin", "spin", "spin", "hub", "hub", "ground", "gf", "entangle", "dense", "batch"])
    if what == "spin":
        return _draw_spin(rng, 8, 29, "apply", dtype=rng.choice(["f64", "f64", "f32"]))
    if what == "hub":
        return _draw_hub(rng, 5, 14, "apply", dtype=rng.choice(["f64", "f64", "f32"]))
    if what == "ground":
        return _draw_spin(rng, 10, 24, "ground", mode=rng.choice(["f64", "mixed"]), steps=0)
    if what == "gf":
        return _draw_hub(rng, 6, 11, "gf", n_iter=rng.randint(40, 200), n_omega=rng.randint(100, 3000), eta=1.0)
    if what == "entangle":
        return _draw_spin(rng, 8, 25, "entangle")
    if what == "dense":
        return {"kind": "dense", "alpha": round(rng.uniform(0.1, 1.2), 3),
                "total": int(round(math.exp(rng.uniform(math.log(60), math.log(3500))))), "nq": rng.randint(3, 21),
                "pairs": rng.randint(1, 2)}
    return {"kind": "batch", "n": int(round(math.exp(rng.uniform(math.log(8), math.log(400)))))}


def _spin(name, lx, ly, j2, n_up, do, **more):
    c = {"kind": do, "model": "spin", "lx": lx, "ly": ly, "j2": j2, "n_up": n_up, **more}
    return {"name": name, **c} if name else c


def _hub(name, geom, lx, ly, U, tp, disorder, n_up, n_dw, do, **more):
    c = {"kind": do, "model": "hubbard", "geom": geom, "lx": lx, "ly": ly, "U": U, "tp": tp, "disorder": disorder,
         "n_up": n_up, "n_dw": n_dw, **more}
    return {"name": name, **c} if name else c


def _draw_spin(rng, n_lo, n_hi, do, **more):
    while True:
        ly = rng.choice([1, 1, 2, 3, 4, 5])
        lx = int(round(rng.randint(n_lo, n_hi) / ly))
        n = lx * ly
        if lx < 2 or not n_lo <= n <= n_hi:
            continue
        j2 = rng.choice([0.0, 0.25, 0.5, 0.3, 0.41])
        return _spin(None, lx, ly, j2, max(1, n // 2 - rng.choice([0, 0, 0, 1, 2, 3])), do, **more)


def _draw_hub(rng, n_lo, n_hi, do, **more):
    geom = rng.choice(["ring", "ring", "open", "impurity"])
    n = rng.randint(n_lo, n_hi)
    lx, ly = (n, 1) if geom == "ring" else (n - 1, 1)
    if geom == "open":
        ly = rng.choice([2, 3])
        lx = max(2, n // ly)
        n = lx * ly
    up, dw = (min(n - 1, max(1, n // 2 + rng.choice([-1, 0, 0, 1]))) for _ in range(2))
    return _hub(None, geom, lx, ly, rng.choice([4.0, 8.0, 3.7]), rng.choice([0.0, 0.0, 0.3, 0.25]),
                rng.choice([0.0, 0.0, 1.0]), up, dw, do, **more)


# --------------------------------------------------------------------------- inputs

def _model(case, seed=0):
    if case["model"] == "spin":
        # side A: the first half of the sites (the cut of the repository's configurations)
        half = (1 << (case["lx"] * case["ly"] // 2)) - 1
        m = wl.j1j2_torus(case["lx"], case["ly"], 1.0, case["j2"], case["n_up"], cut_mask=half)
        if case["kind"] == "ground":
            # a point of an anisotropy scan: the energy is another one for another seed
            m.jz = m.jz * (1.0 + (37 * int(seed) % 32) / 64.0)
        return m
    lx, ly, U, tp, up, dw = (case[k] for k in ("lx", "ly", "U", "tp", "n_up", "n_dw"))
    n = lx + 1 if case["geom"] == "impurity" else lx * ly
    eps = None
    if case["disorder"]:
        eps = np.random.default_rng(n).uniform(-case["disorder"], case["disorder"], size=n)
    if case["geom"] == "ring":
        return wl.hubbard_chain(lx, 1.0, U, up, dw, True, tp=tp, eps=eps)
    if case["geom"] == "open":
        return wl.hubbard_open_cluster(lx, ly, 1.0, U, tp=tp, eps=eps, n_up=up, n_dw=dw)
    if case["geom"] == "torus":
        return wl.hubbard_torus(lx, ly, 1.0, U, up, dw)
    return wl.anderson_impurity(lx, U, -U / 2, 0.5, wl.impurity_bath(lx), up, dw)


def _vector(n, seed, dtype=torch.float64):
    """Seeded uniform [-1, 1) values, normalised."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 17)
    x = torch.rand(n, generator=g, device="cuda", dtype=dtype).mul_(2.0).sub_(1.0)
    return x.div_(torch.linalg.vector_norm(x))


def _torch_dtype(case):
    return torch.float32 if case.get("dtype") == "f32" else torch.float64


def _dense_blocks(case):
    # the operator of a fixed Hamiltonian; the state is what changes with the seed
    chi = wd.block_dims(case["total"], case["alpha"], case["nq"])
    return wd.dense_block_operator(chi, case["pairs"], 20260507)


def _omega(case):
    return np.linspace(-15.0, 15.0, case["n_omega"])


def prepare(case, seed):
    st = {"case": case}
    if case["kind"] == "dense":
        st["op"] = gb.DenseOperator(_dense_blocks(case))
        st["x"] = _vector(st["op"].dim, seed)
        st["y"] = torch.empty_like(st["x"])
        return st
    if case["kind"] == "batch":
        st["b"] = gb.batch_create(wl.batched_hubbard_instances(case["n"]))
        st["x"] = _vector(st["b"].dim, seed, torch.float32)
        st["y"] = torch.empty_like(st["x"])
        return st
    ctx = gb.build_local_ops(gb.build_sectors(_model(case, seed)))
    st["ctx"] = ctx
    st["x"] = _vector(ctx.dim, seed, _torch_dtype(case))
    if case["kind"] == "apply":
        st["y"] = torch.empty_like(st["x"])
    return st


def run(state):
    case, x = state["case"], state["x"]
    if case["kind"] == "apply":
        return gb.apply_H(state["ctx"], x, state["y"])
    if case["kind"] == "dense":
        state["op"].apply(x, state["y"])
        return state["y"]
    if case["kind"] == "batch":
        return gb.batch_apply(state["b"], x, state["y"])
    if case["kind"] == "ground":
        fixed = case["steps"] > 0
        return gb.lanczos_ground(state["ctx"], case["mode"], max_iter=case["steps"] or 400, fixed_iter=fixed,
                                 v0=x).e0
    if case["kind"] == "gf":
        return gb.lanczos_gf(state["ctx"], x, -6.0, _omega(case), case["eta"], n_iter=case["n_iter"])[0]
    es = gb.entanglement_spectrum(state["ctx"], x)
    return {"lam": np.concatenate(es.lam), "weight": es.weight, "entropy": es.entropy}


# --------------------------------------------------------------------------- work

def _terms(m):
    """(states, off-diagonal matrix elements of H) of one model's sector."""
    if m.kind == "spin":
        return math.comb(m.n_sites, m.n_up), m.n_bonds * 2 * math.comb(m.n_sites - 2, m.n_up - 1)
    S, u, d = m.n_sites, m.n_up, m.n_dw
    a, b = math.comb(S, u), math.comb(S, d)
    hop = lambda k: 2 * math.comb(S - 2, k - 1) if 1 <= k <= S - 1 else 0  # noqa: E731
    return a * b, m.n_bonds * (hop(u) * b + hop(d) * a)


def _block_dims(m):
    n, k = m.n_sites, m.n_up
    nA = bin(m.cut_mask).count("1")
    return [(math.comb(nA, s), math.comb(n - nA, k - s)) for s in range(max(0, k - (n - nA)), min(nA, k) + 1)]


def work(case):
    if case["kind"] == "dense":
        chi = [int(c) for c in wd.block_dims(case["total"], case["alpha"], case["nq"])]
        n, fl, ops = sum(c * c for c in chi), 0, 0
        for c in chi:
            fl += 4 * c ** 3
            ops += 2 * c * c
        for a, b in list(zip(chi, chi[1:])) + list(zip(chi[1:], chi)):
            fl += case["pairs"] * 2 * (b * a * a + b * a * b)
            ops += case["pairs"] * 2 * a * b
        return {"bytes": 8 * (2 * n + ops), "flops": fl}
    if case["kind"] == "batch":
        t = [_terms(m) for m in wl.batched_hubbard_instances(case["n"])]
        return {"bytes": 8 * sum(d for d, _ in t), "flops": sum(2 * (d + e) for d, e in t)}
    m = _model(case)
    D, nnz = _terms(m)
    if case["kind"] == "apply":
        return {"bytes": (8 if case["dtype"] == "f32" else 16) * D, "flops": 2 * (D + nnz)}
    if case["kind"] == "ground":
        # per step: one H|psi> and the three-term update (about 60 steps to convergence)
        k, w = case["steps"] or 60, 4 if case["mode"] == "mixed" else 8
        return {"bytes": 6 * w * D * k, "flops": (2 * (D + nnz) + 10 * D) * k}
    if case["kind"] == "gf":
        # two shifted sectors: H|psi>, the update and one projection against the basis per step
        k, by, fl = case["n_iter"], 0, 0
        for d in (1, -1):
            if not 0 <= m.n_up + d <= m.n_sites:
                continue
            D2, nnz2 = _terms(m.with_sector(m.n_up + d, m.n_dw))
            kk = min(k, D2)
            by += 8 * D2 * (6 * kk + kk * kk // 2)
            fl += (2 * (D2 + nnz2) + 10 * D2) * kk + 4 * D2 * (kk * kk // 2)
        return {"bytes": by, "flops": fl}
    fl = 0
    for a, b in _block_dims(m):
        s, L = min(a, b), max(a, b)
        fl += s * s * L + 4 * s ** 3 // 3
    return {"bytes": 8 * D + 8 * sum(min(a, b) for a, b in _block_dims(m)), "flops": fl}


# --------------------------------------------------------------------------- the same in plain FP64

def _popcount(x):
    c = np.zeros_like(x)
    for i in range(32):
        c += (x >> i) & 1
    return c


class _Side:
    """States of one side grouped by popcount, ascending, and their ranks."""

    def __init__(self, sites):
        self.sites = list(sites)
        self.n = len(self.sites)
        self.bit = {s: p for p, s in enumerate(self.sites)}
        w = np.arange(1 << self.n, dtype=np.int64)
        pc = _popcount(w)
        self.states = [w[pc == k] for k in range(self.n + 1)]
        self.rank = np.zeros(1 << self.n, np.int64)
        for st in self.states:
            self.rank[st] = np.arange(len(st))


def _csr(rows, cols, vals, n):
    if not rows:
        return None
    r, c, v = (torch.as_tensor(np.concatenate(a), device="cuda") for a in (rows, cols, vals))
    if not len(r):
        return None
    return torch.sparse_coo_tensor(torch.stack([r, c]), v, (n, n)).coalesce().to_sparse_csr()


class _Exact:
    """H of one sector applied block by block with torch sparse products, FP64."""

    def __init__(self, m):
        self.m, spin = m, m.kind == "spin"
        S = m.n_sites
        if spin:
            inA = [(m.cut_mask >> i) & 1 for i in range(S)]
            at_cut = [0] * S
            for i, j in m.bonds:
                if inA[i] != inA[j]:
                    at_cut[i] = at_cut[j] = 1
            A = [i for i in range(S) if inA[i]]
            B = [i for i in range(S) if not inA[i]]
            self.A = _Side([i for i in A if at_cut[i]] + [i for i in A if not at_cut[i]])
            self.B = _Side([i for i in B if not at_cut[i]] + [i for i in B if at_cut[i]])
            ks = [(s, m.n_up - s) for s in range(self.A.n + 1) if 0 <= m.n_up - s <= self.B.n]
            self.cross = [(int(i), int(j), b) if inA[i] else (int(j), int(i), b)
                          for b, (i, j) in enumerate(m.bonds) if inA[i] != inA[j]]
        else:
            self.A, self.B = _Side(range(S)), _Side(range(S))
            ks = [(m.n_up, m.n_dw)]
            self.cross = []
        self.ks, self.off = ks, [0]
        for s, k in ks:
            self.off.append(self.off[-1] + len(self.A.states[s]) * len(self.B.states[k]))
        self.dim = self.off[-1]
        self.ops = {}

    def side(self, sd, k):
        """(sparse off-diagonal part, diagonal) of one side's operator at charge k."""
        key = (id(sd), k)
        if key in self.ops:
            return self.ops[key]
        m, st = self.m, sd.states[k]
        rows, cols, vals, diag = [], [], [], np.zeros(len(st))
        for b, (i, j) in enumerate(m.bonds):
            if int(i) not in sd.bit or int(j) not in sd.bit:
                continue
            p, q = sorted((sd.bit[int(i)], sd.bit[int(j)]))
            bp, bq = (st >> p) & 1, (st >> q) & 1
            on = np.flatnonzero(bp != bq)
            to = sd.rank[st[on] ^ ((1 << p) | (1 << q))]
            if m.kind == "spin":
                v = np.full(len(on), 0.5 * m.jxy[b])
                diag += m.jz[b] * np.where(bp == bq, 0.25, -0.25)
            else:
                between = ((1 << q) - 1) & ~((1 << (p + 1)) - 1)
                v = -m.t[b] * (1 - 2 * (_popcount(st[on] & between) & 1))
            rows.append(on), cols.append(to), vals.append(v.astype(np.float64))
        if m.kind == "hubbard":
            for p, i in enumerate(sd.sites):
                diag += m.eps[i] * ((st >> p) & 1)
        self.ops[key] = _csr(rows, cols, vals, len(st)), torch.as_tensor(diag, device="cuda")
        return self.ops[key]

    def apply(self, x):
        y = torch.empty_like(x)
        blk = [x[self.off[i]:self.off[i + 1]].view(len(self.A.states[s]), len(self.B.states[k]))
               for i, (s, k) in enumerate(self.ks)]
        for i, (s, k) in enumerate(self.ks):
            X, sa, sb = blk[i], self.A.states[s], self.B.states[k]
            (HA, dA), (HB, dB) = self.side(self.A, s), self.side(self.B, k)
            if self.m.kind == "spin":
                L = np.stack([((sa >> self.A.bit[a]) & 1) - 0.5 for a, _, _ in self.cross], 1) if self.cross else None
                R = np.stack([self.m.jz[e] * (((sb >> self.B.bit[b]) & 1) - 0.5) for _, b, e in self.cross], 1) \
                    if self.cross else None
            else:
                L = np.stack([((sa >> p) & 1).astype(float) for p in range(self.A.n)], 1)
                R = np.stack([self.m.U[p] * ((sb >> p) & 1) for p in range(self.B.n)], 1)
            V = dA[:, None] + dB[None, :]
            if L is not None:
                V = V.addmm_(torch.as_tensor(L, device="cuda"), torch.as_tensor(R.T.copy(), device="cuda"))
            Y = V.mul_(X)
            if HA is not None:
                Y += HA @ X
            if HB is not None:
                Y += (HB @ X.t().contiguous()).t()
            for a, b, e in self.cross:
                p, q = self.A.bit[a], self.B.bit[b]
                for up in (0, 1):  # bit of a; the B bit is the other
                    j = i - 1 if up else i + 1
                    r = np.flatnonzero(((sa >> p) & 1) == up)
                    c = np.flatnonzero(((sb >> q) & 1) == 1 - up)
                    if not 0 <= j < len(self.ks) or not len(r) or not len(c):
                        continue
                    rs = torch.as_tensor(self.A.rank[sa[r] ^ (1 << p)], device="cuda")
                    cs = torch.as_tensor(self.B.rank[sb[c] ^ (1 << q)], device="cuda")
                    r, c = torch.as_tensor(r, device="cuda"), torch.as_tensor(c, device="cuda")
                    Z = torch.zeros(len(r), X.shape[1], device="cuda", dtype=x.dtype)
                    Z[:, c] = blk[j].index_select(0, rs).index_select(1, cs).mul_(0.5 * self.m.jxy[e])
                    Y.index_add_(0, r, Z)
            y[self.off[i]:self.off[i + 1]] = Y.reshape(-1)
        return y


def _lanczos(H, v0, steps):
    """alpha, beta of a fully re-orthogonalised run from v0."""
    steps = min(steps, len(v0))
    V = torch.empty(steps, len(v0), device="cuda", dtype=torch.float64)
    V[0] = v0 / torch.linalg.vector_norm(v0)
    al, be = [], []
    for j in range(steps):
        w = H.apply(V[j])
        al.append(float(torch.dot(V[j], w)))
        for _ in range(2):
            w -= V[: j + 1].t() @ (V[: j + 1] @ w)
        be.append(float(torch.linalg.vector_norm(w)))
        if j + 1 == steps or be[-1] < 1e-12:
            break
        V[j + 1] = w / be[-1]
    return np.array(al), np.array(be)


def _lowest(H, v0):
    al, be = _lanczos(H, v0, 100)
    T = np.diag(al) + np.diag(be[: len(al) - 1], 1) + np.diag(be[: len(al) - 1], -1)
    return float(np.linalg.eigvalsh(T)[0])


def _remap(m, psi, H1, create):
    """c^dag_{0,up} psi or c_{0,up} psi (site 0 is the first operator: no sign), the shifted model and its H."""
    m2 = m.with_sector(m.n_up + (1 if create else -1), m.n_dw)
    H2 = _Exact(m2)
    dst = H2.A.states[m2.n_up]
    on = np.flatnonzero((dst & 1) == (1 if create else 0))
    src = H1.A.rank[dst[on] ^ 1]
    X = psi.view(len(H1.A.states[m.n_up]), -1)
    out = torch.zeros(len(dst), X.shape[1], device="cuda", dtype=torch.float64)
    out[torch.as_tensor(on, device="cuda")] = X[torch.as_tensor(src, device="cuda")]
    return H2, out.view(-1)


def _continued(z, al, be, w0):
    t = np.zeros_like(z)
    for n in range(len(al) - 1, 0, -1):
        t = be[n - 1] ** 2 / (z - al[n] - t)
    return w0 / (z - al[0] - t)


def exact(case, seed):
    if case["kind"] == "dense":
        B = _dense_blocks(case)
        chi, off = [int(c) for c in B.chi], B.offsets()
        x = _vector(int(off[-1]), seed)
        up = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")  # noqa: E731
        X = [x[off[q]:off[q + 1]].view(c, c) for q, c in enumerate(chi)]
        Y = [up(B.HL[q]) @ X[q] + X[q] @ up(B.HR[q]).t() for q in range(len(chi))]
        for t, d in enumerate(B.delta):
            for q in range(len(chi)):
                if B.Lm[t][q] is not None:
                    Y[q + d] += up(B.Lm[t][q]) @ X[q] @ up(B.Rm[t][q]).t()
        return torch.cat([y.reshape(-1) for y in Y])
    if case["kind"] == "batch":
        models = wl.batched_hubbard_instances(case["n"])
        x = _vector(sum(_terms(m)[0] for m in models), seed, torch.float32).double()
        out, o = [], 0
        for m in models:
            H = _Exact(m)
            out.append(H.apply(x[o:o + H.dim]))
            o += H.dim
        return torch.cat(out)
    m = _model(case, seed)
    D, _ = _terms(m)
    if case["kind"] == "entangle":
        x = _vector(D, seed)
        lam, wt, o = [], [], 0
        for a, b in _block_dims(m):
            X = x[o:o + a * b].view(a, b)
            o += a * b
            e = torch.linalg.eigvalsh(X @ X.t() if a <= b else X.t() @ X)
            lam.append(e.flip(0).cpu().numpy())
            wt.append(float((X * X).sum()))
        lam, wt = np.concatenate(lam), np.array(wt)
        p = lam[lam > 0] / wt.sum()
        return {"lam": lam, "weight": wt, "entropy": float(-(p * np.log(p)).sum())}
    H = _Exact(m)
    x = _vector(D, seed, _torch_dtype(case)).double()
    if case["kind"] == "apply":
        return H.apply(x)
    if case["kind"] == "ground":
        # the basis of a re-orthogonalised run is kept: up to 50 M states fit
        return _lowest(H, x) if D <= 50_000_000 else None
    w, G = _omega(case), 0.0
    for create in (True, False):
        if not 0 <= m.n_up + (1 if create else -1) <= m.n_sites:
            continue
        H2, phi = _remap(m, x, H, create)
        w0 = float(torch.dot(phi, phi))
        if w0 <= 0.0:
            continue
        al, be = _lanczos(H2, phi, case["n_iter"])
        z = w + 1j * case["eta"]
        G = G + (_continued(z - 6.0, al, be, w0) if create else -_continued(-6.0 - z, al, be, w0))
    return G
