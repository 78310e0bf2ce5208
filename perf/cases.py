"""What this library is asked to do, as cases that can be timed and compared.

An evaluation case is one call of a plan: energy, forces and stress of a
periodic cell at a geometry 0.01 A away from the one the plan was made for,
as a relaxation or molecular-dynamics loop issues it step after step.  The
shapes are the library's own workloads (8-atom diamond cell, Si-like diamond
supercells, CsSnI3-like perovskite cells) and cells with other orbital and
auxiliary counts on the same two lattices.  An LRI case is one call of the
block preparation for a batch of atom pairs.

FP64 plans return their FP64 results.  The split-precision plans contract in
FP32-accumulated tensor-core products (their contract is 1e-5 relative), and
a program that picks them keeps forces and stress in single precision; so
their results are handed on as float32.
"""
import math

import numpy as np
import torch

from paper_2412_11081_gb300 import hfx, inputs

PRECISION = {"fp64": hfx.HFX_FP64, "bf16x3": hfx.HFX_BF16X3, "bf16x6": hfx.HFX_BF16X6}
SPACING = {"diamond": 5.43, "perovskite": 6.2}


def _eval(name, lattice, n_rep, n_ao, n_abf, r_c, precision, **kw):
    """Plain values only: the per-species shapes are texts such as "18,13,13"."""
    case = {"name": name, "what": "evaluate", "lattice": lattice, "n_rep": n_rep, "n_ao": n_ao, "n_abf": n_abf,
            "r_c": r_c, "precision": precision, "strain": 0.0, "entry": "host", "graph": False, "deterministic": False}
    case.update(kw)
    return case


def listed():
    return [
        # the smallest calls: an 8-atom cell of a minimal basis, in FP64 and,
        # in an MD loop with frozen lists, replayed from the plan's CUDA graph
        _eval("cell8_fp64", "diamond", 1, "4", "9", 2.6, "fp64"),
        _eval("cell8_graph", "diamond", 1, "4", "9", 2.6, "bf16x6", graph=True),
        # FP64 at a real basis: the reference result of a small three-species cell
        _eval("perovskite5_fp64", "perovskite", 1, "18,13,13", "75,60,60", 4.2, "fp64"),
        # Si at a double-zeta basis: unit cell, the ordinary 64-atom cell (both
        # split precisions), and the largest that a server holds several of
        _eval("si8", "diamond", 1, "13", "50", 3.7, "bf16x6"),
        _eval("si64", "diamond", 2, "13", "50", 3.7, "bf16x6", entry="device"),
        _eval("si64_x3", "diamond", 2, "13", "50", 3.7, "bf16x3", strain=0.03),
        _eval("si216", "diamond", 3, "13", "50", 3.7, "bf16x6", entry="device", strain=0.03),
        # ragged blocks of three species, bit-reproducible sums
        _eval("ragged40", "perovskite", 2, "5,9,13", "14,40,50", 3.7, "bf16x6", deterministic=True),
        # more than 16 orbitals on one species (Cs): unit-cell doubling and a relaxation-size cell
        _eval("perovskite40", "perovskite", 2, "18,13,13", "75,60,60", 4.2, "bf16x6"),
        _eval("perovskite135", "perovskite", 3, "18,13,13", "75,60,60", 4.2, "bf16x6", entry="device"),
        # block preparation: a few small pairs (coefficients only), and the pairs of a Si shell with gradients
        {"name": "lri_small", "what": "lri", "batch": 6, "m_i": 7, "m_k": 5, "n_i": 3, "n_k": 2, "gradient": False},
        {"name": "lri_si", "what": "lri", "batch": 128, "m_i": 50, "m_k": 50, "n_i": 13, "n_k": 13, "gradient": True},
    ]


def draw(rng):
    what = rng.choice(["fp64", "split", "split", "ragged", "wide", "lri"])
    if what == "lri":
        m_i, m_k = rng.randint(4, 64), rng.randint(4, 64)
        n_i, n_k = rng.randint(2, 13), rng.randint(2, 13)
        batch = int(math.exp(rng.uniform(math.log(2), math.log(129))))
        return {"what": "lri", "batch": batch, "m_i": m_i, "m_k": m_k, "n_i": n_i, "n_k": n_k,
                "gradient": rng.random() < 0.6}
    if what == "fp64":
        big = rng.random() < 0.3
        c = _eval("", "diamond", 1, str(rng.randint(7, 13) if big else rng.randint(2, 6)),
                  str(rng.randint(17, 50) if big else rng.randint(3, 16)), round(rng.uniform(2.2, 2.8), 2), "fp64")
    elif what == "split":
        n_rep = rng.choice([1, 1, 2, 2, 3])
        over = rng.random() < 0.15   # auxiliary sets beyond 64, with small orbital sets
        c = _eval("", "diamond", min(n_rep, 2) if over else n_rep, str(rng.randint(3, 9) if over else rng.randint(4, 15 if n_rep < 3 else 13)),
                  str(rng.randint(65, 80) if over else rng.randint(9, 64 if n_rep < 3 else 50)),
                  round(rng.uniform(2.6, 3.7), 2), rng.choice(["bf16x6", "bf16x6", "bf16x3"]),
                  graph=rng.random() < 0.2, strain=rng.choice([0.0, 0.03]))
    elif what == "ragged":
        c = _eval("", "perovskite", rng.choice([1, 2, 2]), ",".join(str(rng.randint(3, 15)) for _ in range(3)),
                  ",".join(str(rng.randint(9, 64)) for _ in range(3)), round(rng.uniform(3.0, 4.2), 2), "bf16x6",
                  deterministic=rng.random() < 0.3)
    else:
        c = _eval("", "perovskite", rng.choice([1, 2, 2, 3]), "%d,%d,%d" % (rng.randint(17, 18), rng.randint(9, 13),
                                                                            rng.randint(9, 13)),
                  "%d,%d,%d" % (rng.randint(50, 75), rng.randint(30, 60), rng.randint(30, 60)),
                  round(rng.uniform(3.4, 4.2), 2), "bf16x6", strain=rng.choice([0.0, 0.03]))
    c["entry"] = rng.choice(["host", "device"])
    del c["name"]
    return c


def _ints(text):
    return [int(x) for x in text.split(",")]


def _workload(case, seed, n_rep=None):
    return inputs.make_workload(case["lattice"], n_rep or case["n_rep"], SPACING[case["lattice"]],
                                _ints(case["n_ao"]), _ints(case["n_abf"]), case["r_c"], 1000 + seed,
                                strain_amp=case["strain"])


def _inputs(case, seed):
    """The cell and the geometry of the step."""
    w = _workload(case, seed)
    return w, inputs.geometry_sequence(w, 1, seed=seed + 17)[0]


def _pairs(case, seed):
    return inputs.lri_pairs(case["batch"], case["m_i"], case["m_k"], case["n_i"], case["n_k"], seed=5 + seed)


def prepare(case, seed):
    if case["what"] == "lri":
        _, A, B, dA, dB, _ = _pairs(case, seed)
        return {"what": "lri", "args": (A, B, dA, dB) if case["gradient"] else (A, B)}
    w, pos = _inputs(case, seed)
    plan = hfx.Plan(w, precision=PRECISION[case["precision"]], freeze_lists=case["graph"], graph=case["graph"],
                    deterministic=case["deterministic"])
    state = {"what": case["entry"], "plan": plan, "lattice": w.lattice, "positions": pos, "n": w.n_atoms,
             "single": case["precision"] != "fp64"}
    if case["entry"] == "device":
        state["d_pos"] = torch.tensor(pos, dtype=torch.float64, device="cuda")
        state["d_out"] = torch.zeros(1 + 3 * w.n_atoms + 9, dtype=torch.float64, device="cuda")
    return state


def run(state):
    if state["what"] == "lri":
        return hfx.lri_fit(*state["args"])
    if state["what"] == "device":   # positions and results in device memory
        out, n = state["d_out"], state["n"]
        state["plan"].evaluate_device(state["lattice"], state["d_pos"].data_ptr(), out.data_ptr())
        res = out.to(torch.float32) if state["single"] else out
        return {"E": res[:1], "F": res[1:1 + 3 * n].view(n, 3), "sigma": res[1 + 3 * n:].view(3, 3)}
    E, F, sigma = state["plan"].evaluate(state["lattice"], state["positions"])
    kind = np.float32 if state["single"] else np.float64
    return {"E": np.array([E], kind), "F": F.astype(kind, copy=False), "sigma": sigma.astype(kind, copy=False)}


# ---------------------------------------------------------------- the same in 64 bits
# Written from the method: C = G f(r), V = M h(r); items screened by norm and
# by Cauchy-Schwarz bound; Y^{XZ} = sum_W C_XW D_WZ; E and its derivatives in
# the pair vectors.  Blocks are padded to the largest shape with zeros.
class _Cell:
    """Pairs, radial factors and kept items of a cell."""

    def __init__(self, w, pos):
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        t = lambda a, k=torch.float64: torch.as_tensor(np.ascontiguousarray(a), dtype=k, device=self.dev)  # noqa: E731
        self.w, self.N, self.S = w, w.n_atoms, w.n_species
        self.na, self.ma = int(w.n_ao.max()), int(w.n_abf.max())
        self.sp = t(w.species, torch.long)
        self.pos, self.L = t(pos), t(w.lattice)
        self.G = torch.zeros(self.S, self.S, self.ma, self.na, self.na, dtype=torch.float64, device=self.dev)
        self.M = torch.zeros(self.S, self.S, self.ma, self.ma, dtype=torch.float64, device=self.dev)
        for s in range(self.S):
            for u in range(self.S):
                g, m = w.G[s * self.S + u], w.M[s * self.S + u]
                self.G[s, u, :g.shape[0], :g.shape[1], :g.shape[2]] = t(g)
                self.M[s, u, :m.shape[0], :m.shape[1]] = t(m)
        self.Gn, self.Mn = self.G.flatten(2).norm(dim=2), self.M.flatten(2).norm(dim=2)
        # D blocks, padded, and the table (i, j, R) -> block (the last block is zero)
        idx = t(w.d_index, torch.long)
        nd = idx.shape[0]
        self.D = torch.zeros(nd + 1, self.na, self.na, dtype=torch.float64, device=self.dev)
        off, vals = t(w.d_offset, torch.long), t(w.d_values)
        nao = t(w.n_ao, torch.long)
        ni, nj = nao[self.sp[idx[:, 0]]], nao[self.sp[idx[:, 1]]]
        for a in range(self.na):
            for b in range(self.na):
                k = torch.nonzero((ni > a) & (nj > b))[:, 0]
                self.D[k, a, b] = vals[off[k] + a * nj[k] + b]
        self.Dn = self.D.flatten(1).norm(dim=1)
        self.Dn[self.Dn <= w.theta["D"]] = 0.0
        self.D[self.Dn == 0.0] = 0.0
        self.HD = int(idx[:, 2:].abs().max())
        n = 2 * self.HD + 1
        self.dlut = torch.full((self.N * self.N * n ** 3,), nd, dtype=torch.long, device=self.dev)
        self.dlut[self._at(idx[:, 0], idx[:, 1], idx[:, 2:], self.HD)] = torch.arange(nd, device=self.dev)
        d = self.pos[idx[:, 1]] + idx[:, 2:].double() @ self.L - self.pos[idx[:, 0]]
        reach = float(d.norm(dim=1).max())
        RC = 2.0 * w.r_c
        self.images = t(_images(w.lattice, RC + reach + 1.0), torch.long)
        # C pairs
        self.c = self._near(RC)
        r = self.c["r"]
        x, e = 1.0 - (r / RC) ** 2, torch.exp(-0.5 * r * r)
        f, fp = x ** 3 * e, (-6.0 * r / RC ** 2) * x * x * e - r * x ** 3 * e
        site = self.c["site"]
        self.c["f"] = torch.where(site, 1.0, f)
        self.c["g"] = torch.where(site, 0.0, fp / r.clamp_min(1e-300))[:, None] * self.c["d"]
        gn = self.Gn[self.sp[self.c["i"]], self.sp[self.c["j"]]]
        nC, nG = self.c["f"].abs() * gn, torch.where(site, 0.0, fp.abs()) * gn
        keep = (nC > w.theta["C"]) | (nG > w.theta["dC"])
        self.c["n"] = torch.where(keep, torch.maximum(nC, nG), 0.0)
        self.c = {k: v[keep] for k, v in self.c.items()}
        # V pairs
        self.v = self._near(RC + reach + 1.0)
        r, om = self.v["r"], w.omega
        ec = torch.erfc(om * r)
        h, hp = ec / (r + 1.0), (-2.0 * om / math.sqrt(math.pi)) * torch.exp(-(om * r) ** 2) / (r + 1.0) - ec / (r + 1.0) ** 2
        site = self.v["site"]
        self.v["h"] = torch.where(site, 1.0, h)
        self.v["g"] = torch.where(site, 0.0, hp / r.clamp_min(1e-300))[:, None] * self.v["d"]
        mn = self.Mn[self.sp[self.v["i"]], self.sp[self.v["j"]]]
        nV, nG = self.v["h"].abs() * mn, torch.where(site, torch.zeros_like(hp), hp.abs()) * mn
        self.v["n"] = torch.where((nV > w.theta["V"]) | (nG > w.theta["dV"]), torch.maximum(nV, nG), 0.0)
        # the bound's inner factor of every key (X; Z) is made on demand from the V pairs, which hold every key in reach
        self.HY = int(self.v["R"].abs().max())
        n = 2 * self.HY + 1
        self.ylut = torch.full((self.N * self.N * n ** 3,), -1, dtype=torch.long, device=self.dev)
        self.ylut[self._at(self.v["i"], self.v["j"], self.v["R"], self.HY)] = torch.arange(len(self.v["i"]), device=self.dev)
        self.cp = torch.searchsorted(self.c["i"], torch.arange(self.N + 1, device=self.dev)).tolist()
        self.vp = torch.searchsorted(self.v["i"], torch.arange(self.N + 1, device=self.dev)).tolist()
        self.yhat = torch.zeros(len(self.v["i"]), dtype=torch.float64, device=self.dev)
        for X in range(self.N):
            c, v = self.home(self.c, self.cp, X), self.home(self.v, self.vp, X)
            di = self.d_of(c["j"][None, :], v["j"][:, None], v["R"][:, None] - c["R"][None])
            self.yhat[self.vp[X]:self.vp[X + 1]] = self.Dn[di] @ c["n"]

    def _at(self, i, j, R, H):
        n = 2 * H + 1
        R = R + H
        return (((i * self.N + j) * n + R[..., 0]) * n + R[..., 1]) * n + R[..., 2]

    def _near(self, rmax):
        """Pairs (i -> j, R) closer than rmax, by i."""
        parts = []
        for i in range(self.N):
            d = self.pos[None] + (self.images.double() @ self.L)[:, None] - self.pos[i]
            r = d.norm(dim=2)
            kR, kj = torch.nonzero(r < rmax, as_tuple=True)
            parts.append((torch.full_like(kj, i), kj, self.images[kR], d[kR, kj], r[kR, kj]))
        i, j, R, d, r = (torch.cat(x) for x in zip(*parts))
        return {"i": i, "j": j, "R": R, "d": d, "r": r, "site": (i == j) & (R == 0).all(dim=1)}

    def home(self, pairs, ptr, A):
        return {k: v[ptr[A]:ptr[A + 1]] for k, v in pairs.items()}

    def d_of(self, i, j, R):
        """Block numbers of D_{ij}(R); the zero block where there is none."""
        inside = (R.abs() <= self.HD).all(dim=-1)
        got = self.dlut[torch.where(inside, self._at(i, j, R.clamp(-self.HD, self.HD), self.HD), 0)]
        return torch.where(inside, got, self.D.shape[0] - 1)

    def y_of(self, i, j, R):
        inside = (R.abs() <= self.HY).all(dim=-1)
        got = self.ylut[torch.where(inside, self._at(i, j, R.clamp(-self.HY, self.HY), self.HY), 0)]
        return torch.where(inside, got, -1)

    def items(self, A):
        """Kept triplets (V pair, C pair, key of Y^{BF}) and kept pairs of the second product of home atom A."""
        c, v, cs = self.home(self.c, self.cp, A), self.home(self.v, self.vp, A), self.w.theta["CS"]
        dn = self.Dn[self.d_of(v["i"], v["j"], v["R"])] * v["n"]
        q = torch.nonzero(dn > 0.0)[:, 0]
        y = self.y_of(v["j"][q][:, None], c["j"][None], c["R"][None] - v["R"][q][:, None])
        bound = dn[q][:, None] * c["n"][None] * torch.where(y >= 0, self.yhat[y.clamp_min(0)], 0.0)
        kv, kc = torch.nonzero(bound > cs, as_tuple=True)
        y1 = torch.arange(self.vp[A], self.vp[A + 1], device=self.dev)
        y2 = self.y_of(v["j"], v["i"], -v["R"])
        pairs = torch.nonzero((y2 >= 0) & (v["n"] * self.yhat[y1] * self.yhat[y2.clamp_min(0)] > cs))[:, 0]
        return (self.vp[A] + q[kv], self.cp[A] + kc, y[kv, kc]), (self.vp[A] + pairs, y2[pairs])


def _images(lattice, rmax):
    recip = np.linalg.inv(lattice).T
    n = [int(math.ceil(rmax * np.linalg.norm(recip[k]))) + 1 for k in range(3)]
    return np.stack(np.meshgrid(*[np.arange(-k, k + 1) for k in n], indexing="ij"), -1).reshape(-1, 3)


def _exact_evaluate(w, pos):
    C = _Cell(w, pos)
    N, na, ma, dev = C.N, C.na, C.ma, C.dev
    items = [C.items(A) for A in range(N)]
    need = torch.zeros(len(C.v["i"]), dtype=torch.bool, device=dev)
    for A, ((_, _, y), (p, y2)) in enumerate(items):
        need[y] = True
        need[p] = True
        need[y2] = True
    slot = torch.cumsum(need, 0) - 1
    Y = torch.zeros(int(need.sum()), na, ma, na, dtype=torch.float64, device=dev)   # [key][x][alpha][z]
    for X in range(N):
        c = C.home(C.c, C.cp, X)
        blocks = C.G[C.sp[X], C.sp[c["j"]]] * c["f"][:, None, None, None]           # [W][alpha][x][w]
        Cx = blocks.permute(2, 1, 0, 3).reshape(na * ma, -1)
        keys = torch.nonzero(need[C.vp[X]:C.vp[X + 1]])[:, 0] + C.vp[X]
        for k in keys.split(256):
            di = C.d_of(c["j"][:, None], C.v["j"][k][None], C.v["R"][k][None] - c["R"][:, None])
            Dx = C.D[di].permute(0, 2, 1, 3).reshape(len(c["j"]) * na, -1)          # [(W, w)][(Z, z)]
            Y[slot[k]] = (Cx @ Dx).view(na, ma, len(k), na).permute(2, 0, 1, 3)
    E = torch.zeros((), dtype=torch.float64, device=dev)
    gC = torch.zeros(len(C.c["i"]), 3, dtype=torch.float64, device=dev)
    s = torch.zeros(len(C.v["i"]), dtype=torch.float64, device=dev)                 # <M, R_AB>
    for A in range(N):
        (tv, tc, ty), (pv, y2) = items[A]
        sA = int(C.sp[A])
        if len(pv):
            Yba = Y[slot[y2]].permute(0, 2, 1, 3)                                   # [B][beta][b][a]
            MY = C.M[sA, C.sp[C.v["j"][pv]]] @ Yba.reshape(len(pv), ma, na * na)
            MY = MY.view(-1, ma, na, na).transpose(2, 3)                            # [B][alpha][a][b]
            s[pv] += (MY * Y[slot[pv]].transpose(1, 2)).sum(dim=(1, 2, 3))
            Z = (MY * C.v["h"][pv][:, None, None, None]).permute(1, 2, 0, 3).reshape(ma * na, -1)
        order = torch.argsort(tc, stable=True)
        tv, tc, ty = tv[order], tc[order], ty[order]
        ends = torch.searchsorted(tc, torch.arange(C.cp[A], C.cp[A + 1] + 1, device=dev)).tolist()
        for k, q in enumerate(range(C.cp[A], C.cp[A + 1])):
            f = int(C.c["j"][q])
            Gt = C.G[sA, C.sp[f]]
            Q = torch.zeros(ma, na, na, dtype=torch.float64, device=dev)
            a, b = ends[k], ends[k + 1]
            if b > a:
                p, n = tv[a:b], b - a
                Dab = C.D[C.d_of(C.v["i"][p], C.v["j"][p], C.v["R"][p])]
                U = torch.bmm(Dab, Y[slot[ty[a:b]]].view(n, na, ma * na))           # [B][a][(beta, f)]
                U = U.view(n, na, ma, na).transpose(1, 2).reshape(n, ma, na * na)
                W = torch.bmm(C.M[sA, C.sp[C.v["j"][p]]], U)                        # [B][alpha][(a, f)]
                s[p] += C.c["f"][q] * (W * Gt.reshape(ma, na * na)).sum(dim=(1, 2))
                Q += torch.einsum("n,nxy->xy", C.v["h"][p], W).view(ma, na, na)
            if len(pv):
                di = C.d_of(torch.full_like(pv, f), C.v["j"][pv], C.v["R"][pv] - C.c["R"][q])
                Q += (Z @ C.D[di].transpose(1, 2).reshape(-1, na)).view(ma, na, na)
            gC[q] = -2.0 * (Gt * Q).sum() * C.c["g"][q]
    E -= (C.v["h"] * s).sum()
    F = torch.zeros(N, 3, dtype=torch.float64, device=dev)
    W = torch.zeros(3, 3, dtype=torch.float64, device=dev)
    for pairs, g in ((C.c, gC), (C.v, -s[:, None] * C.v["g"])):
        F.index_add_(0, pairs["i"], g)
        F.index_add_(0, pairs["j"], -g)
        W += g.T @ pairs["d"]
    sigma = -W / abs(float(np.linalg.det(w.lattice)))
    return {"E": E.view(1), "F": F, "sigma": sigma}


def exact(case, seed):
    if case["what"] == "lri":
        _, A, B, dA, dB, _ = (torch.as_tensor(x) if isinstance(x, np.ndarray) else x for x in _pairs(case, seed))
        X = torch.linalg.solve(A, B)
        return (X, torch.linalg.solve(A[:, None], dB - dA @ X[:, None])) if case["gradient"] else X
    return _exact_evaluate(*_inputs(case, seed))


_counted = {}


def _per_cell(case):
    """Contraction FLOPs and D bytes per unit cell of the lattice (every
    supercell has the same pairs per atom): 2 n_abf(X) n_ao(X) n_ao(W) n_ao(Z)
    per term of a Y block, and per kept item of the two exchange products."""
    key = (case["lattice"], case["n_ao"], case["n_abf"], case["r_c"])
    if key not in _counted:
        w = _workload(dict(case, strain=0.0), 0, n_rep=1)
        C = _Cell(w, w.positions)
        na = torch.as_tensor(w.n_ao, dtype=torch.float64, device=C.dev)[C.sp]
        nb = torch.as_tensor(w.n_abf, dtype=torch.float64, device=C.dev)[C.sp]
        flops, need = 0.0, torch.zeros(len(C.v["i"]), dtype=torch.bool, device=C.dev)
        for A in range(C.N):
            (tv, tc, ty), (pv, y2) = C.items(A)
            need[ty] = True
            need[pv] = True
            need[y2] = True
            B, F = C.v["j"][tv], C.c["j"][tc]
            flops += float((2 * nb[B] * na[A] * na[B] * na[F] + 4 * nb[A] * nb[B] * na[A] * na[F]).sum())
            B = C.v["j"][pv]
            flops += float((4 * nb[A] * nb[B] * na[A] * na[B]).sum())
            c = C.home(C.c, C.cp, A)
            di = C.d_of(c["j"][:, None], B[None], C.v["R"][pv][None] - c["R"][:, None])
            flops += float((2 * nb[A] * na[A] * na[c["j"]][:, None] * na[B][None] * (C.Dn[di] > 0)).sum())
        for X in range(C.N):
            c, k = C.home(C.c, C.cp, X), torch.nonzero(need[C.vp[X]:C.vp[X + 1]])[:, 0] + C.vp[X]
            di = C.d_of(c["j"][:, None], C.v["j"][k][None], C.v["R"][k][None] - c["R"][:, None])
            flops += float((2 * nb[X] * na[X] * na[c["j"]][:, None] * na[C.v["j"][k]][None] * (C.Dn[di] > 0)).sum())
        _counted[key] = (flops, 8.0 * w.d_values.size)
    return _counted[key]


def work(case):
    if case["what"] == "lri":
        b, n, w = case["batch"], case["m_i"] + case["m_k"], case["n_i"] * case["n_k"]
        k = 4 if case["gradient"] else 1
        flops = b * (n ** 3 / 3 + 2.0 * n * n * w + (k - 1) * 4.0 * n * n * w)
        return {"bytes": 8.0 * b * k * (n * n + 2 * n * w), "flops": flops}
    cells = case["n_rep"] ** 3
    flops, d_bytes = _per_cell(case)
    n_ao, n_abf = _ints(case["n_ao"]), _ints(case["n_abf"])
    templates = sum(8.0 * b * (a * a2 + b2) for a, b in zip(n_ao, n_abf) for a2, b2 in zip(n_ao, n_abf))
    atoms = cells * (8 if case["lattice"] == "diamond" else 5)
    return {"bytes": cells * d_bytes + templates + 48.0 * atoms + 80.0, "flops": cells * flops}
