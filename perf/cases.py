"""Timed workloads of the library, one pass each through its public calls.

A case is a lattice, a bond dimension, a precision and one of the calls that
a ground-state search is made of:

  product   y = H_eff x at one node (ttn_apply_heff_device), the inner call of
            every eigensolver step
  gradient  E, dE/dpsi and dE/dcouplings at one node (ttn_energy_grad: the
            forward products and the adjoint one)
  move      the isometry centre taken to another node and back
            (ttn_move_center: QR, absorption, operator updates), with one
            product at each end, as a sweep uses the operators
  update    one node update from a given tensor (ttn_node_import,
            ttn_optimize_node, ttn_node_export)
  sweep     a whole sweep from host tensors with the energies and the
            site probabilities (ttn_load_tensors, ttn_sweep, ttn_energy,
            ttn_measure)
  batch     the same for two charge sectors swept together (ttn_batch_sweep)

Products of a mixed-precision state carry FP32 accuracy, and the vector of an
eigensolver (with the probabilities read off it) is fixed by its tolerance
only: they are handed on as FP32, every FP64 quantity as FP64.

``exact`` restates each call in dense FP64 torch (charge blocks ignored, every
operator a plain matrix or a row selection) from the same tensors.
"""
import numpy as np
import torch

import paper_2011_10658_gb300 as qed

D = 267            # dressed-site dimension
KRYLOV = 64        # eigensolver basis
MIXED = ("tf32x3", "tf32", "bf16")


def _case(name, kind, L, chi, Q, precision, layer=0, to=-1, g2=1.0, tol=0.0):
    c = dict(kind=kind, Lx=L[0], Ly=L[1], Lz=L[2], chi=chi, Q=Q, precision=precision, layer=layer, to=to, g2=g2, tol=tol)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: the one-block product at the root of a small tree
        _case("root_4x2x2_chi16", "product", (4, 2, 2), 16, 0, "tf32x3", layer=3),
        # the plain FP64 method's product, on narrow sectors
        _case("product_2x2x2_chi8_fp64", "product", (2, 2, 2), 8, 0, "fp64"),
        # the benchmark state's bottom and upper products, split TF32
        _case("product_4x4x4_chi64", "product", (4, 4, 4), 64, 0, "tf32x3"),
        _case("upper_4x4x4_chi64", "product", (4, 4, 4), 64, 0, "tf32x3", layer=2),
        # a problem of the finite-density batch, BF16 operands, odd sector widths
        _case("product_4x4x4_chi48_bf16", "product", (4, 4, 4), 48, 8, "bf16", g2=0.5),
        # the FP64 path that every mixed result is checked against
        _case("product_4x4x4_chi64_fp64", "product", (4, 4, 4), 64, 0, "fp64"),
        # forward and adjoint products of the gradient node update
        _case("gradient_4x4x4_chi32", "gradient", (4, 4, 4), 32, 4, "fp64"),
        # centre moves between neighbouring bottom nodes, as a sweep does them
        _case("move_4x4x4_chi64", "move", (4, 4, 4), 64, 0, "tf32x3", to=0),
        # node updates inside a sweep: the widest (bottom) and a narrow one
        _case("update_4x4x4_chi64", "update", (4, 4, 4), 64, 0, "tf32x3", tol=1e-6),
        _case("update_4x4x4_chi32_layer3", "update", (4, 4, 4), 32, 4, "tf32x3", layer=3, tol=1e-8),
        # the plain method as a whole: one FP64 sweep and its observables
        _case("sweep_2x2x2_chi8", "sweep", (2, 2, 2), 8, 0, "fp64", tol=1e-12),
        # two charge sectors of it together
        _case("batch_2x2x2_chi8", "batch", (2, 2, 2), 8, 0, "fp64", tol=1e-12),
    ]


LATTICES = {(2, 2, 2): 3, (4, 2, 2): 4, (4, 4, 2): 5, (4, 4, 4): 6}   # layers of the tree


def draw(rng):
    kind = rng.choice(["product"] * 5 + ["gradient", "move", "move", "update", "update", "sweep"])
    g2 = rng.choice([0.5, 1.0, 2.0, 4.0])
    if kind == "sweep":
        return _case(None, "sweep", (2, 2, 2), rng.randint(5, 8), rng.choice([0, 1, 2]), "fp64", g2=rng.choice([0.5, 1.0, 2.0]), tol=1e-12)
    L = rng.choice([(2, 2, 2), (4, 2, 2), (4, 4, 2), (4, 4, 4), (4, 4, 4)])
    chi = int(round(np.exp(rng.uniform(np.log(7), np.log({3: 16, 4: 32, 5: 64, 6: 64}[LATTICES[L]])))))
    Q = rng.choice([0, 0, 1, 2, 4])
    layer = rng.choice([0, 0, rng.randrange(LATTICES[L])])
    precision = rng.choice(["tf32x3", "tf32x3", "fp64", "tf32", "bf16"])
    if kind == "product":
        if L == (4, 4, 4) and precision != "fp64":
            chi = int(round(np.exp(rng.uniform(np.log(12), np.log(96)))))
        return _case(None, kind, L, chi, Q, precision, layer=layer, g2=g2)
    if kind == "gradient":
        return _case(None, kind, L, min(chi, 32), Q, "fp64", layer=layer, g2=g2)
    if kind == "move":
        to = rng.choice([0, 1])
        return _case(None, kind, L, chi, Q, rng.choice(["tf32x3", "fp64", "bf16"]), layer=to and rng.choice([0, 2]), to=to, g2=g2)
    return _case(None, kind, L, min(chi, 48), Q, rng.choice(["tf32x3", "tf32x3", "fp64"]), layer=layer, g2=g2, tol=1e-8)


# ---------------------------------------------------------------- the problem
def _couplings(g2):
    """t = m = 1, electric g^2, plaquette 1 / (2 g^2), penalty ten times the largest."""
    cB = 1.0 / (2.0 * g2)
    return dict(t=1.0, m=1.0, ge2=float(g2), cB=cB, nu=10.0 * max(1.0, g2 / 2.0, cB))


class Tables:
    """Lattice, terms, tree and sectors of a case: the problem's statement."""

    def __init__(self, case, Q=None):
        self.couplings = _couplings(case["g2"])
        self.shape = (case["Lx"], case["Ly"], case["Lz"])
        self.model = qed.Model(*self.shape, Q=case["Q"] if Q is None else Q, **self.couplings)
        self.chi = case["chi"]
        coef, cls, nops, ops = self.model.terms()
        self.terms = [(float(coef[k]), int(cls[k]), {int(o[0]): (int(o[1]), int(o[2]), int(o[3])) for o in ops[k][: nops[k]]})
                      for k in range(len(coef))]
        tree = self.model.tree()
        self.layer = [int(r[0]) for r in tree]
        self.kids = [((int(r[2]), int(r[3])), (int(r[4]), int(r[5]))) for r in tree]
        self.parent = [int(r[6]) for r in tree]
        self.bonds = [sorted(b.items()) for b in self.model.sectors(self.chi)]
        self.sites = []
        for kid in self.kids:
            s = []
            for kind, i in kid:
                s += [i] if kind == 0 else self.sites[i]
            self.sites.append(s)
        self.charge = {p: qed.basis(p)[:, 8].astype(int) for p in (1, -1)}
        self._ops = {}
        self._touch = {}

    def node(self, case, where="layer"):
        """First node of a layer (-1: none); the second one where the case starts there too."""
        at = [i for i, l in enumerate(self.layer) if l == case[where]]
        return at[1 if where == "to" and case["to"] == case["layer"] else 0]

    def parity(self, site):
        x, y, z = site % self.shape[0], site // self.shape[0] % self.shape[1], site // (self.shape[0] * self.shape[1])
        return 1 if (x + y + z) % 2 == 0 else -1

    def op(self, site, key):
        """(src, val, charge shift) of a site operator."""
        k = (self.parity(site),) + key
        if k not in self._ops:
            src, val = qed.local_op(k[0], *key)
            src = src.astype(np.int64)
            rows = np.nonzero((src >= 0) & (val != 0))[0]
            q = self.charge[k[0]]
            self._ops[k] = (src, val, int(q[rows[0]] - q[src[rows[0]]]) if rows.size else 0)
        return self._ops[k]

    def leg(self, node, leg):
        """[(charge, dimension)] of a leg."""
        if leg == 2:
            return self.bonds[node]
        kind, i = self.kids[node][leg]
        if kind == 1:
            return self.bonds[i]
        q = self.charge[self.parity(i)]
        return [(int(c), int((q == c).sum())) for c in np.unique(q)]

    def blocks(self, node):
        """(left, right, parent sector indices) in storage order."""
        la, lb, lc = (self.leg(node, i) for i in range(3))
        b = {q: i for i, (q, _) in enumerate(lb)}
        return [(ia, b[qc - qa], ic) for ic, (qc, _) in enumerate(lc) for ia, (qa, _) in enumerate(la) if qc - qa in b]

    def index(self, node):
        """Dense (a, b, c) index of every stored entry."""
        legs = [self.leg(node, i) for i in range(3)]
        off = [np.concatenate([[0], np.cumsum([d for _, d in l])]) for l in legs]
        at = []
        for blk in self.blocks(node):
            r = [np.arange(off[i][blk[i]], off[i][blk[i] + 1]) for i in range(3)]
            at.append(((r[0][:, None, None] * off[1][-1] + r[1][:, None]) * off[2][-1] + r[2]).reshape(-1))
        return np.concatenate(at), tuple(int(o[-1]) for o in off)

    def region(self, node, leg):
        if leg == 2:
            return set(range(int(np.prod(self.shape)))) - set(self.sites[node])
        kind, i = self.kids[node][leg]
        return {i} if kind == 0 else set(self.sites[i])

    def touched(self, k, node):
        """Which of the three regions around a node term k acts on."""
        if node not in self._touch:
            around = [self.region(node, leg) for leg in range(3)]
            self._touch[node] = [tuple(any(s in r for s in ops) for r in around) for _, _, ops in self.terms]
        return self._touch[node][k]

    def shift(self, k, sites):
        return sum(self.op(s, o)[2] for s, o in self.terms[k][2].items() if s in sites)


# ---------------------------------------------------------------- states
_kept = {}


def _tables(case):
    key = ("tables",) + tuple(case[k] for k in ("Lx", "Ly", "Lz", "chi", "Q", "g2"))
    if _kept.get("tables", (None,))[0] != key:
        _kept["tables"] = (key, Tables(case))
    return _kept["tables"][1]


def _handle(case):
    """The tensor network that the calls work on, kept as a program keeps it
    (one at a time); an update's has one loose sweep behind it."""
    key = tuple(case[k] for k in ("Lx", "Ly", "Lz", "chi", "Q", "g2", "precision")) + (case["kind"] == "update",)
    if _kept.get("handle", (None,))[0] != key:
        _kept.pop("handle", None)
        ttn = qed.TTN(_tables(case).model, case["chi"], seed=1, precision=case["precision"],
                      stream=torch.cuda.current_stream().cuda_stream)
        if case["kind"] == "update":
            ttn.sweep(1, tol=1e-3, max_krylov=KRYLOV, allow_noconv=True)
        if case["kind"] == "move":
            tab = _tables(case)
            a, b, root = tab.node(case), tab.node(case, "to"), len(tab.parent) - 1
            ttn.move_center(a)
            d = Dense(tab, [ttn.node_export(n) for n in range(root + 1)])
            d.move(a, b, schmidt=True)
            d.move(b, root)
            ttn.load_tensors([d.packed(n, t).cpu().numpy() for n, t in enumerate(d.T)])
            for n in (a, b, a, b):
                ttn.move_center(n)
        _kept["handle"] = (key, ttn)
    return _kept["handle"][1]


class State:
    pass


def _randn(n, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(n, dtype=torch.float64, device="cuda", generator=g)


def prepare(case, seed):
    s = State()
    s.case, s.kind = case, case["kind"]
    if s.kind in ("sweep", "batch"):
        s.ttn, s.start = [], []
        for i in range(2 if s.kind == "batch" else 1):
            tab = Tables(case, Q=case["Q"] + 2 * i)
            ttn = qed.TTN(tab.model, case["chi"], seed=seed + i, precision=case["precision"],
                          stream=torch.cuda.current_stream().cuda_stream)
            s.ttn.append(ttn)
            s.start.append([ttn.node_export(n) for n in range(len(tab.parent))])
        return s
    tab = _tables(case)
    s.ttn = _handle(case)
    s.node = tab.node(case)
    if s.kind == "move":
        s.far = tab.node(case, "to")
        s.x = [_randn(s.ttn.node_size(n), seed + 7919 * i) for i, n in enumerate((s.far, s.node))]
        s.y = [torch.empty_like(x) for x in s.x]
    s.ttn.move_center(s.node)
    s.n = s.ttn.node_size(s.node)
    if s.kind == "update":
        now = torch.from_numpy(s.ttn.node_export(s.node)).cuda()
        start = now / now.norm() + 0.3 * _randn(s.n, seed) / s.n ** 0.5
        s.start = (start / start.norm()).cpu().numpy()
    elif s.kind in ("product", "gradient"):
        s.x = _randn(s.n, seed)
        s.y = torch.empty_like(s.x)
    return s


def _out(y, precision):
    return y.to(torch.float32) if precision in MIXED else y


def run(s):
    c = s.case
    if s.kind == "product":
        s.ttn.apply_heff_device(s.x.data_ptr(), s.y.data_ptr(), s.n)
        return _out(s.y, c["precision"])
    if s.kind == "gradient":
        e, dc = s.ttn.energy_grad_device(s.node, s.x.data_ptr(), s.y.data_ptr(), s.n)
        return {"energy": e, "couplings": dc, "psi": s.y}
    if s.kind == "move":
        out = []
        for n, x, y in zip((s.far, s.node), s.x, s.y):
            s.ttn.move_center(n)
            s.ttn.apply_heff_device(x.data_ptr(), y.data_ptr(), x.numel())
            out.append(_out(y, c["precision"]))
        return out
    if s.kind == "update":
        s.ttn.node_import(s.node, s.start)
        e = s.ttn.optimize_node(s.node, tol=c["tol"], max_krylov=KRYLOV)
        return {"energy": e, "tensor": s.ttn.node_export(s.node).astype(np.float32)}
    for ttn, start in zip(s.ttn, s.start):
        ttn.load_tensors(start)
    if s.kind == "batch":
        stats = qed.batch_sweep(s.ttn, 1, tol=c["tol"], max_krylov=KRYLOV)
    else:
        stats = [s.ttn[0].sweep(1, tol=c["tol"], max_krylov=KRYLOV)]
    out = []
    for ttn, st in zip(s.ttn, stats):
        total, bare, parts = ttn.energy()
        out.append({"eigenvalue": st["energy"], "total": total, "bare": bare, "parts": parts, "probs": ttn.measure("probs").astype(np.float32)})
    return out


# ---------------------------------------------------------------- work
def _product_work(tab, node):
    """(flops, operator entries) of one product: every term's operators applied
    leg by leg to the blocks they act on, site operators as row selections."""
    legs = [tab.leg(node, i) for i in range(3)]
    dim = [dict(l) for l in legs]
    bottom = tab.kids[node][0][0] == 0
    flops, entries = 0, 0
    rows = {qc: sum(da * dim[1].get(qc - qa, 0) for qa, da in legs[0]) for qc, _ in legs[2]}
    jobs = [((True, False, False), None), ((False, True, False), None)]
    if tab.parent[node] >= 0:
        jobs.append(((False, False, True), None))
    jobs += [(tab.touched(k, node), k) for k in range(len(tab.terms)) if sum(tab.touched(k, node)) >= 2]
    for touch, k in jobs:
        sh = [tab.shift(k, tab.region(node, i)) if k is not None and touch[i] else 0 for i in range(3)]
        if bottom:
            for qc, dc in legs[2]:
                qi = qc - sh[0] - sh[1]
                if qi not in dim[2]:
                    continue
                n = rows[qc]
                if k is not None:
                    n = 0
                    hit = []
                    for leg in range(2):
                        site = tab.kids[node][leg][1]
                        q = tab.charge[tab.parity(site)]
                        ok = np.ones(D, bool)
                        if site in tab.terms[k][2]:
                            src, val, _ = tab.op(site, tab.terms[k][2][site])
                            ok = (src >= 0) & (val != 0)
                        hit.append({c: int(ok[q == c].sum()) for c in np.unique(q)})
                    n = sum(h * hit[1].get(qc - qa, 0) for qa, h in hit[0].items())
                flops += 2 * n * dc * (dim[2][qi] if touch[2] else 1)
                entries += dc * dim[2][qi] if touch[2] else 0
            continue
        shape = [[dict(l) for l in legs] for _ in range(2)]
        for qa, da in legs[0]:
            for qc, dc in legs[2]:
                qb = qc - qa
                if qb not in dim[1]:
                    continue
                at, size = [qa, qb, qc], [da, dim[1][qb], dc]
                for leg in range(3):
                    if not touch[leg]:
                        continue
                    to = at[leg] + sh[leg]
                    if to not in dim[leg]:
                        break
                    new = dim[leg][to]
                    flops += 2 * size[0] * size[1] * size[2] * new
                    at[leg], size[leg] = to, new
        for leg in range(3):
            if touch[leg]:
                entries += sum(d * dim[leg].get(q + sh[leg], 0) for q, d in legs[leg])
    return flops, entries


def _update_work(tab, node, leg):
    """Flops of the operators of one bond: every term that crosses it, and the
    block Hamiltonian, from the node they are contracted with."""
    legs = [tab.leg(node, i) for i in range(3)]
    n = sum(legs[0][a][1] * legs[1][b][1] * legs[2][c][1] for a, b, c in tab.blocks(node))
    width = max(d for _, d in legs[leg])
    ops = sum(1 for k in range(len(tab.terms)) if tab.touched(k, node)[leg] and sum(tab.touched(k, node)) >= 2)
    share = 0.2 if tab.kids[node][0][0] == 0 else 3.0   # nonzero rows of a selection, or three legs
    return int(2 * n * width * share * (ops + 1)) + 6 * n * width


def work(case):
    tab = _tables(case)
    if case["kind"] in ("sweep", "batch"):
        f = b = 0
        for i in range(2 if case["kind"] == "batch" else 1):
            for node in range(len(tab.parent)):
                pf, pe = _product_work(tab, node)
                n = len(tab.index(node)[0])
                f += 40 * pf + 4 * 40 * 40 * n
                b += 16 * n + 8 * pe
        return {"bytes": b, "flops": f}
    node = tab.node(case)
    n = len(tab.index(node)[0])
    f, e = _product_work(tab, node)
    if case["kind"] == "product":
        return {"bytes": 16 * n + 8 * e, "flops": f}
    if case["kind"] == "gradient":   # the class-resolved products add up to the whole one
        return {"bytes": 16 * n + 8 * e, "flops": 2 * f + 10 * n}
    if case["kind"] == "update":     # about 40 products, each against the basis so far
        return {"bytes": 16 * n + 8 * e, "flops": 40 * f + 4 * 40 * 40 * n}
    far = tab.node(case, "to")
    ff, fe = _product_work(tab, far)
    b = 16 * n + 8 * e + 8 * fe + 16 * len(tab.index(far)[0])
    f += ff
    path = _path(tab, node, far)
    for a, t in list(zip(path, path[1:])) + list(zip(path[::-1], path[::-1][1:])):
        f += _update_work(tab, a, 2 if tab.parent[a] == t else [i for _, i in tab.kids[a]].index(t))
        b += 16 * len(tab.index(a)[0])
    return {"bytes": b, "flops": f}


def _path(tab, a, b):
    up = {a: [a]}
    x = a
    while tab.parent[x] >= 0:
        up[tab.parent[x]] = up[x] + [tab.parent[x]]
        x = tab.parent[x]
    down = [b]
    while down[-1] not in up:
        down.append(tab.parent[down[-1]])
    return up[down[-1]] + down[-2::-1]


# ---------------------------------------------------------------- exact
class Dense:
    """The same problem in dense FP64 torch: T[node] are (left, right, parent)
    arrays, every tensor isometric towards the centre."""

    def __init__(self, tab, packed):
        self.tab = tab
        self.T = []
        for n, v in enumerate(packed):
            at, shape = tab.index(n)
            t = torch.zeros(int(np.prod(shape)), dtype=torch.float64, device="cuda")
            t[torch.from_numpy(at).cuda()] = torch.as_tensor(v, dtype=torch.float64, device="cuda")
            self.T.append(t.view(shape))
        self.memo = {}

    def view(self, node, packed):
        at, shape = self.tab.index(node)
        t = torch.zeros(int(np.prod(shape)), dtype=torch.float64, device="cuda")
        t[torch.from_numpy(at).cuda()] = packed
        return t.view(shape)

    def packed(self, node, t):
        return t.reshape(-1)[torch.from_numpy(self.tab.index(node)[0]).cuda()]

    def inside(self, node, t):
        """t without what rounding put outside the charge blocks."""
        return self.view(node, self.packed(node, t))

    def site_op(self, site, key):
        k = ("site", self.tab.parity(site)) + key
        if k not in self.memo:
            src, val, _ = self.tab.op(site, key)
            self.memo[k] = (torch.from_numpy(np.maximum(src, 0)).cuda(), torch.from_numpy(np.where(src >= 0, val, 0.0)).cuda())
        return self.memo[k]

    @staticmethod
    def on(t, leg, op):
        """op applied to one leg: a matrix, or a row selection (src, val)."""
        if isinstance(op, tuple):
            shape = [1, 1, 1]
            shape[leg] = -1
            return t.index_select(leg, op[0]) * op[1].view(shape)
        return torch.movedim(torch.tensordot(op, t, dims=([1], [leg])), 0, leg)

    @staticmethod
    def gram(t, z, leg):
        other = [i for i in range(3) if i != leg]
        return torch.tensordot(t, z, dims=(other, other))

    def term_op(self, node, leg, k):
        if leg == 2:
            return self.down(node)[0][k]
        kind, i = self.tab.kids[node][leg]
        return self.site_op(i, self.tab.terms[k][2][i]) if kind == 0 else self.up(i)[0][k]

    def ham(self, node, leg, cls):
        """Block Hamiltonian of a leg, of one class or of all."""
        if leg == 2:
            return self.total(self.down(node)[1], cls)
        kind, i = self.tab.kids[node][leg]
        if kind == 1:
            return self.total(self.up(i)[1], cls)
        key = ("diag", i, cls)
        if key not in self.memo:
            d = torch.zeros(D, dtype=torch.float64, device="cuda")
            for coef, cl, ops in self.tab.terms:
                if list(ops) == [i] and cls in (None, cl):
                    d += coef * self.site_op(i, ops[i])[1]
            self.memo[key] = (torch.arange(D, device="cuda"), d)
        return self.memo[key]

    @staticmethod
    def total(parts, cls):
        return sum(parts) if cls is None else parts[cls]

    def _operators(self, node, leg):
        """Operators of `node`'s bond on `leg`, from the terms on its other legs."""
        tab, t = self.tab, self.T[node]
        rest = [i for i in range(3) if i != leg and (i < 2 or tab.parent[node] >= 0)]
        ops, parts = {}, [torch.zeros_like(t) for _ in range(6)]
        for k, (coef, cls, where) in enumerate(tab.terms):
            touch = tab.touched(k, node)
            act = [i for i in rest if touch[i]]
            if not act or (not touch[leg] and len(act) < 2):
                continue
            z = t
            for i in act:
                z = self.on(z, i, self.term_op(node, i, k))
            if touch[leg]:
                ops[k] = self.gram(t, z, leg)
            else:
                parts[cls] += coef * z
        for i in rest:
            for cls in range(6):
                parts[cls] += self.on(t, i, self.ham(node, i, cls))
        return ops, [self.gram(t, p, leg) for p in parts]

    def up(self, node):
        if ("up", node) not in self.memo:
            self.memo[("up", node)] = self._operators(node, 2)
        return self.memo[("up", node)]

    def down(self, node):
        if ("down", node) not in self.memo:
            p = self.tab.parent[node]
            self.memo[("down", node)] = self._operators(p, [i if kind else -1 for kind, i in self.tab.kids[p]].index(node))
        return self.memo[("down", node)]

    def heff(self, node, x, cls=None):
        tab = self.tab
        legs = [i for i in range(3) if i < 2 or tab.parent[node] >= 0]
        y = sum(self.on(x, i, self.ham(node, i, cls)) for i in legs)
        for k, (coef, cl, _) in enumerate(tab.terms):
            touch = tab.touched(k, node)
            if sum(touch) < 2 or cls not in (None, cl):
                continue
            z = x
            for i in range(3):
                if touch[i]:
                    z = self.on(z, i, self.term_op(node, i, k))
            y = torch.add(y, z, alpha=coef)
        return y

    def move(self, a, b, schmidt=False):
        """The isometry centre from a to b: QR with positive diagonal per bond
        (schmidt: singular vectors per charge instead)."""
        tab = self.tab
        path = _path(tab, a, b)
        for c, t in zip(path, path[1:]):
            lc = 2 if tab.parent[c] == t else [i if kind else -1 for kind, i in tab.kids[c]].index(t)
            lt = 2 if tab.parent[t] == c else [i if kind else -1 for kind, i in tab.kids[t]].index(c)
            m = torch.movedim(self.T[c], lc, 2)
            q, r = torch.linalg.qr(m.reshape(-1, m.shape[2]))
            if schmidt:
                at = 0
                for _, d in tab.leg(c, lc):
                    col = slice(at, at + d)
                    u, sv, vh = torch.linalg.svd(r[col, col])
                    q[:, col], r[col, col] = q[:, col] @ u, sv[:, None] * vh
                    at += d
            else:
                sign = torch.where(torch.diagonal(r) < 0, -1.0, 1.0).to(r)
                q, r = q * sign, r * sign[:, None]
            self.T[c] = self.inside(c, torch.movedim(q.view(m.shape), 2, lc).contiguous())
            self.T[t] = self.inside(t, self.on(self.T[t], lt, r).contiguous())
            self.memo = {k: v for k, v in self.memo.items() if k[0] in ("site", "diag") or
                         (k[0] == "up" and not self._below(c, k[1]) and not self._below(t, k[1])) or
                         (k[0] == "down" and self._below(c, k[1]) and self._below(t, k[1]))}

    def _below(self, node, top):
        while node >= 0 and node != top:
            node = self.tab.parent[node]
        return node == top

    def lowest(self, node, x, steps=200):
        """Lowest eigenpair of H_eff by Lanczos with full reorthogonalisation."""
        v = [x / x.norm()]
        a, b = [], []
        for j in range(steps):
            w = self.inside(node, self.heff(node, v[j]))
            a.append(float((w * v[j]).sum()))
            basis = torch.stack(v).view(len(v), -1)
            for _ in range(2):
                w = w - (basis.T @ (basis @ w.reshape(-1))).view(w.shape)
            b.append(float(w.norm()))
            e, s = np.linalg.eigh(np.diag(a) + np.diag(b[:-1], 1) + np.diag(b[:-1], -1))
            if b[-1] * abs(s[-1, 0]) < 1e-13 * abs(e[0]) or b[-1] < 1e-13 or j == steps - 1:
                break
            v.append(w / b[-1])
        out = torch.tensordot(torch.from_numpy(s[:, 0]).cuda(), torch.stack(v[: len(a)]), dims=1)
        out = out / out.norm()
        return float(e[0]), out if float((out * v[0]).sum()) >= 0 else -out


def _exact_sweep(case, Q, start):
    tab = Tables(case, Q=Q)
    d = Dense(tab, start)
    at = len(tab.parent) - 1
    for node in tab.model.sweep_order():
        d.move(at, int(node))
        at = int(node)
        e, d.T[at] = d.lowest(at, d.T[at])
    psi = d.T[at] / d.T[at].norm()
    parts = [float((psi * d.heff(at, psi, cls)).sum()) for cls in range(5)]
    probs = np.zeros((int(np.prod(tab.shape)), D))
    for node, kid in enumerate(tab.kids):
        if kid[0][0] == 0:
            d.move(at, node)
            at = node
            p = d.T[at].square().sum(2)
            probs[kid[0][1]], probs[kid[1][1]] = p.sum(1).cpu().numpy(), p.sum(0).cpu().numpy()
    return {"eigenvalue": e, "total": sum(parts), "bare": sum(parts[:4]), "parts": dict(zip(qed.CLASSES, parts)),
            "probs": probs.reshape(-1)}


def exact(case, seed):
    torch.cuda.empty_cache()
    s = prepare(case, seed)
    if s.kind in ("sweep", "batch"):
        return [_exact_sweep(case, case["Q"] + 2 * i, start) for i, start in enumerate(s.start)]
    tab = _tables(case)
    d = Dense(tab, [s.ttn.node_export(n) for n in range(len(tab.parent))])
    if s.kind == "product":
        return d.packed(s.node, d.heff(s.node, d.view(s.node, s.x)))
    if s.kind == "gradient":
        x = d.view(s.node, s.x)
        hx = [d.heff(s.node, x, cls) for cls in range(5)]
        nrm = float((x * x).sum())
        part = [float((x * h).sum()) / nrm for h in hx]
        e = sum(part)
        c = tab.couplings
        return {"energy": e, "couplings": {n: p / c[n] for n, p in zip(qed.CLASSES, part)},
                "psi": d.packed(s.node, 2.0 * (sum(hx) - e * x) / nrm)}
    if s.kind == "move":
        out, at = [], s.node
        for n, x in zip((s.far, s.node), s.x):
            d.move(at, n)
            at = n
            out.append(d.packed(n, d.heff(n, d.view(n, x))))
        return out
    # the eigenvector itself is fixed by the solver's tolerance only
    return {"energy": d.lowest(s.node, d.view(s.node, torch.from_numpy(s.start).cuda()))[0], "tensor": None}
