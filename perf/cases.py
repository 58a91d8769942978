"""The measured cases: helicity- and colour-summed |M|^2 through the package's
public entry points (``mea.Process.evaluate``, ``evaluate_host``, ``mea.Server``).

A case names a process, the number of events, the precision and the entry
point.  Processes, sqrt(s) ranges and cuts are those of the package's
benchmark and tests; events come from its seeded generator (RAMBO, the jet
cuts).  A program keeps one process handle per subprocess for its whole life,
tuned once when it evaluates thousands of events, so handles are made (and
tuned) once per process here too; inputs and output buffers belong to the
state of one ``prepare``.
"""
import itertools
import math

import numpy as np
import torch

from paper_0909_5257_gb300 import mea

# name: (PDG codes, sqrt(s) range in GeV)
PROCESSES = {
    "gg_gg": ([21, 21, 21, 21], 200.0, 2000.0),
    "uux_gg": ([2, -2, 21, 21], 200.0, 2000.0),
    "gg_3g": ([21] * 5, 200.0, 2000.0),
    "uux_3g": ([2, -2, 21, 21, 21], 200.0, 2000.0),
    "uu_uug": ([2, 2, 2, 2, 21], 200.0, 2000.0),
    "gg_4g": ([21] * 6, 300.0, 3000.0),
    "uux_4g": ([2, -2, 21, 21, 21, 21], 300.0, 3000.0),
    "gg_5g": ([21] * 7, 500.0, 5000.0),
    "uux_5g": ([2, -2] + [21] * 5, 500.0, 5000.0),
    "uu_uu3g": ([2, 2, 2, 2, 21, 21, 21], 500.0, 5000.0),
}
ALPHA_S = 0.118
SEED = 0x09095257
TUNE_FROM = 4096  # a program with this many events per call tunes its handle once

# largest number of events of a drawn case, per process and precision
MOST = {
    "gg_gg": (1 << 20, 1 << 18), "uux_gg": (1 << 20, 1 << 18), "gg_3g": (1 << 20, 1 << 16),
    "uux_3g": (1 << 20, 1 << 17), "uu_uug": (1 << 20, 1 << 17), "gg_4g": (1 << 17, 1 << 12),
    "uux_4g": (300001, 1 << 14), "gg_5g": (9000, 128), "uux_5g": (20011, 1 << 10), "uu_uu3g": (1 << 15, 1 << 11),
}
# requests of one served case: the serving workload's processes and 40/40/20
# mix, sizes spread over its range's lower half, submitted at once
SERVED = [("gg_5g", 1024), ("uux_5g", 9001), ("uu_uu3g", 2048), ("uux_5g", 1500), ("gg_5g", 3333), ("uu_uu3g", 5000),
          ("uux_5g", 4096), ("gg_5g", 1200)]


def listed():
    def case(name, process, n, precision, call="evaluate"):
        return {"name": name, "process": process, "n": n, "precision": precision, "call": call}

    return [
        # 2 -> 2 in double precision, the smallest benchmark configuration: launch latency
        case("gg_gg_fp64", "gg_gg", 1 << 14, "fp64"),
        # an interactive call of a few hundred events, odd count: launches and host path
        case("uux_3g_small", "uux_3g", 777, "mixed"),
        # three jets at production size: the fused straight-line kernels
        case("gg_3g", "gg_3g", 1 << 20, "mixed"),
        # three jets in double precision, ragged count
        case("uu_uug_fp64", "uu_uug", 100003, "fp64"),
        # events that live on the host, page-locked: copies in and out included
        case("gg_3g_host", "gg_3g", 1 << 19, "mixed", "host"),
        # four jets, the tensor-core path at medium size
        case("gg_4g", "gg_4g", 1 << 17, "mixed"),
        # four jets with a quark line, ragged count, many chunks
        case("uux_4g", "uux_4g", 300001, "mixed"),
        # four jets in double precision: the reference values of a study
        case("gg_4g_fp64", "gg_4g", 1 << 12, "fp64"),
        # the heaviest subprocess: 7245 diagrams, 720 colours
        case("gg_5g", "gg_5g", 9000, "mixed"),
        # five jets with one quark line, ragged count
        case("uux_5g", "uux_5g", 20011, "mixed"),
        # five jets with two quark lines
        case("uu_uu3g", "uu_uu3g", 1 << 15, "mixed"),
        # a served mix of the three five-jet subprocesses: the whole request loop
        case("served_5jet", "mix", sum(n for _, n in SERVED), "mixed", "server"),
    ]


def draw(rng):
    """One more case: any process, either precision, either entry point, the
    event count log-uniform from 16 to the process's largest."""
    process = rng.choice(sorted(PROCESSES))
    precision = rng.choice(["mixed", "mixed", "fp64"])
    n = int(round(math.exp(rng.uniform(math.log(16.0), math.log(MOST[process][precision == "fp64"])))))
    call = "host" if rng.random() < 0.2 else "evaluate"
    return {"process": process, "n": n, "precision": precision, "call": call}


_handles = {}
_servers = {}


def _precision(case):
    return mea.PREC_FP64 if case["precision"] == "fp64" else mea.PREC_MIXED


def _momenta(process, n, seed, first=0):
    pdg, lo, hi = PROCESSES[process]
    mom = torch.empty((n, len(pdg), 4), dtype=torch.float64, device="cuda")
    mea.generate_phase_space(len(pdg) - 2, n, mom, first_event=first, seed=SEED + seed, rs_lo=lo, rs_hi=hi)
    return mom


def _handle(process, precision, mom):
    """The process handle a program keeps; tuned once where it evaluates many events per call."""
    tune = mom.shape[0] >= TUNE_FROM
    key = (process, precision if tune else None)
    if key not in _handles:
        P = mea.Process(PROCESSES[process][0], alpha_s=ALPHA_S, auto_tune=False)
        if tune:
            n = min(int(mom.shape[0]), 1 << 20)
            P.autotune(mom, torch.empty(n, dtype=torch.float64, device="cuda"), n_sample=n, precision=precision)
        _handles[key] = P
    return _handles[key]


def prepare(case, seed):
    prec = _precision(case)
    if case["call"] == "server":
        reqs, first = [], 0
        for process, n in SERVED:
            mom = _momenta(process, n, seed, first)
            first += n
            # one handle per process, tuned on a request of this size
            if ("served", process) not in _handles:
                P = mea.Process(PROCESSES[process][0], alpha_s=ALPHA_S, auto_tune=False)
                P.autotune(mom, torch.empty(n, dtype=torch.float64, device="cuda"), precision=prec)
                _handles[("served", process)] = P
            reqs.append((_handles[("served", process)], mom, torch.empty(n, dtype=torch.float64, device="cuda"),
                         torch.empty(n, dtype=torch.uint8, device="cuda")))
        if "mix" not in _servers:
            _servers["mix"] = mea.Server(mem_budget_bytes=100 << 30, n_slots=4)
        torch.cuda.synchronize()  # the server's streams read the inputs
        return {"call": "server", "server": _servers["mix"], "requests": reqs, "prec": prec}
    n = case["n"]
    mom = _momenta(case["process"], n, seed)
    P = _handle(case["process"], prec, mom)
    state = {"call": case["call"], "P": P, "prec": prec}
    if case["call"] == "host":
        state["mom"] = mom.cpu().pin_memory().numpy()
        state["me2"] = torch.empty(n, dtype=torch.float64).pin_memory().numpy()
        state["flags"] = torch.empty(n, dtype=torch.uint8).pin_memory().numpy()
    else:
        state["mom"] = mom
        state["me2"] = torch.empty(n, dtype=torch.float64, device="cuda")
        state["flags"] = torch.empty(n, dtype=torch.uint8, device="cuda")
    return state


def run(state):
    prec = state["prec"]
    if state["call"] == "server":
        srv = state["server"]
        ids = [srv.submit(P, mom, me2, flags=flags, precision=prec) for P, mom, me2, flags in state["requests"]]
        for i in ids:
            srv.wait(i, timeout_ms=120000)
        return [(me2, flags) for _, _, me2, flags in state["requests"]]
    if state["call"] == "host":
        return state["P"].evaluate_host(state["mom"], precision=prec, out=state["me2"], flags=state["flags"])
    state["P"].evaluate(state["mom"], state["me2"], precision=prec, flags=state["flags"])
    return state["me2"], state["flags"]


# ---------------------------------------------------------------- 64-bit values
# |M|^2 by colour-ordered off-shell recursion (Berends and Giele 1988) in
# double precision, plain torch: every current of an ordered word of legs is
# computed once per helicity pattern of those legs.  Word currents obey
#   P^2 J(w) = sum_{w=uv} [J(u), J(v)] + sum_{w=uvt} {J(u), J(v), J(t)},
#   [a, b] = ((2 Pb + Pa).a) b - ((2 Pa + Pb).b) a + (Pa - Pb) (a.b),
#   {a, b, c} = 2 (a.c) b - (a.b) c - (b.c) a,
# quark words  P^2 psi(w) = Pslash sum_{w=uv} Jslash(u) psi(v)  and barred ones
# with the order reversed and the opposite sign; all momenta flow one way.

G5 = torch.diag(torch.tensor([1.0, -1.0, -1.0, -1.0], dtype=torch.float64))


def _gammas(dev):
    s = np.array([[[1, 0], [0, 1]], [[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]]], dtype=complex)
    g = np.zeros((4, 4, 4), dtype=complex)
    for mu in range(4):
        g[mu, :2, 2:] = s[mu]
        g[mu, 2:, :2] = s[mu] if mu == 0 else -s[mu]
    return torch.tensor(g, device=dev)


def _vdot(a, b):
    return a[..., 0] * b[..., 0] - a[..., 1] * b[..., 1] - a[..., 2] * b[..., 2] - a[..., 3] * b[..., 3]


class _Ordered:
    """Word currents of one chunk of events; every tensor is [helicity patterns, E, 4]
    with the patterns in word order (first letter slowest, index 0 = helicity -1)."""

    def __init__(self, pdg, mom):
        self.dev = mom.device
        sign = torch.tensor([-1.0, -1.0] + [1.0] * (len(pdg) - 2), dtype=torch.float64, device=self.dev)
        self.k = mom * sign[None, :, None]  # all flowing out
        self.p = mom
        self.pdg, self.E = pdg, mom.shape[0]
        self.gam = _gammas(self.dev)
        metric = torch.tensor([1.0, -1.0, -1.0, -1.0], dtype=torch.complex128, device=self.dev)
        self.gam_low = self.gam * metric[:, None, None]
        self.J, self.F, self.B, self.extra = {}, {}, {}, {}

    def mom_of(self, w):
        legs = [l for x in w for l in (self.extra[x][0] if x in self.extra else (x,))]
        return self.k[:, legs, :].sum(1)

    def pol(self, l):
        p = self.p[:, l]
        kk = p[:, 1:].norm(dim=1)
        kt = p[:, 1:3].norm(dim=1)
        safe = torch.where(kt > 0, kt, torch.ones_like(kt))
        cp = torch.where(kt > 0, p[:, 1] / safe, torch.ones_like(kt))
        sp = torch.where(kt > 0, p[:, 2] / safe, torch.zeros_like(kt))
        ct, st = p[:, 3] / kk, kt / kk
        z = torch.zeros_like(ct)
        e1 = torch.stack([z, ct * cp, ct * sp, -st], 1).to(torch.complex128)
        e2 = torch.stack([z, -sp, cp, z], 1).to(torch.complex128)
        s = 1.0 if l >= 2 else -1.0  # outgoing: conjugated
        r = math.sqrt(0.5)
        return torch.stack([r * (e1 + s * 1j * e2), r * (-e1 + s * 1j * e2)], 0)

    def spinor(self, l, barred):
        """Column u / v or barred row of quark leg l for its two helicities: the
        massless solutions of pslash w = 0, |w|^2 = 2E, one per chirality."""
        p = self.p[:, l]
        kk = p[:, 1:].norm(dim=1)
        up = torch.where(p[:, 3] >= 0, kk + p[:, 3], (p[:, 1] ** 2 + p[:, 2] ** 2) / (kk - p[:, 3]))
        a = torch.sqrt(up).to(torch.complex128)
        safe = torch.where(up > 0, torch.sqrt(up), torch.ones_like(up))
        b = torch.where(up > 0, torch.complex(p[:, 1], p[:, 2]) / safe, torch.sqrt(2 * kk).to(torch.complex128))
        z = torch.zeros_like(a)
        right = torch.stack([z, z, a, b], 1)
        left = torch.stack([-b.conj(), a, z, z], 1)
        w = torch.stack([left, right], 0)
        if barred:
            w = torch.einsum("hei,ij->hej", w.conj(), self.gam[0])
        return w

    def gluon(self, w):
        """J(w): [2^|w|, E, 4]."""
        if w in self.J:
            return self.J[w]
        if len(w) == 1:
            x = w[0]
            r = self.extra[x][1] if x in self.extra else self.pol(x)
        else:
            kk = self.mom_of(w)
            r = self.gluon_sum(w) / _vdot(kk, kk)[None, :, None]
        self.J[w] = r
        return r

    def gluon_sum(self, w):
        tot = 0
        for i in range(1, len(w)):
            a, b = self.gluon(w[:i])[:, None], self.gluon(w[i:])[None, :]
            pa, pb = self.mom_of(w[:i]), self.mom_of(w[i:])
            tot = tot + (_vdot(2 * pb + pa, a)[..., None] * b - _vdot(2 * pa + pb, b)[..., None] * a
                         + (pa - pb) * _vdot(a, b)[..., None]).flatten(0, 1)
        for i in range(1, len(w) - 1):
            for j in range(i + 1, len(w)):
                a = self.gluon(w[:i])[:, None, None]
                b = self.gluon(w[i:j])[None, :, None]
                c = self.gluon(w[j:])[None, None, :]
                tot = tot + (2 * _vdot(a, c)[..., None] * b - _vdot(a, b)[..., None] * c
                             - _vdot(b, c)[..., None] * a).flatten(0, 2)
        return tot

    def slash(self, v):
        return torch.einsum("...m,mij->...ij", v.to(torch.complex128), self.gam_low)

    def psi_sum(self, q, w):
        tot = 0
        for i in range(1, len(w) + 1):
            tot = tot + torch.einsum("aeij,bej->abei", self.slash(self.gluon(w[:i])), self.psi(q, w[i:])).flatten(0, 1)
        return tot

    def psi(self, q, w):
        """Quark word: [2^|w| (gluons) * 2 (quark), E, 4], the quark's helicity last."""
        if (q, w) not in self.F:
            if not w:
                r = self.spinor(q, False)
            else:
                kk = self.k[:, q] + self.mom_of(w)
                r = torch.einsum("eij,hej->hei", self.slash(kk), self.psi_sum(q, w)) / _vdot(kk, kk)[None, :, None]
            self.F[(q, w)] = r
        return self.F[(q, w)]

    def bar(self, q, w):
        """Barred quark word: [2 (quark) * 2^|w| (gluons), E, 4], the quark's helicity first."""
        if (q, w) not in self.B:
            if not w:
                r = self.spinor(q, True)
            else:
                kk = self.k[:, q] + self.mom_of(w)
                tot = 0
                for i in range(len(w)):
                    tot = tot - torch.einsum("aei,beij->abej", self.bar(q, w[:i]), self.slash(self.gluon(w[i:]))).flatten(0, 1)
                r = torch.einsum("hei,eij->hej", tot, self.slash(kk)) / _vdot(kk, kk)[None, :, None]
            self.B[(q, w)] = r
        return self.B[(q, w)]

    def pair_current(self, qbar, t, u, q):
        """Gluon current of a quark line's ordered word t x u at the exchanged
        gluon x: [2 * 2^|t| * 2^|u| * 2, E, 4] (patterns qbar, t, u, q)."""
        c = torch.einsum("aei,mij,bej->abem", self.bar(qbar, t), self.gam, self.psi(q, u)).flatten(0, 1)
        kk = self.mom_of(t + u) + self.k[:, qbar] + self.k[:, q]
        return c / _vdot(kk, kk)[None, :, None]


def _su3():
    lam = np.zeros((8, 3, 3), dtype=complex)
    lam[0][0, 1] = lam[0][1, 0] = 1
    lam[1][0, 1], lam[1][1, 0] = -1j, 1j
    lam[2][0, 0], lam[2][1, 1] = 1, -1
    lam[3][0, 2] = lam[3][2, 0] = 1
    lam[4][0, 2], lam[4][2, 0] = -1j, 1j
    lam[5][1, 2] = lam[5][2, 1] = 1
    lam[6][1, 2], lam[6][2, 1] = -1j, 1j
    lam[7] = np.diag([1, 1, -2]) / math.sqrt(3)
    return lam / 2


_colour = {}


def _gluon_colour(n):
    """C[s, s'] of the adjoint chains (F^{s1} ... F^{s(n-2)})_{0,n-1} over the permutations s."""
    if ("g", n) not in _colour:
        T = _su3()
        F = np.real(-2j * np.einsum("aij,bjk,cki->abc", T, T, T) + 2j * np.einsum("bij,ajk,cki->abc", T, T, T))
        chain = F  # [x, a1, y]
        for _ in range(n - 3):
            chain = np.tensordot(chain, F, axes=([-1], [0]))
        perms = list(itertools.permutations(range(n - 2)))
        where = {s: i for i, s in enumerate(perms)}
        base = []
        for s in perms:  # <identity | s>
            base.append(float(np.vdot(chain, np.transpose(chain, [0] + [1 + x for x in s] + [n - 1]))))
        C = np.empty((len(perms),) * 2)
        # <s|t> depends on t relative to s: position x of t holds letter t[x] = s[y], y its place in s
        for i, s in enumerate(perms):
            inv = np.argsort(s)
            for j, t in enumerate(perms):
                C[i, j] = base[where[tuple(int(inv[t[x]]) for x in range(n - 2))]]
        _colour[("g", n)] = (perms, C)
    return _colour[("g", n)]


def _line_colour(ng):
    """Strings (T^{s1} ... T^{sn})_{ij} over the permutations of the gluons."""
    if ("q", ng) not in _colour:
        T = _su3()
        perms = list(itertools.permutations(range(ng)))
        V = np.eye(3, dtype=complex)
        for _ in range(ng):
            V = np.tensordot(V, T, axes=([-1], [1]))  # [i, a1, .., an, j]
        flat = np.stack([np.transpose(V, [0] + [1 + int(x) for x in np.argsort(s)] + [ng + 1]).reshape(-1) for s in perms])
        _colour[("q", ng)] = (perms, np.real(flat.conj() @ flat.T))
    return _colour[("q", ng)]


def _two_line_basis(ng):
    """(pairing, word on line A with the exchanged gluon 'x', word before and
    after x on line B) and the colour matrix of those products of strings."""
    if ("qq", ng) not in _colour:
        T = _su3()
        basis, vecs = [], []
        for pairing in range(2):
            for r in range(ng + 1):
                for S in itertools.combinations(range(ng), r):
                    rest = [g for g in range(ng) if g not in S]
                    for wa in itertools.permutations(list(S) + ["x"]):
                        for wb in itertools.permutations(rest + ["x"]):
                            basis.append((pairing, wa, wb))
        for pairing, wa, wb in basis:
            def string(w):
                t, names = np.eye(3, dtype=complex), []
                for a in w:
                    t = np.tensordot(t, T, axes=([-1], [1]))
                    names.append(a)
                return t, names

            ta, na = string(wa)
            tb, nb = string(wb)
            t = np.tensordot(ta, tb, axes=([1 + na.index("x")], [1 + nb.index("x")]))
            na2 = [a for a in na if a != "x"]
            nb2 = [a for a in nb if a != "x"]
            # axes now: i, na2.., j, k, nb2.., l
            names = ["i"] + na2 + ["j", "k"] + nb2 + ["l"]
            order = (["i", "j", "k", "l"] if pairing == 0 else ["k", "j", "i", "l"]) + list(range(ng))
            vecs.append(np.transpose(t, [names.index(x) for x in order]).reshape(-1))
        V = np.stack(vecs)
        _colour[("qq", ng)] = (basis, np.real(V.conj() @ V.T))
    return _colour[("qq", ng)]


def _to_legs(amp, letters, n, E):
    """[2^n, E] with the patterns of `letters` -> leg order."""
    return amp.reshape([2] * n + [E]).permute([letters.index(l) for l in range(n)] + [n]).reshape(-1)


def _me2(process, mom):
    pdg = PROCESSES[process][0]
    n, E = len(pdg), mom.shape[0]
    W = _Ordered(pdg, mom)
    rows, ng = [], sum(c == 21 for c in pdg)
    if ng == n:
        perms, C = _gluon_colour(n)
        last = W.gluon((n - 1,))
        for s in perms:
            w = (0,) + tuple(1 + x for x in s)
            a = _vdot(W.gluon_sum(w)[:, None], last[None, :]).flatten(0, 1)
            rows.append(_to_legs(a, list(w) + [n - 1], n, E))
        colours = 64.0
    elif n - ng == 2:
        perms, C = _line_colour(ng)
        # u u~ -> n g: leg 0 the incoming quark (column), leg 1 the incoming antiquark (row)
        row = W.spinor(1, True)
        for s in perms:
            w = tuple(2 + x for x in s)
            a = torch.einsum("aei,bei->abe", row, W.psi_sum(0, w)).flatten(0, 1)
            rows.append(_to_legs(a, [1] + list(w) + [0], n, E))
        colours = 9.0
    else:
        # u u -> u u + n g: lines (2 <- 0), (3 <- 1) and, with the Fermi sign, (3 <- 0), (2 <- 1)
        basis, C = _two_line_basis(ng)
        for pairing, wa, wb in basis:
            oa, ob = (2, 3) if pairing == 0 else (3, 2)
            i = wb.index("x")
            t, u = tuple(4 + g for g in wb[:i]), tuple(4 + g for g in wb[i + 1:])
            x = ("x", ob, t, u)
            if x not in W.extra:
                W.extra[x] = ((ob,) + t + u + (1,), W.pair_current(ob, t, u, 1))
            w = tuple(x if g == "x" else 4 + g for g in wa)
            a = torch.einsum("aei,bei->abe", W.spinor(oa, True), W.psi_sum(0, w)).flatten(0, 1)
            letters = [oa] + [l for g in w for l in (W.extra[g][0] if g in W.extra else (g,))] + [0]
            a = _to_legs(a, letters, n, E)
            rows.append(a if pairing == 0 else -a)
        colours = 9.0
    A = torch.stack(rows)
    C = torch.tensor(C, dtype=torch.complex128, device=mom.device)
    tot = (A.conj() * (C @ A)).real.sum(0).reshape(-1, E).sum(0)
    g2 = 4.0 * math.pi * ALPHA_S
    return tot * g2 ** (n - 2) / (4.0 * colours)


# events per chunk: bounds the working set of the word tensors to a few GB
CHUNK = {4: 1 << 17, 5: 1 << 16, 6: 1 << 13, 7: 1 << 11}


def _exact_me2(process, mom):
    c = CHUNK[mom.shape[1]]
    return torch.cat([_me2(process, mom[i:i + c]) for i in range(0, mom.shape[0], c)])


def exact(case, seed):
    if case["call"] == "server":
        out, first = [], 0
        for process, n in SERVED:
            out.append((_exact_me2(process, _momenta(process, n, seed, first)), None))
            first += n
        return out
    me2 = _exact_me2(case["process"], _momenta(case["process"], case["n"], seed))
    return (me2.cpu().numpy() if case["call"] == "host" else me2), None


# ---------------------------------------------------------------------- work
# Non-vanishing helicity combinations and FLOPs per event of the ordered
# recursion above with every word current once per helicity pattern of its
# legs (three-vertex 150, four-vertex 100, quark vertex 60, quark propagator 50,
# closing contraction 30 FLOPs) and of the colour sum over independent ordered
# amplitudes (4 m^2 / 2 per combination).

def _words(n, k):
    return math.perm(n, k)


def _gluon_words_flops(n, k_max, fixed):
    """Words of up to k_max of n letters (reversed ones are equal up to a sign)
    plus, with `fixed`, those ending in one more fixed letter."""
    f = 0.0
    for k in range(2, k_max + 1):
        w = _words(n, k) / 2 + (_words(n, k - 1) if fixed else 0)
        f += w * 2 ** k * ((k - 1) * 150 + math.comb(k - 1, 2) * 100)
    return f


def _flops_per_event(process):
    pdg = PROCESSES[process][0]
    n = len(pdg)
    ng = sum(c == 21 for c in pdg)
    if ng == n:
        H, m = 2 ** n - 2 * (n + 1), math.factorial(n - 2)
        f = _gluon_words_flops(n - 2, n - 2, True) + m * H * 30 * (n - 2 + math.comb(n - 2, 2))
    elif n - ng == 2:
        H, m = 2 ** (ng + 1) - 4, math.factorial(ng)
        f = _gluon_words_flops(ng, ng, False)
        for k in range(1, ng):
            f += _words(ng, k) * 2 ** (k + 1) * (60 * k + 50)
        f += m * H * 60 * ng / 2
    else:
        H, m = 6 * 2 ** ng, 2 * math.factorial(ng + 1)
        f = 2 * (_gluon_words_flops(ng + 1, ng + 1, False) + m * H * 60 * (ng + 1) / 2)
    return f + H * 2.0 * m * m


def work(case):
    if case["call"] == "server":
        parts = SERVED
    else:
        parts = [(case["process"], case["n"])]
    nbytes = sum(n * (32 * len(PROCESSES[p][0]) + 9) for p, n in parts)
    return {"bytes": float(nbytes), "flops": float(sum(n * _flops_per_event(p) for p, n in parts))}
