"""Cases by which the speed of this library is measured.

Each case is one call (or one whole solve) through the public Python binding,
at sizes of this repository's workloads (``synthetic.CONFIGS``, the batched
workload's ranges nocc 10..40, nvir 50..250, naux = 6 nvir) or a little below,
odd ones among them. Inputs follow the recipe of ``synthetic``: circular complex Gaussian
Cholesky vectors with Hermitian B[Q], uniform orbital energies, unit trial
vectors; here they are drawn on the GPU, from the seed alone.

``exact`` states the IP and EA equations of ADC(2)+x(3) and those of EE-ADC(2)
once more in plain 64-bit torch (dense integrals, no packing), and takes the
gradients from torch's autograd.
"""
import math

import numpy as np
import torch

import paper_2511_21640_gb300 as adc

SIGMA = 0.05  # standard deviation of the elements of B (the workloads' value)


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest workload (IP-ADC(3), o=8, v=24, Q=96): one product of four vectors, bound by latency
        {"name": "ip_small_sigma", "op": "sigma", "kind": "IP", "order": 3, "x": 1.0, "nocc": 8, "nvir": 24,
         "naux": 96, "k": 4, "precision": "fp64"},
        # the same workload solved whole: four roots, FP64, residual 1e-8
        {"name": "ip_small_solve", "op": "solve", "kind": "IP", "order": 3, "x": 1.0, "nocc": 8, "nvir": 24,
         "naux": 96, "k": 4, "precision": "fp64"},
        # FP64 products of a block of trial vectors, IP, odd sizes of the batched workload's range
        {"name": "ip_sigma_fp64", "op": "sigma", "kind": "IP", "order": 3, "x": 0.5, "nocc": 33, "nvir": 147,
         "naux": 882, "k": 6, "precision": "fp64"},
        # FP64 products, EA-ADC(2)+x(3): the plain FP64 Davidson's step, and every FP64 residual check
        {"name": "ea_sigma_fp64", "op": "sigma", "kind": "EA", "order": 3, "x": 0.5, "nocc": 30, "nvir": 150,
         "naux": 900, "k": 8, "precision": "fp64"},
        # the refinement products of the mixed Davidson (FP64-accurate, sliced), EA, odd sizes
        {"name": "ea_sigma_sliced", "op": "sigma", "kind": "EA", "order": 3, "x": 0.5, "nocc": 31, "nvir": 163,
         "naux": 978, "k": 8, "precision": "sliced"},
        # the headline workload's product: one block of 8 vectors in the mixed Davidson's BF16x3 split
        {"name": "ea_sigma_bf16x3", "op": "sigma", "kind": "EA", "order": 3, "x": 0.5, "nocc": 40, "nvir": 200,
         "naux": 1200, "k": 8, "precision": "bf16x3"},
        # ADC(2): the coupling block alone, a product bound by reading it; the SS-FNS procedure's canonical solve
        {"name": "ea_adc2_sigma_fp64", "op": "sigma", "kind": "EA", "order": 2, "x": 0.0, "nocc": 25, "nvir": 180,
         "naux": 1080, "k": 6, "precision": "fp64"},
        # excitations at second order, FP64
        {"name": "ee_adc2_sigma_fp64", "op": "sigma", "kind": "EE", "order": 2, "x": 0.0, "nocc": 17, "nvir": 85,
         "naux": 510, "k": 4, "precision": "fp64"},
        # excitations with the scaled third order, the mixed Davidson's product (o=12, v=60, Q=360 workload)
        {"name": "ee_sigma_bf16x3", "op": "sigma", "kind": "EE", "order": 3, "x": 0.4, "nocc": 12, "nvir": 60,
         "naux": 360, "k": 4, "precision": "bf16x3"},
        # what a user pays for each new problem: amplitudes, operators and the diagonal from the Cholesky vectors
        {"name": "ea_setup", "op": "setup", "kind": "EA", "order": 3, "x": 0.5, "nocc": 18, "nvir": 90,
         "naux": 540, "k": 0, "precision": "fp64"},
        # the backward pass of two roots: gradients with respect to B, the orbital energies and x
        {"name": "ea_gradient", "op": "gradient", "kind": "EA", "order": 3, "x": 0.4, "nocc": 10, "nvir": 50,
         "naux": 300, "k": 2, "precision": "fp64"},
        # six IP and EA problems of the batched workload's smaller sizes in one grouped launch
        {"name": "batch_sigma_bf16x3", "op": "batch", "kind": "IPEA", "order": 3, "x": 0.5, "nocc": 22, "nvir": 100,
         "naux": 600, "k": 6, "precision": "bf16x3"},
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    op = rng.choice(["sigma"] * 7 + ["solve", "setup", "gradient", "batch"])
    if op == "sigma":
        kind = rng.choice(["IP", "EA", "EA", "EE"])
        if kind == "EE":
            order = rng.choice([2, 3])
            nocc = log_int(4, 17 if order == 2 else 12)
            nvir = 5 * nocc + rng.randint(-3, 3)
            precision = rng.choice(["fp64", "bf16x3", "sliced"])
            k = rng.randint(1, 6)
        else:
            order = rng.choice([2, 3, 3, 3])
            nocc, nvir = log_int(8, 33), log_int(24, 150)
            precision = rng.choice(["fp64", "fp64", "bf16x3", "sliced"])
            k = rng.randint(1, 12)
    elif op == "solve":
        kind, order, precision, k = rng.choice(["IP", "EA"]), 3, "fp64", 4
        nocc, nvir = rng.randint(5, 9), rng.randint(16, 28)
    elif op == "setup":
        kind, order, precision, k = rng.choice(["IP", "EA"]), rng.choice([2, 3]), "fp64", 0
        nocc, nvir = log_int(8, 24), log_int(24, 90)
    elif op == "gradient":
        kind, order, precision, k = rng.choice(["IP", "EA"]), 3, "fp64", rng.randint(1, 4)
        nocc, nvir = log_int(5, 12), log_int(16, 50)
    else:
        kind, order, precision, k = "IPEA", 3, "bf16x3", rng.randint(2, 8)
        nocc, nvir = rng.randint(10, 24), rng.randint(50, 100)
    x = 0.0 if order == 2 else rng.choice([0.4, 0.5, 1.0])
    return {"op": op, "kind": kind, "order": order, "x": x, "nocc": nocc, "nvir": nvir, "naux": 6 * nvir,
            "k": k, "precision": precision}


# ------------------------------------------------------------------ inputs
def _members(case):
    """The problems of a batch: sizes around the case's, IP and EA in turn."""
    o, v = case["nocc"], case["nvir"]
    sizes = [(o, v), (o - 3, v - 11), (o - 9, v // 2 + 1), (o + 2, v - 30), (o - 6, v + 9), (o - 1, v // 2 + 17)]
    return [dict(case, op="sigma", kind="IP" if i % 2 == 0 else "EA", nocc=p, nvir=q, naux=6 * q)
            for i, (p, q) in enumerate(sizes)]


def _dims(case):
    o, v = case["nocc"], case["nvir"]
    po, pv = o * (o - 1) // 2, v * (v - 1) // 2
    return {"IP": (o, po * v), "EA": (v, o * pv), "EE": (o * v, po * pv)}[case["kind"]]


def _problem(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    o, v, q = case["nocc"], case["nvir"], case["naux"]
    n = o + v
    eo = torch.sort(torch.rand(o, generator=g, device="cuda", dtype=torch.float64) * 2.7 - 3.0).values
    ev = torch.sort(torch.rand(v, generator=g, device="cuda", dtype=torch.float64) * 4.9 + 0.1).values
    B = torch.view_as_complex(torch.randn(q, n, n, 2, generator=g, device="cuda", dtype=torch.float64))
    B = (B + B.mH) * (SIGMA / 2.0)  # Hermitian, variance SIGMA^2 off the diagonal
    return B.contiguous(), eo, ev


def _vectors(case, seed):
    """Unit trial vectors as a Davidson run has them: spread-out ones, and ones led by few configurations."""
    n1, n2 = _dims(case)
    k, n = case["k"], n1 + n2
    g = torch.Generator(device="cuda").manual_seed(seed + 7919)
    X = torch.view_as_complex(torch.randn(k, n, 2, generator=g, device="cuda", dtype=torch.float64))
    lead = torch.randint(0, n, (k, 8), generator=g, device="cuda")
    for r in range(1, k, 2):
        X[r, lead[r]] *= 0.1 * math.sqrt(n)
        X[r, r % n1] += math.sqrt(n)
    return X / torch.linalg.vector_norm(X, dim=1, keepdim=True)


def _context(case, B, eo, ev):
    # the operators of the larger problems are built as the benchmark's end-to-end runs build them
    setup = "sliced" if case["op"] in ("sigma", "batch") and case["nvir"] >= 64 else "fp64"
    return adc.Context(B, eo, ev, kind=case["kind"], order=case["order"], x=case["x"], setup=setup)


def prepare(case, seed):
    if case["op"] == "batch":
        members = _members(case)
        ctxs = [_context(m, *_problem(m, seed + 101 * i)) for i, m in enumerate(members)]
        return {"case": case, "ctxs": ctxs, "batch": adc.Batch(ctxs),
                "X": [_vectors(m, seed + 101 * i) for i, m in enumerate(members)]}
    B, eo, ev = _problem(case, seed)
    if case["op"] == "setup":
        return {"case": case, "B": B, "eo": eo, "ev": ev}
    state = {"case": case, "ctx": _context(case, B, eo, ev)}
    if case["op"] in ("sigma", "gradient"):
        state["X"] = _vectors(case, seed)
    return state


def run(state):
    case = state["case"]
    if case["op"] == "sigma":
        return state["ctx"].sigma(state["X"], case["precision"])
    if case["op"] == "solve":
        omega, _, _, _, _ = state["ctx"].davidson(case["k"], tol=1e-8, precision=case["precision"],
                                                  want_vectors=False)
        return omega
    if case["op"] == "setup":
        with _context(case, state["B"], state["eo"], state["ev"]) as ctx:
            return {"main": ctx.main_block(), "diagonal": ctx.diagonal()}
    if case["op"] == "gradient":
        gB, geo, gev, gx = state["ctx"].sigma_adjoint(state["X"], _weights(case))
        return {"B": gB, "eps_occ": geo, "eps_vir": gev, "x": gx}
    return state["batch"].sigma(state["X"], case["precision"])


def _weights(case):
    return np.array([1.0 - 0.4 * r for r in range(case["k"])])


# ------------------------------------------------------------------ bytes and operations
def _sigma_work(case):
    """One product: operators and vectors read once, the products written once; 8 flops per complex multiply-add."""
    o, v, k = case["nocc"], case["nvir"], case["k"]
    n1, n2 = _dims(case)
    po, pv = o * (o - 1) // 2, v * (v - 1) // 2
    third = case["order"] == 3 and case["x"] != 0.0
    if case["kind"] == "EE":
        ops = n1 * n1 + o * pv * v + o * po * v
        macs = n1 * n1 + 4 * n2 * (o + v)
        if third:
            ops += pv * pv + po * po + n1 * n1 + o * v * (o * o + v * v)
            macs += n2 * (pv + po) + n1 * n1 * n1 + 2 * n1 * (o * o + v * v) + 4 * n2 * (o + v)
    else:
        ops = n1 * n1 + n1 * n2
        macs = n1 * n1 + 2 * n1 * n2
        if third:
            pairs = po if case["kind"] == "IP" else pv
            ops += pairs * pairs + (o * v) ** 2
            macs += n2 * pairs + (o * v) ** 2 * (o if case["kind"] == "IP" else v)
    return {"bytes": 16.0 * (ops + 2 * k * (n1 + n2)), "flops": 8.0 * k * macs}


def _setup_work(case):
    """Integrals from B, amplitudes, main block and coupling (leading terms)."""
    o, v, q = case["nocc"], case["nvir"], case["naux"]
    n1, n2 = _dims(case)
    po, pv = o * (o - 1) // 2, v * (v - 1) // 2
    macs = 2 * q * (o * v) ** 2 + (q * o * v ** 3 if case["kind"] == "EA" else q * o ** 3 * v)
    if case["order"] == 3:
        macs += q * v ** 4 // 2 + po * pv * pv + (o * v) ** 3 + q * o * o * v * v
        macs += 2 * o * o * v ** 4 if case["kind"] == "EA" else q * o * v ** 3 + o ** 3 * v ** 3
    ops = n1 * n1 + (pv * pv if case["order"] == 3 and case["kind"] == "EA" else 0)
    return {"bytes": 16.0 * (q * (o + v) ** 2 + n1 * n2 + ops), "flops": 8.0 * macs}


def work(case):
    if case["op"] == "sigma":
        return _sigma_work(case)
    if case["op"] == "batch":
        each = [_sigma_work(m) for m in _members(case)]
        return {"bytes": sum(w["bytes"] for w in each), "flops": sum(w["flops"] for w in each)}
    if case["op"] == "solve":  # about eight expansions of the subspace from its 2 k starting vectors
        one = _sigma_work(dict(case, k=2 * case["k"]))
        return {"bytes": 8.0 * one["bytes"], "flops": 5.0 * one["flops"]}
    one = _setup_work(case)
    if case["op"] == "gradient":  # the setup's contractions again, and two for each in the backward pass
        return {"bytes": 2.0 * one["bytes"], "flops": 3.0 * one["flops"]}
    return one


# ------------------------------------------------------------------ 64-bit values
def _ein(spec, *ops):
    return torch.einsum(spec, *ops)


class _Plain:
    """Integrals, amplitudes and densities of one problem, dense, as the ISR equations name them."""

    def __init__(self, B, eo, ev, third):
        o = self.o = eo.shape[0]
        self.B, self.eo, self.ev = B, eo, ev
        self.D = eo[:, None, None, None] + eo[None, :, None, None] - ev[:, None] - ev[None, :]
        self.t = self.eri("vvoo").permute(2, 3, 0, 1) / self.D
        t, tc = self.t, self.t.conj()
        self.g = 0.5 * _ein("ijdf,ijef->de", tc, t)
        self.h = 0.5 * _ein("njef,mjef->nm", tc, t)
        if not third:
            return
        self.s2 = (0.5 * _ein("ajcd,ijcd->ia", self.eri("vovv"), t)
                   - 0.5 * _ein("jkic,jkac->ia", self.eri("ooov"), t)) / (eo[:, None] - ev[None, :])
        ring = _ein("kbcj,ikac->ijab", self.eri("ovvo"), t)
        ring = ring - ring.transpose(0, 1)
        ring = ring - ring.transpose(2, 3)
        self.lad = self.ladder(t.reshape(o * o, *t.shape[2:])).reshape(t.shape)
        self.t2 = (self.lad + 0.5 * _ein("klij,klab->ijab", self.eri("oooo"), t) + ring) / self.D

    def eri(self, spec):
        o = self.o
        p, q, r, s = (slice(0, o) if c == "o" else slice(o, None) for c in spec)
        B = self.B
        return _ein("Qpr,Qqs->pqrs", B[:, p, r], B[:, q, s]) - _ein("Qps,Qqr->pqrs", B[:, p, s], B[:, q, r])

    def ladder(self, T):
        """1/2 sum_cd <ab||cd> T_cd for antisymmetric T [n][c][d], over the pairs c < d, in slabs of a."""
        v = self.ev.shape[0]
        c, d = torch.triu_indices(v, v, 1, device=T.device)
        Bv = self.B[:, self.o:, self.o:]
        Tp = T[:, c, d]
        step = max(1, int(5e8 / v ** 3))
        out = []
        for a in range(0, v, step):
            J = _ein("Qac,Qbd->abcd", Bv[:, a:a + step], Bv)
            out.append(_ein("abp,np->nab", J[:, :, c, d] - J[:, :, d, c], Tp))
        return torch.cat(out, 1)

    def main_block(self, kind, x):
        t, tc, eo, ev, g, h = self.t, self.t.conj(), self.eo, self.ev, self.g, self.h
        oovv = self.eri("oovv")
        if kind == "EA":
            M = -0.5 * _ein("klac,klbc->ab", t, oovv) + 0.5 * (ev[:, None] - ev[None, :]) * g.T
            M = M + torch.diag(ev)
            if x is None:
                return M
            t2, s2, Bv, o = self.t2, self.s2, self.B, self.o
            R = _ein("njcf,mjaf->canm", tc, t)
            g3 = 0.5 * (_ein("ijdf,ijef->de", tc, t2) + _ein("ijdf,ijef->de", t2.conj(), t))
            ovvo = self.eri("ovvo")
            vv = Bv[:, o:, o:]
            coul = _ein("Qab,Q->ab", vv, _ein("Qde,de->Q", vv, g))
            exch = _ein("Qae,Qeb->ab", vv, _ein("Qdb,de->Qeb", vv, g))
            Y = (-0.5 * _ein("klac,klbc->ab", t2, oovv) - _ein("mabd,md->ab", self.eri("ovvv"), s2)
                 + _ein("adbk,kd->ab", self.eri("vvvo"), s2.conj()) + coul - exch
                 + 0.5 * _ein("ijbe,ijea->ab", self.lad.conj(), t)
                 + _ein("mabn,nm->ab", ovvo, h) - _ein("mcbn,canm->ab", ovvo, R))
            return M + x * (Y + 0.5 * (ev[:, None] - ev[None, :]) * g3.T)
        M = 0.5 * _ein("kjcd,ikcd->ij", oovv, t) - 0.5 * (eo[:, None] - eo[None, :]) * h.T - torch.diag(eo)
        if x is None:
            return M
        t2, s2 = self.t2, self.s2
        h3 = 0.5 * (_ein("jkcd,ikcd->ji", tc, t2) + _ein("jkcd,ikcd->ji", t2.conj(), t))
        oooo, vovo = self.eri("oooo"), self.eri("vovo")
        Y = (0.5 * _ein("kjcd,ikcd->ij", oovv, t2) - _ein("kjei,ke->ij", self.eri("oovo"), s2)
             + _ein("cjik,kc->ij", self.eri("vooo"), s2.conj()) + _ein("kjli,lk->ij", oooo, h)
             + 0.25 * _ein("kjlm,lmik->ij", oooo, _ein("lmef,ikef->lmik", tc, t)) - _ein("cjdi,cd->ij", vovo, g)
             + _ein("cjdk,kicd->ij", vovo, _ein("klcf,ildf->kicd", tc, t)))
        return M + x * (Y - 0.5 * (eo[:, None] - eo[None, :]) * h3.T)

    def sigma(self, kind, x, X):
        """M X (x None: ADC(2)) with the satellites as full antisymmetric arrays."""
        eo, ev, o, v, k = self.eo, self.ev, self.o, self.ev.shape[0], X.shape[0]
        tc = self.t.conj()
        if kind == "EE":
            return self.sigma_ee(X)
        n = v if kind == "EA" else o
        p, q = torch.triu_indices(n, n, 1, device=X.device)
        X1, X2 = X[:, :n], X[:, n:]
        S1 = X1 @ self.main_block(kind, x).T
        if kind == "EA":
            F = X.new_zeros(k, o, v, v)
            F[:, :, p, q] = X2.reshape(k, o, -1)
            F = F - F.transpose(2, 3)
            C = self.eri("vovv")
            if x is not None:
                U = _ein("cgem,kmgd->ckde", self.eri("vvvo"), tc)
                C = C + x * (0.5 * _ein("ckmn,mnde->ckde", self.eri("vooo"), tc) + U - U.transpose(2, 3))
            S2 = _ein("ckde,nc->nkde", C.conj(), X1) + (ev[:, None] + ev[None, :] - eo[:, None, None]) * F
            S1 = S1 + 0.5 * _ein("ckde,nkde->nc", C, F)
            if x is not None:
                ring = _ein("dlfk,nlfe->nkde", self.eri("vovo"), F)
                S2 = S2 + x * (self.ladder(F.reshape(k * o, v, v)).reshape(F.shape) - ring + ring.transpose(2, 3))
            return torch.cat([S1, S2[:, :, p, q].reshape(k, -1)], 1)
        F = X.new_zeros(k, o, o, v)
        F[:, p, q] = X2.reshape(k, -1, v)
        F = F - F.transpose(1, 2)
        C = self.eri("oovo").permute(3, 1, 0, 2)
        if x is not None:
            U = _ein("fimk,jmfa->kija", self.eri("vooo"), tc)
            C = C + x * (0.5 * _ein("efak,jief->kija", self.eri("vvvo"), tc) - U + U.transpose(1, 2))
        S2 = _ein("kija,nk->nija", C.conj(), X1) + (ev - eo[:, None, None] - eo[None, :, None]) * F
        S1 = S1 + 0.5 * _ein("kija,nija->nk", C, F)
        if x is not None:
            ring = _ein("akbj,nkib->nija", self.eri("vovo"), F)
            S2 = S2 + x * (0.5 * _ein("klij,nkla->nija", self.eri("oooo"), F) + ring - ring.transpose(1, 2))
        return torch.cat([S1, S2[:, p, q].reshape(k, -1)], 1)

    def sigma_ee(self, X):
        """EE-ADC(2)."""
        eo, ev, t, o, v, k = self.eo, self.ev, self.t, self.o, self.ev.shape[0], X.shape[0]
        p, q = torch.triu_indices(o, o, 1, device=X.device)
        r, s = torch.triu_indices(v, v, 1, device=X.device)
        X1 = X[:, :o * v].reshape(k, o, v)
        F = X.new_zeros(k, o, o, v, v)
        F[:, p[:, None], q[:, None], r, s] = X[:, o * v:].reshape(k, p.numel(), -1)
        F = F - F.transpose(1, 2)
        F = F - F.transpose(3, 4)
        io, iv = torch.eye(o, device=X.device), torch.eye(v, device=X.device)
        oovv, tc = self.eri("oovv"), t.conj()
        dS = ev[None, :] - eo[:, None]
        over = (_ein("iMaA,jMbA->iajb", t, tc) - _ein("ba,ij->iajb", self.g, io)
                - _ein("ji,ab->iajb", self.h, iv))
        M = (0.5 * (dS[None, None] - dS[:, :, None, None]) * over - self.eri("vovo").permute(3, 0, 1, 2)
             + _ein("iMaA,jMbA->iajb", t, oovv) - 0.5 * _ein("MNaA,MNbA,ij->iajb", t, oovv, io)
             - 0.5 * _ein("iMAB,jMAB,ab->iajb", t, oovv, iv))
        vovv, oovo = self.eri("vovv"), self.eri("oovo")
        S1 = (_ein("iajb,njb->nia", M, X1) + dS * X1 + 0.5 * _ein("alcd,nilcd->nia", vovv, F)
              + 0.5 * _ein("kldi,nklad->nia", oovo, F))
        f = _ein("alcd,nka->nklcd", vovv.conj(), X1)
        w = _ein("kldi,nic->nklcd", oovo.conj(), X1)
        S2 = f - f.transpose(1, 2) + w - w.transpose(3, 4)
        S2 = S2 + (ev[:, None] + ev[None, :] - eo[:, None, None, None] - eo[None, :, None, None]) * F
        return torch.cat([S1.reshape(k, -1), S2[:, p[:, None], q[:, None], r, s].reshape(k, -1)], 1)

    def diagonal(self, kind, x):
        eo, ev, o, v = self.eo, self.ev, self.o, self.ev.shape[0]
        B = self.B
        d = torch.diagonal(B, dim1=1, dim2=2)
        G = (d.T @ d - _ein("Qpq,Qqp->pq", B, B)).real * (0.0 if x is None else x)
        n = v if kind == "EA" else o
        p, q = torch.triu_indices(n, n, 1, device=B.device)
        goo, gvo, gvv = G[:o, :o], G[o:, :o], G[o:, o:]
        if kind == "EA":
            sat = ev[p] + ev[q] - eo[:, None] + gvv[p, q] - gvo[p].T - gvo[q].T
        else:
            sat = ev - eo[p][:, None] - eo[q][:, None] + goo[p, q][:, None] - gvo[:, p].T - gvo[:, q].T
        return torch.cat([torch.diagonal(self.main_block(kind, x)).real, sat.reshape(-1)])


def _exact_sigma(case, seed):
    P = _Plain(*_problem(case, seed), case["order"] == 3)
    return P.sigma(case["kind"], case["x"] if case["order"] == 3 else None, _vectors(case, seed))


def exact(case, seed):
    # dense 64-bit contractions: beyond these sizes (about 15 teraflop) they take longer than 20 seconds;
    # the third-order EE singles block has dozens of terms and no short form
    if case["kind"] == "EE" and case["order"] == 3:
        return None
    third = case["order"] == 3
    if third and 8.0 * (case["naux"] * case["nvir"] ** 4 + (case["nocc"] * case["nvir"]) ** 2 * case["nvir"] ** 2) > 2e13:
        return None
    with torch.set_grad_enabled(case["op"] == "gradient"):
        if case["op"] == "batch":
            return [_exact_sigma(m, seed + 101 * i) for i, m in enumerate(_members(case))]
        if case["op"] == "sigma":
            return _exact_sigma(case, seed)
        B, eo, ev = _problem(case, seed)
        x = case["x"] if third else None
        if case["op"] == "solve":
            n = sum(_dims(case))
            M = _Plain(B, eo, ev, third).sigma(case["kind"], x, torch.eye(n, dtype=B.dtype, device="cuda"))
            return torch.linalg.eigvalsh(M)[:case["k"]].cpu().numpy()
        if case["op"] == "setup":
            P = _Plain(B, eo, ev, third)
            return {"main": P.main_block(case["kind"], x).cpu().numpy(),
                    "diagonal": P.diagonal(case["kind"], x).cpu().numpy()}
        for a in (eo, ev):
            a.requires_grad_()
        xt = torch.tensor(x, dtype=torch.float64, device="cuda", requires_grad=True)
        Y = _vectors(case, seed)
        S = _Plain(B, eo, ev, True).sigma(case["kind"], xt, Y)
        w = torch.from_numpy(_weights(case)).cuda()
        (w * (Y.conj() * S).sum(1).real).sum().backward()
        # the gradient of B is fixed only on Hermitian changes (adc_sigma_adjoint), not element by element
        return {"B": None, "eps_occ": eo.grad, "eps_vir": ev.grad, "x": float(xt.grad)}
