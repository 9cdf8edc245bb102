"""The calls that a user of the density-fitted EA/IP-ADC library makes, as cases that can be timed.

Three kinds of call, all through the public binding (``ADC``):

* ``sigma``: one sigma = M X for a block of trial vectors, the call that a Davidson solver (the
  library's own or a program's) repeats tens to hundreds of times per molecule;
* ``setup``: a new molecule, from orbital energies and density-fitting factors to its first sigma;
* ``davidson``: the lowest roots and their spectroscopic factors, as one call.

Inputs follow the repository's recipe (``adc_inputs.py``: orbital energies, B^Q = s (G + G^T) / 2 with
s = 0.3 / sqrt(naux), trial vectors N(0, 1) / sqrt(dim)), drawn here on the GPU from the seed.

Vectors of the mixed-precision calls are kept in single precision by the calling program: a sigma of
precision 'bf16x3' carries about six digits (split-BF16 products, FP32 accumulation), and a block of
vectors is the largest thing such a program holds.  It converts a block to the float64 that the entry
point takes and the result back, and both conversions are part of the pass.  FP64 calls are float64
throughout.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2012_06714_gb300 import ADC


def _case(name, call, kind, order, precision, nocc, nvir, naux, nvec, host=False):
    return dict(name=name, call=call, kind=kind, order=order, precision=precision, nocc=nocc, nvir=nvir, naux=naux,
                nvec=nvec, host=host)


def listed():
    return [
        # the smallest workload of the repository (EA-ADC(2), 25 orbitals): launches and host work only
        _case("sigma_ea2_fp64_tiny", "sigma", "ea", 2, "fp64", 5, 20, 80, 4),
        # the same workload solved: four roots in one call
        _case("davidson_ea2_fp64_tiny", "davidson", "ea", 2, "fp64", 5, 20, 80, 4),
        # a small molecule at the reference precision, solved (subspace algebra and FP64 sigma)
        _case("davidson_ea3_fp64_small", "davidson", "ea", 3, "fp64", 8, 45, 187, 4),
        # reference-precision products of a mid-sized molecule, both directions (attachment, ionisation)
        _case("sigma_ea3_fp64_mid", "sigma", "ea", 3, "fp64", 12, 97, 381, 4),
        _case("sigma_ip3_fp64_mid", "sigma", "ip", 3, "fp64", 14, 113, 445, 5),
        # mixed precision, attachment: a small molecule with odd sizes and two unconverged roots, the
        # medium workload, and the large one that the benchmark is quoted on
        _case("sigma_ea3_mixed_small", "sigma", "ea", 3, "bf16x3", 9, 61, 245, 2),
        _case("sigma_ea3_mixed_medium", "sigma", "ea", 3, "bf16x3", 20, 180, 600, 4),
        _case("sigma_ea3_mixed_large", "sigma", "ea", 3, "bf16x3", 40, 400, 1400, 4),
        # mixed precision, ionisation: a molecule of the 64-molecule batch (six roots each) and the
        # medium workload with five roots
        _case("sigma_ip3_mixed_small", "sigma", "ip", 3, "bf16x3", 13, 97, 385, 6),
        _case("sigma_ip3_mixed_medium", "sigma", "ip", 3, "bf16x3", 20, 180, 600, 5),
        # a new molecule to its first product: medium workload from device arrays, and a molecule of
        # the batch from host arrays (how the batch hands them over)
        _case("setup_ea3_mixed_medium", "setup", "ea", 3, "bf16x3", 20, 180, 600, 4),
        _case("setup_ip3_mixed_small", "setup", "ip", 3, "bf16x3", 17, 121, 483, 6, host=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the same calls over molecules of 25 to 440 orbitals and blocks of 1 to 8 vectors."""
    call = rng.choice(["sigma", "sigma", "sigma", "setup", "davidson"])
    kind = rng.choice(["ea", "ip"])
    if call == "davidson":
        precision, order = "fp64", rng.choice([2, 3])
        nocc, nvir, nvec = _log(rng, 4, 10), _log(rng, 16, 50), rng.randint(2, 5)
    else:
        precision = rng.choice(["bf16x3", "bf16x3", "fp64"])
        order = 3 if precision == "bf16x3" else rng.choice([2, 3, 3])
        nvec = rng.randint(1, 8)
        if call == "setup":
            top = 200 if precision == "bf16x3" else 90
            nocc, nvir = _log(rng, 5, 22), _log(rng, 20, top)
        elif precision == "fp64":
            nocc, nvir = _log(rng, 5, 20), _log(rng, 20, 120)
        elif kind == "ip":
            nocc, nvir = _log(rng, 8, 30), _log(rng, 40, 250)
        else:
            nocc, nvir = _log(rng, 5, 40), _log(rng, 20, 320)
            nvec = rng.randint(1, 4) if nvir > 250 else nvec
    naux = int(round(rng.uniform(3.0, 3.5) * (nocc + nvir)))
    host = call == "setup" and rng.random() < 0.5
    c = _case("", call, kind, order, precision, nocc, nvir, naux, nvec, host=host)
    del c["name"]
    return c


def _system(case, seed):
    """(eps, B, generator) on the GPU: the repository's synthetic molecule, from the seed alone."""
    o, v, Q = case["nocc"], case["nvir"], case["naux"]
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 1000003 + 12345)

    def uniform(n):
        return torch.rand(n, dtype=torch.float64, device="cuda", generator=g)

    eps_o = torch.sort(-1.5 + 1.2 * uniform(o)).values
    eps_v = torch.sort(0.05 + 4.95 * uniform(v) ** 2).values
    B = torch.randn(Q, o + v, o + v, dtype=torch.float64, device="cuda", generator=g)
    s = 0.15 / math.sqrt(Q)
    for q0 in range(0, Q, 64):  # a block at a time: no second array of B's size
        b = B[q0:q0 + 64]
        b.copy_(s * (b + b.transpose(1, 2)))
    return torch.cat([eps_o, eps_v]), B, g


def _dim(case):
    o, v = case["nocc"], case["nvir"]
    return v + o * v * v if case["kind"] == "ea" else o + o * o * v


def _vectors(case, g):
    X = torch.randn(case["nvec"], _dim(case), dtype=torch.float64, device="cuda", generator=g) / math.sqrt(_dim(case))
    return X.float() if case["precision"] == "bf16x3" else X


def _open(case, eps, B):
    return ADC(eps, B, case["nocc"], order=case["order"], kind=case["kind"], precision=case["precision"])


def prepare(case, seed):
    eps, B, g = _system(case, seed)
    X = None if case["call"] == "davidson" else _vectors(case, g)
    if case["call"] == "setup":
        if case["host"]:
            eps, B = eps.cpu().numpy(), B.cpu().numpy()
        return dict(case=case, eps=eps, B=B, X=X)
    return dict(case=case, h=_open(case, eps, B), X=X)


def _sigma(h, X):
    if X.dtype == torch.float32:
        return h.sigma(X.double()).float()
    return h.sigma(X)


def run(state):
    case = state["case"]
    if case["call"] == "sigma":
        return _sigma(state["h"], state["X"])
    if case["call"] == "setup":
        h = _open(case, state["eps"], state["B"])
        S = _sigma(h, state["X"])
        h.close()
        return S
    e, p, _, _ = state["h"].davidson(case["nvec"], tol=1e-8)
    return e, p


def _sigma_flops(case):
    """Multiply-adds (x 2) of one sigma over the cheapest orders of its contractions."""
    o, v, Q, n = (float(case[k]) for k in ("nocc", "nvir", "naux", "nvec"))
    if case["kind"] == "ea":
        f = 2 * n * Q * (o * v * v * 2 + v * v * 2)  # first-order coupling, row and column
        if case["order"] == 3:
            # vv|vv term: over auxiliary functions, or over symmetric and antisymmetric pairs
            f += n * o * v ** 3 * min(4 * Q, v) + 2 * n * 3 * o * o * v ** 3  # and three ring contractions
            f += 2 * n * 5 * o * o * v ** 3  # second-order coupling, row (3) and column (2) with t
    else:
        f = 2 * n * Q * (o * o * v * 2 + o * o * 2)
        if case["order"] == 3:
            f += 2 * n * (o ** 4 * v + 3 * o ** 3 * v * v)  # hole-hole and ring contractions
            f += 2 * n * (2 * o * o * v ** 3 + 2 * 3 * o ** 3 * v * v + 2 * Q * v ** 3)  # second-order coupling
    return f


def work(case):
    o, v, Q, n = (float(case[k]) for k in ("nocc", "nvir", "naux", "nvec"))
    nmo = o + v
    word = 4 if case["precision"] == "bf16x3" else 8
    vec = 2 * n * _dim(case) * word
    held = 8 * Q * nmo * nmo / 2  # the symmetric factors; order 3 adds (ia|jb), (ij|ab) and t, a word each
    if case["order"] == 3:
        held += 3 * o * o * v * v * word
    if case["call"] == "sigma":
        return dict(bytes=vec + held, flops=_sigma_flops(case))
    if case["call"] == "setup":
        f = _sigma_flops(case) + 2 * Q * o * o * v * v * 2
        if case["order"] == 3:
            f += o * o * v ** 3 * min(4 * Q, v) + 2 * 10 * o ** 3 * v ** 3
        return dict(bytes=vec + 8 * Q * nmo * nmo, flops=f)
    # a solve needs at least a handful of products per root
    return dict(bytes=5 * (vec + held), flops=5 * _sigma_flops(case))


# ---- the same results in 64 bits from plain torch ---------------------------------------------------


class _Plain:
    """Spin-adapted EA/IP-ADC(2)/(3) from its working equations, four-index integrals, float64."""

    def __init__(self, case, eps, B):
        o, v = case["nocc"], case["nvir"]
        self.o, self.v, self.kind, self.order = o, v, case["kind"], case["order"]
        self.eo, self.ev = eps[:o], eps[o:]
        self.Boo, self.Bov, self.Bvv = B[:, :o, :o], B[:, :o, o:], B[:, o:, o:].contiguous()
        e = torch.einsum
        self.ovov = e("Qia,Qjb->iajb", self.Bov, self.Bov)
        self.oovv = e("Qij,Qab->ijab", self.Boo, self.Bvv)
        self.oooo = e("Qij,Qkl->ijkl", self.Boo, self.Boo)
        self.ooov = e("Qij,Qka->ijka", self.Boo, self.Bov)
        D2 = self.eo[:, None, None, None] + self.eo[:, None, None] - self.ev[:, None] - self.ev
        D1 = self.eo[:, None] - self.ev
        t = self.t = self.ovov.transpose(1, 2) / D2
        self.tau = 2 * t - t.transpose(2, 3)
        # second-order singles (part of the transition moments also at order 2)
        self.t1 = (e("Qid,Qad->ia", e("Qkc,ikdc->Qid", self.Bov, self.tau), self.Bvv)
                   - e("kilc,klac->ia", self.ooov, self.tau)) / D1
        if self.order == 3:
            W = (e("kcjb,ikac->ijab", self.ovov, 2 * t - t.transpose(2, 3)) - e("kjbc,ikac->ijab", self.oovv, t)
                 - e("kjac,ikcb->ijab", self.oovv, t))
            self.Lt = self.ladder(t.reshape(o * o, v, v)).reshape(o, o, v, v)
            self.t2 = (self.Lt + e("kilj,klab->ijab", self.oooo, t) + W + W.permute(1, 0, 3, 2)) / D2
        self.M11 = self._ea11() if self.kind == "ea" else -self._ip11()

    def ladder(self, X):
        """sum_cd (ac|bd) X[m, c, d], one row a of the integrals at a time."""
        v, Q = self.v, self.Bvv.shape[0]
        out = torch.empty_like(X)
        flat, B2 = X.reshape(X.shape[0], v * v), self.Bvv.reshape(Q, v * v)
        for a in range(v):
            acbd = (self.Bvv[:, a, :].T @ B2).reshape(v, v, v)  # [c][b][d]
            out[:, a, :] = flat @ acbd.permute(0, 2, 1).reshape(v * v, v)
        return out

    def _ea11(self):
        e, t, ovov, oovv = torch.einsum, self.t, self.ovov, self.oovv

        def both(x):  # -x_kl^ac [(kb|lc) - 1/2 (kc|lb)]
            return -e("klac,kblc->ab", x, ovov) + 0.5 * e("klac,kclb->ab", x, ovov)

        X = both(t)
        M = torch.diag(self.ev)
        if self.order == 3:
            g = e("Qkc,kc->Q", self.Bov, self.t1)
            X = X + both(self.t2) + 2 * e("Q,Qab->ab", g, self.Bvv)
            X = X - e("Qkb,Qka->ab", self.Bov, e("kc,Qac->Qka", self.t1, self.Bvv))
            X = X - e("klac,klbc->ab", t, self.Lt - 0.5 * self.Lt.transpose(2, 3))
            tT = t.transpose(2, 3)  # t_lm^dc
            G = e("kldb,lmcd->kmbc", oovv, tT - 0.5 * t) + e("kbld,lmcd->kmbc", ovov, t - 2 * tT)
            X = X + e("kmac,kmbc->ab", t, G)
            G = e("kldb,lmcd->kmbc", oovv, t - 0.5 * tT) + e("kbld,lmcd->kmbc", ovov, tT - 0.5 * t)
            X = X + e("kmca,kmbc->ab", t, G)
            Z = e("klce,klde->cd", t, 2 * t - t.transpose(2, 3))
            M = M + 2 * e("Q,Qab->ab", e("Qcd,cd->Q", self.Bvv, Z), self.Bvv)
            M = M - e("Qac,Qcb->ab", e("Qad,cd->Qac", self.Bvv, Z), self.Bvv)
            U = e("kmcd,lmcd->kl", t, self.tau)
            M = M - 2 * e("klab,kl->ab", oovv, U) + e("kbla,kl->ab", ovov, U)
        return M + X + X.T

    def _ip11(self):
        e, t, ovov, oovv, oooo = torch.einsum, self.t, self.ovov, self.oovv, self.oooo

        def both(x):  # x_il^cd [(jc|ld) - 1/2 (jd|lc)]
            return e("ilcd,jcld->ij", x, ovov) - 0.5 * e("ilcd,jdlc->ij", x, ovov)

        X = both(t)
        M = torch.diag(self.eo)
        if self.order == 3:
            X = X + both(self.t2) + 2 * e("kc,ijkc->ij", self.t1, self.ooov) - e("kc,ikjc->ij", self.t1, self.ooov)
            X = X + e("ikcd,jkcd->ij", t, e("jlkm,lmcd->jkcd", oooo, t - 0.5 * t.transpose(2, 3)))
            tT = t.transpose(2, 3)  # t_kl^ed
            G = e("ljcd,klde->kecj", oovv, 0.5 * t - tT) + e("jcld,klde->kecj", ovov, 2 * tT - t)
            X = X + e("ikce,kecj->ij", t, G)
            G = e("ljcd,klde->kecj", oovv, 0.5 * tT - t) + e("jcld,klde->kecj", ovov, 0.5 * t - tT)
            X = X + e("ikec,kecj->ij", t, G)
            U = e("kmcd,lmcd->kl", t, self.tau)
            M = M - 2 * e("ijkl,kl->ij", oooo, U) + e("ilkj,kl->ij", oooo, U)
            Z = e("klce,klde->cd", t, 2 * t - t.transpose(2, 3))
            M = M + 2 * e("ijcd,cd->ij", oovv, Z) - e("jcid,cd->ij", ovov, Z)
        return M + X + X.T

    def sigma(self, Y):
        e, o, v, n = torch.einsum, self.o, self.v, Y.shape[0]
        n1 = v if self.kind == "ea" else o
        y1 = Y[:, :n1]
        s1 = y1 @ self.M11.T
        t, tau, Boo, Bov, Bvv = self.t, self.tau, self.Boo, self.Bov, self.Bvv
        if self.kind == "ea":
            Y2 = Y[:, n1:].reshape(n, o, v, v)
            Yt = 2 * Y2 - Y2.transpose(2, 3)
            W = e("Qjc,njcd->nQd", Bov, Yt)
            hq = e("nc,Qcb->nQb", y1, Bvv)
            s2 = (self.ev[:, None] + self.ev - self.eo[:, None, None]) * Y2 + e("Qia,nQb->niab", Bov, hq)
            if self.order == 3:
                P = e("Qjm,nlmj->nQl", Boo, e("lmdc,njcd->nlmj", t, Yt))
                W = W + e("nmed,Qme->nQd", e("jmce,njcd->nmed", tau, Yt), Bov)
                V = e("jmce,njcd->nmed", t, Yt) + e("jmec,njdc->nmed", t, Yt)
                P = P - e("nmed,Qed->nQm", V, Bvv)
                s1 = s1 + e("nQl,Qla->na", P, Bov)
                p = e("nc,Qlc->nQl", y1, Bov)
                s2 = s2 + e("nlim,lmba->niab", e("nQl,Qim->nlim", p, Boo), t)
                s2 = s2 + e("nbme,imae->niab", e("nQb,Qme->nbme", hq, Bov), tau)
                q = e("nQm,Qeb->nmeb", p, Bvv)
                s2 = s2 - e("nmeb,imae->niab", q, t) - e("nmea,imeb->niab", q, t)
                s2 = s2 + self.ladder(Y2.reshape(n * o, v, v)).reshape(n, o, v, v)
                s2 = s2 - e("jiac,njcb->niab", self.oovv, Y2) - e("jibd,njad->niab", self.oovv, Y2)
                s2 = s2 + e("iajc,njcb->niab", self.ovov, 2 * Y2 - Y2.transpose(2, 3))
            s1 = s1 + e("nQd,Qda->na", W, Bvv)
        else:
            Y2 = Y[:, n1:].reshape(n, o, o, v)
            Yt = 2 * Y2 - Y2.transpose(1, 2)
            s1 = s1 + e("nQk,Qki->ni", e("Qja,njka->nQk", Bov, Yt), Boo)
            s2 = e("nQk,Qja->njka", e("ni,Qki->nQk", y1, Boo), Bov)
            s2 = s2 + (self.ev - self.eo[:, None, None] - self.eo[:, None]) * Y2
            if self.order == 3:
                Z = e("jkde,njka->ndea", t, Yt)
                s1 = s1 + e("nQe,Qie->ni", e("ndea,Qad->nQe", Z, Bvv), Bov)
                s1 = s1 + e("iklc,nklc->ni", self.ooov, e("jlac,njka->nklc", tau, Yt))
                s1 = s1 - e("lkic,nlkc->ni", self.ooov, e("jlac,njka->nlkc", t, Yt))
                s1 = s1 - e("ljic,nljc->ni", self.ooov, e("klca,njka->nljc", t, Yt))
                w = e("nQe,Qad->nead", e("ni,Qie->nQe", y1, Bov), Bvv)
                s2 = s2 + e("nead,jkde->njka", w, t)
                s2 = s2 + e("nklc,jlac->njka", e("ni,iklc->nklc", y1, self.ooov), tau)
                s2 = s2 - e("nlkc,jlac->njka", e("ni,lkic->nlkc", y1, self.ooov), t)
                s2 = s2 - e("nljc,klca->njka", e("ni,ljic->nljc", y1, self.ooov), t)
                s2 = s2 + e("kilj,nkla->nija", self.oooo, Y2) - e("kiab,nkjb->nija", self.oovv, Y2)
                s2 = s2 + e("iakb,nkjb->nija", self.ovov, 2 * Y2 - Y2.transpose(1, 2))
                s2 = s2 - e("kjab,nikb->nija", self.oovv, Y2)
        return torch.cat([s1, s2.reshape(n, -1)], dim=1)

    def root_s(self, Y, power):
        """S^power Y for S = diag(1, 2 - P): eigenvalue 1 on swap-symmetric pairs, 3 on the antisymmetric."""
        n, o, v = Y.shape[0], self.o, self.v
        n1 = v if self.kind == "ea" else o
        y2 = Y[:, n1:].reshape((n, o, v, v) if self.kind == "ea" else (n, o, o, v))
        sw = y2.transpose(2, 3) if self.kind == "ea" else y2.transpose(1, 2)
        y2 = 0.5 * (y2 + sw) + 0.5 * 3.0 ** power * (y2 - sw)
        return torch.cat([Y[:, :n1], y2.reshape(n, -1)], dim=1)

    def roots(self, nroots):
        """Lowest eigenvalues by dense diagonalisation; spectroscopic factors with T through second order."""
        n1 = self.v if self.kind == "ea" else self.o
        dim = n1 + (self.o * self.v * self.v if self.kind == "ea" else self.o * self.o * self.v)
        eye = torch.eye(dim, dtype=torch.float64, device=self.t.device)
        A = self.root_s(self.sigma(self.root_s(eye, -0.5)), 0.5)
        w, U = torch.linalg.eigh(0.5 * (A + A.T))
        SY = self.root_s(U[:, :nroots].T.contiguous(), 0.5)  # S Y of the S-normalised vectors
        e, t, o, v, n = torch.einsum, self.t, self.o, self.v, nroots
        u = t - 0.5 * t.transpose(2, 3)
        y1 = SY[:, :n1]
        if self.kind == "ea":
            y2 = SY[:, n1:].reshape(n, o, v, v)
            a = y1 - e("rb,cb->rc", y1, e("klcd,klbd->cb", t, u))
            b = -e("rb,kb->rk", y1, self.t1) - e("rjcd,kjdc->rk", y2, t)
        else:
            y2 = SY[:, n1:].reshape(n, o, o, v)
            a = y1 - e("rj,kj->rk", y1, e("klcd,jlcd->kj", t, u))
            b = e("rj,jc->rc", y1, self.t1) - e("rija,ijac->rc", y2, t)
        return w[:nroots], 2 * ((a * a).sum(1) + (b * b).sum(1))


def exact(case, seed):
    o, v, Q, n = (float(case[k]) for k in ("nocc", "nvir", "naux", "nvec"))
    # FP64 arithmetic of about one TFLOP/s: what would take over about 20 seconds is left out
    flops = 20 * o * o * v * v * Q + 24 * n * o * o * v ** 3
    if case["order"] == 3:
        flops += 2 * Q * v ** 4 * (2 if case["kind"] == "ea" else 1) + 2 * (o * o + n * o) * v ** 4 + 24 * o ** 3 * v ** 3
    if flops > 1.2e13 or (case["call"] == "davidson" and _dim(case) > 8000):
        return None
    eps, B, g = _system(case, seed)
    ref = _Plain(case, eps, B)
    if case["call"] != "davidson":
        return ref.sigma(_vectors(case, g).double())
    w, p = ref.roots(case["nvec"])
    # order 3 takes its spectroscopic factors from third-order moments, which are not restated here
    return w.cpu().numpy(), (p.cpu().numpy() if case["order"] == 2 else None)
