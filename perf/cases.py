"""The work a user of the library has it do, as a list of timed cases.

Every case goes through the Python binding (``paper_2311_10048_gb300.lno_ot``):
a context per program, domains as device tensors, outputs in the caller's
buffers.  Inputs follow the package's synthetic recipe (``synth.py``): random
DF factors with a decaying auxiliary index, sorted orbital energies, MP2-like
doubles; here they are drawn on the GPU so that a domain costs milliseconds.

Kinds of case
  energy   one domain, ``Context.energy`` with per-triplet outputs (and with an
           f_ov block: the orbital contributions too); ``sel`` > 0 computes a
           seeded sample of that many triplets per spin case
  closed   the same for a closed-shell domain (both spins share their arrays)
  batch    ``Context.energy_batched`` over several domains of different sizes
  central  ``Context.energy_central`` for central orbitals of one spin
  grad     ``triples_energy`` and its gradients by ``torch.autograd``
  naf      ``Context.naf``
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2311_10048_gb300 import lno_ot

DEV = "cuda"
F64 = torch.float64


# ---------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------
def _energy(name, nbas, na, nb, naux, prec, fov=False, sel=0):
    return dict(name=name, kind="energy", nbas=nbas, na=na, nb=nb, naux=naux, prec=prec,
                fov=fov, sel=sel)


def listed():
    return [
        # the smallest domain of the test suite: launch and latency bound
        _energy("small_x10", 40, 6, 4, 120, "bf16x10"),
        # the same in the binding's default precision (the float64 comparator)
        _energy("small_fp64", 40, 6, 4, 120, "fp64"),
        # a below-average LNO domain, nothing a multiple of a tile
        _energy("ragged_x10", 121, 14, 11, 363, "bf16x10"),
        # the medium domain of the test suite, all its triplets
        _energy("medium_x10", 200, 20, 18, 600, "bf16x10"),
        # the virtual space of the benchmark's domain with few occupied orbitals
        _energy("wide_x10", 368, 8, 6, 1200, "bf16x10"),
        # the faster precision on an average domain
        _energy("average_x6", 150, 12, 10, 450, "bf16x6"),
        # a restricted open-shell reference: the f_ov term, orbital contributions
        _energy("open_shell_fov_x10", 100, 11, 9, 300, "bf16x10", fov=True),
        # a closed-shell domain: spin-flip images computed once
        dict(name="closed_shell_x10", kind="closed", nbas=112, na=12, nb=12, naux=336,
             prec="bf16x10"),
        # the small end of the many-domain batch of a large molecule
        dict(name="batch_x10", kind="batch", prec="bf16x10",
             shapes="68x8x7x204,77x9x7x231,83x9x6x249,95x11x9x285,104x12x11x312,126x14x13x378"),
        # what an LNO program takes from each domain: its central orbital's share
        dict(name="central_x10", kind="central", nbas=140, na=14, nb=12, naux=420, spin=0,
             nlmo=1, prec="bf16x10"),
        # energy and all gradients of a small domain
        dict(name="gradient_x10", kind="grad", nbas=60, na=7, nb=5, naux=180, prec="bf16x10",
             sel=0),
        # NAF compression of the medium domain's DF factors
        dict(name="naf", kind="naf", nbas=200, na=20, nb=18, naux=600, prec="bf16x10"),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["energy", "fov", "closed", "batch", "central", "grad", "naf"],
                       [10, 2, 2, 2, 2, 3, 2])[0]

    def occ(hi):
        na = rng.randint(3, hi)
        return na, max(1, na - rng.randint(0, 3))

    if kind in ("energy", "fov"):
        prec = rng.choice(["bf16x10", "bf16x10", "bf16x10", "bf16x6", "bf16x3", "fp64"])
        cap = 4e11 if prec == "fp64" else 3e13
        sel = 0
        for _ in range(1000):
            v = _logint(rng, 20, 70 if prec == "fp64" else 330)
            na, nb = occ(24)
            c = _energy("", v + na, na, nb, rng.randint(2, 4) * (v + na) + rng.randint(0, 7), prec,
                        fov=kind == "fov", sel=sel)
            if _alg_flops(c) <= cap:
                break
            if rng.random() < 0.3:
                sel = rng.randint(3, 12)
    elif kind == "closed":
        for _ in range(1000):
            v, n = _logint(rng, 24, 200), rng.randint(3, 18)
            c = dict(kind="closed", nbas=v + n, na=n, nb=n, naux=3 * (v + n) + rng.randint(0, 5),
                     prec="bf16x10")
            if _alg_flops(c) <= 1.5e13:
                break
    elif kind == "batch":
        rows = []
        for _ in range(rng.randint(2, 6)):
            na = rng.randint(8, 13)
            nv = max(60, int(round(8 * na * rng.uniform(0.8, 1.2))))
            rows.append("%dx%dx%dx%d" % (na + nv, na, na - rng.randint(1, 3), 3 * (na + nv)))
        c = dict(kind="batch", prec="bf16x10", shapes=",".join(rows))
    elif kind == "central":
        v = _logint(rng, 30, 160)
        na, nb = occ(14)
        c = dict(kind="central", nbas=v + na, na=na, nb=nb, naux=3 * (v + na) + rng.randint(0, 5),
                 spin=rng.randint(0, 1), nlmo=rng.randint(1, 2), prec="bf16x10")
    elif kind == "grad":
        prec = rng.choice(["bf16x10", "bf16x10", "fp64"])
        v = _logint(rng, 12, 60)
        na, nb = occ(6)
        c = dict(kind="grad", nbas=v + na, na=na, nb=nb, naux=2 * (v + na) + rng.randint(0, 9),
                 prec=prec, sel=0 if v < 40 else rng.randint(2, 9))
    else:
        v = _logint(rng, 24, 180)
        na, nb = occ(20)
        c = dict(kind="naf", nbas=v + na, na=na, nb=nb,
                 naux=min(640, 2 * (v + na) + rng.randint(0, 99)), prec="bf16x10")
    c.pop("name", None)
    return c


# ---------------------------------------------------------------------------
# Sizes
# ---------------------------------------------------------------------------
def _c2(n):
    return n * (n - 1) // 2


def _c3(n):
    return n * (n - 1) * (n - 2) // 6


def _ntrip(na, nb):
    """Restricted triplets of the cases aaa, aab, abb, bbb."""
    return [_c3(na), _c2(na) * nb, _c2(nb) * na, _c3(nb)]


def _shapes(case):
    if case["kind"] == "batch":
        return [tuple(int(x) for x in s.split("x")) for s in case["shapes"].split(",")]
    return [(case["nbas"], case["na"], case["nb"], case["naux"])]


def _selection(case):
    """Seeded triplet samples per spin case (host int64 arrays), or None."""
    if not case.get("sel"):
        return None
    out = []
    for c, n in enumerate(_ntrip(case["na"], case["nb"])):
        r = np.random.default_rng([n, c, case["sel"]])
        out.append(np.sort(r.choice(n, size=min(case["sel"], n), replace=False)).astype(np.int64))
    return out


def _counts(case, na, nb):
    n = _ntrip(na, nb)
    return [min(case["sel"], x) for x in n] if case.get("sel") else n


def _method_flops(nbas, na, nb, n):
    """W contractions of n[case] triplets, every restricted output once."""
    va, vb = nbas - na, nbas - nb

    def same(v, o):
        return 6 * v * _c2(v) * (v + o)

    def mixed(vs, vt, os_, ot):
        return 2 * vs * vs * vt * (2 * (vt + ot) + vs + os_) + 4 * vt * _c2(vs) * (vs + os_)

    return (n[0] * same(va, na) + n[3] * same(vb, nb) + n[1] * mixed(va, vb, na, nb)
            + n[2] * mixed(vb, va, nb, na))


def _alg_flops(case):
    return sum(_method_flops(n, na, nb, _counts(case, na, nb)) for n, na, nb, _ in _shapes(case))


def _input_bytes(nbas, na, nb, naux, spins=2):
    va, vb = nbas - na, nbas - nb
    n = spins * (naux * nbas * nbas + nbas) + na * va + (nb * vb if spins == 2 else 0)
    n += na * na * va * va + (nb * nb * vb * vb if spins == 2 else 0) + na * nb * va * vb
    return 8 * n


def work(case):
    kind = case["kind"]
    b = f = 0.0
    for nbas, na, nb, naux in _shapes(case):
        va, vb = nbas - na, nbas - nb
        inp = _input_bytes(nbas, na, nb, naux, 1 if kind == "closed" else 2)
        # the three-external integrals, once per occupied orbital and spin pair
        df = 2.0 * naux * (na * va * _c2(va) + nb * vb * _c2(vb)
                           + na * va * vb * vb / 2 + nb * vb * va * va / 2)
        n = _counts(case, na, nb)
        if kind == "closed":
            n = [n[0], n[1], 0, 0]
            df /= 2
        if kind == "naf":
            npair = nbas * (nbas + 1) / 2
            b += 2 * 8 * naux * nbas * nbas * 2
            f += 2 * naux * naux * npair + 10.0 * naux ** 3 + 4.0 * naux * naux * npair
            continue
        if kind == "central":
            os_, ot = (na, nb) if case["spin"] == 0 else (nb, na)
            p = case["nlmo"]
            m = [0, 0, 0, 0]
            m[0 if case["spin"] == 0 else 3] = p * _c2(os_)
            m[1 if case["spin"] == 0 else 2] = p * os_ * ot
            m[2 if case["spin"] == 0 else 1] = p * _c2(ot)
            f += df + _NQ * _method_flops(nbas, na, nb, m)
            b += inp
            continue
        fw = _method_flops(nbas, na, nb, n)
        b += inp + 8 * sum(n)
        f += df + fw
        if kind == "grad":   # recomputation and two products per contraction
            b += inp
            f += 2 * df + 3 * fw
    return dict(bytes=float(b), flops=float(f))


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
_NQ = 4              # quadrature points of the central-orbital cases
_LAP = (1.2, 22.0)   # denominator range the quadrature covers (Eh)


def _spin(gen, nbas, nocc, naux):
    b = torch.randn(naux, nbas, nbas, dtype=F64, device=DEV, generator=gen)
    b = b.triu() + b.triu(1).transpose(1, 2)
    q = torch.arange(naux, dtype=F64, device=DEV)
    b *= (torch.exp(-q * (4.0 / naux)) / math.sqrt(naux))[:, None, None]

    def uni(n, lo, hi):
        x = torch.rand(n, dtype=F64, device=DEV, generator=gen)
        return (lo + (hi - lo) * x).sort().values

    eps = torch.cat([uni(nocc, -2.0, -0.3), uni(nbas - nocc, 0.1, 5.0)])
    t1 = torch.randn(nocc, nbas - nocc, dtype=F64, device=DEV, generator=gen) * 1e-3
    return b.contiguous(), eps, t1


def _ovov(bp, op, bq, oq):
    """(ia|jb) as [i][j][a][b]."""
    naux, nbas = bp.shape[:2]
    x = bp[:, :op, op:].reshape(naux, -1)
    y = bq[:, :oq, oq:].reshape(naux, -1)
    return (x.t() @ y).view(op, nbas - op, oq, nbas - oq).permute(0, 2, 1, 3)


def _d2(ep, op, eq, oq):
    return (ep[:op, None, None, None] + eq[None, :oq, None, None]
            - ep[None, None, op:, None] - eq[None, None, None, oq:])


def _domain(gen, nbas, na, nb, naux, fov=False, closed=False):
    up = _spin(gen, nbas, na, naux)
    dn = up if closed else _spin(gen, nbas, nb, naux)
    t2 = []
    for b, e, n in ((up[0], up[1], na), (dn[0], dn[1], nb)):
        g = _ovov(b, n, b, n)
        t2.append(((g - g.transpose(2, 3)) / _d2(e, n, e, n)).contiguous())
    t2ab = (_ovov(up[0], na, dn[0], nb) / _d2(up[1], na, dn[1], nb)).contiguous()
    d = dict(nbas=nbas, naux=naux, nocc=(na, nb), B=[up[0], dn[0]], eps=[up[1], dn[1]],
             t1=[up[2], dn[2]], t2aa=t2[0], t2bb=t2[0] if closed else t2[1], t2ab=t2ab)
    if fov:
        d["fov"] = [torch.randn(n, nbas - n, dtype=F64, device=DEV, generator=gen) * 0.02
                    for n in (na, nb)]
    return d


def _inputs(case, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    doms = [_domain(gen, n, na, nb, naux, bool(case.get("fov")), case["kind"] == "closed")
            for n, na, nb, naux in _shapes(case)]
    u = None
    if case["kind"] == "central":
        n = (case["na"], case["nb"])[case["spin"]]
        u = torch.randn(n, n, dtype=F64, device=DEV, generator=gen)
        u = torch.linalg.qr(u)[0][:case["nlmo"]].contiguous()
    return doms, u


def prepare(case, seed):
    lno_ot.load_library()
    doms, u = _inputs(case, seed)
    ctx = lno_ot.Context(0, case["prec"])
    st = dict(kind=case["kind"], ctx=ctx, doms=doms, u=u, sel=_selection(case))
    if case["kind"] in ("energy", "closed"):
        n = _counts(case, case["na"], case["nb"])
        st["e_trip"] = [torch.zeros(x, dtype=F64, device=DEV) if x else None for x in n]
        st["e_orb"] = ([torch.zeros(x, dtype=F64, device=DEV) for x in (case["na"], case["nb"])]
                       if case.get("fov") else None)
    elif case["kind"] == "central":
        st["spin"] = case["spin"]
        st["quad"] = _quadrature()
    elif case["kind"] == "grad":
        d = doms[0]
        st["leaves"] = [*d["B"], *d["eps"], *d["t1"], d["t2aa"], d["t2bb"], d["t2ab"]]
        for x in st["leaves"]:
            x.requires_grad_(True)
    torch.cuda.synchronize()
    return st


def _quadrature():
    """_NQ points of 1/x = int exp(-x s) ds on _LAP: trapezoid rule in log s, weights by
    least squares on the relative error."""
    x = np.geomspace(*_LAP, 400)
    s = np.geomspace(0.35 / _LAP[1], 2.2 / _LAP[0], _NQ)
    w = np.linalg.lstsq(x[:, None] * np.exp(-x[:, None] * s), np.ones_like(x), rcond=None)[0]
    return s, w


def run(state):
    ctx, d, kind = state["ctx"], state["doms"][0], state["kind"]
    if kind in ("energy", "closed"):
        out = ctx.energy(d, e_trip=state["e_trip"], trip_sel=state["sel"], e_orb=state["e_orb"])
        out["e_trip"] = state["e_trip"]
        out["e_orb"] = state["e_orb"]
        return out
    if kind == "batch":
        return ctx.energy_batched(state["doms"])
    if kind == "central":
        return ctx.energy_central(d, state["spin"], state["u"], *state["quad"])
    if kind == "grad":
        e = lno_ot.triples_energy(ctx, d, trip_sel=state["sel"])
        return [e, *torch.autograd.grad(e, state["leaves"])]
    out, lam = ctx.naf(d)
    return dict(B=out["B"], naux=out["naux"], lam=lam)


# ---------------------------------------------------------------------------
# The same quantities in plain float64 torch
# ---------------------------------------------------------------------------
class _Ref:
    """(T) energies per triplet, spin-case equations with full virtual cubes.

    The occupied indices of a triplet run over the rows the arrays hold, the
    summed occupied index over the first ``noi`` of them (they differ when
    pseudo-orbitals follow the real ones); ``lap`` = (s, w) weights elements by
    -w exp(s D) instead of 1/D."""

    def __init__(self, d, noi=None, lap=None):
        self.lap = lap
        self.no = d["nocc"]
        self.noi = noi or d["nocc"]
        o = self.no
        self.oo = [d["B"][s][:, :self.noi[s], :o[s]] for s in (0, 1)]
        self.ov = [d["B"][s][:, :o[s], o[s]:] for s in (0, 1)]
        self.vv = [d["B"][s][:, o[s]:, o[s]:] for s in (0, 1)]
        self.eo = [d["eps"][s][:o[s]] for s in (0, 1)]
        self.ev = [d["eps"][s][o[s]:] for s in (0, 1)]
        self.t1 = d["t1"]
        self.tss = [d["t2aa"], d["t2bb"]]
        self.tst = [d["t2ab"], d["t2ab"].permute(1, 0, 3, 2)]
        self.fov = d.get("fov")
        self.memo = {}

    def _once(self, key, make):
        if key not in self.memo:
            self.memo[key] = make()
        return self.memo[key]

    # K-concatenated operands: rows of the virtual index, columns of the pair
    def at(self, s, p, q):
        def make():
            x = torch.einsum("Qm,Qa->ma", self.oo[s][:, :, q], self.ov[s][:, p])
            x = x - torch.einsum("Qm,Qa->ma", self.oo[s][:, :, p], self.ov[s][:, q])
            return torch.cat([self.tss[s][p, q], x.t()], 1)
        return self._once(("at", s, p, q), make)

    def bt(self, s, x):
        def make():
            g = torch.einsum("Qeb,Qc->ebc", self.vv[s], self.ov[s][:, x])
            g = g - g.transpose(1, 2)
            return torch.cat([g, self.tss[s][x, :self.noi[s]]], 0).flatten(1)
        return self._once(("bt", s, x), make)

    def a1(self, s, p, k):
        t = 1 - s
        return self._once(("a1", s, p, k), lambda: torch.cat(
            [-self.tst[s][p, k],
             torch.einsum("Qa,QM->aM", self.ov[s][:, p], self.oo[t][:, :, k])], 1))

    def bg(self, s, x):
        t = 1 - s
        return self._once(("bg", s, x), lambda: torch.cat(
            [torch.einsum("Qb,QEC->EbC", self.ov[s][:, x], self.vv[t]),
             self.tst[s][x, :self.noi[t]]], 0).flatten(1))

    def bf(self, s, k):
        t = 1 - s
        return self._once(("bf", s, k), lambda: torch.cat(
            [torch.einsum("Qbe,QC->ebC", self.vv[s], self.ov[t][:, k]),
             -self.tst[s][:self.noi[s], k]], 0).flatten(1))

    def at2(self, s, p, k):
        t = 1 - s
        return self._once(("at2", s, p, k), lambda: torch.cat(
            [self.tst[s][p, k].t(),
             torch.einsum("Qm,QC->Cm", self.oo[s][:, :, p], self.ov[t][:, k])], 1))

    def kss(self, s, p, q):
        def make():
            g = torch.einsum("Qa,Qb->ab", self.ov[s][:, p], self.ov[s][:, q])
            return g - g.t()
        return self._once(("kss", s, p, q), make)

    def kst(self, s, p, k):
        return self._once(("kst", s, p, k), lambda: torch.einsum(
            "Qa,QC->aC", self.ov[s][:, p], self.ov[1 - s][:, k]))

    def _weigh(self, w, v, dd):
        if self.lap is None:
            return (w * (w + v) / dd).sum()
        return (w * (w + v) * (-self.lap[1] * torch.exp(self.lap[0] * dd))).sum()

    def same(self, s, i, j, k):
        nv = self.ev[s].numel()
        x = (self.at(s, j, k) @ self.bt(s, i) + self.at(s, k, i) @ self.bt(s, j)
             + self.at(s, i, j) @ self.bt(s, k)).view(nv, nv, nv)
        w = x - x.transpose(0, 1) + x.permute(1, 2, 0)
        sets = [(self.t1[s], lambda p, q: self.kss(s, p, q))]
        if self.fov is not None:
            sets.append((self.fov[s], lambda p, q: self.tss[s][p, q]))
        v = 0
        for c, pl in sets:
            y = (c[i][:, None, None] * pl(j, k) + c[j][:, None, None] * pl(k, i)
                 + c[k][:, None, None] * pl(i, j))
            v = v + y - y.transpose(0, 1) + y.permute(1, 2, 0)
        ev = self.ev[s]
        dd = (self.eo[s][i] + self.eo[s][j] + self.eo[s][k] - ev[:, None, None]
              - ev[None, :, None] - ev[None, None, :])
        return self._weigh(w, v, dd) / 6

    def mixed(self, s, i, j, k):
        t = 1 - s
        vs, vt = self.ev[s].numel(), self.ev[t].numel()
        y = (self.a1(s, j, k) @ self.bg(s, i) - self.a1(s, i, k) @ self.bg(s, j)
             + self.at(s, i, j) @ self.bf(s, k)).view(vs, vs, vt)
        z = (self.at2(s, i, k) @ self.bt(s, j) - self.at2(s, j, k) @ self.bt(s, i)).view(
            vt, vs, vs)
        w = y - y.transpose(0, 1) + z.permute(1, 2, 0)
        sets = [(self.t1[s], self.t1[t], lambda p: self.kst(s, p, k), self.kss(s, i, j))]
        if self.fov is not None:
            sets.append((self.fov[s], self.fov[t], lambda p: self.tst[s][p, k],
                         self.tss[s][i, j]))
        v = 0
        for cs, ct, pl, kab in sets:
            u = cs[i][:, None, None] * pl(j) - cs[j][:, None, None] * pl(i)
            v = v + u - u.transpose(0, 1) + kab[:, :, None] * ct[k]
        dd = (self.eo[s][i] + self.eo[s][j] + self.eo[t][k] - self.ev[s][:, None, None]
              - self.ev[s][None, :, None] - self.ev[t][None, None, :])
        return self._weigh(w, v, dd) / 2


def _triplets(na, nb, sel=None):
    """Restricted triplets (i, j, k) of the four cases in lexicographic order."""
    def same(n):
        return [(i, j, k) for i in range(n) for j in range(i + 1, n) for k in range(j + 1, n)]

    def mixed(n2, n1):
        return [(i, j, k) for i in range(n2) for j in range(i + 1, n2) for k in range(n1)]

    out = [same(na), mixed(na, nb), mixed(nb, na), same(nb)]
    return [[t[int(q)] for q in sel[c]] for c, t in enumerate(out)] if sel else out


def _energies(ref, trips):
    fn = [lambda *t: ref.same(0, *t), lambda *t: ref.mixed(0, *t), lambda *t: ref.mixed(1, *t),
          lambda *t: ref.same(1, *t)]
    return [torch.stack([fn[c](*t) for t in trips[c]]) if trips[c] else None for c in range(4)]


def _totals(e):
    s = [0.0 if x is None else math.fsum(x.tolist()) for x in e]
    return dict(aaa=s[0], aab=s[1], abb=s[2], bbb=s[3], total=math.fsum(s), status=0)


def _orbitals(e, trips, na, nb):
    out = [np.zeros(na), np.zeros(nb)]
    for c, x in enumerate(e):
        s = 0 if c < 2 else 1
        for (i, j, k), v in zip(trips[c], [] if x is None else x.tolist()):
            if c in (0, 3):
                for p in (i, j, k):
                    out[s][p] += v / 3
            else:
                out[s][i] += v / 4
                out[s][j] += v / 4
                out[1 - s][k] += v / 2
    return [torch.from_numpy(x) for x in out]


def _augmented(d, spin, u, s):
    """The domain with one pseudo-orbital per row of u after spin's occupied orbitals."""
    n = d["nocc"][spin]
    c = u * torch.exp(d["eps"][spin][:n] * (s / 2))
    b = d["B"][spin]
    row = torch.einsum("li,Qip->Qlp", c, b[:, :n])
    b = torch.cat([b[:, :n], row, b[:, n:]], 1)
    col = torch.einsum("li,Qpi->Qpl", c, b[:, :, :n])
    b = torch.cat([b[:, :, :n], col, b[:, :, n:]], 2)
    out = dict(d)
    e = d["eps"][spin]
    eps = torch.cat([e[:n], torch.zeros(u.shape[0], dtype=F64, device=e.device), e[n:]])
    t1 = torch.cat([d["t1"][spin], c @ d["t1"][spin]], 0)
    key = ("t2aa", "t2bb")[spin]
    t = d[key]
    t = torch.cat([t, torch.einsum("li,ijab->ljab", c, t)], 0)
    t = torch.cat([t, torch.einsum("lj,ijab->ilab", c, t)], 1)
    x = d["t2ab"]
    y = torch.einsum("li,ijab->ljab" if spin == 0 else "lj,ijab->ilab", c, x)
    for k, val in (("B", b), ("eps", eps), ("t1", t1)):
        out[k] = [val if q == spin else d[k][q] for q in (0, 1)]
    out[key], out["t2ab"] = t, torch.cat([x, y], spin)
    out["nocc"] = tuple(d["nocc"][q] + (u.shape[0] if q == spin else 0) for q in (0, 1))
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind != "naf" and _alg_flops(case) > 6e12:
        return None
    doms, u = _inputs(case, seed)
    d = doms[0]
    if kind in ("energy", "closed"):
        trips = _triplets(case["na"], case["nb"], _selection(case))
        e = _energies(_Ref(d), trips)
        return dict(_totals(e), e_trip=e,
                    e_orb=_orbitals(e, trips, case["na"], case["nb"]) if case.get("fov") else None)
    if kind == "batch":
        return 0, [_totals(_energies(_Ref(x), _triplets(*x["nocc"]))) for x in doms]
    if kind == "central":
        sp, o, n = case["spin"], d["nocc"][case["spin"]], d["nocc"][1 - case["spin"]]
        out = np.zeros(case["nlmo"])
        for s, w in zip(*_quadrature()):
            ref = _Ref(_augmented(d, sp, u, s), d["nocc"], (s, w))
            for p in range(case["nlmo"]):
                x = [ref.same(sp, j, k, o + p) for j in range(o) for k in range(j + 1, o)]
                x += [ref.mixed(sp, j, o + p, k) for j in range(o) for k in range(n)]
                x += [ref.mixed(1 - sp, j, k, o + p) for j in range(n) for k in range(j + 1, n)]
                out[p] += math.fsum(torch.stack(x).tolist()) / 3 if x else 0.0
        return out
    if kind == "grad":
        leaves = [*d["B"], *d["eps"], *d["t1"], d["t2aa"], d["t2bb"], d["t2ab"]]
        for x in leaves:
            x.requires_grad_(True)
        f = dict(d, B=[(b + b.transpose(1, 2)) / 2 for b in d["B"]])
        for k in ("t2aa", "t2bb"):
            x = (d[k] - d[k].transpose(2, 3)) / 2
            f[k] = (x - x.transpose(0, 1)) / 2
        e = _energies(_Ref(f), _triplets(case["na"], case["nb"], _selection(case)))
        e = sum(x.sum() for x in e if x is not None)
        g = torch.autograd.grad(e, leaves, allow_unused=True)
        g = [torch.zeros_like(x) if y is None else y for x, y in zip(leaves, g)]
        return [e.detach(), *g]
    j = []
    for b in d["B"]:
        p, q = torch.triu_indices(case["nbas"], case["nbas"], device=DEV)
        j.append(b[:, p, q])
    lam = torch.linalg.eigvalsh((j[0] @ j[0].t() + j[1] @ j[1].t()) / 2).flip(0)
    return dict(B=None, naux=int((lam > 1e-2).sum()), lam=lam.cpu().numpy())
