"""Inputs at the edges of what the entry points accept: factors whose sums over the
auxiliary index are large in every slice, sizes at a launch's limits, bounded and
nearly full memory."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2311_10048_gb300 import lno_ot
from paper_2311_10048_gb300.synth import make_domain

pytestmark = pytest.mark.gpu


def all_trips(na, nb):
    return [na * (na - 1) * (na - 2) // 6, na * (na - 1) // 2 * nb, nb * (nb - 1) // 2 * na,
            nb * (nb - 1) * (nb - 2) // 6]


def e_trips(prec, dd, **kw):
    ctx = lno_ot.Context(0, prec, **kw)
    n = all_trips(*dd["nocc"])
    et = [torch.zeros(max(x, 1), dtype=torch.float64, device="cuda") for x in n]
    ctx.energy(dd, e_trip=et)
    ctx.close()
    return np.concatenate([e[:x].cpu().numpy() for e, x in zip(et, n)])


@pytest.mark.parametrize("naux", [150, 300, 1200])
@pytest.mark.parametrize("prec,tol", [("bf16x15", 2e-8), ("bf16x10", 2e-8), ("bf16x6", 1e-6)])
def test_flat_factors(naux, prec, tol):
    """Factors of one size along the auxiliary index: (pq|rs) = h_pq h_rs sum_Q g_Q^2
    reaches naux times the square of the scale, so the leading class sum of the DF
    products passes 2^21 (where five slices need more than 53 bits) and comes near
    2^24.  |h| <= 1 with both signs keeps the antisymmetrised integrals as large, so
    the tolerances are those of test_gpu_contract.py."""
    nbas, na, nb = 30, 4, 3
    d = make_domain(nbas, (na, nb), naux=naux, L=naux / 3, seed=21, t1_sd=0.02)
    rng = np.random.default_rng(naux)
    g = rng.uniform(0.09, 0.1, naux) * rng.choice([-1.0, 1.0], naux)
    for s in (0, 1):
        h = rng.uniform(-1.0, 1.0, (nbas, nbas))
        h = np.triu(h) + np.triu(h, 1).T
        d["B"][s] = np.ascontiguousarray(g[:, None, None] * h[None])
    dd = lno_ot.to_device(d)
    ref = e_trips("fp64", dd)
    assert np.abs(e_trips(prec, dd) - ref).max() <= tol * np.abs(ref).max()


def test_gradient_of_a_domain_whose_slicing_exceeds_one_grid(lib):
    """1449 virtuals: the v^2 rows of a DF block are more than 65535 32-row tiles.  One
    aaa triplet; E is homogeneous of degree -1 in the orbital energies, 4 in the DF
    factors and 2 in (T1, T2) together, so sum x dE/dx is -E, 4 E and 2 E: float32 in
    the forward's elements leaves ~1e-9 of E, the adjoint's 32-bit operands less."""
    v = 1449
    d = make_domain(v + 3, (3, 0), naux=8, L=6.0, seed=13, t1_sd=0.02)
    dd = lno_ot.to_device(d)
    torch.cuda.empty_cache()
    ctx = lno_ot.Context(0, "bf16x10")
    E = ctx.energy(dd)["total"]
    z = torch.zeros_like
    g = dict(dB=[z(dd["B"][0]), None], deps=[z(dd["eps"][0]), None], dt1=[z(dd["t1"][0]), None],
             dt2aa=z(dd["t2aa"]))
    ctx.backward(dd, 1.0, g)
    ctx.close()
    dot = lambda x, y: float((x * y).sum())
    assert abs(dot(dd["eps"][0], g["deps"][0]) + E) <= 1e-6 * abs(E)
    assert abs(dot(dd["B"][0], g["dB"][0]) - 4 * E) <= 1e-6 * abs(E)
    amp = dot(dd["t1"][0], g["dt1"][0]) + dot(dd["t2aa"], g["dt2aa"])
    assert abs(amp - 2 * E) <= 1e-6 * abs(E)


class PoolHigh:
    """Most bytes in use in the device's default pool (what cudaMallocAsync takes)."""
    USED, HIGH = 7, 8   # CU_MEMPOOL_ATTR_USED_MEM_CURRENT, _HIGH

    def __init__(self):
        self.cu = ctypes.CDLL("libcuda.so.1")
        self.pool = ctypes.c_void_p()
        assert self.cu.cuDeviceGetDefaultMemPool(ctypes.byref(self.pool), 0) == 0

    def _get(self, attr):
        x = ctypes.c_uint64()
        assert self.cu.cuMemPoolGetAttribute(self.pool, attr, ctypes.byref(x)) == 0
        return x.value

    def reset(self):
        torch.cuda.synchronize()
        x = ctypes.c_uint64(0)
        assert self.cu.cuMemPoolSetAttribute(self.pool, self.HIGH, ctypes.byref(x)) == 0
        self.base = self._get(self.USED)

    def high(self):
        torch.cuda.synchronize()
        return self._get(self.HIGH) - self.base


@pytest.mark.parametrize("prec", ["bf16x10", "bf16x15", "tf32", "fp64"])
@pytest.mark.parametrize("naux", [8, 33])
def test_workspace_bound_holds_for_what_is_allocated(prec, naux):
    """A domain without triplets only stages its DF blocks: at the smallest bound that
    is accepted, no more than that is allocated (rows of few auxiliary functions were
    charged at a quarter of what they took)."""
    dd = lno_ot.to_device(make_domain(150, (1, 0), naux=naux, L=15.0, seed=5))
    pool = PoolHigh()

    def run(bound):
        ctx = lno_ot.Context(0, prec, workspace_bytes=bound)
        pool.reset()
        rc = ctx.energy(dd, raise_on_error=False)["status"]
        high = pool.high()
        ctx.close()
        assert rc in (lno_ot.OK, lno_ot.ENOMEM)
        return rc == lno_ot.OK, high

    lo, hi = 256, 256 << 20
    while hi - lo > 256:
        mid = (lo + hi) // 2
        ok, high = run(mid)
        if ok:
            hi = mid
            assert high <= mid + 4096   # the pool's own rounding of a dozen blocks
        else:
            lo = mid
    assert run(hi)[0]


@pytest.mark.parametrize("flat", [False, True])
def test_fp16_slices_refused_by_the_second_spin_only(flat):
    """Doubles of the second spin near the largest magnitude throughout: its leading FP16
    sums are not provably exact, so its operands are laid out again on the BF16 slices.
    What the first spin has computed is not computed again (triplets and products of the
    call), at any point of the quadrature."""
    v, n = 256, 3
    d = make_domain(v + n, (n, n), naux=150, L=50.0, seed=77, t1_sd=0.02)
    if flat:
        top = max(np.abs(d[k]).max() for k in ("t2aa", "t2bb", "t2ab"))
        d["t2bb"] = np.sign(d["t2bb"]) * 0.99 * 2.0 ** np.ceil(np.log2(top))
    dd = lno_ot.to_device(d)
    ref = e_trips("fp64", dd)
    got = e_trips("bf16x10", dd)
    assert np.abs(got - ref).max() <= 2e-8 * np.abs(ref).max()
    U = torch.eye(n, dtype=torch.float64, device="cuda")[:1].contiguous()
    s, w = [0.05, 0.4], [0.2, 0.5]
    dE = []
    for prec in ("fp64", "bf16x10"):
        ctx = lno_ot.Context(0, prec)
        dE.append(ctx.energy_central(dd, 0, U, s, w)[0])
        st = ctx.stats()
        ctx.close()
    assert abs(dE[0] - dE[1]) <= 2e-8 * abs(dE[0])
    # holding the central orbital: C(3,2) aaa and 3 x 3 aab triplets in the first spin's
    # pass, C(3,2) abb ones in the second's
    assert st["triplets"] == len(s) * 15
    k16 = lambda k: (k + 15) // 16 * 16
    pairs, K = v * (v - 1) // 2, k16(v + n)
    same = 2.0 * v * pairs * 3 * K
    mixed = 2.0 * v * v * v * 3 * K + 2.0 * v * pairs * 2 * K
    want = 6 * (3 * same + 9 * mixed) + (10 if flat else 6) * 3 * mixed
    assert abs(st["tensor_flops"] - len(s) * want) <= 1e-9 * want


@pytest.mark.parametrize("prec", ["bf16x10", "bf16x6", "fp64"])
def test_small_pieces_give_the_same_triplets_and_gradients(lib, prec):
    """What a call does after it ran out of device memory: the triplets' energies are
    the same bit for bit (a triplet is cut into chunks by the domain's shape alone), and
    the gradients agree within the 32-bit operands of their products."""
    dd = lno_ot.to_device(make_domain(100, (8, 6), naux=120, L=40.0, seed=3, t1_sd=0.02))
    n = all_trips(8, 6)
    z = torch.zeros_like
    e, grads = [], []
    for on in (0, 1):
        ctx = lno_ot.Context(0, prec)
        assert lib.lno_ot_selftest_small_pieces(ctx.h, on) == 0
        et = [torch.zeros(x, dtype=torch.float64, device="cuda") for x in n]
        out = ctx.energy(dd, e_trip=et)
        e.append([out["total"]] + [x.cpu().numpy() for x in et])
        g = dict(dB=[z(x) for x in dd["B"]], deps=[z(x) for x in dd["eps"]],
                 dt1=[z(x) for x in dd["t1"]], dt2aa=z(dd["t2aa"]), dt2bb=z(dd["t2bb"]),
                 dt2ab=z(dd["t2ab"]))
        ctx.backward(dd, 1.0, g)
        ctx.close()
        grads.append(g["dB"] + g["deps"] + g["dt1"] + [g["dt2aa"], g["dt2bb"], g["dt2ab"]])
    assert e[0][0] == e[1][0]
    for x, y in zip(e[0][1:], e[1][1:]):
        assert np.array_equal(x, y)
    for x, y in zip(*grads):
        assert float((x - y).abs().max()) <= 1e-7 * float(x.abs().max())


def test_many_triplets_take_little_memory_each(lib):
    """1.27 million triplets of a few virtuals: the contraction problems are on the device a
    window at a time, so a triplet costs its index and its energy (20 bytes, and as much
    again for slack), and those beyond the first window are what they are alone, bit for
    bit and against the float64 path."""
    na, nb = 100, 98
    dd = lno_ot.to_device(make_domain(103, (na, nb), naux=20, L=10.0, seed=4, t1_sd=0.02))
    n = all_trips(na, nb)
    rng = np.random.default_rng(0)
    part = [np.sort(rng.choice(x, x // 5, replace=False)) for x in n]
    pool = PoolHigh()

    def run(prec, sel):
        ctx = lno_ot.Context(0, prec)
        m = n if sel is None else [len(x) for x in sel]
        et = [torch.zeros(x, dtype=torch.float64, device="cuda") for x in m]
        pool.reset()
        ctx.energy(dd, e_trip=et, trip_sel=sel)
        high = pool.high()
        ctx.close()
        return [e.cpu().numpy() for e in et], high

    full, hi_full = run("bf16x10", None)
    some, hi_some = run("bf16x10", part)
    assert hi_full - hi_some <= 40 * (sum(n) - sum(len(x) for x in part))
    for f, s, x in zip(full, some, part):
        assert np.array_equal(f[x], s)
    few = [x[::997] for x in part]
    ref, _ = run("fp64", few)
    for f, r, x in zip(full, ref, few):
        assert np.abs(f[x] - r).max() <= 1e-7 * np.abs(r).max()


@pytest.mark.parametrize("prec,v,n,short", [("bf16x10", 256, (3, 3), 1536),
                                            ("bf16x10", 24, (4, 3), 16384),
                                            ("bf16x15", 24, (4, 3), 16384)])
def test_long_auxiliary_index(prec, v, n, short):
    """Auxiliary bases beyond the lengths whose class sums need no checks (1536 on FP16
    slices, 16384 on BF16 ones): with zero factors there they give the shorter basis's
    energies bit for bit.  Beyond 16384 the adjoint splits its products; its gradients
    agree with the float64 path's within the 32-bit operands."""
    d = make_domain(v + n[0], n, naux=short, L=short / 3, seed=6, t1_sd=0.02)
    e = [e_trips(prec, lno_ot.to_device(d))]
    d["naux"] = short + 40
    d["B"] = [np.concatenate([b, np.zeros((40,) + b.shape[1:])]) for b in d["B"]]
    dd = lno_ot.to_device(d)
    e.append(e_trips(prec, dd))
    assert np.array_equal(e[0], e[1])
    if v > 100:
        return
    g = []
    for p in ("fp64", prec):
        ctx = lno_ot.Context(0, p)
        x = dict(dB=[torch.zeros_like(b) for b in dd["B"]], dt2ab=torch.zeros_like(dd["t2ab"]))
        ctx.backward(dd, 1.0, x)
        ctx.close()
        g.append(x["dB"] + [x["dt2ab"]])
    for x, y in zip(*g):
        assert float((x - y).abs().max()) <= 1e-7 * float(x.abs().max())


@pytest.mark.parametrize("prec", ["bf16x10", "fp64"])
def test_every_bound_above_the_smallest_is_accepted(prec):
    """Rows are packed tightly only where the wide ones (and the lists that the orbital
    contributions take afterwards) do not fit: no bound in between is refused, and the
    results are the same bit for bit."""
    dd = lno_ot.to_device(make_domain(40, (12, 10), naux=41, L=15.0, seed=5))

    def run(bound):
        ctx = lno_ot.Context(0, prec, workspace_bytes=bound)
        orb = [torch.zeros(n, dtype=torch.float64, device="cuda") for n in (12, 10)]
        out = ctx.energy(dd, raise_on_error=False, e_orb=orb)
        ctx.close()
        return out["total"] if out["status"] == lno_ot.OK else None

    want = run(0)
    lo, hi = 256, 64 << 20
    while hi - lo > 256:
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if run(mid) is not None else (mid, hi)
    for bound in np.linspace(hi, 2.2 * hi, 60).astype(int):
        assert run(int(bound)) == want, bound
