"""W contraction on CTA pairs (csrc/tc_pair.cu) at the edges of its tiles.

Per-triplet energies of a few triplets per case against the float64 path of
the library (itself pinned to the oracle elsewhere), for virtual counts around
one and two n-tiles of each slice count, row counts around 256-row tiles, k
lengths around the 32-element blocks, and tuned tile caps.

Tolerances: the slices of a precision with S slices of 8 bits leave 2^(-8 S)
of the largest operand product per term, and the float32 rounding of the W
intermediates and of the energy sums leaves ~1e-9 of a triplet's energy for
the smallest virtual spaces here; 16 (S = 2), 24 (S = 3) and >= 32 bits give
1e-3, 1e-6 and 2e-8 relative to the largest triplet energy with a margin of at
least 4 over the worst per-triplet errors the larger suites see."""
import numpy as np
import pytest
import torch

from paper_2311_10048_gb300 import lno_ot
from paper_2311_10048_gb300.synth import make_domain

pytestmark = pytest.mark.gpu
TOL = {"bf16x3": 1e-3, "tf32": 1e-3, "bf16x6": 1e-6, "bf16x10": 2e-8, "bf16x15": 2e-8}


def e_trips(prec, dd, sel, tune=None):
    ctx = lno_ot.Context(0, prec, tune_cache=tune)
    et = [torch.zeros(max(x.size, 1), dtype=torch.float64, device="cuda") for x in sel]
    ctx.energy(dd, e_trip=et, trip_sel=sel)
    ctx.close()
    return np.concatenate([e[:x.size].cpu().numpy() for e, x in zip(et, sel)])


def sample(na, nb):
    n = [na * (na - 1) * (na - 2) // 6, na * (na - 1) // 2 * nb, nb * (nb - 1) // 2 * na,
         nb * (nb - 1) * (nb - 2) // 6]
    return [np.unique(np.array([0, x // 2, x - 1]) if x else np.zeros(0)).astype(np.int64)
            for x in n]


@pytest.mark.parametrize("v,na,nb", [(15, 4, 3), (16, 4, 4), (23, 5, 4), (33, 3, 3), (65, 4, 3),
                                     (80, 3, 3), (81, 4, 3), (97, 5, 3), (128, 4, 3),
                                     (129, 3, 3), (160, 4, 4), (161, 3, 3), (257, 3, 3)])
def test_tile_edges(v, na, nb):
    d = make_domain(v + na, (na, nb), naux=v + na + 5, L=(v + na) / 3, seed=100 + v, t1_sd=0.02)
    dd = lno_ot.to_device(d)
    sel = sample(na, nb)
    ref = e_trips("fp64", dd, sel)
    for prec, tol in TOL.items():
        got = e_trips(prec, dd, sel)
        assert np.abs(got - ref).max() <= tol * np.abs(ref).max(), prec


@pytest.mark.parametrize("cap", [16, 48, 80])
def test_tile_caps_are_bitwise_equal(tmp_path, cap):
    d = make_domain(101, (4, 3), naux=90, L=30.0, seed=9, t1_sd=0.02)
    dd = lno_ot.to_device(d)
    sel = sample(4, 3)
    p = tmp_path / "t.txt"
    p.write_text(f"100000 {cap} 3\n")
    for prec in ("bf16x3", "bf16x6", "bf16x10", "bf16x15"):
        assert np.array_equal(e_trips(prec, dd, sel, str(p)), e_trips(prec, dd, sel)), prec


@pytest.mark.parametrize("off", [0.0, 2e-3, -2e-3, 0.02, -0.02])
def test_integral_scale_near_a_power_of_two(off):
    """The integral scale is measured on two slices of the DF factors and settled
    in full when the largest integral is within 1% of a power of two."""
    d = make_domain(26, (4, 3), naux=40, L=14.0, seed=31, t1_sd=0.02)
    va, vb = 22, 23
    m = 0.0
    for s, o in ((0, 4), (1, 3)):
        for t, p in ((0, 4), (1, 3)):
            g = np.einsum("Qab,Qic->abic", d["B"][s][:, o:, o:], d["B"][t][:, :p, p:])
            h = np.einsum("Qij,Qka->ijka", d["B"][s][:, :o, :o], d["B"][t][:, :p, p:])
            m = max(m, np.abs(g).max(), np.abs(h).max())
    f = np.sqrt(2.0 ** np.ceil(np.log2(2 * m)) * (1 + off) / (2 * m))
    d["B"] = [b * f for b in d["B"]]
    dd = lno_ot.to_device(d)
    sel = sample(4, 3)
    ref = e_trips("fp64", dd, sel)
    for prec in ("bf16x10", "bf16x15", "bf16x6"):
        assert np.abs(e_trips(prec, dd, sel) - ref).max() <= TOL[prec] * np.abs(ref).max(), prec


@pytest.mark.parametrize("key", ["B", "t2aa", "t2ab"])
def test_nan_reaches_the_energy(key):
    d = make_domain(20, (4, 3), naux=30, L=10.0, seed=8)
    dd = lno_ot.to_device(d)
    x = dd["B"][0] if key == "B" else dd[key]
    x.view(-1)[x.numel() // 2 + 3] = float("nan")
    for prec in ("fp64", "bf16x6", "bf16x10"):
        ctx = lno_ot.Context(0, prec)
        assert np.isnan(ctx.energy(dd)["total"]), prec
        ctx.close()


@pytest.mark.parametrize("kind", ["plain", "B", "t2", "occupied"])
def test_fp16_slices_and_their_fallback(kind):
    """BF16X10 on FP16 slices (256 virtuals, or 160 with 8 occupied), and the data
    for which their leading sums are not provably exact: DF factors (or doubles)
    all near the largest magnitude, which run on the BF16 slices."""
    v, na, nb = (160, 8, 8) if kind == "occupied" else (256, 3, 3)
    d = make_domain(v + na, (na, nb), naux=150, L=50.0, seed=77, t1_sd=0.02)
    rng = np.random.default_rng(1)
    if kind == "B":
        d["B"] = [np.where(b < 0, -1.0, 1.0) * rng.uniform(0.09, 0.1) for b in d["B"]]
    if kind == "t2":
        for k in ("t2aa", "t2bb", "t2ab"):
            d[k] = np.sign(d[k]) * 0.03
    dd = lno_ot.to_device(d)
    sel = sample(na, nb)
    ref = e_trips("fp64", dd, sel)
    assert np.abs(e_trips("bf16x10", dd, sel) - ref).max() <= TOL["bf16x10"] * np.abs(ref).max()
    ctx = lno_ot.Context(0, "bf16x10", keep_operands=True)
    for _ in range(2):
        et = [torch.zeros(max(x.size, 1), dtype=torch.float64, device="cuda") for x in sel]
        ctx.energy(dd, e_trip=et, trip_sel=sel)
        got = np.concatenate([e[:x.size].cpu().numpy() for e, x in zip(et, sel)])
        assert np.abs(got - ref).max() <= TOL["bf16x10"] * np.abs(ref).max()
    ctx.close()


@pytest.mark.parametrize("prec,nbas,na,nb,naux,limit", [
    ("bf16x10", 33, 5, 3, 67, 1139968), ("bf16x15", 33, 5, 3, 67, 1420800),
    ("tf32", 40, 6, 4, 120, 2758912), ("fp64", 40, 6, 4, 120, 2749696)])
def test_workspace_bound_counts_the_data_not_the_pitch(prec, nbas, na, nb, naux, limit):
    """workspace_bytes that held a domain when its rows were padded to 16 bytes holds
    it with 64-byte rows (the smallest accepted bounds of that layout)."""
    dd = lno_ot.to_device(make_domain(nbas, (na, nb), naux=naux, L=15.0, seed=5))
    e = []
    for bound in (limit, 0):
        ctx = lno_ot.Context(0, prec, workspace_bytes=bound)
        e.append(ctx.energy(dd)["total"])
        ctx.close()
    assert e[0] == e[1]


def test_naf_workspace_bound():
    dd = lno_ot.to_device(make_domain(24, (4, 3), naux=100, L=15.0, seed=5))
    lam = []
    for bound in (1160704, 0):
        ctx = lno_ot.Context(0, "fp64", workspace_bytes=bound)
        lam.append(ctx.naf(dd)[1])
        ctx.close()
    assert np.array_equal(lam[0], lam[1])
