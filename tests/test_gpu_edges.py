"""Inputs at the edges of what the entry points accept: factors whose sums over the
auxiliary index are large in every slice, sizes at a launch's limits, bounded and
nearly full memory."""
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
