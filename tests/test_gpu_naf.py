"""NAF compression on the GPU (lno_ot_naf, Sec. 3.6, eq naf_w) against the
oracle: the eigenvalues of W, the number of kept NAFs, the compressed factors
up to the sign of each NAF, and E(T) of the compressed domain (float64 path),
for thresholds that keep everything, about half, and few NAFs."""
import numpy as np
import pytest
import torch

from oracle import naf as N
from oracle import triples as T
from paper_2311_10048_gb300 import lno_ot
from paper_2311_10048_gb300.synth import config_domain, make_domain

pytestmark = pytest.mark.gpu


def sign_fixed(B):
    """Each NAF block times the sign of its largest-magnitude element."""
    B = np.array(B)
    flat = B.reshape(B.shape[0], -1)
    idx = np.abs(flat).argmax(axis=1)
    return B * np.sign(flat[np.arange(len(idx)), idx])[:, None, None]


CASES = [("small", dict(nbas=14, nocc=(4, 2), naux=40, L=6.0, seed=3), (0.0, 1e-3, 1e-1)),
         ("c0", None, (1e-2, 1.0))]


@pytest.mark.parametrize("name,kw,epss", CASES)
def test_naf_matches_oracle(lib, name, kw, epss):
    d = config_domain("c0") if kw is None else make_domain(t1_sd=0.02, **kw)
    dd = lno_ot.to_device(d)
    ctx = lno_ot.Context(0, "fp64")
    for eps in epss:
        lam_ref, V, Bu, Bd = N.naf(d["B"][0], d["B"][1], eps)
        comp, lam = ctx.naf(dd, eps)
        np.testing.assert_allclose(lam, lam_ref, rtol=0, atol=1e-12 * lam_ref[0])
        assert comp["naux"] == V.shape[1]
        for s, ref in ((0, Bu), (1, Bd)):
            got = comp["B"][s].cpu().numpy()
            np.testing.assert_allclose(sign_fixed(got), sign_fixed(ref), rtol=0,
                                       atol=1e-11 * np.abs(ref).max())
        e_gpu = ctx.energy(comp)["total"]
        oc, _ = N.compressed_domain(d, eps)
        e_ref = T.energy(oc)["total"]
        assert abs(e_gpu - e_ref) <= 1e-10 * abs(e_ref), (eps, e_gpu, e_ref)
    ctx.close()


@pytest.mark.parametrize("n,naux", [(7, 5), (9, 33), (18, 47), (33, 130)])
def test_naf_of_odd_sizes_and_of_asymmetric_factors(n, naux):
    """Odd auxiliary counts (padded rotations), and factors that are not symmetric
    in (p, q): W takes p <= q, the compression every element."""
    rng = np.random.default_rng(n)
    B = [rng.normal(size=(naux, n, n)) * np.exp(-3 * np.arange(naux) / naux)[:, None, None]
         for _ in range(2)]
    for sym in (True, False):
        b = [np.triu(x) + np.triu(x, 1).transpose(0, 2, 1) if sym else x for x in B]
        iu = np.triu_indices(n)
        j = [x[:, iu[0], iu[1]] for x in b]
        lam, vec = np.linalg.eigh((j[0] @ j[0].T + j[1] @ j[1].T) / 2)
        lam, vec = lam[::-1], vec[:, ::-1]
        eps = float(np.sqrt(lam[naux // 2] * lam[naux // 2 + 1]))
        d = lno_ot.to_device(dict(make_domain(n, (2, 1), naux=naux, L=naux / 3, seed=1), B=b))
        ctx = lno_ot.Context(0, "fp64")
        out, got = ctx.naf(d, eps)
        ctx.close()
        assert np.abs(got - lam).max() <= 1e-12 * lam[0]
        assert out["naux"] == naux // 2 + 1
        for s in (0, 1):
            want = np.einsum("Xk,Xpq->kpq", vec[:, :out["naux"]], b[s])
            # eigenvectors to ~1e-15 over the relative gaps (>= 1e-5 in these draws)
            assert np.abs(sign_fixed(out["B"][s].cpu().numpy()) - sign_fixed(want)).max() \
                <= 1e-8 * np.abs(want).max()
