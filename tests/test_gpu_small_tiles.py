"""Tiles below 8 KB (dacp_set_launch takes them down to 1 KB): more partial sums than at the default tiles.

Moments of every precision, with and without pair couplings, against the oracle, and the parameter choice (Lanczos
sums and kernel-polynomial moments over the same tiles) against 8 KB tiles. Tolerances as derived in
test_gpu_resident: 8 (N + 8) u (orders)^2 for the moments, u = 2^-24 for float32; pairs add N (N - 1) / 2 products.
"""

import numpy as np
import pytest

import workloads as W
from oracle import dacp as DA
from oracle import hamiltonian as Hm

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
P = pytest.importorskip("paper_2011_02107_gb300")

PRECS = [("fp64", P.DACP_FP64, 2.0 ** -53), ("fp32", P.DACP_FP32, 2.0 ** -24), ("df32", P.DACP_DF32, 2.0 ** -44)]


@pytest.mark.parametrize("name,prec,unit", PRECS)
@pytest.mark.parametrize("pairs", [False, True])
@pytest.mark.parametrize("b", [1, 4])
@pytest.mark.parametrize("tile", [1024, 2048, 4096])
def test_moments_on_small_tiles(tile, b, pairs, name, prec, unit):
    Ns = (12, 9, 11)
    models = [W.random_model(N, seed=140 + i) for i, N in enumerate(Ns)]
    if pairs:
        rng = np.random.default_rng(7)
        models = [dict(m, Jxx=np.triu(rng.uniform(-0.3, 0.3, m["J"].shape), 1),
                       Jyy=np.triu(rng.uniform(-0.3, 0.3, m["J"].shape), 1)) for m in models]
    psis = [W.start_vectors(N, b, seed=16, r=i) for i, N in enumerate(Ns)]
    emax = np.array([Hm.pauli_norm_bound(m) for m in models])
    d = P.Dacp(models, psis, block_b=b, precision=prec)
    try:
        d.set_launch(0, tile)
        d.set_params(emax, 0.3 * emax, 0, 3)
        d.filter()
        d.basis_moments()
        kn = d.params()["kn"]
        for r, m in enumerate(models):
            mu = d.moments(r)
            ref, _ = DA.chebyshev_moments(m, d.filtered(r), emax[r], mu.shape[0] - 1)
            ref = 0.5 * (ref + ref.transpose(0, 2, 1))
            terms = m["N"] + 8 + (m["N"] * (m["N"] - 1) // 2 if pairs else 0)
            assert np.abs(mu - ref).max() <= 8 * terms * unit * (kn[r] + 2) ** 2, (r, m["N"])
    finally:
        d.close()


@pytest.mark.parametrize("name,prec,unit", PRECS)
def test_parameters_on_small_tiles(name, prec, unit):
    """E_max from 20 Lanczos steps and the window: the same sums in another partition."""
    models = [W.spin_glass_shard(N, seed=150 + N) for N in (12, 10)]
    psis = [W.start_vectors(m["N"], 4, seed=17, r=r) for r, m in enumerate(models)]
    out = []
    for tile in (8192, 1024):
        d = P.Dacp(models, psis, block_b=4, precision=prec)
        try:
            d.set_launch(0, tile)
            d.choose_params(20)
            out.append(d.params())
        finally:
            d.close()
    tol = 1e-3 if name == "fp32" else 1e-9
    for key in ("emax", "a"):
        assert np.allclose(out[0][key], out[1][key], rtol=tol, atol=0), key
