"""The resident evolution (csrc/resident.cu) against the oracle's directly recorded moments.

One case per way a realization is laid out: tiles below one CTA's least size, one CTA, clusters of
2 to 8 CTAs, CTAs on a counter barrier; every block size; with and without the global flip; and the
start vectors and couplings the fixed-point form hands to the floating-point kernels.

Tolerance, from the recurrence: an order adds a rounding error of norm at most (N + 8) u to w_k
(N + 2 products and sums, one store), u = 2^-53 for float64 and 2^-44 for double-float; an error made
at order j reaches order k through U_{k-j}(G), of norm at most k - j + 1; and mu_j comes from products
of two such vectors, doubled. With n orders that is at most 4 (N + 8) u n^2; the reference adds as much.
"""

import numpy as np
import pytest

import workloads as W
from oracle import dacp as DA
from oracle import hamiltonian as Hm

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
P = pytest.importorskip("paper_2011_02107_gb300")


def _bound(m):
    return float(np.abs(Hm.diagonal(m)).max() + np.abs(m["gamma"]).sum() + abs(m.get("gflip", 0.0)))


def _check(models, psis, b, orders, prec, unit, emax=None):
    emax = np.array([_bound(m) for m in models]) if emax is None else emax
    n = max(1, int(orders * 0.2 / np.pi))                 # a = 0.2 E_max: k_n = floor(n pi / 0.2)
    d = P.Dacp(models, psis, block_b=b, precision=prec)
    try:
        d.set_params(emax, 0.2 * emax, 0, n)              # K = 0: psi_E is the start block, normalised
        d.filter()
        d.basis_moments()
        kn = d.params()["kn"]
        for r, m in enumerate(models):
            mu = d.moments(r)
            ref, _ = DA.chebyshev_moments(m, d.filtered(r), emax[r], mu.shape[0] - 1)
            ref = 0.5 * (ref + ref.transpose(0, 2, 1))
            tol = 8 * (m["N"] + 8) * unit * (kn[r] + 2) ** 2
            err = np.abs(mu - ref).max()
            assert err <= tol, (r, m["N"], err, tol)
    finally:
        d.close()


def _flip(m, c):
    return dict(m, gflip=c)


PRECS = [("fp64", P.DACP_FP64, 2.0 ** -53), ("df32", P.DACP_DF32, 2.0 ** -44)]


@pytest.mark.parametrize("name,prec,unit", PRECS)
@pytest.mark.parametrize("flip", [False, True])
@pytest.mark.parametrize("b", [1, 2, 4])
@pytest.mark.parametrize("Ns", [(1, 2, 3, 4), (5, 9, 12, 7, 10), (6, 6), (13,), (8,)])
def test_resident_evolution_on_small_batches(Ns, b, flip, name, prec, unit):
    models = [W.random_model(N, seed=70 + i) for i, N in enumerate(Ns)]
    if flip:
        models = [_flip(m, 0.41 * (-1) ** i) for i, m in enumerate(models)]
    psis = [W.start_vectors(N, b, seed=3, r=i) for i, N in enumerate(Ns)]
    _check(models, psis, b, 40, prec, unit)


@pytest.mark.parametrize("name,prec,unit", PRECS)
@pytest.mark.parametrize("N,b,count", [(14, 4, 2), (13, 4, 40), (16, 2, 1), (16, 4, 1), (15, 1, 1)])
def test_resident_evolution_over_many_ctas(N, b, count, name, prec, unit):
    models = [_flip(W.spin_glass_shard(N, seed=5 + r), 0.3) for r in range(count)]
    psis = [W.start_vectors(N, b, seed=4, r=r) for r in range(count)]
    _check(models, psis, b, 24, prec, unit)


@pytest.mark.parametrize("name,prec,unit", PRECS)
@pytest.mark.parametrize("N", [6, 11])
def test_start_vectors_of_one_state_and_of_uneven_size(N, name, prec, unit):
    """A basis state (all the norm in one element), a smooth vector with elements down to 1e-30, and an
    ordinary block in one batch: those the fixed point does not suit go through the other kernels."""
    one = np.zeros((1 << N, 2))
    one[3, 0] = one[5, 1] = 1.0
    decay = np.exp(-np.arange(1 << N) * 69.0 / (1 << N))[:, None] * np.array([[1.0, -1.0]])
    decay[::2, 1] *= 0.5
    models = [W.random_model(N, seed=80 + i) for i in range(3)]
    _check(models, [one, W.start_vectors(N, 2, seed=6), decay], 2, 30, prec, unit)


@pytest.mark.parametrize("flip", [False, True])
@pytest.mark.parametrize("N,tile", [(13, 32768), (14, 65536)])
def test_double_float_clusters_keep_the_bits_of_the_per_order_launch(N, tile, flip):
    """16 realizations of 8 tiles take the per-order launch, the first two of them alone a cluster each: their
    moments equal to the last bit."""
    models = [W.spin_glass_shard(N, seed=20 + r) for r in range(16)]
    if flip:
        models = [_flip(m, 0.7 - 0.01 * r) for r, m in enumerate(models)]
    psis = [W.start_vectors(N, 4, seed=8, r=r) for r in range(16)]
    emax = np.array([_bound(m) for m in models])
    mu = []
    for count in (16, 2):
        d = P.Dacp(models[:count], psis[:count], block_b=4, precision=P.DACP_DF32)
        try:
            d.set_launch(0, tile)
            d.set_params(emax[:count], 0.1 * emax[:count], 5, 2 + np.arange(count) % 2)
            d.filter()
            d.basis_moments()
            mu.append([d.moments(r) for r in range(2)])
        finally:
            d.close()
    for a, b in zip(*mu):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("flip", [False, True])
@pytest.mark.parametrize("N", [10, 11, 12, 13])
def test_kpm_moments_of_one_cta_keep_the_bits_of_the_per_order_launch(N, flip):
    """A 14-spin realization beside it takes the whole batch through the per-order launches: the parameters and
    the features, which hold 32 of the moments, of the smaller one are equal to the last bit."""
    models = [W.spin_glass_shard(n, seed=30 + n) for n in (N, 14)]
    if flip:
        models = [_flip(m, 0.6 - 0.1 * r) for r, m in enumerate(models)]
    psis = [W.start_vectors(m["N"], 4, seed=9, r=r) for r, m in enumerate(models)]
    out = []
    for count in (1, 2):
        d = P.Dacp(models[:count], psis[:count], block_b=4, precision=P.DACP_DF32)
        try:
            d.choose_params(20)
            p = d.params()
            out.append([np.asarray(p["a"])[0], np.asarray(p["emax"])[0], np.asarray(d.features())[0]])
        finally:
            d.close()
    assert all(np.array_equal(x, y) for x, y in zip(*out))


@pytest.mark.parametrize("name,prec,unit", PRECS)
def test_bound_far_below_the_radius_is_reported_as_before(name, prec, unit):
    """Coefficients beyond the limbs, and vectors that outgrow the fixed point, end as DACP_ERR_NUMERIC."""
    m = W.chain(9)
    for shrink in (0.02, 0.6):
        em = shrink * np.abs(np.linalg.eigvalsh(Hm.dense_h(m))).max()
        d = P.Dacp([m, m], [W.start_vectors(9, 2, seed=0, r=r) for r in range(2)], block_b=2, precision=prec)
        try:
            d.set_params(em, 0.3 * em, 0, 8)
            d.filter()
            d.basis_moments()
            assert (d.central_eigs(4)[1] == -4).all()
        finally:
            d.close()


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("b,Ns", [(1, (1, 3, 8, 14, 17)), (2, (2, 9, 12, 16)), (4, (1, 5, 10, 13, 15, 18)), (4, (11,))])
def test_apply_h_on_the_default_tiles(Ns, b, prec):
    """Default tiles shrink with the batch (float64) and the vector (float32): every element within a rounding
    per term, N flips, the global flip and the diagonal (itself summed from N (N + 1) / 2 terms), taken four
    times, of the sum of the magnitudes."""
    torch = pytest.importorskip("torch")
    models = [_flip(W.random_model(N, seed=90 + i), 0.3 * (i % 2)) for i, N in enumerate(Ns)]
    psis = [W.start_vectors(N, b, seed=13, r=i) for i, N in enumerate(Ns)]
    f32 = prec == "fp32"
    d = P.Dacp(models, psis, block_b=b, precision=P.DACP_FP32 if f32 else P.DACP_FP64)
    try:
        for r, m in enumerate(models):
            N = m["N"]
            xd = torch.from_numpy(np.ascontiguousarray(W.start_vectors(N, b, seed=14, r=r))).cuda()
            xd = xd.float() if f32 else xd.double()
            yd = torch.zeros_like(xd)
            d.apply_h(r, xd.data_ptr(), yd.data_ptr())
            x = xd.double().cpu().numpy()
            ref, scale = Hm.apply_h_rows(m, x, np.arange(1 << N), with_abs=True)
            dscale = (np.abs(np.triu(m["J"], 1)).sum() + np.abs(m["h"]).sum()) * np.abs(x)
            tol = 4 * ((N + 4) * 2.0 ** (-24 if f32 else -53) * scale + (N * (N + 1) // 2 + 1) * 2.0 ** -53 * dscale)
            assert (np.abs(yd.double().cpu().numpy() - ref) <= tol).all(), (r, N)
    finally:
        d.close()


@pytest.mark.parametrize("flip", [False, True])
@pytest.mark.parametrize("b", [1, 2, 4])
@pytest.mark.parametrize("Ns", [(3, 5, 13), (6, 9, 12, 7, 10)])
def test_uneven_batches_have_the_moments_of_each_realization_alone(Ns, b, flip):
    """Realizations with fewer slots than their CTA has threads, beside larger ones: the sums are exact integers, so
    neither the number of CTAs nor that of threads shows in the moments, and none is declined (one launch)."""
    models = [W.random_model(N, seed=110 + i) for i, N in enumerate(Ns)]
    if flip:
        models = [_flip(m, 0.37 * (-1) ** i) for i, m in enumerate(models)]
    psis = [W.start_vectors(N, b, seed=15, r=i) for i, N in enumerate(Ns)]

    def moments(at):
        emax = np.array([_bound(models[i]) for i in at])
        d = P.Dacp([models[i] for i in at], [psis[i] for i in at], block_b=b, precision=P.DACP_FP64)
        try:
            d.set_params(emax, 0.2 * emax, 0, 12)
            d.filter()
            before = d.launch_count()
            d.basis_moments()
            assert d.launch_count() == before + 1
            return [d.moments(r) for r in range(len(at))]
        finally:
            d.close()

    for i, mu in enumerate(moments(range(len(Ns)))):
        assert np.array_equal(mu, moments([i])[0]), Ns[i]


@pytest.mark.parametrize("b", [1, 2, 4])
@pytest.mark.parametrize("N,flip", [(6, 0.0), (9, 0.0), (10, 0.4), (13, 0.0), (14, -0.3)])
def test_even_start_vectors_stay_in_fixed_point(N, flip, b):
    """Starts whose elements are all alike in size concentrate under the evolution and outgrow the first scale: the
    uniform product state, random signs and a constant with one sign changed. The run starts again with more room
    (one launch more), never in floating point (a launch per order)."""
    D = 1 << N
    rng = np.random.default_rng(N)
    cols = np.stack([np.ones(D), rng.choice([-1.0, 1.0], D), np.where(np.arange(D) == D // 3, -1.0, 1.0),
                     rng.choice([-1.0, 1.0], D)], axis=1)[:, :b]
    models = [dict(W.chain(N), gflip=flip), _flip(W.spin_glass_shard(N, seed=160), flip)]
    emax = np.array([_bound(m) for m in models])
    d = P.Dacp(models, [cols, cols], block_b=b, precision=P.DACP_FP64)
    try:
        d.set_params(emax, 0.2 * emax, 0, 19)             # 298 orders
        d.filter()
        before = d.launch_count()
        d.basis_moments()
        assert d.launch_count() == before + 2
        kn = d.params()["kn"]
        for r, m in enumerate(models):
            mu = d.moments(r)
            ref, _ = DA.chebyshev_moments(m, d.filtered(r), emax[r], mu.shape[0] - 1)
            ref = 0.5 * (ref + ref.transpose(0, 2, 1))
            assert np.abs(mu - ref).max() <= 8 * (N + 8) * 2.0 ** -53 * (kn[r] + 2) ** 2, r
    finally:
        d.close()


@pytest.mark.parametrize("b", [1, 4])
def test_declined_realizations_run_side_by_side(b):
    """Basis states (declined by the fixed point) beside ordinary blocks: one launch per order for all of them
    together, as many as the longest takes, and nothing of the others' rows is touched."""
    Ns = (10, 9, 11, 8, 12, 10)
    declined = (0, 2, 3, 4)
    models = [W.random_model(N, seed=170 + i) for i, N in enumerate(Ns)]
    psis = [W.start_vectors(N, b, seed=18, r=i) for i, N in enumerate(Ns)]
    for r in declined:
        psis[r] = np.zeros_like(psis[r])
        psis[r][3 + np.arange(b), np.arange(b)] = 1.0
    emax = np.array([_bound(m) for m in models])
    n = 4 + 2 * np.arange(len(Ns))
    out = []
    for at in (range(len(Ns)), [1], [5]):
        d = P.Dacp([models[i] for i in at], [psis[i] for i in at], block_b=b, precision=P.DACP_FP64)
        try:
            d.set_params(emax[at], 0.2 * emax[at], 0, n[at])
            d.filter()
            before = d.launch_count()
            d.basis_moments()
            kn = d.params()["kn"]
            longest = max([kn[r] + 2 for r in declined], default=0) if len(at) > 1 else 0
            assert d.launch_count() == before + 1 + longest
            out.append([d.moments(r) for r in range(len(at))])
            if len(at) > 1:
                for r in declined:
                    ref, _ = DA.chebyshev_moments(models[r], d.filtered(r), emax[r], out[0][r].shape[0] - 1)
                    ref = 0.5 * (ref + ref.transpose(0, 2, 1))
                    tol = 8 * (Ns[r] + 8) * 2.0 ** -53 * (kn[r] + 2) ** 2
                    assert np.abs(out[0][r] - ref).max() <= tol, r
        finally:
            d.close()
    assert np.array_equal(out[0][1], out[1][0]) and np.array_equal(out[0][5], out[2][0])


def test_window_of_declined_start_vectors():
    """The 256 kernel-polynomial moments of a basis state come from the floating-point kernels, 128 launches for the
    batch; the window agrees with the oracle's. An error e of the moments, at most 8 (N + 8) u 128^2 = 2.6e-10, moves
    the level count by D e sum_j 4 / (pi j) < 2.1e-6 of 40, and the window by as much of itself."""
    from oracle import params as OP
    N, R = 10, 3
    models = [W.spin_glass_shard(N, seed=180 + r) for r in range(R)]
    one = np.zeros((1 << N, 2))
    one[7, 0] = one[8, 1] = 1.0
    launches, p = [], None
    for psis in ([one] * R, [W.start_vectors(N, 2, seed=19, r=r) for r in range(R)]):
        d = P.Dacp(models, psis, block_b=2, precision=P.DACP_FP64)
        try:
            before = d.launch_count()
            d.choose_params(20)
            launches.append(d.launch_count() - before)
            p = p or d.params()
        finally:
            d.close()
    assert launches[0] == launches[1] + 128
    for r, m in enumerate(models):
        mu = OP.kpm_moments(m, one[:, 0], p["emax"][r], 256)
        assert abs(p["a"][r] / OP.kpm_window(mu, 1 << N, p["emax"][r], 40.0) - 1.0) < 1e-7, r


@pytest.mark.parametrize("flip", [False, True])
@pytest.mark.parametrize("Ns,tile", [((11, 13, 12, 13, 11, 12, 11), 65536), ((10, 12, 11, 13, 10), 32768),
                                     ((11, 14, 12), 65536), ((12,) * 9, 65536)])
def test_double_float_clusters_of_every_size_keep_the_bits(Ns, tile, flip):
    """One launch per size, in clusters of as many CTAs as it has tiles, against the per-order launch, which 16
    realizations with one of 8 tiles among them take: filtered vectors and moments equal to the last bit, runs of
    unequal length."""
    big = {65536: 14, 32768: 13}[tile]
    sizes = Ns + (big,) * (16 - len(Ns))
    models = [W.spin_glass_shard(N, seed=190 + r) for r, N in enumerate(sizes)]
    if flip:
        models = [_flip(m, 0.5 - 0.07 * r) for r, m in enumerate(models)]
    psis = [W.start_vectors(N, 4, seed=20, r=r) for r, N in enumerate(sizes)]
    emax = np.array([_bound(m) for m in models])
    K, n = 5 + np.arange(16) % 3, 2 + np.arange(16) % 2
    out = []
    for count in (len(Ns), 16):
        d = P.Dacp(models[:count], psis[:count], block_b=4, precision=P.DACP_DF32)
        try:
            d.set_launch(0, tile)
            d.set_params(emax[:count], 0.1 * emax[:count], K[:count], n[:count])
            d.filter()
            before = d.launch_count()
            d.basis_moments()
            launches = len(set(Ns)) if count == len(Ns) else max(d.params()["kn"]) + 2
            assert d.launch_count() == before + launches
            out.append([d.filtered(r) for r in range(len(Ns))] + [d.moments(r) for r in range(len(Ns))])
        finally:
            d.close()
    for x, y in zip(*out):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("N,R", [(13, 8), (11, 36)])
def test_autotuner_weighs_the_resident_launch(N, R):
    """A few double-float realizations run twice as fast in clusters as with a launch per order: tuned or not, they
    take them, and the tuner leaves run lengths and parameters as they were."""
    models = [W.spin_glass_shard(N, seed=210 + r) for r in range(R)]
    psis = [W.start_vectors(N, 4, seed=21, r=r) for r in range(R)]
    emax = np.array([_bound(m) for m in models])
    d = P.Dacp(models, psis, block_b=4, precision=P.DACP_DF32)
    try:
        d.set_params(emax, 0.05 * emax, 7, 6)                 # 378 orders
        moments = []
        for tune in (False, True):
            if tune:
                d.autotune(64)
            d.filter()
            before = d.launch_count()
            d.basis_moments()
            assert d.launch_count() == before + 1
            moments.append([d.moments(r) for r in range(R)])
        for x, y in zip(*moments):
            assert x.shape == y.shape and np.abs(x - y).max() <= 8 * (N + 8) * 2.0 ** -44 * 378 ** 2
    finally:
        d.close()


@pytest.mark.parametrize("b,N", [(4, 10), (1, 13), (4, 13)])
def test_a_tile_size_that_the_caller_sets_is_the_one_in_use(N, b):
    """Small float64 handles start with smaller tiles than 64 KB, and say so; 64 KB are 64 KB when asked for.
    The filtered vectors do not depend on the tiles, but for the sum of their norm."""
    m = W.chain(N)
    psi = W.start_vectors(N, b, seed=22)
    d = P.Dacp([m], [psi], block_b=b, precision=P.DACP_FP64)
    try:
        first = d.launch()
        assert first == (0, 8192)
        emax = np.array([_bound(m)])
        d.set_params(emax, 0.2 * emax, 6, 2)
        ref = None
        for tile in (first[1], 65536, 16384, 65536):
            d.set_launch(0, tile)
            assert d.launch() == (0, tile)
            d.filter()
            ref = d.filtered(0) if ref is None else ref
            assert np.abs(d.filtered(0) - ref).max() <= 1e-14       # normalised; the norm's sum is regrouped
    finally:
        d.close()


def test_a_barrier_that_ran_out_is_named():
    m = W.spin_glass_shard(9, seed=1)
    d = P.Dacp([m], [W.start_vectors(9, 1, seed=2)], block_b=1, precision=P.DACP_FP32)
    try:
        d.set_params(_bound(m), 0.2 * _bound(m), 4, 2)
        d.set_launch(1, 2048)
        P.dacp_test_poison_barrier(d.handle)
        with pytest.raises(P.DacpError, match="barrier") as e:
            d.filter()
        assert e.value.status == 5
    finally:
        d.close()


@pytest.mark.parametrize("b", [1, 2, 4])
@pytest.mark.parametrize("bits,N", [(9, 9), (9, 12), (10, 11), (10, 13), (11, 13)])
def test_kpm_moments_keep_the_bits_at_every_tile_size(bits, N, b):
    """As above for tiles of 2^9 to 2^11 states, one to eight of them, and every block size."""
    models = [_flip(W.spin_glass_shard(n, seed=220 + n), 0.3) for n in (N, 14)]
    psis = [W.start_vectors(m["N"], b, seed=23, r=r) for r, m in enumerate(models)]
    out = []
    for count in (1, 2):
        d = P.Dacp(models[:count], psis[:count], block_b=b, precision=P.DACP_DF32)
        try:
            d.set_launch(0, (8 * b) << bits)
            before = d.launch_count()
            d.choose_params(12)
            p = d.params()
            out.append([d.launch_count() - before, np.asarray(p["a"])[0], np.asarray(p["emax"])[0],
                        np.asarray(d.features())[0]])
        finally:
            d.close()
    assert out[1][0] == out[0][0] + 127                   # 128 per-order launches in the place of one
    assert all(np.array_equal(x, y) for x, y in zip(out[0][1:], out[1][1:]))
