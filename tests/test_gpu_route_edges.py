"""Kernels behind a rule on sizes, at the sizes where a rule changes its mind.

Tolerances as for the pass variants: an FFT line of 1024 points has 10 radix-2 levels of at
most about 1.5 * 2^-24 in the 2-norm, two axes 1.8e-6 if all errors added up: 2e-6;
interpolation and gridding about eight roundings of 2^-24 per contribution: 1e-6.
"""
import numpy as np
import pytest

import oracle
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL_FFT = 2e-6
TOL_V = 1e-6
TOL_OP = TOL_FFT + TOL_V


@pytest.fixture(scope="module")
def nf():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1710_03197_gb300 as nf
    return nf


def rel(a, b):
    return float(np.linalg.norm(np.ravel(a) - np.ravel(b)) / np.linalg.norm(b))


def cn(shape, seed):
    rng = np.random.default_rng(seed)
    return (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).astype(np.complex64)


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


# strided lines that are no powers of two with CTAs enough for 4 to 16 columns: threads
# that take one butterfly of the smallest radix, and threads that take several
@pytest.mark.parametrize("L,other,nb", [(54, 288, 17), (250, 288, 9), (360, 288, 9), (384, 96, 26), (500, 144, 17),
                                        (750, 96, 13), (1000, 96, 13), (972, 36, 34)])
def test_mixed_radix_columns_of_a_batch(nf, L, other, nb):
    Kd = (L, other)
    Nd = tuple(2 * max(1, K // 3) for K in Kd)
    om = W.uniform_random_om(701, 2, seed=L)
    p = oracle.make_plan(om, Nd, Kd, (4, 4))
    xs, ys = cn((nb,) + Nd, 1), cn((nb, om.shape[0]), 2)
    with nf.NufftPlan(dev(om), Nd, Kd, (4, 4)) as plan:
        yb, xb = plan.forward_batch(dev(xs)).cpu().numpy(), plan.adjoint_batch(dev(ys)).cpu().numpy()
    for b in {0, nb - 1}:
        assert rel(yb[b], oracle.forward(p, xs[b])) < TOL_OP
        assert rel(xb[b], oracle.adjoint(p, ys[b])) < TOL_OP


# V of a 2D batch: CTAs below and above the number from which a thread takes four elements
@pytest.mark.parametrize("J,M,nb", [(4, 41000, 16), (4, 41000, 17), (5, 30000, 17), (6, 25000, 13), (6, 25000, 12),
                                    (7, 17000, 18), (7, 700, 5)])
def test_2d_batch_interpolation(nf, J, M, nb):
    Kd, Nd = (90, 80), (54, 48)
    om = W.uniform_random_om(M, 2, seed=J)
    p = oracle.make_plan(om, Nd, Kd, (J, J))
    xs = cn((nb,) + Nd, 3)
    with nf.NufftPlan(dev(om), Nd, Kd, (J, J)) as plan:
        yb = plan.forward_batch(dev(xs)).cpu().numpy()
    for b in {0, 3, 4, nb - 1}:
        assert rel(yb[b], oracle.forward(p, xs[b])) < TOL_OP


# staged 2D kernels whose coefficients lose the odd pitch for a third CTA per SM, and keep it
@pytest.mark.parametrize("Jd", [(16, 16), (16, 14), (13, 16), (15, 15)])
@pytest.mark.parametrize("Kd", [(360, 288), (64, 80)])
def test_2d_many_neighbours(nf, Jd, Kd):
    Nd = tuple(K // 10 * 8 for K in Kd)   # a lean grid: G is well conditioned
    om = W.uniform_random_om(1500, 2, seed=5)
    p = oracle.make_plan(om, Nd, Kd, Jd)
    z, y = cn(Kd, 5), cn(1500, 6)
    with nf.NufftPlan(dev(om), Nd, Kd, Jd) as plan:
        assert rel(plan.interp(dev(z)).cpu().numpy(), oracle.interp_V(p, z)) < TOL_V
        assert rel(plan.gridding(dev(y)).cpu().numpy(), oracle.gridding_VH(p, y)) < TOL_V


# one transform whose small chunks go to the two-warp gridding kernel
def test_2d_single_transform_of_small_chunks(nf):
    Kd, Nd, M = (1000, 972), (500, 486), 250001
    om = W.uniform_random_om(M, 2, seed=8)
    p = oracle.make_plan(om, Nd, Kd, (4, 4))
    y = cn(M, 7)
    with nf.NufftPlan(dev(om), Nd, Kd, (4, 4)) as plan:
        nch = plan.info()["nchunks"]
        assert nch >= 32 * 152 and M <= 64 * nch   # the rule for that kernel
        assert rel(plan.gridding(dev(y)).cpu().numpy(), oracle.gridding_VH(p, y)) < TOL_V


# 1D: one tile's list of 1 to 40 chunks over four thread groups, three pairs in flight.  A
# chunk's sums round by up to 2^-31 B per contribution, B < 2 max|c| sum(|Re y| + |Im y|) over its
# points; a wrong list is off by whole contributions.
@pytest.mark.parametrize("K,M", [(64, 300), (64, 1025), (500, 2049), (1000, 5000), (64, 7000), (1024, 9001), (96, 40001)])
def test_1d_reduction(nf, K, M):
    om = W.uniform_random_om(M, 1, seed=M)
    p = oracle.make_plan(om, (K // 2,), (K,), (6,))
    y = cn(M, 8)
    with nf.NufftPlan(dev(om), (K // 2,), (K,), (6,)) as plan:
        got = plan.gridding(dev(y)).cpu().numpy()
    ref = oracle.gridding_VH(p, y)
    sums = (np.abs(y.real) + np.abs(y.imag)).sum()
    fixed = min(M, 1024) * 2.0 ** -31 * 2 * np.abs(p.coef[0]).max() * sums
    assert np.abs(got - ref).max() <= fixed + TOL_V * np.linalg.norm(ref)


# 3D tile sums: eight planes per thread, and two for lists of many chunks (1 to about 40 of
# them), whole tiles and remainders of both, one transform and a batch
@pytest.mark.parametrize("Kd,M,spread,nb", [((96, 96, 96), 9000, 3.1, 1), ((48, 48, 48), 9000, 3.1, 1),
                                            ((48, 36, 50), 41000, 0.25, 1), ((32, 48, 32), 20000, 0.1, 1),
                                            ((18, 20, 30), 9001, 3.1, 2), ((40, 64, 36), 21000, 0.3, 3)])
@pytest.mark.parametrize("Jd", [(6, 6, 6), (3, 5, 4)])
def test_3d_reduction(nf, Kd, M, spread, nb, Jd):
    Nd = tuple(2 * (K // 4) for K in Kd)
    om = (np.random.default_rng(M).uniform(-spread, spread, (M, 3))).astype(np.float32)
    p = oracle.make_plan(om, Nd, Kd, Jd)
    ys = cn((nb, M), 9)
    with nf.NufftPlan(dev(om), Nd, Kd, Jd) as plan:
        assert rel(plan.gridding(dev(ys[0])).cpu().numpy(), oracle.gridding_VH(p, ys[0])) < TOL_V
        if nb > 1:
            xb = plan.adjoint_batch(dev(ys)).cpu().numpy()
            assert rel(xb[nb - 1], oracle.adjoint(p, ys[nb - 1])) < TOL_OP


def _kernels(f):
    """Names of the kernels that f launches, empty where the profiler sees none."""
    from torch.profiler import ProfilerActivity, profile
    f()
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        f()
        torch.cuda.synchronize()
    return " ".join(e.key for e in prof.key_averages())


def _first(J):
    """Lowest frequency, in grid cells, whose first neighbour is cell 0."""
    return (J - 1) // 2 - 0.5 * (J % 2)


def _tile(om, K, J, T):
    """Tile of each point's first neighbour on a K^3 grid."""
    t = np.zeros(om.shape[0], dtype=np.int64)
    for a in range(3):
        t = t * (K // T) + (oracle.offsets_1d(om[:, a].astype(np.float64), K, J).astype(np.int64) + 1) % K // T
    return t


# 3D V by staged chunks on tiles of 10, with chunks of one round of the CTA's warps, one point
# more, several rounds and the longest there is; and by points
@pytest.mark.parametrize("J,M,staged", [(4, 1000000, True), (5, 600000, True), (6, 300000, True), (7, 300000, True),
                                        (6, 300, False), (7, 9000, False), (4, 30000, False)])
def test_3d_interpolation_routes(nf, J, M, staged):
    K, N, T = 100, 50, 10
    rng = np.random.default_rng(J)
    om = rng.uniform(-np.pi, np.pi, (M, 3)).astype(np.float32)
    step = 16 * (32 // J)
    picks = []
    if M >= 300000:   # tiles that hold exactly these numbers of points
        sizes = {0: step, 111: step + 1, 222: 3 * step + 5, 333: 1, 444: 2048, 555: 2049}
        om = om[~np.isin(_tile(om, K, J, T), list(sizes))]
        for t, n in sizes.items():
            corner = np.array([t // 100, t // 10 % 10, t % 10]) * T
            u = corner + _first(J) + rng.uniform(0.1, T - 0.1, (n, 3))
            w = (2 * np.pi / K * (u - K * (u > K / 2))).astype(np.float32)
            w = w[_tile(w, K, J, T) == t]
            assert w.shape[0] == n
            picks.append(np.arange(om.shape[0], om.shape[0] + n))
            om = np.concatenate([om, w])
    picks = np.concatenate(picks + [rng.integers(0, om.shape[0], 1000)])
    z = cn((K,) * 3, 10)
    p = oracle.make_plan(om[picks], (N,) * 3, (K,) * 3, (J,) * 3)
    with nf.NufftPlan(dev(om), (N,) * 3, (K,) * 3, (J,) * 3) as plan:
        zd = dev(z)
        got = plan.interp(zd).cpu().numpy()
        plan.set_graphs(False)
        names = _kernels(lambda: plan.interp(zd))
    assert rel(got[picks], oracle.interp_V(p, z)) < TOL_V
    if "k_interp" in names:
        assert ("k_interp_chunk3d" in names) == staged, names


# every J of the two-word bound by magnitudes in a strip of shared memory, samples aligned in
# phase at the most loaded cell, chunks of the largest size inside one tile of 16
@pytest.mark.parametrize("Jd,M", [((6, 5, 4), 2048), ((2, 7, 5), 1500), ((8, 8, 8), 700), ((1, 3, 1), 900),
                                  ((6, 6, 6), 2048), ((6, 6, 6), 2049), ((4, 4, 4), 2048), ((7, 7, 7), 2048)])
def test_3d_gridding_bound_in_one_tile(nf, Jd, M):
    K, N = 32, 16
    rng = np.random.default_rng(M)
    u = np.stack([_first(J) + rng.uniform(0.1, 15.9, M) for J in Jd], 1)
    om = (2 * np.pi / K * (u - K * (u > K / 2))).astype(np.float32)
    p = oracle.make_plan(om, (N,) * 3, (K,) * 3, Jd)
    first = (p.k0 + 1) % K
    assert first.max() < 16    # one tile
    load = np.zeros((K,) * 3)
    for js in np.ndindex(*Jd):
        idx = tuple((p.k0[:, a] + 1 + js[a]) % K for a in range(3))
        np.add.at(load, idx, np.abs(np.prod([p.coef[a][:, js[a]] for a in range(3)], axis=0)))
    cell = np.unravel_index(np.argmax(load), load.shape)
    w = np.ones(M, dtype=np.complex128)
    for a in range(3):
        j = (cell[a] - (p.k0[:, a] + 1)) % K
        w *= np.where(j < Jd[a], p.coef[a][np.arange(M), np.minimum(j, Jd[a] - 1)], 0)
    y = np.where(np.abs(w) > 0, w / np.maximum(np.abs(w), 1e-300), 1.0).astype(np.complex64)
    ref = oracle.gridding_VH(p, y)
    with nf.NufftPlan(dev(om), (N,) * 3, (K,) * 3, Jd) as plan:
        assert plan.info()["nchunks"] == (M + 2047) // 2048
        got = plan.gridding(dev(y)).cpu().numpy()
    assert rel(got, ref) < TOL_V


# the stable sort by tile around the size at which its tile changes
@pytest.mark.parametrize("M", [(1 << 18) - 1, 1 << 18, (1 << 18) + 1, 5])
def test_sort_by_tile(nf, M):
    om = W.uniform_random_om(M, 2, seed=12)
    with nf.NufftPlan(dev(om), (64, 64), (128, 128), (6, 6)) as plan:
        kf, _, _, perm = plan.interpolator()
    k = kf.numpy()[perm.numpy()] // 16
    tile = k[:, 0] * 8 + k[:, 1]
    assert (np.diff(tile) >= 0).all()
    np.testing.assert_array_equal(np.sort(perm.numpy()), np.arange(M))
