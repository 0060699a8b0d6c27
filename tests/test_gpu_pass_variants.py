"""The passes that a size rule chooses, each side of it, against the FP64 oracle.

FFT passes (line lengths, columns per CTA, eight or sixteen values per thread), the 3D
chunk interpolation and tile reduction for every J they are built for, on tiles that are
not 16 wide and with point counts at the edges of a round, and the batched 2D kernels.

Tolerances: an FFT line of 256 points has 8 radix-2 levels, each with at most about
1.5 * 2^-24 of relative rounding in the 2-norm; three axes give 3 * 8 * 1.5 * 2^-24 =
2.1e-6 if all errors added up: 2e-6.  Interpolation and gridding: about eight roundings of
2^-24 per contribution: 1e-6.
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


# (grid, image): axis-0 lines of 128 and 256 above and below the threshold for sixteen
# values per thread, columns that 16 or 8 do not divide, the axis-1 pass with outer
# lines, and images that fill more or less than half of the grid
@pytest.mark.parametrize("Kd,Nd", [
    ((128, 96, 64), (64, 48, 32)), ((256, 48, 64), (200, 24, 32)), ((128, 64, 64), (64, 32, 32)),
    ((64, 128, 128), (64, 64, 100)), ((64, 256, 64), (50, 128, 64)), ((128, 90, 90), (64, 60, 90)),
    ((256, 50, 30), (128, 26, 30)), ((16, 32, 1024), (16, 20, 512)), ((512, 128), (256, 128)), ((1024, 36), (512, 18)),
    ((64, 512), (34, 512)), ((512, 36, 36), (256, 18, 36)),
])
def test_fft_passes(nf, Kd, Nd):
    d = len(Kd)
    om = W.uniform_random_om(7, d, seed=3)
    p = oracle.make_plan(om, Nd, Kd, (6,) * d)
    x, z = cn(Nd, 1), cn(Kd, 2)
    with nf.NufftPlan(dev(om), Nd, Kd, (6,) * d) as plan:
        assert rel(plan.scale_pad_fft(dev(x)).cpu().numpy(), oracle.fft_forward(oracle.scale_pad(p, x))) < TOL_FFT
        assert rel(plan.ifft_crop_rescale(dev(z)).cpu().numpy(), oracle.crop_rescale(p, oracle.fft_adjoint(z))) < TOL_FFT


# lines that are not powers of two: every radix (3 to 16) as the first, the middle
# and the last stage, on a contiguous and on a strided axis
@pytest.mark.parametrize("L", [18, 20, 24, 30, 50, 54, 72, 108, 144, 150, 162, 192, 240, 250, 324, 360, 384, 400, 500,
                               750, 768, 864, 960, 972, 1000])
@pytest.mark.parametrize("other,strided", [(16, True), (80, True), (36, False)])
def test_mixed_radix_lines(nf, L, other, strided):
    Kd = (L, other) if strided else (other, L)
    Nd = tuple(2 * max(1, K // 3) for K in Kd)
    om = W.uniform_random_om(5, 2, seed=4)
    p = oracle.make_plan(om, Nd, Kd, (4, 4))
    x, z = cn(Nd, 8), cn(Kd, 9)
    with nf.NufftPlan(dev(om), Nd, Kd, (4, 4)) as plan:
        assert rel(plan.scale_pad_fft(dev(x)).cpu().numpy(), oracle.fft_forward(oracle.scale_pad(p, x))) < TOL_FFT
        assert rel(plan.ifft_crop_rescale(dev(z)).cpu().numpy(), oracle.crop_rescale(p, oracle.fft_adjoint(z))) < TOL_FFT


# the CG step's sums in the image-side passes, with CTAs of full and of part warps
@pytest.mark.parametrize("Nd,Kd", [((12, 14), (20, 18)), ((24, 30), (36, 60)), ((40, 36), (64, 50)), ((50, 64), (100, 128))])
def test_cg_hooks_in_the_passes(nf, Nd, Kd):
    om = W.uniform_random_om(4 * Nd[0] * Nd[1], 2, seed=6)
    p = oracle.make_plan(om, Nd, Kd, (6, 6))
    y = cn(om.shape[0], 10)
    with nf.NufftPlan(dev(om), Nd, Kd, (6, 6)) as plan:
        got = plan.solve_cg(dev(y), maxiter=3).cpu().numpy()
    assert rel(got, oracle.cg(p, y, np.zeros(Nd), 3)) < 10 * TOL_OP


@pytest.mark.parametrize("J", [4, 5, 6, 7])
@pytest.mark.parametrize("Kd,M", [((32, 32, 32), 1), ((32, 32, 32), 6001), ((20, 24, 36), 1279), ((16, 18, 50), 81)])
def test_3d_interpolation_and_gridding(nf, J, Kd, M):
    Nd = tuple(2 * (K // 4) for K in Kd)
    om = W.uniform_random_om(M, 3, seed=M + J)
    p = oracle.make_plan(om, Nd, Kd, (J,) * 3)
    z, y = cn(Kd, 4), cn(M, 5)
    with nf.NufftPlan(dev(om), Nd, Kd, (J,) * 3) as plan:
        assert rel(plan.interp(dev(z)).cpu().numpy(), oracle.interp_V(p, z)) < TOL_V
        assert rel(plan.gridding(dev(y)).cpu().numpy(), oracle.gridding_VH(p, y)) < TOL_V


# 3D interpolation on both sides of the CTA rule, one transform and a batch
@pytest.mark.parametrize("J", [4, 5, 6, 7])
@pytest.mark.parametrize("K,M,nb", [(48, 9000, 1), (128, 9000, 1), (64, 4001, 3), (64, 4001, 17)])
def test_3d_chunk_and_point_kernels(nf, J, K, M, nb):
    om = W.uniform_random_om(M, 3, seed=15)
    Kd, Nd = (K,) * 3, (K // 4 * 2, K // 4 * 2, K // 4 * 2)
    p = oracle.make_plan(om, Nd, Kd, (J,) * 3)
    xs = cn((nb,) + Nd, 16)
    with nf.NufftPlan(dev(om), Nd, Kd, (J,) * 3) as plan:
        yb = plan.forward_batch(dev(xs)).cpu().numpy()
    for b in {0, nb - 1}:
        assert rel(yb[b], oracle.forward(p, xs[b])) < TOL_OP


# 2D single transforms: tiles of 16 and others, chunk counts at the edges of a chunk
@pytest.mark.parametrize("Jd", [(4, 4), (5, 5), (6, 6), (7, 7), (7, 4), (1, 6)])
@pytest.mark.parametrize("Kd,M", [((64, 48), 255), ((32, 32), 1025), ((36, 90), 4100), ((18, 64), 40)])
def test_2d_single_transforms(nf, Jd, Kd, M):
    Nd = tuple(2 * (K // 4) for K in Kd)
    om = W.uniform_random_om(M, 2, seed=M + 1)
    om[: M // 2] = 0.2 + 0.01 * om[: M // 2]     # more than one chunk in a tile
    p = oracle.make_plan(om, Nd, Kd, Jd)
    x, z, y = cn(Nd, 11), cn(Kd, 12), cn(M, 13)
    with nf.NufftPlan(dev(om), Nd, Kd, Jd) as plan:
        assert rel(plan.interp(dev(z)).cpu().numpy(), oracle.interp_V(p, z)) < TOL_V
        assert rel(plan.gridding(dev(y)).cpu().numpy(), oracle.gridding_VH(p, y)) < TOL_V
        assert rel(plan.selfadjoint(dev(x)).cpu().numpy(), oracle.selfadjoint(p, x)) < 2 * TOL_OP


# the polynomial form of the coefficients, and trajectories around the size at which
# the sort changes its tile
@pytest.mark.parametrize("N,K,J,M", [(64, 128, 8, 300), (64, 128, 6, 300), (40, 60, 5, 300), (16, 16, 3, 300),
                                     (64, 128, 6, (1 << 18) - 1), (64, 128, 6, (1 << 18) + 1)])
def test_coefficients_and_sort(nf, N, K, J, M):
    om = W.uniform_random_om(M, 2, seed=14)
    with nf.NufftPlan(dev(om), (N, N), (K, K), (J, J)) as plan:
        kf, coefs, _, perm = plan.interpolator()
    np.testing.assert_array_equal(np.sort(perm.numpy()), np.arange(M))
    pick = np.arange(0, M, max(1, M // 300))
    p = oracle.make_plan(om[pick], (N, N), (K, K), (J, J))
    for a in range(2):
        np.testing.assert_array_equal(kf.numpy()[pick, a], (p.k0[:, a] + 1) % K)
        err = np.abs(coefs[a].numpy()[pick] - p.coef[a]).max() / np.abs(p.coef[a]).max()
        assert err < 1e-7, (a, err)   # the float32 rounding is at most 2^-24 = 6e-8 of a component


# chunks of few and of many points, CTA counts on both sides of the rule, odd tiles
@pytest.mark.parametrize("Jd", [(4, 4), (5, 5), (6, 6), (7, 7), (5, 7), (6, 1)])
@pytest.mark.parametrize("Kd,M,nb", [((256, 256), 3001, 20), ((256, 256), 17000, 2), ((90, 64), 700, 3),
                                     ((360, 288), 9000, 11)])
def test_2d_batches(nf, Jd, Kd, M, nb):
    Nd = tuple(2 * (K // 4) for K in Kd)
    om = W.uniform_random_om(M, 2, seed=M)
    om[: M // 8] = 0.1 + 0.02 * om[: M // 8]     # a dense tile of several chunks
    p = oracle.make_plan(om, Nd, Kd, Jd)
    xs, ys = cn((nb,) + Nd, 6), cn((nb, M), 7)
    with nf.NufftPlan(dev(om), Nd, Kd, Jd) as plan:
        yb, xb = plan.forward_batch(dev(xs)).cpu().numpy(), plan.adjoint_batch(dev(ys)).cpu().numpy()
        again = plan.adjoint_batch(dev(ys)).cpu().numpy()
    np.testing.assert_array_equal(again, xb)
    for b in {0, 1, nb - 1}:
        assert rel(yb[b], oracle.forward(p, xs[b])) < TOL_OP
        assert rel(xb[b], oracle.adjoint(p, ys[b])) < TOL_OP
