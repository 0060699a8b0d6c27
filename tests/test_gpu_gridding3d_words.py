"""3D gridding with two and with three accumulator words per cell, against the FP64 oracle.

A chunk sums in two words where the bound max|y| * (largest sum of weight magnitudes of a
cell) makes their rounding step no larger than that of three words.  The samples here are
aligned in phase so that the most loaded cell reaches that bound (an overflow would show
as a sign change), on spread points (two words) and on a dense cluster (three), with
chunks of one point, of the largest size and one more, with tiles of 16 and other edges.

Tolerance: a contribution is a product of three float32 coefficients and a sample, about
eight roundings of at most 2^-24 in relative terms, and the fixed-point step is below
2^-24 of the largest contribution; independent errors add up to less than
8 * 2^-24 = 4.8e-7 of the grid's norm, plus the final rounding: 1e-6.
"""
import itertools

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-6


def _tile_points(M, K, width, seed):
    """M points whose frequencies fall into `width` grid cells from cell K/4 + 3 on."""
    rng = np.random.default_rng(seed)
    u = K / 4 + 3.5 + width * rng.random((M, 3))
    return (2 * np.pi / K * (u - K * (u > K / 2))).astype(np.float32)


def _weights(p, cell):
    """Weight of every point at one grid cell."""
    w = np.ones(p.M, dtype=np.complex128)
    for a in range(3):
        j = (cell[a] - (p.k0[:, a] + 1)) % p.Kd[a]
        hit = j < p.Jd[a]
        w *= np.where(hit, p.coef[a][np.arange(p.M), np.minimum(j, p.Jd[a] - 1)], 0)
    return w


@pytest.mark.parametrize("width", [9.0, 0.5], ids=["spread", "cluster"])
@pytest.mark.parametrize("N,K,J,M", [(16, 32, 6, 2048), (16, 32, 6, 2049), (16, 32, 4, 1), (16, 20, 4, 700),
                                     (16, 24, 5, 1501), (16, 32, 5, 33), (20, 40, 7, 2047), (16, 32, 7, 900),
                                     (16, 32, 3, 500)])
def test_most_loaded_cell_at_its_bound(N, K, J, M, width):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1710_03197_gb300 as nf

    om = _tile_points(M, K, width, seed=M + J)
    p = oracle.make_plan(om, (N,) * 3, (K,) * 3, (J,) * 3)
    load = np.zeros((K,) * 3)
    for js in itertools.product(range(J), repeat=3):
        idx = tuple((p.k0[:, a] + 1 + js[a]) % K for a in range(3))
        np.add.at(load, idx, np.abs(np.prod([p.coef[a][:, js[a]] for a in range(3)], axis=0)))
    w = _weights(p, np.unravel_index(np.argmax(load), load.shape))
    y = np.where(np.abs(w) > 0, w / np.maximum(np.abs(w), 1e-300), 1.0).astype(np.complex64)
    ref = oracle.gridding_VH(p, y)
    plan = nf.NufftPlan(torch.from_numpy(om).cuda(), (N,) * 3, (K,) * 3, (J,) * 3)
    for scale in (1.0, 1e-20, 3e15):
        got = plan.gridding(torch.from_numpy(y * np.float32(scale)).cuda()).cpu().numpy().astype(np.complex128) / scale
        assert np.linalg.norm(got - ref) <= TOL * np.linalg.norm(ref), scale
    plan.close()
