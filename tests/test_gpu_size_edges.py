"""Kernels at the sizes where their work splits differently, on the GPU vs the oracle.

Sizes lie at the edges of tiles, of size classes and of table sizes (one below, at and one
above). Integers (labels, counts, cells) are bit-exact; f_l is FP32 (1e-4 relative, as its
sums are), R is 1e-4 max(1, |R|), frames are FP64 sums (1e-10) and the fit agrees to 1e-7
(its stop on a cost change of 1e-15 fixes it to about 3e-8).
"""
import numpy as np
import pytest
import torch

import oracle
from helpers import assert_close_nan, oracle_fl
from test_gpu_coregrow import _check as check_core_grow

pytestmark = pytest.mark.gpu

L = 1 << 21


@pytest.fixture(scope="module")
def ctx():
    from paper_1902_01010_gb300 import Context

    return Context(0)


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _fl(ctx, pos, vel, lab, **kw):
    from paper_1902_01010_gb300 import Params

    f = ctx.velden(_dev(pos), _dev(vel), _dev(lab.astype(np.int32)), Params.default(**kw))
    ctx.sync()
    return f.cpu().numpy()


def _halo(n, seed, spread=40000, step=1):
    """One halo: Gaussian positions on a lattice of `step`, Gaussian velocities."""
    rng = np.random.default_rng(seed)
    p = np.round(rng.normal(0, spread / step, size=(n, 3))).astype(np.int64) * step
    return ((p + 1000) % L).astype(np.int32), rng.normal(0, 80, size=(n, 3)).astype(np.float32)


# ------------------------------------------------------------------------- 3D FOF
# tiles of scans (2048) and of the one-launch sort (4096)
@pytest.mark.parametrize("n", [2, 31, 32, 33, 2047, 2048, 2049, 4095, 4096, 4097, 8193])
@pytest.mark.parametrize("T", [9000 ** 2, 40000 ** 2])
def test_fof_small_counts(ctx, n, T):
    rng = np.random.default_rng(n)
    pos = rng.integers(0, L, size=(n, 3))
    k = n // 3
    pos[:k] = pos[0] + rng.normal(0, 4000, size=(k, 3)).astype(np.int64)
    pos = (pos % L).astype(np.int32)
    lab = ctx.fof3d(_dev(pos), T)
    ctx.sync()
    assert np.array_equal(lab.cpu().numpy(), oracle.fof3d(pos, T))


# sort tiles of 1,024 keys below 2^20 keys and of 4,096 from there on
@pytest.mark.parametrize("n", [(1 << 20) - 1, (1 << 20) + 1])
def test_fof_sort_tile_sizes(ctx, n):
    rng = np.random.default_rng(n)
    pos = rng.integers(0, L, size=(n, 3))
    pos[::3] = pos[::3] // 50000 * 50000 + rng.integers(0, 12000, size=pos[::3].shape)
    pos = (pos % L).astype(np.int32)
    T = 3500 ** 2
    lab = ctx.fof3d(_dev(pos), T)
    ctx.sync()
    assert np.array_equal(lab.cpu().numpy(), oracle.fof3d(pos, T))


# crowded cells: two clumps of `m` in cells that touch, a gap of one more or less than the
# linking length between their nearest members, and members on cell faces
@pytest.mark.parametrize("m", [3, 9, 64, 65, 300, 3000])
@pytest.mark.parametrize("gap", [-1, 0, 1])
def test_fof_crowded_cells(ctx, m, gap):
    rng = np.random.default_rng(m)
    b = 5000
    a = rng.integers(0, 200, size=(m, 3))
    c = rng.integers(0, 200, size=(m, 3))
    a[0], c[0] = [199, 100, 100], [0, 100, 100]
    c += [199 + b + gap, 0, 0]
    grid = np.stack(np.meshgrid(*[np.arange(6) * (b + 1)] * 3, indexing="ij"), -1).reshape(-1, 3) + 300000
    pos = (np.concatenate([a, c, grid]) + [L - 2600, 5, L - 90]) % L
    pos = pos.astype(np.int32)
    lab = ctx.fof3d(_dev(pos), b * b)
    ctx.sync()
    lab = lab.cpu().numpy()
    assert np.array_equal(lab, oracle.fof3d(pos, b * b))
    assert (lab[m] == lab[0]) == (gap < 0)  # d^2 < T links


# ---------------------------------------------------------------------------- f_l
# many halos in mixed order: chunks of 32 slots that span several halos, label counts
# through a table, halos at and above N_se
def test_fl_many_small_halos(ctx):
    rng = np.random.default_rng(5)
    sizes = np.r_[np.full(40, 20), 21, 31, 32, 33, 63, 64, 65, 95, 96, 97, 255, 256, 257, 320, np.full(60, 5)]
    lab = np.repeat(np.arange(len(sizes)), sizes)
    ctr = rng.integers(0, L, size=(len(sizes), 3))
    pos = ((ctr[lab] + rng.normal(0, 3000, size=(len(lab), 3)).astype(np.int64)) % L).astype(np.int32)
    vel = rng.normal(0, 80, size=(len(lab), 3)).astype(np.float32)
    p = rng.permutation(len(lab))
    first = np.full(len(sizes), len(lab))
    np.minimum.at(first, lab[p], np.arange(len(lab)))  # a halo's label is its first member
    lab, pos, vel = first[lab[p]].astype(np.int32), pos[p], vel[p]
    assert_close_nan(_fl(ctx, pos, vel, lab), oracle_fl(pos, vel, lab), 1e-4, what="f_l")


# separations below, around and above what 32-bit squares hold (26,754 an axis), partly
# filled buckets, and a few dense clumps in a wide cloud (curve jumps inside buckets)
@pytest.mark.parametrize("nse,nv", [(256, 32), (64, 16), (33, 33)])
@pytest.mark.parametrize("spread", [3, 300, 9000, 27000, 120000, "clumps"])
def test_fl_separations(ctx, spread, nse, nv):
    rng = np.random.default_rng(nse)
    n = 4001
    if spread == "clumps":
        s = rng.choice([20.0, 400.0, 100000.0], size=(n, 1))
        p = rng.integers(-60000, 60000, size=(7, 3))[rng.integers(0, 7, size=n)] + rng.normal(0, 1, (n, 3)) * s
        pos = (np.round(p).astype(np.int64) % L).astype(np.int32)
        vel = rng.normal(0, 80, size=(n, 3)).astype(np.float32)
    else:
        pos, vel = _halo(n, 3, spread)
    lab = np.zeros(n, np.int32)
    assert_close_nan(_fl(ctx, pos, vel, lab, nse=nse, nv=nv), oracle_fl(pos, vel, lab, nse, nv), 1e-4,
                     what=f"{spread}")


def test_fl_more_keys_below_the_bins_than_16_bits_hold(ctx):
    """A core of 70,000 members beside a sparse cloud: for most of the cloud every core
    member lies in the inner half of the first bound."""
    rng = np.random.default_rng(11)
    core = rng.normal(0, 25, size=(70000, 3))
    cloud = rng.normal(0, 20000, size=(3000, 3)) + [9000, 0, 0]
    pos = (np.round(np.concatenate([core, cloud])).astype(np.int64) % L).astype(np.int32)
    vel = rng.normal(0, 80, size=pos.shape).astype(np.float32)
    lab = np.zeros(len(pos), np.int32)
    got = _fl(ctx, pos, vel, lab)
    m = np.arange(len(pos))
    up = oracle.unwrap(pos, m)
    for k in np.r_[rng.integers(0, 70000, 20), rng.integers(70000, 73000, 150)]:
        ref = oracle.velden_one(up, vel, m, int(k))
        assert abs(got[k] - ref) <= 1e-4 * ref, k


# ------------------------------------------------- background cells, frames, fit
# classes by members: frames by warp, block (1,024) and cluster (16,384), trees by block
# (8,192) and cluster (65,536), histograms by 256 and 1,024 threads (16,384); `step` > 1
# gives equal coordinates on either side of the medians
@pytest.mark.parametrize("n,step", [(160, 1), (161, 1), (1023, 1), (1024, 500), (1025, 1), (4097, 9000),
                                    (8191, 1), (8192, 3000), (8193, 1), (16383, 1), (16384, 2000),
                                    (16385, 1), (65535, 1), (65536, 2500), (65537, 1)])
def test_background_and_fit_size_classes(ctx, n, step):
    from paper_1902_01010_gb300 import Params

    pos, vel = _halo(n, n, step=step)
    lab = np.zeros(n, np.int32)
    P = Params.default()
    fl = ctx.velden(_dev(pos), _dev(vel), _dev(lab), P)
    R, ell, hs = ctx.outlier_ratio(_dev(pos), _dev(vel), fl, _dev(lab), P)
    ctx.sync()
    fl, R, ell, hs = fl.cpu().numpy(), R.cpu().numpy(), ell.cpu().numpy(), hs.cpu().numpy()
    m = np.arange(n)
    ref, leaf, cells = oracle.background_halo(oracle.unwrap(pos, m), vel, m, fl.astype(np.float64))
    fin = np.isfinite(ref)
    assert np.array_equal(np.isfinite(R), fin) and fin.sum() > 0.9 * n
    assert (np.abs(R[fin] - ref[fin]) <= 1e-4 * np.maximum(1.0, np.abs(ref[fin]))).all()
    fr = oracle.halo_frame(vel, m)
    assert np.allclose(hs[0, 5:8], fr[:3], rtol=1e-10, atol=1e-9) and abs(hs[0, 8] - fr[3]) <= 1e-10 * fr[3]
    fit = oracle.ell_fit(R.astype(np.float64))
    assert abs(hs[0, 3] - fit[0]) <= 1e-7 * max(1.0, abs(fit[0])) and abs(hs[0, 4] - fit[1]) <= 1e-7 * fit[1]
    assert np.allclose(ell, (R.astype(np.float64) - hs[0, 3]) / hs[0, 4], rtol=1e-6, atol=1e-6, equal_nan=True)


# fewest and most bins, more bins than members, a bin count that no warp divides
@pytest.mark.parametrize("n,lo,hi", [(160, 10, 10), (300, 400, 400), (700, 33, 33), (5000, 1024, 1024)])
def test_fit_bin_counts(ctx, n, lo, hi):
    from paper_1902_01010_gb300 import Params

    pos, vel = _halo(n, n)
    lab = np.zeros(n, np.int32)
    P = Params.default(fit_nbins_min=lo, fit_nbins_max=hi)
    fl = ctx.velden(_dev(pos), _dev(vel), _dev(lab), P)
    R, ell, hs = ctx.outlier_ratio(_dev(pos), _dev(vel), fl, _dev(lab), P)
    ctx.sync()
    fit = oracle.ell_fit(R.cpu().numpy().astype(np.float64), lo, hi)
    hs = hs.cpu().numpy()
    assert abs(hs[0, 3] - fit[0]) <= 1e-7 * max(1.0, abs(fit[0])) and abs(hs[0, 4] - fit[1]) <= 1e-7 * fit[1]


# ------------------------------------------------------------------- 6D linking
# tiles of 32 candidates, with separations, speed ratios and speed differences that lie
# exactly on their thresholds (lattice positions, velocities from a few integers), where
# the FP32 test must leave the decision to FP64
@pytest.mark.parametrize("n", [31, 32, 33, 63, 65, 160, 1025, 4000])
@pytest.mark.parametrize("use_lv,use_vt", [(1, 1), (0, 1), (1, 0)])
def test_link_tiles_and_exact_thresholds(ctx, n, use_lv, use_vt):
    from paper_1902_01010_gb300 import Params

    rng = np.random.default_rng(n)
    side = int(np.ceil(n ** (1 / 3))) + 1
    pos = (rng.integers(0, side, size=(n, 3)) * 500 + 3000).astype(np.int32)
    vel = (rng.choice([-200, -100, -50, 0, 50, 100, 200, 400], size=(n, 3))).astype(np.float32)
    lab = np.zeros(n, np.int32)
    ell = rng.uniform(1, 4, n).astype(np.float32)
    ell[::5] = 2.5  # on the threshold
    hs = np.zeros((1, 12))
    hs[0, :9] = [0, n, 1, 0, 1, 0, 0, 0, 100]
    hs[0, 9], hs[0, 10] = 500.0 ** 2 * 2, 150.0 ** 2
    P = Params.default(nsearch_min=20, use_lv=use_lv, use_vr_theta=use_vt)
    got = ctx.fof6d(_dev(pos), _dev(vel), _dev(ell), _dev(lab), _dev(hs), P)
    ctx.sync()
    m = np.arange(n)
    cand = (ell >= 2.5).astype(np.uint8)
    ref = oracle.fof6d_halo(oracle.unwrap(pos, m), vel, m, cand, hs[0, [9, 10, 5, 6, 7]], use_lv=use_lv,
                            use_vt=use_vt)
    assert np.array_equal(got.cpu().numpy(), ref)


# ------------------------------------------------------------------ core growth
# moments by block below 4,096 members and by cluster from there on
@pytest.mark.parametrize("diffuse", [600, 3409, 3410, 3411, 9000])
def test_core_growth_team_sizes(ctx, diffuse):
    rng = np.random.default_rng(diffuse)
    g = np.stack(np.meshgrid(*[np.arange(7)] * 3, indexing="ij"), -1).reshape(-1, 3) * 500
    base = np.array([100000, 100000, 100000])
    pos = [g + base, g + base + [3500, 0, 0]]
    vel = [rng.normal(0, 0.3, size=(len(g), 3)) + [s, 0, 0] for s in (200, -200)]
    d = rng.normal(size=(diffuse, 3))
    d = d / np.linalg.norm(d, axis=1)[:, None] * rng.uniform(9000, 90000, (diffuse, 1))
    pos.append(np.round(base + [3250, 1500, 1500] + d))
    vel.append(rng.normal(0, 60, size=(diffuse, 3)))
    pos, vel = np.vstack(pos).astype(np.int32), np.vstack(vel).astype(np.float32)
    check_core_grow(ctx, pos, vel, np.zeros(len(pos), np.int32), None, 700.0)
