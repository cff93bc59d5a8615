"""Calls at the ends of what the library accepts and at the hand-overs inside its kernels,
on the GPU vs the oracle or a plain numpy form of the same step. No case faults the GPU:
what is out of range is refused by the host or by a kernel's own check.
"""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

L = 1 << 21


@pytest.fixture(scope="module")
def ctx():
    from paper_1902_01010_gb300 import Context

    return Context(0)


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


# ------------------------------------------------------------ trees built by a cluster
def test_cluster_trees_hand_over_to_their_blocks(ctx):
    """Halos whose nodes a cluster splits together before each block takes subtrees of its
    own: equal coordinates make the halves uneven, so the cluster's last split comes at
    another node in each halo and the blocks start on subtrees of different sizes. Every
    build gives the same cells and the same bits of R; the cells are the oracle's."""
    from paper_1902_01010_gb300 import Params

    rng = np.random.default_rng(2)
    sizes, steps = [65536, 70001, 90000, 131072], [1, 9000, 2500, 20000]
    pos, vel, lab, at = [], [], [], 0
    for k, (n, step) in enumerate(zip(sizes, steps)):
        p = np.round(rng.normal(0, 40000 / step, size=(n, 3))).astype(np.int64) * step
        pos.append((p + 400000 * k) % L)
        vel.append(rng.normal(0, 80, size=(n, 3)))
        lab.append(np.full(n, at))
        at += n
    pos = np.concatenate(pos).astype(np.int32)
    vel = np.concatenate(vel).astype(np.float32)
    lab = np.concatenate(lab).astype(np.int32)
    fl = np.exp(rng.normal(-12, 1, at)).astype(np.float32)
    d = [_dev(pos), _dev(vel), _dev(fl), _dev(lab)]
    first = None
    for _ in range(20):
        R, _, hs = ctx.outlier_ratio(*d, Params.default())
        ctx.sync()
        got = R.cpu().numpy(), hs.cpu().numpy()[:, 11]
        if first is None:
            first = got
        assert np.array_equal(got[0], first[0], equal_nan=True) and np.array_equal(got[1], first[1])
    o = 0
    for k, n in enumerate(sizes):
        m = np.arange(o, o + n)
        ref, leaf, _ = oracle.background_halo(oracle.unwrap(pos, m), vel, m, fl[m].astype(np.float64))
        assert first[1][k] == len(np.unique(leaf))
        fin = np.isfinite(ref)
        assert np.array_equal(np.isfinite(first[0][m]), fin)
        assert (np.abs(first[0][m][fin] - ref[fin]) <= 1e-4 * np.maximum(1.0, np.abs(ref[fin]))).all()
        o += n


# ------------------------------------------------------------------ labels out of range
@pytest.mark.parametrize("bad", [-1, -(1 << 31), 5000, (1 << 31) - 1])
@pytest.mark.parametrize("call", ["velden", "fof6d_field", "find_substructure"])
def test_label_out_of_range_is_refused(ctx, call, bad):
    """One label outside [0, n) among 5,000: VR_ERR_INVALID_ARG, and the next call on the
    context works."""
    from paper_1902_01010_gb300 import VrError

    rng = np.random.default_rng(3)
    n = 5000
    pos = _dev(rng.integers(0, 40000, size=(n, 3)).astype(np.int32))
    vel = _dev(rng.normal(0, 50, (n, 3)).astype(np.float32))
    good = np.zeros(n, np.int32)
    want = ctx.velden(pos, vel, _dev(good))
    ctx.sync()
    lab = good.copy()
    lab[3777] = bad
    with pytest.raises(VrError) as e:
        if call == "velden":
            ctx.velden(pos, vel, _dev(lab))
        elif call == "fof6d_field":
            ctx.fof6d_field(pos, vel, _dev(lab), 1000.0)
        else:
            ctx.find_substructure(pos, vel, _dev(lab), 1000.0, 1.0)
        ctx.sync()
    assert e.value.code == 1 and "label" in str(e.value)
    got = ctx.velden(pos, vel, _dev(good))
    ctx.sync()
    assert torch.equal(got, want)


# ------------------------------------------------- 3D FOF with the shortest linking lengths
@pytest.mark.parametrize("T", [1, 2, 3, 4])
@pytest.mark.parametrize("n", [0, 3000, 40000])
def test_fof_shortest_linking_lengths(ctx, T, n):
    """Sub-cells of one lattice point. Points that differ by half the box along any axes share
    all but the top bit of each coordinate; around them clumps of lattice neighbours, across
    the periodic edge too, and cells of more members than one warp tests at once."""
    rng = np.random.default_rng(10 * T + n)
    h = 1 << 20
    corners = np.stack(np.meshgrid(*[[0, h]] * 3, indexing="ij"), -1).reshape(-1, 3) + 5
    pos = [corners, corners, corners + [1, 0, 0], corners + [0, 1, 1], corners - 6]
    if n:
        ctr = np.concatenate([rng.integers(0, L, size=(20, 3)), [[0, 0, 0], [h, h, h], [L - 1, 3, h - 1]]])
        pos.append(ctr[rng.integers(0, len(ctr), n)] + rng.integers(-6, 7, size=(n, 3)))
        pos.append(rng.integers(0, L, size=(n // 3, 3)))
    pos = (np.concatenate(pos) % L).astype(np.int32)
    pos = pos[rng.permutation(len(pos))]
    lab = ctx.fof3d(_dev(pos), T)
    ctx.sync()
    assert np.array_equal(lab.cpu().numpy(), oracle.fof3d(pos, T))


# ---------------------------------------- f_l: more members in one bin than 16 bits count
@pytest.mark.parametrize("n,near,gap,spread", [
    (65536, 0, 0, 0), (70000, 0, 0, 0), (131072, 0, 0, 0),          # all at one point
    (65600, 100, 5000, 0), (65600, 100, 40000, 0),                  # all at one distance
    (65700, 40, 5000, 2), (131200, 100, 40000, 2), (66000, 255, 20000, 30)])
def test_fl_bins_of_more_than_16_bits(ctx, n, near, gap, spread):
    """`n` members in a clump and `near` others at a distance of `gap`, for which the whole clump
    lies in one bin of a level; N_se = 256 of them decided by the particle index where the
    separations are equal."""
    from paper_1902_01010_gb300 import Params

    rng = np.random.default_rng(n + gap)
    p = np.concatenate([[gap, 0, 0] + np.round(rng.uniform(-spread, spread, (n, 3))),
                        np.round(rng.uniform(-20, 20, (near, 3)))]).astype(np.int64)
    p = p[rng.permutation(len(p))]
    pos = ((p + 700000) % L).astype(np.int32)
    vel = rng.normal(0, 80, size=pos.shape).astype(np.float32)
    lab = np.zeros(len(pos), np.int32)
    got = ctx.velden(_dev(pos), _dev(vel), _dev(lab), Params.default())
    ctx.sync()
    got = got.cpu().numpy()
    m = np.arange(len(pos))
    up = oracle.unwrap(pos, m)
    few = np.flatnonzero(p[:, 0] < gap - spread)
    for k in np.r_[rng.integers(0, len(pos), 12), few[:24]].astype(int):
        ref = oracle.velden_one(up, vel, m, int(k))
        assert abs(got[k] - ref) <= 1e-4 * ref, k


# ------------------------------------------------------- contexts on several host threads
def test_contexts_on_host_threads_with_different_bin_counts():
    """One context per host thread is a documented use: calls with few and with many fit bins
    at the same time all succeed and give what each gives alone."""
    import ctypes
    import threading

    from paper_1902_01010_gb300 import Context, Params, lib
    from paper_1902_01010_gb300.vr import HALO_COLS, _ptr

    rng = np.random.default_rng(9)
    n = 300
    pos = _dev((np.round(rng.normal(0, 30000, (n, 3))).astype(np.int64) % L).astype(np.int32))
    vel = _dev(rng.normal(0, 80, (n, 3)).astype(np.float32))
    fl = _dev(np.exp(rng.normal(-12, 1, n)).astype(np.float32))
    lab = torch.zeros(n, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    bins = [1024, 1024] + 6 * [200]
    alone = {b: Context(0).outlier_ratio(pos, vel, fl, lab, Params.default(fit_nbins_max=b))[1].cpu()
             for b in set(bins)}
    errors, call = [], lib().vr_outlier_ratio
    start = threading.Barrier(len(bins))

    def work(b):
        try:
            c, s, P, nh = Context(0), torch.cuda.Stream(), Params.default(fit_nbins_max=b), ctypes.c_int64()
            with torch.cuda.stream(s):
                ws = c.workspace(n, P)
                R, ell = (torch.empty(n, dtype=torch.float32, device="cuda") for _ in range(2))
                hs = torch.empty((n // P.nmin + 1, HALO_COLS), dtype=torch.float64, device="cuda")
            args = (c.h, _ptr(pos), _ptr(vel), _ptr(fl), n, _ptr(lab), ctypes.byref(P), _ptr(R), _ptr(ell),
                    _ptr(hs), ctypes.byref(nh), _ptr(ws), ws.numel(), ctypes.c_void_p(s.cuda_stream))
            start.wait()
            for _ in range(1000):
                c.check(call(*args))
            s.synchronize()
            assert torch.equal(ell.cpu(), alone[b])
        except Exception as e:  # noqa: BLE001
            errors.append(f"{b} bins: {e}")

    threads = [threading.Thread(target=work, args=(b,)) for b in bins]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors


# --------------------------------------------------- the fit's median and MAD, to the last bit
def _mad(x):
    """1.4826 median |x - median(x)| of the finite values, in FP64 as the fit defines it."""
    x = np.sort(x[np.isfinite(x)].astype(np.float64))
    n = len(x)
    med = x[n // 2] if n & 1 else 0.5 * (x[n // 2 - 1] + x[n // 2])
    d = np.sort(np.abs(x - med))
    return 1.4826 * (d[n // 2] if n & 1 else 0.5 * (d[n // 2 - 1] + d[n // 2]))


def _ratio_of(ctx, target, seed):
    """A halo with f_l chosen such that R comes out as `target` to the last FP32 bit, with no
    iterations of the fit: sigma_R is MAD' then. Returns (R, halo rows)."""
    from paper_1902_01010_gb300 import Params

    n = len(target)
    rng = np.random.default_rng(seed)
    pos = (np.round(rng.normal(0, 30000, (n, 3))).astype(np.int64) % L).astype(np.int32)
    d = [_dev(pos), _dev(rng.normal(0, 0.4, (n, 3)).astype(np.float32)), None,
         torch.zeros(n, dtype=torch.int32, device="cuda")]
    P = Params.default(fit_iters=0)
    ln_fl = np.zeros(n)
    for _ in range(4):
        d[2] = _dev(np.exp(ln_fl).astype(np.float32))
        R, _, hs = ctx.outlier_ratio(d[0], d[1], d[2], d[3], P)
        ctx.sync()
        R = R.cpu().numpy()
        if np.array_equal(R, target.astype(np.float32)):
            break
        ln_fl += target - R.astype(np.float64)
    return R, hs.cpu().numpy()


@pytest.mark.parametrize("n", [160, 161, 400, 1001, 4000, 16384, 20001, 40000])
@pytest.mark.parametrize("centre,width", [(0.05, 0.4), (3.0, 4.0), (-20.0, 0.05), (0.0, 12.0)])
def test_mad_is_exact(ctx, n, centre, width):
    """Odd and even counts, with MADs well below and above 1 and far from the median's size."""
    rng = np.random.default_rng(n)
    R, hs = _ratio_of(ctx, rng.normal(centre, width, n), n)
    assert hs[0, 4] == _mad(R)


def test_mad_of_values_on_either_side_of_a_key_edge(ctx):
    """An even count whose median lies half an ulp off the FP32 grid: of the two values next
    below the middle distance, one below and one above the median, the FP32 distances have
    the order that the exact ones have not."""
    u = 2.0 ** -18                      # spacing of FP32 in [32, 64)
    b = 32.0 + 2 * u                    # even mantissa: the median b + u/2 rounds down to it
    edge, top = 0.75 - 2.0 ** -15, 0.75
    up = lambda dist: b + dist
    dn = lambda dist: b - dist
    rng = np.random.default_rng(4)
    grid = lambda x, g: np.round(x / g) * g
    small = grid(rng.uniform(0.1, 0.6, 96), u)
    big = grid(rng.uniform(1.2, 1.9, 99), u)
    x = np.r_[b, b + u, up(edge), dn(edge - u / 2), up(top + 3 * u),
              up(small[:48]), dn(small[48:]), up(big[:49]), dn(big[49:])]
    assert len(x) == 200 and (x > b + u / 2).sum() == 100 and np.array_equal(x, x.astype(np.float32))
    R, hs = _ratio_of(ctx, x, 1)
    assert np.array_equal(R, x.astype(np.float32))
    assert hs[0, 4] == _mad(R)


# -------------------------------------------------------- the shape that a launch takes
def test_tuning_report_names_the_shapes_of_untuned_launches():
    """1.1 M members in one halo are more than 32,768 buckets, 5,000 are few: each takes the
    shape of its size, and the report names it; a forced shape is named instead."""
    from paper_1902_01010_gb300 import Context

    c = Context(0)
    assert c.tuning_report()["f_l"]["chosen"] == [0, 0, 0]
    rng = np.random.default_rng(8)

    def call(n):
        pos = _dev((np.round(rng.normal(0, 60000, (n, 3))).astype(np.int64) % L).astype(np.int32))
        c.velden(pos, _dev(rng.normal(0, 80, (n, 3)).astype(np.float32)),
                 torch.zeros(n, dtype=torch.int32, device="cuda"))
        c.sync()
        rep = c.tuning_report()["f_l"]
        return [rep["shapes"][k]["warps"] for k in rep["chosen"]]

    assert call(1_100_000) == [2, 4, 4]
    assert call(5000) == [2, 4, 4]  # the middle bin's; the first had no launch
    c.tuning_force(1, -1)
    assert call(5000) == [8, 8, 8]
    c.tuning_force(-1, -1)
    assert call(5000) == [2, 4, 4]


# ------------------------------------------- core moments: clusters for large halos' cores
@pytest.mark.parametrize("small", [300, 5000])
def test_core_moments_of_many_halos_beside_a_large_one(ctx, small):
    """300 halos of two cores, whose moments a block takes each (also where a halo alone in the
    box, of 5,000 members, would have a cluster), and one of 13,000 members, which has."""
    from test_gpu_coregrow import _check

    rng = np.random.default_rng(small)
    g = np.stack(np.meshgrid(*[np.arange(5)] * 3, indexing="ij"), -1).reshape(-1, 3) * 500
    sizes, pos, vel, lab = [13000] + 300 * [small], [], [], []
    for n in sizes:
        base = np.array([100000, 100000, 100000])
        d = rng.normal(size=(n - 2 * len(g), 3))
        d = d / np.linalg.norm(d, axis=1)[:, None] * rng.uniform(9000, 90000, (len(d), 1))
        pos += [g + base, g + base + [3500, 0, 0], np.round(base + [3250, 1500, 1500] + d)]
        vel += [rng.normal(0, 0.3, size=(len(g), 3)) + [s, 0, 0] for s in (200, -200)]
        vel.append(rng.normal(0, 60, size=(len(d), 3)))
        lab.append(np.full(n, sum(map(len, lab))))
    pos, vel = np.vstack(pos).astype(np.int32), np.vstack(vel).astype(np.float32)
    core, grown, kept = _check(ctx, pos, vel, np.concatenate(lab).astype(np.int32), None, 700.0,
                               halos=[0, 1, 150, 300], f_c=0.005)
    assert kept == 2 * len(sizes) and (grown != core).any()


# ---------------------------------------------- 3D FOF: thousands of particles a sub-cell
@pytest.mark.parametrize("n,spread,T", [(40000, 100, 5000 ** 2), (33, 1, 9), (50000, 2000, 5000 ** 2),
                                        (4097, 300, 900 ** 2)])
def test_fof_crowded_sub_cells(ctx, n, spread, T):
    """A clump across the corner where eight sub-cells (and the box's periodic edges) meet, a
    second one out of reach, and single particles between sub-cells of many."""
    rng = np.random.default_rng(n)
    p = np.concatenate([rng.normal(0, spread, (n, 3)), rng.normal(300000, spread, (n // 2, 3)),
                        rng.integers(0, L, (200, 3))])
    pos = (np.round(p).astype(np.int64) % L).astype(np.int32)
    pos = pos[rng.permutation(len(pos))]
    lab = ctx.fof3d(_dev(pos), T)
    ctx.sync()
    assert np.array_equal(lab.cpu().numpy(), oracle.fof3d(pos, T))


# ------------------------------------------------ 6D links far from the halo frame's origin
@pytest.mark.parametrize("bulk", [3000.0, 1.0e6])
@pytest.mark.parametrize("v_ratio,theta,use_lv", [(2.0, 0.314, 1), (1.2, 0.9, 0), (1.05, 1.5, 0), (5.0, 1.57, 1)])
def test_links_with_a_bulk_velocity_far_above_the_dispersion(ctx, bulk, v_ratio, theta, use_lv):
    """Velocities a few FP32 spacings from a halo velocity that lies between them: the rounding
    of the frame is a good part of every member's velocity in it."""
    from paper_1902_01010_gb300 import Params

    rng = np.random.default_rng(int(bulk))
    ulp = float(np.spacing(np.float32(bulk)))
    n = 1500
    pos = (rng.integers(0, 9, (n, 3)) * 500 + 3000).astype(np.int32)
    k = np.where(rng.random((n, 1)) < 0.5, rng.integers(-9, 10, (n, 3)), rng.integers(-60, 61, (n, 3)))
    vel = (bulk + k * ulp).astype(np.float32)
    ell = np.where(rng.random(n) < 0.8, 3.0, 1.0).astype(np.float32)
    for frac in ([0.5, 0.5, 0.5], [0.49, -0.5, 0.26], [0.0, 0.5, -0.37]):
        hs = np.zeros((1, 12))
        hs[0, :3] = [0, n, 1]
        hs[0, 5:8] = bulk + np.array(frac) * ulp
        hs[0, 9], hs[0, 10] = 500.0 ** 2 * 1.5, (14 * ulp) ** 2
        P = Params.default(nsearch_min=20, nmin=2, use_lv=use_lv, v_ratio=v_ratio, theta_op=theta)
        got = ctx.fof6d(_dev(pos), _dev(vel), _dev(ell), _dev(np.zeros(n, np.int32)), _dev(hs), P)
        ctx.sync()
        m = np.arange(n)
        ref = oracle.fof6d_halo(oracle.unwrap(pos, m), vel, m, (ell >= 2.5).astype(np.uint8),
                                hs[0, [9, 10, 5, 6, 7]], v_ratio, theta, use_lv=use_lv, nmin=2)
        assert np.array_equal(got.cpu().numpy(), ref)
        assert len(np.unique(ref)) > 2


@pytest.mark.parametrize("bad", [600, (1 << 31) - 1])
def test_stage_1_label_out_of_range_is_refused(ctx, bad):
    """A label6 of n or more among the groups to grow: VR_ERR_INVALID_ARG, and the next call works."""
    from paper_1902_01010_gb300 import VrError

    rng = np.random.default_rng(5)
    n = 600
    pos, vel = _dev(rng.integers(0, 4000, (n, 3)).astype(np.int32)), _dev(rng.normal(0, 50, (n, 3)).astype(np.float32))
    ell, lab = _dev(np.full(n, 3.0, np.float32)), torch.zeros(n, dtype=torch.int32, device="cuda")
    hs = np.zeros((1, 12))
    hs[0, :3] = [0, n, 1]
    hs[0, 9], hs[0, 10] = 300.0 ** 2, 40.0 ** 2
    good = ctx.fof6d(pos, vel, ell, lab, _dev(hs))
    ctx.sync()
    want = good.clone()
    ctx.grow_groups(pos, vel, ell, lab, _dev(hs), want)
    l6 = good.clone()
    l6[123] = bad
    with pytest.raises(VrError) as e:
        ctx.grow_groups(pos, vel, ell, lab, _dev(hs), l6)
        ctx.sync()
    assert e.value.code == 1 and "stage-1 label" in str(e.value)
    got = good.clone()
    ctx.grow_groups(pos, vel, ell, lab, _dev(hs), got)
    ctx.sync()
    assert torch.equal(got, want)


# ------------------------------------- 6D links in flat, elongated and clumped-up halos
@pytest.mark.parametrize("shape", ["line", "plane", "filament", "two clumps", "duplicates"])
@pytest.mark.parametrize("n", [33, 1000, 5000])
def test_links_in_flat_and_elongated_halos(ctx, shape, n):
    """Halos that fill few cells of their bounding cube, where a tile of 32 members may lie on a
    jump of the curve: the field 6DFOF, and the two-stage linking of its smaller groups."""
    from paper_1902_01010_gb300 import GrowParams, Params

    rng = np.random.default_rng(n)
    z = np.zeros(n)
    p = {"line": np.stack([rng.integers(0, 2 * n, n), z, z], 1),
         "plane": np.stack([rng.integers(0, 9000, n), rng.integers(0, 9000, n), z], 1),
         "filament": np.stack([rng.integers(0, 3 * n, n), rng.normal(0, 300, n), rng.normal(0, 300, n)], 1),
         "two clumps": rng.normal(0, 500, (n, 3)) + rng.choice([0, 300000], (n, 1)),
         "duplicates": np.repeat(rng.integers(0, 5000, (n // 7 + 1, 3)), 7, 0)[:n]}[shape]
    pos = ((np.round(p).astype(np.int64) + 1000) % L).astype(np.int32)[rng.permutation(n)]
    vel = rng.normal(0, 80, (n, 3)).astype(np.float32)
    lab = np.zeros(n, np.int32)
    P = Params.default(nsearch_min=20, nmin=4)
    got, hs = ctx.fof6d_field(_dev(pos), _dev(vel), _dev(lab), 400.0, 1.25, P)
    ctx.sync()
    m = np.arange(n)
    up = oracle.unwrap(pos, m)
    row = hs[0].cpu().numpy()
    ref = oracle.fof6d_halo(up, vel, m, np.ones(n, np.uint8), row[[9, 10, 5, 6, 7]], use_vt=0, nmin=4)
    assert np.array_equal(got.cpu().numpy(), ref)
    # two-stage linking: outliers of a tighter linking, grown with the relaxed criteria
    ell = rng.uniform(1.5, 4.0, n).astype(np.float32)
    prm = np.array([250.0 ** 2, 60.0 ** 2, 0, 0, 0])
    hs2 = np.zeros((1, 12))
    hs2[0, :3] = [0, n, 1]
    hs2[0, 9:11] = prm[:2]
    args = dict(v_ratio=3.0, theta_op=1.2)
    P = Params.default(nsearch_min=20, nmin=4, **args)
    l6 = ctx.fof6d(_dev(pos), _dev(vel), _dev(ell), _dev(lab), _dev(hs2), P)
    ctx.sync()
    one = oracle.fof6d_halo(up, vel, m, (ell >= 2.5).astype(np.uint8), prm, nmin=4, **args)
    assert np.array_equal(l6.cpu().numpy(), one)
    ctx.grow_groups(_dev(pos), _dev(vel), _dev(ell), _dev(lab), _dev(hs2), l6, P, GrowParams.default())
    ctx.sync()
    two = oracle.grow_halo(up, vel, m, ell, one, prm, ell_th=2.5, **args)
    assert np.array_equal(l6.cpu().numpy(), two)
