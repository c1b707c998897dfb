"""Imported offsets that leave the frame, as a matcher marks pixels it found no match for."""
import numpy as np
import pytest

from paper_1804_03787_gb300 import gpm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("zoom", [1.0, 1.9])
@pytest.mark.parametrize("mark", [(1 << 30, 1 << 30), (1 << 30, 0), (-(1 << 31), 1 << 30), (5, -9)])
def test_recost_of_far_offsets_on_a_frame_narrower_than_the_patch(mark, zoom):
    """A plane of scale 1.9 spreads the taps of a 9 x 9 patch wider than an 8 x 8 frame: no offset keeps them inside, and
    every one of these offsets puts every sample (tap displacements stay below 8 px) beyond the frame on each axis that is
    far, where it reads the border texels."""
    import torch
    W = H = 8
    gp = gpm.default_params(patch_radius=4, cells=(8,), pm_iters=0, num_hyp=32, gain_normalize=0)
    rng = np.random.default_rng(8)
    f1, f2 = (rng.random((H, W, 3)).astype(np.float32) for _ in range(2))
    ctx = gpm.Context(gp, W, H)
    ctx.match([(torch.from_numpy(f1).cuda(), torch.from_numpy(f2).cuda())])
    n, m = W * H, ctx.export(gpm.MODELS).shape[1]
    c = 3.5 - 3.5 * zoom
    mh = np.tile(np.array([zoom, 0, c, 0, zoom, c, 0, 0, 1.0]), (2, m, 1))
    mi = ctx.export(gpm.MODEL_INFO).copy()
    mi[:, :, 0] = 1
    nnf = np.tile(np.array(mark, np.int32), (2, n, 1))
    for what, data in ((gpm.NNF, nnf), (gpm.MODELS, mh), (gpm.MODEL_INFO, mi),
                       (gpm.LABELS, (np.full((2, n), -1, np.int32), np.full((2, n), 0.06, np.float32), np.zeros((2, n, 2))))):
        ctx.import_state(what, data, 1, after_fit=True)
    ctx.match(None, 1)
    got = ctx.export(gpm.COST)
    ctx.close()
    d = np.arange(-4, 5)
    p = np.arange(8)
    tap = np.clip(p[:, None] + d, 0, 7)                                  # [pixel][tap] on one axis
    at = [np.clip(p[:, None] + v + zoom * (tap - p[:, None]), 0, 7) for v in map(float, mark)]
    lo = [np.minimum(np.floor(a).astype(int), 6) for a in at]
    for k, (a, b) in enumerate(((f1, f2), (f2, f1))):
        a, b = a.astype(np.float64), b.astype(np.float64)
        rows = b[lo[1]] * (1 - (at[1] - lo[1]))[..., None, None] + b[lo[1] + 1] * (at[1] - lo[1])[..., None, None]
        wx = (at[0] - lo[0])[:, None, None, :, None]
        s = rows[:, :, lo[0]].transpose(2, 0, 1, 3, 4) * (1 - wx) + rows[:, :, lo[0] + 1].transpose(2, 0, 1, 3, 4) * wx
        src = a[tap[:, :, None, None], tap[None, None]].transpose(2, 0, 1, 3, 4)  # [x][y][ty][tx][channel]
        want = np.abs(src - s).mean((2, 3, 4)).T.reshape(-1)
        # tap positions to 1e-6 px, blends and sums to some 1e-6: far below the differences of wrong texels (0.1)
        assert np.abs(np.asarray(got[k]).reshape(-1) - want).max() < 1e-5


@pytest.mark.parametrize("mark,motion", [((1 << 20, 1 << 20), 0), ((65536 + 3, 0), 3)])
def test_level0_sweeps_replace_far_incumbents(mark, motion):
    """Half the pixels start from a marker equal to the motion modulo 2^16, among neighbours that hold the motion: a pixel that
    takes it over must store it."""
    import torch

    import oracle as O

    from _parity import TIE, dilate, oracle_frames, oracle_params
    W, H = 61, 43
    gp = gpm.default_params(patch_radius=2, cells=(), pm_iters=2, num_hyp=64, pm_init=0, gain_normalize=0)
    P = oracle_params(gp, W, H)
    rng = np.random.default_rng(5)
    f1 = rng.random((H, W, 3)).astype(np.float32)
    f2 = (np.roll(f1, motion, 1) * 0.99 + 0.01 * rng.random((H, W, 3))).astype(np.float32)
    truth = np.stack([np.tile((m, 0), (W * H, 1)) for m in (motion, -motion)])
    far = np.stack([np.tile(mark, (W * H, 1)), np.tile((mark[0] - 2 * motion, mark[1]), (W * H, 1))])
    nnf = np.where(rng.random((2, W * H, 1)) < 0.5, far, truth).astype(np.int32)
    ctx = gpm.Context(gp, W, H)
    pair = (torch.from_numpy(f1).cuda(), torch.from_numpy(f2).cuda())
    ctx.match([pair])
    ctx.import_state(gpm.NNF, nnf, level=0)
    ctx.match([pair])
    got = ctx.export(gpm.NNF)
    ctx.close()
    frames, _ = oracle_frames(P, f1, f2)
    for d in range(2):
        vx, vy = (np.ascontiguousarray(nnf[d][:, c]) for c in range(2))
        c = np.zeros(W * H)
        O.pm_recost(P, *frames[d], 0, None, None, None, vx, vy, c)
        cone = np.zeros((H, W), bool)
        for k in range(2 * P.pm_iters):
            amb = np.full(W * H, np.inf)
            O.pm_sweep(P, *frames[d], d, 0, k >> 1, k & 1, None, None, None, vx, vy, c, amb)
            cone |= dilate((amb < TIE).reshape(H, W), 2 * P.pm_iters - 1 - k)
        sure = ~cone.reshape(-1)
        assert sure.mean() > 0.5
        assert (got[d][:, 0] == vx)[sure].all() and (got[d][:, 1] == vy)[sure].all()


def _marked(W, H, seed, mark, share):
    """Two motions (left and right part) with a sixth of the offsets random, and a share of the pixels marked."""
    rng = np.random.default_rng(seed)
    y, x = np.mgrid[0:H, 0:W].astype(np.float64)
    t = np.where((x < 0.6 * W)[..., None], np.stack([1.01 * x + 0.02 * y + 3, 0.99 * y - 0.015 * x - 2], -1),
                 np.stack([x - 11 + 0.05 * y, y * 1.04 + 6], -1)) + rng.normal(0, 0.4, (H, W, 2))
    t = np.where((rng.random((H, W)) < 1 / 6)[..., None], rng.random((H, W, 2)) * (W, H), t)
    v = np.rint(t - np.stack([x, y], -1)).astype(np.int64)
    v[rng.random((H, W)) < share] = mark
    return np.ascontiguousarray(v.reshape(-1, 2).astype(np.int32))


# windows of 8 and 16 px (a warp each), 18 px with 512 threads a window, and 18 px with 256 (more than 456 windows)
@pytest.mark.parametrize("W,H,s,hyp", [(37, 29, 8, 96), (53, 41, 16, 128), (41, 30, 18, 96), (200, 160, 18, 257)])
@pytest.mark.parametrize("share", [0.1, 0.55, 0.75])
@pytest.mark.parametrize("mark", [1 << 20, -(1 << 20), 1 << 23, -(1 << 23), 1 << 30, -(1 << 30), -(1 << 31)])
def test_planes_of_marked_fields_equal_oracle(mark, share, W, H, s, hyp):
    """Markers are matches like any other: outliers of a window's motion, or its plane where they prevail."""
    import torch

    import oracle as O

    from _parity import oracle_params, ransac_equal
    gp = gpm.default_params(patch_radius=2, cells=(s,), pm_iters=0, num_hyp=hyp)
    P = oracle_params(gp, W, H)
    f = np.random.default_rng(s).random((H, W, 3)).astype(np.float32) * 0.2 + 0.4
    nnf = np.stack([_marked(W, H, 10 * s + d, mark, share) for d in range(2)])
    ctx = gpm.Context(gp, W, H)
    fr = torch.from_numpy(f).cuda()
    ctx.match([(fr, fr.clone())])
    ctx.import_state(gpm.NNF, nnf, level=0)
    ctx.fit_planes(1)
    gmh, gmi = ctx.export(gpm.MODELS), ctx.export(gpm.MODEL_INFO)
    ctx.close()
    frame = np.asarray(f, np.float64)
    first = np.arange(int(O.cell_base(P)[1])) * 2
    for d in range(2):
        mh, mi = O.empty_models(P)
        vx, vy = (np.ascontiguousarray(nnf[d][:, c]) for c in range(2))
        O.fit_level(P, frame, frame, d, 1, 1, vx, vy, None, mh, mi)
        sure = first[(mi[first, O.MI_FLAGS] & O.F_AMBIG) == 0]
        assert len(sure) > len(first) // 4
        bad = sure[~ransac_equal(gmh[d], gmi[d], mh, mi, sure)]
        assert len(bad) == 0, f"dir {d}: windows {bad // 2} differ"


def test_far_windows_are_fitted_by_graphs_captured_before_an_import():
    """A fit captured before the field is imported serves far windows all the same; whole runs, which replace the field, take
    the launches of before once more afterwards."""
    import torch
    W, H, s = 53, 41, 16
    gp = gpm.default_params(patch_radius=2, cells=(s,), pm_iters=0, num_hyp=64)
    f = torch.from_numpy(np.random.default_rng(3).random((H, W, 3)).astype(np.float32)).cuda()
    nnf = np.stack([_marked(W, H, 7 + d, 1 << 20, 0.2) for d in range(2)])
    st = torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(st):
        ctx = gpm.Context(gp, W, H, stream=st)
        counts = []
        for _ in range(2):
            n = ctx.launch_count()
            ctx.run([(f, f)])
            counts.append(ctx.launch_count() - n)
            ctx.match([(f, f)])
            ctx.import_state(gpm.NNF, nnf, level=0)
            ctx.fit_planes(1)
            want = ctx.export(gpm.MODEL_INFO), ctx.export(gpm.MODELS)
        assert counts[0] == counts[1]
        ctx.close()
        ctx = gpm.Context(gp, W, H, stream=st)
        ctx.match([(f, f)])
        ctx.sync()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            ctx.fit_planes(1)
        ctx.import_state(gpm.NNF, nnf, level=0)
        g.replay()
        got = ctx.export(gpm.MODEL_INFO), ctx.export(gpm.MODELS)
        ctx.close()
    assert (want[0][:, ::2, 1] > 0).any()  # inliers: the cues drop these planes later
    assert (got[0] == want[0]).all() and (got[1] == want[1]).all()


def test_far_flows_of_imported_labels_reach_the_next_level_exactly():
    """A merge makes the flows of imported labels the pixels' offsets: the fit after it takes them as it takes an imported
    field with the same offsets."""
    import torch

    import oracle as O

    from _parity import oracle_params
    W, H = 53, 41
    gp = gpm.default_params(patch_radius=2, cells=(16, 8), pm_iters=2, num_hyp=64)
    rng = np.random.default_rng(9)
    f = torch.from_numpy(rng.random((H, W, 3)).astype(np.float32)).cuda()
    far = rng.random((2, W * H)) < 0.3
    labels = (np.where(far, 0, -1).astype(np.int32), np.zeros((2, W * H), np.float32),
              np.where(far[..., None], 2.0**29, 0.0) + np.zeros(2))
    got = []
    for again in (False, True):
        ctx = gpm.Context(gp, W, H)
        ctx.match([(f, f)])
        ctx.import_state(gpm.LABELS, labels, level=0)
        ctx.fit_planes(1)
        ctx.match(None, 1)
        field = ctx.export(gpm.NNF)
        assert (field[far] == 1 << 29).all()
        if again:
            ctx.import_state(gpm.NNF, field, level=1)
        ctx.fit_planes(2)
        got.append((ctx.export(gpm.MODEL_INFO), ctx.export(gpm.MODELS)))
        ctx.close()
    level2 = 2 * int(O.cell_base(oracle_params(gp, W, H))[1])
    assert (got[1][0][:, level2::2, 1] >= 32).any()  # planes of the near matches, half of a window and more
    assert (got[0][0] == got[1][0]).all() and (got[0][1] == got[1][1]).all()


@pytest.mark.parametrize("W,H,s,hyp", [(53, 41, 16, 128), (37, 29, 8, 96), (41, 30, 18, 96), (200, 160, 18, 257)])
@pytest.mark.parametrize("gain", [30.0, 300.0])
def test_planes_that_reach_far_equal_oracle(gain, W, H, s, hyp):
    """A projective motion whose vanishing line passes just beyond the right border: inliers of one plane lie 10^4 to 10^6 px
    apart, too far for 32-bit sums."""
    import torch

    import oracle as O

    from _parity import oracle_params, ransac_equal
    gp = gpm.default_params(patch_radius=2, cells=(s,), pm_iters=0, num_hyp=hyp, min_inliers=4)
    P = oracle_params(gp, W, H)
    f = np.random.default_rng(s).random((H, W, 3)).astype(np.float32) * 0.2 + 0.4
    y, x = np.mgrid[0:H, 0:W].astype(np.float64)
    den = 1 - (x + 0.1 * y) / (W + 0.1 * H)
    v = np.stack([np.rint(gain * (x - W / 2) / den) - x, np.rint(gain * (y - H / 2) / den) - y], -1).reshape(-1, 2).astype(np.int32)
    assert np.abs(v).max() > 16383  # beyond what a window holds as near
    nnf = np.stack([v, v[::-1]])
    ctx = gpm.Context(gp, W, H)
    fr = torch.from_numpy(f).cuda()
    ctx.match([(fr, fr.clone())])
    ctx.import_state(gpm.NNF, nnf, level=0)
    ctx.fit_planes(1)
    gmh, gmi = ctx.export(gpm.MODELS), ctx.export(gpm.MODEL_INFO)
    ctx.close()
    frame = np.asarray(f, np.float64)
    first = np.arange(int(O.cell_base(P)[1])) * 2
    for d in range(2):
        mh, mi = O.empty_models(P)
        vx, vy = (np.ascontiguousarray(nnf[d][:, c]) for c in range(2))
        O.fit_level(P, frame, frame, d, 1, 1, vx, vy, None, mh, mi)
        sure = first[(mi[first, O.MI_FLAGS] & O.F_AMBIG) == 0]
        assert len(sure) > len(first) // 4
        bad = sure[~ransac_equal(gmh[d], gmi[d], mh, mi, sure)]
        assert len(bad) == 0, f"dir {d}: windows {bad // 2} differ"


@pytest.mark.parametrize("mark", [(1 << 24) + 3, -(1 << 30) - 12345, (1 << 31) - 129])
def test_planes_of_markers_that_are_no_floats_equal_oracle(mark):
    """Far offsets that FP32 rounds by more than the inlier radius: the refit is tested on the matches as they are."""
    test_planes_of_marked_fields_equal_oracle(mark, 0.75, 53, 41, 16, 128)
    test_planes_of_marked_fields_equal_oracle(mark, 0.75, 41, 30, 18, 96)
