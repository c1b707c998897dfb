"""The per-window RANSAC search (both stages) against the oracle, at the sizes where its paths meet: window sides
around the one-warp limits (8, 16) and with ragged quads and chunks of matches, hypothesis counts around a batch of
32 and a round of 256, and windows whose imported offsets reach too far for the FP32 solve."""
import numpy as np
import pytest

import oracle as O
from paper_1804_03787_gb300 import gpm

from _parity import oracle_params

pytestmark = pytest.mark.gpu


def _matches(W, H, seed, far):
    """Two projective motions (left and right part), a sixth of the offsets random, a few far out of the frame."""
    rng = np.random.default_rng(seed)
    y, x = np.mgrid[0:H, 0:W].astype(np.float64)
    den = 1 + 4e-4 * (x - W / 2) - 3e-4 * y
    a = np.stack([(1.01 * x + 0.02 * y + 3) / den, (0.99 * y - 0.015 * x - 2) / den], -1)
    b = np.stack([x - 11 + 0.05 * y, y * 1.04 + 6], -1)
    t = np.where((x < 0.6 * W)[..., None], a, b) + rng.normal(0, 0.4, (H, W, 2))
    v = np.rint(t - np.stack([x, y], -1)).astype(np.int32)
    r = rng.random((H, W)) < 1 / 6
    rnd = np.stack([rng.integers(0, W, (H, W)), rng.integers(0, H, (H, W))], -1) - np.stack([x, y], -1).astype(np.int64)
    v[r] = rnd[r]
    if far:
        v[rng.random((H, W)) < 0.02] = (40000, -30000)
    return np.ascontiguousarray(v.reshape(-1, 2).astype(np.int32))


@pytest.mark.parametrize("s,hyp,far", [(4, 33, False), (6, 64, False), (8, 257, False), (8, 96, True), (10, 31, False),
                                       (16, 600, False), (16, 64, True), (18, 1, False), (18, 257, False),
                                       (34, 256, False), (34, 300, True), (64, 512, False), (96, 64, False)])
def test_ransac_search_equals_oracle(s, hyp, far):
    import torch
    W, H = max(2 * s + 5, 20), max(s + s // 2 + 3, 17)
    gp = gpm.default_params(patch_radius=2, cells=(s,), pm_iters=0, num_hyp=hyp)
    P = oracle_params(gp, W, H)
    f = np.random.default_rng(s).random((H, W, 3)).astype(np.float32) * 0.2 + 0.4
    nnf = np.stack([_matches(W, H, 10 * s + d, far) for d in range(2)])
    ctx = gpm.Context(gp, W, H)
    fr = torch.from_numpy(f).cuda()
    ctx.match([(fr, fr.clone())])
    ctx.import_state(gpm.NNF, nnf, level=0)
    ctx.fit_planes(1)
    gmi = ctx.export(gpm.MODEL_INFO)
    resid = ctx.export(gpm.STAGE1_LABELS)[0] < 0
    ctx.close()
    frame = np.asarray(f, np.float64)
    ncell = int(O.cell_base(P)[1])
    for d in range(2):
        mh, mi = O.empty_models(P)
        vx, vy = (np.ascontiguousarray(nnf[d][:, c]) for c in range(2))
        for stage in (1, 2):
            mask = None if stage == 1 else np.ascontiguousarray(resid[d].astype(np.uint8))
            O.fit_level(P, frame, frame, d, 1, stage, vx, vy, mask, mh, mi)
            ids = np.arange(ncell) * 2 + stage - 1
            tie = (mi[ids, O.MI_FLAGS] & O.F_AMBIG) > 0
            assert (gmi[d][ids, O.MI_NIN] == mi[ids, O.MI_NIN]).all()
            for f in (O.MI_BESTK, O.MI_BESTSCORE):  # the winner and its support
                bad = (gmi[d][ids, f] != mi[ids, f]) & ~tie
                assert not bad.any(), f"dir {d} stage {stage}: windows {np.flatnonzero(bad)} differ"
            assert (~tie).any()
