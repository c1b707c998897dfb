"""The edge-aware fill's geodesic seeds at line lengths around the scans' chunks (32 pixels of a row, 32 sections of the
rows), with few seeds, against the oracle's sweeps: each model is its own translation, so a pixel's flow names its seed's."""
import numpy as np
import pytest

import oracle as O
from paper_1804_03787_gb300 import gpm

from _parity import oracle_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,seeds,flat", [(31, 9, 1, False), (32, 33, 2, False), (33, 64, 3, True), (65, 31, 7, False),
                                            (97, 130, 20, True), (300, 70, 40, False), (70, 300, 40, False), (64, 48, 0, False)])
def test_seeds_equal_oracle(W, H, seeds, flat):
    import torch
    gp = gpm.default_params(patch_radius=1, cells=(8,), pm_iters=0, num_hyp=32, fill_iters=0, interp=1)
    P = oracle_params(gp, W, H)
    rng = np.random.default_rng(W + H)
    f = rng.random((H, W, 3)).astype(np.float32)
    if flat:  # equal steps everywhere: every tie is decided by the seeds' order
        f[:] = 0.5
    ctx = gpm.Context(gp, W, H)
    fr = torch.from_numpy(f).cuda()
    ctx.match([(fr, fr.clone())])
    m, n = ctx.export(gpm.MODELS).shape[1], W * H
    used = min(m, seeds)
    t = np.stack([np.arange(m) % 7 - 3 + np.arange(m) / 64, np.arange(m) // 7], 1)
    mh = np.tile(np.eye(3).reshape(9), (2, m, 1))
    mh[:, :, 2], mh[:, :, 5] = t[:, 0], t[:, 1]
    mi = ctx.export(gpm.MODEL_INFO).copy()
    mi[:, :, O.MI_VALID] = 1
    at = rng.choice(n, seeds, replace=False)
    lab = np.full((2, n), -1, np.int32)
    if seeds:
        lab[:, at] = np.arange(seeds) % used
    flow = np.where((lab >= 0)[..., None], t[np.maximum(lab, 0)], 0.0)
    for what, data in ((gpm.NNF, np.zeros((2, n, 2), np.int32)), (gpm.MODELS, mh), (gpm.MODEL_INFO, mi),
                       (gpm.LABELS, (lab, np.full((2, n), 0.01, np.float32), flow)), (gpm.CUES, np.zeros((2, n), np.uint8))):
        ctx.import_state(what, data, 1)
    got = ctx.flow_and_occlusion()[0][0].cpu().numpy().reshape(n, 2)
    ctx.close()
    s = O.interp_seeds(P, f, lab[0])
    assert (s >= 0).all() if seeds else (s < 0).all()
    want = t[lab[0][s]] if seeds else np.zeros((n, 2))
    assert np.abs(got - want).max() < 1e-4
