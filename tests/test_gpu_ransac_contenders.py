"""The block kernels' search (256 and 512 threads a window) where many hypotheses contend for a window while its warps raise
the bound: one noisy motion per window, so that supports are close together and often equal, against the oracle.  A launch
of more than 456 windows of at most 60 px takes 256 threads a window, others 512."""
import numpy as np
import pytest

import oracle as O
from paper_1804_03787_gb300 import gpm

from _parity import oracle_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,s,hyp,noise", [(200, 160, 18, 257, 2), (200, 160, 18, 600, 1), (400, 240, 34, 256, 2),
                                             (70, 52, 34, 512, 2), (64, 64, 64, 600, 2), (150, 100, 62, 300, 1)])
def test_contending_hypotheses_equal_oracle(W, H, s, hyp, noise):
    import torch
    gp = gpm.default_params(patch_radius=2, cells=(s,), pm_iters=0, num_hyp=hyp)
    P = oracle_params(gp, W, H)
    rng = np.random.default_rng(W + hyp)
    f = rng.random((H, W, 3)).astype(np.float32) * 0.2 + 0.4
    y, x = np.mgrid[0:H, 0:W]
    motion = np.stack([3 + np.rint(0.03 * x), np.rint(0.02 * y) - 2], -1)
    nnf = np.stack([(motion + rng.integers(-noise, noise + 1, (H, W, 2))).reshape(-1, 2) for _ in range(2)]).astype(np.int32)
    ctx = gpm.Context(gp, W, H)
    fr = torch.from_numpy(f).cuda()
    ctx.match([(fr, fr.clone())])
    ctx.import_state(gpm.NNF, nnf, level=0)
    ctx.fit_planes(1)
    gmi = ctx.export(gpm.MODEL_INFO)
    ctx.close()
    frame = np.asarray(f, np.float64)
    ncell = int(O.cell_base(P)[1])
    assert (2 * ncell > 456) == (W > 150)
    first = np.arange(ncell) * 2
    for d in range(2):
        mh, mi = O.empty_models(P)
        vx, vy = (np.ascontiguousarray(nnf[d][:, c]) for c in range(2))
        O.fit_level(P, frame, frame, d, 1, 1, vx, vy, None, mh, mi)
        sure = (mi[first, O.MI_FLAGS] & O.F_AMBIG) == 0
        assert sure.any()
        for k in (O.MI_BESTK, O.MI_BESTSCORE):
            assert (gmi[d][first, k] == mi[first, k])[sure].all()
