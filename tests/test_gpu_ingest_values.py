"""The gain's sums and its product at values where their integer and FP32 forms give way to FP64: below 2^-16, at 2 and
above, zeros, negative ones; rows shorter and longer than a block of the sums."""
import math

import numpy as np
import pytest

from paper_1804_03787_gb300 import gpm

pytestmark = pytest.mark.gpu

KINDS = {"unit": lambda r, s: r.random(s), "dark": lambda r, s: r.random(s) * 2.0 ** -15,
         "bright": lambda r, s: r.random(s) * 50, "edges": lambda r, s: r.choice([0.0, 2.0 ** -16, 2.0, 1.9999999, 1.0], s),
         "signed": lambda r, s: r.random(s) - 0.25, "wide": lambda r, s: 10.0 ** r.uniform(-30, 3, s)}


@pytest.mark.parametrize("W,H", [(37, 29), (8, 300), (1500, 5), (129, 128)])
@pytest.mark.parametrize("kind", sorted(KINDS))
def test_ingest_gain_and_products(kind, W, H):
    import torch
    rng = np.random.default_rng(W + len(kind))
    f1, f2 = (KINDS[kind](rng, (H, W, 3)).astype(np.float32) for _ in range(2))
    f2 *= np.float32(0.7)
    ctx = gpm.Context(gpm.default_params(cells=(), pm_iters=0), W, H)
    ctx.match([(torch.from_numpy(f1).cuda(), torch.from_numpy(f2).cuda())])
    got = ctx.export(gpm.FRAMES)
    ctx.close()
    a, b = (math.fsum(f.reshape(-1).tolist()) for f in (f1, f2))
    want = [f1, (f2.astype(np.float64) * (a / b)).astype(np.float32)]
    for d in range(2):
        g = np.asarray(got[d]).reshape(H, W, 4)[..., :3]
        # FP64 sums carry at most n 2^-53: the product's rounding may flip, no more
        assert (np.abs(g - want[d]) <= np.spacing(np.abs(want[d]))).all()
        assert (g != want[d]).mean() < 1e-3
