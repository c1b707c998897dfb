"""The restricted sweeps' shortcuts (the interval lower bound, candidates tested at the last visit) at the radii and
sizes where their conditions change, against the oracle's full evaluation."""
import pytest

from paper_1804_03787_gb300 import gpm

import test_gpu_parity as parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,r,cells", [(61, 43, 4, (16, 8)), (96, 33, 4, (32, 16)), (40, 40, 3, (8,)),
                                         (35, 67, 2, (16,)), (129, 21, 1, (8,))])
def test_restricted_sweeps_equal_oracle(W, H, r, cells):
    import torch
    gpm.load()
    parity.test_restricted_patchmatch_level1_lockstep(torch, W, H, r, cells)
