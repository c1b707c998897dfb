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


@pytest.mark.parametrize("W,H", [(61, 43), (40, 97), (129, 21), (24, 17)])
def test_level0_sweeps_with_region_bound_equal_oracle(W, H):
    """Radius 4 with FP32 texels, where list B is tested by the 3 x 3 regions' sums too: ragged tiles, and frames with
    few or no pixels whose patch stays inside."""
    import torch
    gpm.load()
    parity.test_level0_patchmatch_matches_oracle_up_to_near_ties(torch, W, H, 4, (8,))
