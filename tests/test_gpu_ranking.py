"""The remainder ranking at the frame counts where its form changes (several lanes per frame, a lane per
frame, several frames per thread, an odd last frame): equal remainders everywhere (ties go to the earlier
frame) and a few distinct ones among equal ones."""

import numpy as np
import pytest
import torch

import workload as wl
from helpers import oracle_run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [2, 31, 63, 128, 129, 256, 257, 511, 512, 513, 545, 1023, 1025, 3001])
@pytest.mark.parametrize("levels", [1, 3])
def test_ties(T, levels):
    import paper_2607_23265_gb300 as wz
    X, Q = wl.random_video(T, 2, 3, 8, 1, seed=T)
    # whole quarters: equal weights, hence exactly equal remainders, in long runs
    r = (np.arange(T) * 7 % 5 % levels + 1) / 4
    kw = dict(temporal_mode="raw")
    out = wz.wz_condense_ex(X.cuda(), Q.cuda(), 0.3, frame_scores=torch.from_numpy(r).float().cuda(), **kw)
    ref = oracle_run(X, Q, 0.3, frame_scores=r, token_frames=[], **kw)
    assert np.array_equal(out["budgets"].cpu().numpy(), ref["budgets"])
