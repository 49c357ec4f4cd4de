"""The max-over-query scorer on batches: the fused pass with every place its unit query rows can
take in the workspace, tiles cut at video ends, clusters of the statistics kernel with fewer than
eight frames, and the per-video path where the fused pass does not apply."""

import ctypes as C

import pytest
import torch

from helpers import accepted_random, compare_condense, oracle_run

pytestmark = pytest.mark.gpu

BY_VIDEO, OWN, SLOTS, OPERATOR = range(4)   # where the unit query rows go

CASES = [
    # V, T, H, W, D, query rows, their place
    (2, 3, 11, 12, 128, [5, 64], OWN),
    (3, 5, 12, 12, 192, [1, 128, 33], SLOTS),              # past the column partials in use
    (16, 11, 12, 12, 64, [128] * 16, OPERATOR),            # 176 frames
    (16, 4, 12, 12, 512, [128, 120] * 8, BY_VIDEO),        # no room
    (5, 4, 9, 9, 128, [3, 17, 128, 64, 1], BY_VIDEO),      # frames of fewer than 128 tokens
    (4, 45, 13, 10, 64, [16, 15, 90, 2], SLOTS),           # several videos inside a CTA's range
    (2, 9, 16, 16, 1024, [127, 100], SLOTS),               # long queries: small query-row stages
    (2, 4, 13, 13, 4160, [40, 24], BY_VIDEO),              # too wide for the fused pass
]


def _place(wz, V, T, H, W, D, Lqs, ratios):
    """The place that the library chooses (the checked build says)."""
    fn = C.CDLL(wz.LIB_CHECKED_PATH).wz_check_query_rows
    return fn(V, T, H, W, D, (C.c_int32 * V)(*Lqs), (C.c_float * V)(*ratios))


@pytest.mark.parametrize("V,T,H,W,D,Lqs,place", CASES)
def test_maxsim_batch_shapes(V, T, H, W, D, Lqs, place):
    import paper_2607_23265_gb300 as wz
    ratios = [(0.2, 0.1, 0.3)[v % 3] for v in range(V)]
    assert _place(wz, V, T, H, W, D, Lqs, ratios) == place
    vids = [accepted_random(T, H, W, D, lq, r, seed=500 + 7 * k, relevance="maxsim")
            for k, (lq, r) in enumerate(zip(Lqs, ratios))]
    X = torch.stack([x for x, _ in vids]).cuda()
    Q = torch.cat([q for _, q in vids]).cuda()
    status = torch.zeros((1,), dtype=torch.int32, device="cuda")
    out = wz.wz_condense_batch(X, Q, Lqs, ratios, relevance="maxsim", device_status=status)
    assert int(status.item()) == 0
    offs = out["row_offsets"]
    for v, (x, q) in enumerate(vids):
        ref = oracle_run(x, q, ratios[v], relevance="maxsim")
        one = {k: out[k][offs[v]:offs[v + 1]] for k in ("tokens", "index")}
        one.update(budgets=out["budgets"][v], count=out["count"][v:v + 1], relevance=out["relevance"][v])
        compare_condense(one, ref, x.dtype)


@pytest.mark.parametrize("T,D", [(480, 64), (300, 192)])
def test_maxsim_short_tiles(T, D):
    """Narrow rows: a tile is one or a few ring stages, many tiles per CTA."""
    import paper_2607_23265_gb300 as wz
    H = W = 16
    X, Q = accepted_random(T, H, W, D, 40, 0.05, seed=D, relevance="maxsim")
    out = wz.wz_condense_ex(X.cuda(), Q.cuda(), 0.05, relevance="maxsim")
    ref = oracle_run(X, Q, 0.05, relevance="maxsim", token_frames=range(0, T, 37))
    compare_condense(out, ref, X.dtype, frames=range(0, T, 37))
