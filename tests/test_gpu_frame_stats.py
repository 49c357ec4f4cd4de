"""Frame statistics of many frames: several frames per CTA or cluster (the last of a video not full, rows
of more vectors than threads), gates by warps and by CTAs."""

import pytest
import torch

from helpers import accepted_random, compare_condense, oracle_run

pytestmark = pytest.mark.gpu

CASES = [
    # V, T, H, W, D, query rows, scorer
    (130, 5, 8, 8, 64, 3, "mean"),        # one frame left for a video's last CTA
    (1, 650, 8, 9, 72, 2, "mean"),
    (10, 64, 8, 8, 1032, 4, "mean"),      # two vectors per thread
    (9, 70, 23, 23, 64, 2, "mean"),       # 529 tokens: a CTA per gate
    (1, 201, 8, 8, 2112, 9, "maxsim"),    # clusters of eight, one frame in the last
    (33, 19, 12, 12, 64, 17, "maxsim"),   # clusters of four
]


@pytest.mark.parametrize("V,T,H,W,D,Lq,scorer", CASES)
def test_many_frames(V, T, H, W, D, Lq, scorer):
    import paper_2607_23265_gb300 as wz
    vids = [accepted_random(T, H, W, D, Lq, 0.1, seed=900 + 31 * v, relevance=scorer) for v in range(min(V, 3))]
    pick = [v % len(vids) for v in range(V)]
    X = torch.stack([vids[p][0] for p in pick]).cuda()
    Q = torch.cat([vids[p][1] for p in pick]).cuda()
    out = wz.wz_condense_batch(X, Q, [Lq] * V, [0.1] * V, relevance=scorer)
    offs = out["row_offsets"]
    refs = [oracle_run(x, q, 0.1, relevance=scorer) for x, q in vids]
    for v in sorted({0, 1, 2, V // 2, V - 1} & set(range(V))):
        one = {k: out[k][offs[v]:offs[v + 1]] for k in ("tokens", "index")}
        one.update(budgets=out["budgets"][v], count=out["count"][v:v + 1], relevance=out["relevance"][v])
        compare_condense(one, refs[pick[v]], X.dtype)
