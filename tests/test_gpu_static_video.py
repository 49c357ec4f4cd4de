"""Videos whose frames are all the same: delta_t is exactly 0 although the cosine of equal vectors is rounded, so
gamma_t is 0 too and the WTA keeps no detail."""

import pytest
import torch

pytestmark = pytest.mark.gpu

CASES = [
    # V, T, D, scorer: each kernel of the frame statistics
    (24, 8, 192, "mean"),       # a CTA per frame
    (80, 9, 72, "mean"),        # four frames per CTA
    (24, 8, 192, "maxsim"),     # clusters of eight
    (40, 9, 128, "maxsim"),     # clusters of four
]


def _still(V, T, D, seed):
    """V videos of T equal frames; whole numbers, so that every channel sum is exact in fp32."""
    g = torch.Generator().manual_seed(seed)
    frame = torch.randint(-6, 7, (V, 1, 9, 9, D), generator=g).expand(V, T, 9, 9, D)
    return frame.to(torch.bfloat16).contiguous().cuda()


@pytest.mark.parametrize("V,T,D,scorer", CASES)
def test_still_batch(V, T, D, scorer):
    import paper_2607_23265_gb300 as wz
    X = _still(V, T, D, seed=V + D)
    Q = torch.randn(3 * V, D, generator=torch.Generator().manual_seed(5)).to(torch.bfloat16).cuda()
    out = wz.wz_condense_batch(X, Q, [3] * V, [0.2] * V, relevance=scorer)
    rel = out["relevance"].cpu()
    assert torch.count_nonzero(rel[:, :, 1]) == 0, "delta"
    assert torch.count_nonzero(rel[:, :, 2]) == 0, "gamma"


def test_still_with_external_frame_scores():
    import paper_2607_23265_gb300 as wz
    V, T, D = 24, 8, 192
    X = _still(V, T, D, seed=3)
    Q = torch.ones(1, D, dtype=torch.bfloat16).cuda()
    r = torch.rand(V, T, generator=torch.Generator().manual_seed(4))
    for v in range(V):
        out = wz.wz_condense_ex(X[v], Q, 0.2, frame_scores=r[v].cuda())
        # no detail passes a gate of 0: r~ is the mean of each pair (one ulp of fp32 for the output)
        pair = r[v].double().reshape(T // 2, 2).mean(1).repeat_interleave(2)
        assert torch.allclose(out["relevance"].cpu()[:, 3].double(), pair, rtol=2 ** -23, atol=0)
