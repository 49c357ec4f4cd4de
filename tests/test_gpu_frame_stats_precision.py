"""How exact the frame statistics' squares and neighbour products are: no further from 64 bits than fp32 sums over
a sixteenth of the channels each (one chain per thread of 512, a tree per warp) with the sixteen totals in fp64."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _fma(a, b, c):
    # exact product of two floats in 64 bits, one rounding to 32
    return (a.astype(np.float64) * b + c).astype(np.float32)


def _sixteen_totals(a, b):
    """Row sums of a * b over [F, D] float32 in the order described above."""
    F, D = a.shape
    pad = -D % 2048
    a, b = (np.pad(x, ((0, 0), (0, pad))).reshape(F, -1, 512, 4) for x in (a, b))
    p = np.zeros((F, 512), np.float32)
    for i in range(a.shape[1]):
        for e in (3, 2, 1, 0):
            p = _fma(a[:, i, :, e], b[:, i, :, e], p)
    p = p.reshape(F, 16, 32)
    while p.shape[2] > 1:
        p = p[:, :, :p.shape[2] // 2] + p[:, :, p.shape[2] // 2:]
    return p[:, :, 0].astype(np.float64).sum(1)


CASES = [
    # T, D, scorer, spatial mode
    (400, 3584, "mean", "none"),     # no gates, more frames than a wave of 512 threads
    (640, 3584, "mean", "wsm"),      # four frames per CTA
    (200, 3584, "mean", "wsm"),      # a CTA per frame
    (264, 1152, "mean", "none"),
    (160, 3584, "maxsim", "wsm"),    # clusters of eight
    (300, 3584, "maxsim", "wsm"),    # clusters of four
    (300, 8192, "maxsim", "wsm"),
    (160, 1152, "maxsim", "wsm"),
]


@pytest.mark.parametrize("T,D,scorer,mode", CASES)
def test_delta_error(T, D, scorer, mode):
    import paper_2607_23265_gb300 as wz
    g = torch.Generator().manual_seed(T + D)
    # a quiet video of one token per frame, so that the frame sums are the tokens themselves
    X = torch.randn(1, D, generator=g) * (1 + 0.01 * torch.randn(T, D, generator=g))
    X = X.to(torch.bfloat16).reshape(T, 1, 1, D)
    Q = torch.randn(5, D, generator=g).to(torch.bfloat16)
    out = wz.wz_condense_ex(X.cuda(), Q.cuda(), 0.1, relevance=scorer, spatial_mode=mode)
    got = out["relevance"].cpu()[1:, 1].double().numpy()
    S = X.reshape(T, D).double().numpy()
    s32 = S.astype(np.float32)

    def delta(dot):
        cur, prev = dot(slice(1, None), slice(1, None)), dot(slice(0, -1), slice(0, -1))
        return 1.0 - dot(slice(1, None), slice(0, -1)) / np.sqrt(cur * prev)

    want = delta(lambda i, j: (S[i] * S[j]).sum(1))
    ref = delta(lambda i, j: _sixteen_totals(s32[i], s32[j]))
    rms = lambda e: float(np.sqrt(np.mean(e * e)))  # noqa: E731
    assert rms(got - want) <= rms(ref - want), (rms(got - want), rms(ref - want))
