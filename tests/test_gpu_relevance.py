"""The relevance pass at the edges of its launch shapes: one and several consumer groups, rows
of one to many vectors per thread, chunks cut by short frames, windows and frames that end
inside a CTA's range, a query change between videos inside it."""

import numpy as np
import pytest
import torch

import oracle as O
import workload as wl

pytestmark = pytest.mark.gpu

CASES = [
    # T, H, W, D, dtype
    (1, 1, 1, 8, "bf16"),
    (300, 1, 3, 64, "bf16"),       # frames shorter than a chunk, several groups
    (40, 23, 23, 264, "bf16"),
    (9, 24, 25, 512, "f32"),
    (11, 23, 23, 896, "bf16"),
    (37, 16, 17, 1152, "bf16"),
    (24, 15, 15, 1160, "f32"),
    (23, 20, 15, 2304, "bf16"),    # 24 consumer warps
    (5, 13, 13, 2816, "bf16"),
    (16, 13, 13, 896, "f32"),      # few tokens per CTA
    (3, 27, 27, 3584, "bf16"),
    (7, 9, 9, 4096, "bf16"),
    (6, 9, 9, 4104, "bf16"),       # two vectors per thread
    (4, 8, 9, 8200, "bf16"),
    (5, 8, 9, 2056, "f32"),
    (2100, 4, 4, 64, "f32"),       # rows of one warp: four groups, frames of two chunks
    (700, 6, 6, 256, "bf16"),
    (300, 7, 9, 136, "bf16"),
    (4, 5, 5, 16392, "bf16"),      # eight vectors per thread: two tokens per chunk, then one
    (3, 6, 7, 32768, "bf16"),
    (3, 7, 7, 16384, "f32"),
    (5, 6, 6, 8192, "f32"),        # four vectors per thread
]


@pytest.mark.parametrize("T,H,W,D,dtype", CASES)
def test_relevance_shapes(T, H, W, D, dtype):
    import paper_2607_23265_gb300 as wz
    X, Q = wl.random_video(T, H, W, D, 3, dtype=dtype, seed=D)
    ts, fs, fm = wz.wz_relevance(X.cuda(), Q.cuda(), frame_mean=True)
    x, q = X.double().numpy().reshape(T, H * W, D), O.query_embedding(Q.double().numpy())
    a = np.stack([O.token_saliency(x[t], q) for t in range(T)])
    r, mean = zip(*[O.frame_relevance(x[t], q) for t in range(T)])
    # a cosine from fp32 sums: each addend passes at most 8 (thread) + 5 (warp) + 32 (warps)
    # roundings, in the dot and in half of the squared norm, relative to |x||q|
    bound = 1.5 * 45 * 2.0 ** -24
    assert np.abs(ts.cpu().double().numpy() - a).max() <= bound
    # fp32 sums over the H W tokens of a frame
    scale = np.abs(x).sum(axis=1).max() / (H * W)
    assert np.abs(fm.cpu().double().numpy() - np.stack(mean)).max() <= (H * W + 4) * 2.0 ** -24 * scale
    assert np.abs(fs.cpu().double().numpy() - np.array(r)).max() <= 1e-5


@pytest.mark.parametrize("V,T,H,W,D", [(7, 6, 16, 16, 512), (40, 1, 13, 13, 1792), (9, 4, 16, 16, 3584)])
def test_relevance_of_a_batch(V, T, H, W, D):
    """Videos change inside a CTA's range: its groups take the next query together."""
    import paper_2607_23265_gb300 as wz
    X, _ = wl.random_video(V * T, H, W, D, 1, seed=V)
    Q = torch.randn((2 * V, D), generator=torch.Generator().manual_seed(V), dtype=torch.float64).to(X.dtype)
    out = wz.wz_condense_batch(X.view(V, T, H, W, D).cuda(), Q.cuda(), [2] * V, [0.1] * V)
    got = out["relevance"].cpu().double().numpy().reshape(V * T, 4)
    x, q = X.double().numpy().reshape(V * T, H * W, D), Q.double().numpy()
    r = [O.frame_relevance(x[f], O.query_embedding(q[2 * (f // T):2 * (f // T) + 2]))[0] for f in range(V * T)]
    assert np.abs(got[:, 0] - np.array(r)).max() <= 1e-5
