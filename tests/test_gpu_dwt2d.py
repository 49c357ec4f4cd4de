"""wz_dwt2d / wz_idwt2d at the edges of their tiles: maps shorter than the filter, every filter
length, channel counts around the channel chunk, odd widths and rows that are not aligned for a
channel pair (one channel per thread), the largest map."""

import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu

CASES = [
    # H, W, D, wavelet, mode, dtype, elements the features are off a 16-byte boundary
    (1, 1, 8, 4, "symmetric", "bf16", 0),
    (1, 9, 2, 10, "zero", "f32", 0),
    (5, 3, 70, 7, "symmetric", "f32", 0),
    (7, 27, 33, 4, "periodic", "bf16", 0),
    (13, 13, 64, 1, "symmetric", "bf16", 0),
    (13, 12, 66, 2, "zero", "bf16", 1),
    (16, 16, 40, 3, "periodic", "f32", 1),
    (27, 27, 24, 4, "symmetric", "bf16", 2),
    (24, 25, 48, 5, "symmetric", "f32", 0),
    (14, 31, 16, 6, "symmetric", "f32", 0),
    (20, 11, 18, 8, "zero", "bf16", 0),
    (33, 17, 12, 9, "symmetric", "bf16", 0),
    (64, 64, 11, 10, "symmetric", "f32", 0),
    (64, 63, 10, 10, "periodic", "bf16", 0),
    (27, 26, 34, 44, "symmetric", "bf16", 0),
    (4, 4, 1, 1, "symmetric", "bf16", 0),        # few channels: chunks of 8, 16, 32, 64
    (4, 5, 3, 1, "zero", "f32", 0),
    (2, 4, 8, 4, "symmetric", "bf16", 0),
    (4, 4, 9, 1, "periodic", "f32", 0),
    (3, 2, 17, 2, "symmetric", "bf16", 0),
    (4, 2, 32, 1, "symmetric", "f32", 0),
]


@pytest.mark.parametrize("H,W,D,wavelet,mode,dtype,off", CASES)
def test_dwt2d_edges(H, W, D, wavelet, mode, dtype, off):
    import paper_2607_23265_gb300 as wz
    T = 2
    dt = {"bf16": torch.bfloat16, "f32": torch.float32}[dtype]
    g = torch.Generator().manual_seed(H * 64 + W)
    X = torch.randn((T, H, W, D), generator=g).to(dt)
    buf = torch.empty((X.numel() + off,), dtype=dt, device="cuda")
    Xd = buf[off:].view(T, H, W, D)
    Xd.copy_(X)
    f = O.wavelet_filters(wavelet)
    F = f["F"]
    bands = wz.wz_dwt2d(Xd, wavelet, mode)
    x = X.double().numpy()
    ref = [np.stack(b) for b in zip(*[O.dwt2d(x[t], f, mode) for t in range(T)])]
    # two passes of F fused multiply-adds with taps rounded to fp32: each adds at most
    # (F + 2) 2^-24 of the sum of the magnitudes of its terms
    u = 2.0 ** -24
    S = max(np.abs(f["dec_lo"]).sum(), np.abs(f["dec_hi"]).sum())
    bound = 2 * (F + 2) * u * S * S * np.abs(x).max()
    for k in range(4):
        err = np.abs(bands[k].cpu().double().numpy() - ref[k]).max()
        assert err <= bound, (k, err, bound)
    y = wz.wz_idwt2d(*bands, H, W, wavelet)
    got = [b.cpu().double().numpy() for b in bands]
    back = np.stack([O.idwt2d(*[b[t] for b in got], H, W, f) for t in range(T)])
    S = np.abs(f["rec_lo"]).sum() + np.abs(f["rec_hi"]).sum()
    bound = 2 * (F + 2) * u * S * S * max(np.abs(b).max() for b in got)
    err = np.abs(y.cpu().double().numpy() - back).max()
    assert err <= bound, (err, bound)
