"""The CUDA-core condensation in each of its tile shapes (rows per frame, number of tiles), with
channel counts and token counts that no tile divides, in fp32 and bf16, and frames without rows."""

import numpy as np
import pytest
import torch

from helpers import accepted_random, compare_condense, oracle_run, to_np64

pytestmark = pytest.mark.gpu

CASES = [
    # T, H, W, D, ratio, dtype
    (1, 1, 1, 8, 1.0, "f32"),
    (9, 7, 9, 136, 0.3, "f32"),          # 32 x 64 tiles
    (6, 13, 10, 264, 0.6, "bf16"),
    (32, 13, 13, 3584, 0.135, "f32"),    # 32 x 128
    (12, 13, 13, 3592, 0.36, "f32"),     # 64 x 128
    (8, 16, 16, 3592, 0.7, "f32"),       # 128 x 128
    (8, 16, 15, 3600, 0.75, "bf16"),
]


@pytest.mark.parametrize("T,H,W,D,ratio,dtype", CASES)
def test_simt_tiles(T, H, W, D, ratio, dtype):
    import paper_2607_23265_gb300 as wz
    X, Q = accepted_random(T, H, W, D, 5, ratio, seed=T * H, dtype=dtype)
    out = wz.wz_condense_ex(X.cuda(), Q.cuda(), ratio, path="simt")
    ref = oracle_run(X, Q, ratio)
    compare_condense(out, ref, X.dtype)
    if dtype == "f32":
        # chains of H W fused multiply-adds on independent roundings of 2^-24, plus the operator's own
        got, want = to_np64(out["tokens"]), ref["out_tokens"]
        assert np.linalg.norm(got - want) <= (np.sqrt(H * W) + 16) * 2.0 ** -24 * np.linalg.norm(want)
