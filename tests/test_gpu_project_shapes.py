"""The projector in each of its tile shapes: 128 x 32 .. 256 on one SM and 256 x 256 on a pair of
SMs, with rows and columns that end inside a tile (and inside either half of a pair's), one K step
and more K steps than the ring has stages."""

import pytest

from test_gpu_project import _case, _check, _hidden_ok, _np, _run, wz  # noqa: F401  (wz: the module's fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,D,C,E", [
    (4100, 64, 320, 512),       # pairs: one K step; columns end in the second tile's first half
    (300, 192, 3584, 3584),     # pairs: rows end in the first half of the second tile
    (1500, 640, 1152, 576),     # pairs, then 128 x 64
    (129, 128, 3584, 64),       # 128 x 64, then 128 x 32
    (1000, 448, 1152, 3520),    # 128 x 64, then pairs
    (2500, 128, 320, 4864),     # 128 x 64, then pairs with more tiles than pairs
    (9800, 64, 256, 256),       # pairs in two rounds' reach, 39 tiles of 256 rows
])
def test_project_tiles(wz, B, D, C, E):  # noqa: F811
    Z, W1, b1, W2, b2 = _case(B, D, C, E, seed=B + C)
    out, hidden = _run(wz, Z, W1, b1, W2, b2)
    hg = _np(hidden)
    _hidden_ok(hg, _np(Z), _np(W1), _np(b1))
    _check(out, hg, _np(W2), _np(b2))
