"""The projector in each of its tile shapes: 128 x 32, 64 and 256 on one SM and 256 x 256 on a pair of
SMs, with rows and columns that end inside a tile (and inside either half of a pair's), one K step
and more K steps than the ring has stages.  (Pairs need many K steps: their start takes three.)"""

import ctypes as C

import pytest

from test_gpu_project import _case, _check, _hidden_ok, _np, _run, wz  # noqa: F401  (wz: the module's fixture)

pytestmark = pytest.mark.gpu

PAIR = 512   # the library's name for 256 x 256 on a pair


def _tile(wz, rows, cols, k):
    """The tile columns that a layer of `rows` x `cols`, `k` deep, takes (the checked library says)."""
    return C.CDLL(wz.LIB_CHECKED_PATH).wz_check_project_tile(rows, cols, k)


@pytest.mark.parametrize("B,D,C,E,tiles", [
    (4100, 5760, 320, 512, (PAIR, 256)),      # columns end in the second tile's first half
    (300, 5760, 3584, 3584, (PAIR, 256)),     # rows end in the first half of the second tile
    (2500, 128, 1856, 4864, (256, PAIR)),     # more tiles than pairs
    (4100, 64, 320, 512, (256, 256)),         # one K step
    (1500, 640, 1152, 576, (256, 64)),
    (129, 128, 3584, 64, (64, 32)),
    (1000, 448, 1152, 3520, (64, 256)),
    (9800, 64, 256, 256, (256, 256)),
    (2688, 256, 3584, 320, (256, 64)),        # an odd number of 128-row blocks
    (100, 64, 64, 20480, (32, 256)),          # fewer rows than a tile's, 80 tiles of 256 columns
    (300, 128, 10048, 192, (256, 32)),        # rows and columns end inside the last tiles
    (31, 512, 4096, 64, (64, 32)),            # few rows, many columns
    (32, 512, 4096, 64, (32, 32)),
])
def test_project_tiles(wz, B, D, C, E, tiles):  # noqa: F811
    assert (_tile(wz, B, C, D), _tile(wz, B, E, C)) == tiles
    Z, W1, b1, W2, b2 = _case(B, D, C, E, seed=B + C)
    out, hidden = _run(wz, Z, W1, b1, W2, b2)
    hg = _np(hidden)
    _hidden_ok(hg, _np(Z), _np(W1), _np(b1))
    _check(out, hg, _np(W2), _np(b2))
