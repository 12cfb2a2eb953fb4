"""The CTA-pair kernel where its tiles, its T' and the converters' turns come out differently."""
import pytest

from paper_2410_09615_b200 import binding as K
from helpers import run_case

pytestmark = pytest.mark.gpu

CASES = [  # d_in, d_out, r, b, token tile
    (2176, 8192, 272, 40, 64),         # T' tiles of ranks, the second of them with 16
    (320, 8208, 272, 64, 64),          # the same in two parts, and half a packed tile at the end
    (1088, 1024, 208, 250, 64),        # T' by the ranks in more chunks than its width asks for
    (1024, 10240, 0, 120, 128),        # stages of 256 columns, one token tile
    (1152, 1024, 16, 1000, 128),       # an odd number of 128-column blocks in stages of 256
    (384, 20016, 0, 300, 256),         # three stages a tile, several tiles a pair: the turns shift from tile to tile
    (640, 20016, 80, 300, 256),        # five stages and adapter stages in two parts
    (4160, 8192, 64, 333, 256),        # tiles of 176 tokens that share T' tiles of 256; index bytes by cp.async
]


@pytest.mark.parametrize("d_in,d_out,r,b,tile", CASES)
def test_pair_plans(d_in, d_out, r, b, tile):
    res = run_case(d_in, d_out, r, b, seed=61, rows=None if b * d_out * d_in < 1 << 33 else range(0, b, 5))
    assert res["ok"] and res["launches"] == 1 and res["token_tile"] == tile, res
