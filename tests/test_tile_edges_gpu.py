"""Sizes at the edges of the kernels' tiles and dispatch rules, all elements against the oracle: the small-batch kernel on
64-, 128- and 256-row tiles (bf16 and int4 adapters), the CTA-pair kernel on 64-, 128- and 256-token tiles, and the compression
kernels where rows are no multiples of their vector widths.  The tolerances are those of ``parity`` (bf16 result, one bf16
rounding of T); bytes are equal."""
import numpy as np
import pytest
import torch

import oracle
from paper_2410_09615_b200 import binding as K, inputs
from helpers import run_case, to_dev
from test_adapter_q_gpu import long_tailed, run_q

pytestmark = pytest.mark.gpu

SMALL = [  # d_in, d_out, r, b
    (64, 256, 16, 2),          # one unit, a quarter of it; one row tile of 16 in all of T
    (192, 272, 16, 9),         # units end in the middle; the last row tile has 16 rows
    (2048, 1040, 208, 8),      # 128- or 64-row tiles, the last with 16 rows; codes of L without tensor map (r % 32 = 16)
    (1024, 4112, 64, 16),      # a row tile more than 64 x 64
    (8192, 1552, 288, 3),      # clusters of eight, four units each; stages of 64 codes: the last has one step
    (8256, 3600, 96, 5),       # d_in % 128 = 64, 33 units over four CTAs
    (832, 20016, 48, 1),       # 256-row tiles, the last with 48 rows
    (448, 19008, 0, 16),
    (512, 512, 64, 17),        # three token tiles
    (448, 784, 208, 32),
    (1728, 528, 80, 33),
    (320, 304, 1008, 64),      # the largest batch; T region nearly half full
]


@pytest.mark.parametrize("d_in,d_out,r,b", SMALL)
def test_small_batch_tile_edges(d_in, d_out, r, b):
    res = run_case(d_in, d_out, r, b, seed=51)
    assert res["ok"] and res["launches"] == 1 and res["token_tile"] == 0, res
    if r:
        res = run_q(d_in, d_out, r, b, seed=52, wseed=51)
        assert res["ok"] and res["launches"] == 1, res


PAIR = [  # d_in, d_out, r, b, token tile
    (320, 528, 32, 300, 64),           # d_in % 128 = 64; five row tiles, an odd number
    (1728, 5120, 16, 65, 64),          # one token in the second token tile; no tile left over for T'
    (512, 8208, 48, 64, 64),           # the small batches of layers with 8192 rows and more
    (448, 2000, 48, 1000, 128),
    (448, 9616, 48, 300, 256),
    (192, 20016, 16, 600, 256),        # several tiles a pair, odd number of row tiles
    (256, 38016, 0, 257, 256),
]


@pytest.mark.parametrize("d_in,d_out,r,b,tile", PAIR)
def test_pair_tile_edges(d_in, d_out, r, b, tile):
    res = run_case(d_in, d_out, r, b, seed=53)
    assert res["ok"] and res["launches"] == 1 and res["token_tile"] == tile, res


# (below: rows a block has lanes for, one and several rows a thread, a last block that is not full)
@pytest.mark.parametrize("rows,d_in", [(1, 4), (7, 20), (33, 1028), (16, 64), (5, 4112), (9475, 64), (1000, 192), (70001, 12), (300, 4100), (1187, 4112), (2500, 1028)])
def test_mask_row_widths(rows, d_in):
    rng = np.random.default_rng([rows, d_in])
    codes = rng.integers(-8, 8, size=(rows, d_in)).astype(np.int8)
    xbar = rng.random(d_in).astype(np.float32)
    for x in (xbar, None):
        got = K.slim_mask_top2(to_dev(codes), None if x is None else to_dev(x))
        assert np.array_equal(got.cpu().numpy(), oracle.mask_top2(codes, x))


def test_mask_takes_a_negative_zero_magnitude_for_zero():
    # -0 is a legal magnitude (not below zero) and ties with +0: the lower index is kept
    group = np.array([(5, 0, 0, 3), (0, 7, 0, 0), (0, 0, 0, -8), (1, 1, 1, 1), (0, 0, 0, 0), (2, -2, 0, 1)], np.int8)
    codes = np.tile(group, (1, 16))
    ones = np.array([[(-0.0 if i >> k & 1 else 1.0) for k in range(4)] for i in range(16)], np.float32).reshape(64)
    for xbar in (ones, np.copysign(np.float32(0.0), np.where(np.signbit(ones), -1, 1)).astype(np.float32)):
        got = K.slim_mask_top2(to_dev(codes), to_dev(xbar)).cpu().numpy()
        assert np.array_equal(got, oracle.mask_top2(codes, xbar))
    assert np.array_equal(oracle.mask_top2(group[:1], np.array([-0.0, 1, 1, 1], np.float32)), [[1, 0, 0, 1]])


@pytest.mark.parametrize("rows,cols", [(3, 130), (9, 1002), (2, 6), (5, 136), (7, 1004), (601, 12), (1025, 2)])
def test_adapter_row_widths(rows, cols):
    A = long_tailed(rows, cols, 54)
    codes, scales = K.slim_pack_adapter(K.bf16_from_bits(A))
    ocodes, oscales = oracle.quant_adapter(A)
    assert np.array_equal(codes.cpu().numpy(), ocodes) and np.array_equal(K.bits_from_bf16(scales), oscales)
    back = K.bits_from_bf16(K.slim_unpack_adapter(codes, scales))
    assert np.array_equal(back, inputs.f32_to_bf16_bits(oracle.dequant_adapter(ocodes, oscales).astype(np.float32)))


def test_scale_search_where_the_sum_leaves_binades_slowly_and_fast():
    # nearly all weights in the first bins, and nearly all in the last: the two ways a candidate's error sum can grow
    for seed, w in ((1, 1e-3), (2, 1.0)):
        rng = np.random.default_rng(seed)
        W = (w * rng.uniform(0.9, 1.0, (640, 1600)) * rng.choice([-1, 1], (640, 1600))).astype(np.float32)
        W[0, 0] = 1.0
        codes, sa, table, alpha = K.slim_quant(to_dev(W))
        ocodes, oscale, oalpha, otable = oracle.slim_quant(W)
        assert float(alpha) == oalpha and np.array_equal(table.cpu().numpy().view(np.uint64), otable.view(np.uint64))
        assert float(sa[0]) == oscale and np.array_equal(codes.cpu().numpy(), ocodes)
