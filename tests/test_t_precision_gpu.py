"""T = X R^T keeps 32 bits on the shapes that always had it in 32 bits: rows that are no multiple of 256 columns (up to 16 tokens), of
128 columns or outputs (above), and ranks above 2560 at 9 to 16 tokens.  The inputs make columns of T that are equal in their high
bits, up to 44807, and L subtracts them from one another, so that Y is a small integer that is right only if both kept their last
bit; every value is an int4 code times a scale that is a power of two or one, so bf16 and int4 adapters give the same Y."""
import numpy as np
import pytest
import torch

from paper_2410_09615_b200 import binding as K, inputs
from helpers import to_dev

pytestmark = pytest.mark.gpu

A, P = K.KERNEL_AUTO, K.KERNEL_PREFILL
SHAPES = [  # d_in, d_out, r, b, kernel (of the call with bf16 adapters)
    (320, 1040, 48, 1, A),         # small batches: index bytes without tensor map, narrow row tiles
    (1408, 528, 80, 5, A),         # with tensor map
    (832, 20016, 48, 12, A),       # 256-row tiles
    (384, 20016, 144, 9, A),
    (1728, 528, 80, 24, A),        # three and five tiles of eight tokens
    (512, 784, 208, 20, A),
    (1728, 528, 80, 33, A),
    (512, 784, 208, 40, A),
    (512, 272, 2576, 10, A),       # a rank that the 32-bit kernel always took
    (320, 528, 32, 300, A),        # CTA pairs, 64-token tiles
    (448, 9616, 48, 300, A),       # 256-token tiles
    (1728, 5120, 176, 600, A),     # parts of T' from several pairs
    (448, 272, 48, 100, P),        # one CTA a tile, T' in one slice
    (4160, 272, 48, 70, P),        # and in several
]


@pytest.mark.parametrize("s", [1.0, 0.0])
@pytest.mark.parametrize("d_in,d_out,r,b,kernel", SHAPES)
def test_columns_of_T_that_differ_in_their_last_bits(d_in, d_out, r, b, kernel, s):
    rng = np.random.default_rng([d_in, d_out, r, b])
    codes = rng.integers(-8, 8, size=(d_out, d_in)).astype(np.int8)
    mask = inputs.top2_mask(rng.standard_normal((d_out, d_in)).astype(np.float32))
    X = np.zeros((b, d_in), np.int64)
    X[:, 0], X[:, 129] = 100, rng.integers(-1, 2, b)
    R = np.zeros((r, d_in), np.int64)
    R[:, 0], R[:, 129] = 64 * np.repeat(rng.integers(-7, 8, r // 2), 2), rng.integers(-7, 8, r)      # columns 2 i and 2 i + 1 differ in the second term
    R[:, 2], R[:, 130] = 448, 7                                                                      # the groups' largest: scales 64 and 1
    L = np.zeros((d_out, r), np.int64)
    i = rng.integers(0, r // 2, d_out)
    L[np.arange(d_out), 2 * i], L[np.arange(d_out), 2 * i + 1] = 7, -7
    codes[:, 0] = 0                                                                                   # the large activation meets R alone
    exact = (X @ R.T) @ L.T + int(s) * (X[:, [129]] * (codes.astype(np.int64) * mask)[:, 129])
    assert np.abs(exact).max() <= 256                                                                # bf16 holds it
    bf = lambda a: K.bf16_from_bits(inputs.f32_to_bf16_bits(a.astype(np.float32)))
    vals, meta = K.slim_pack(to_dev(codes), to_dev(mask))
    Y = K.slim_linear_fwd(bf(X), vals, meta, s, bf(L), bf(R), kernel=kernel)
    assert np.array_equal(inputs.bf16_bits_to_f64(K.bits_from_bf16(Y)), exact)
    Lq, Ls = K.slim_pack_adapter(bf(L))
    Rq, Rs = K.slim_pack_adapter(bf(R))
    Y = K.slim_linear_fwd_q(bf(X), vals, meta, s, Lq, Ls, Rq, Rs)
    assert np.array_equal(inputs.bf16_bits_to_f64(K.bits_from_bf16(Y)), exact)
