"""slim_pack on masks of any non-zero bytes and on groups that are refused beside others that are not."""
import numpy as np
import pytest
import torch

import oracle
from paper_2410_09615_b200 import binding as K
from helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d_out,d_in", [(16, 64), (48, 1088), (1008, 320)])
def test_any_non_zero_mask_byte_keeps(d_out, d_in):
    rng = np.random.default_rng([d_out, d_in])
    codes = rng.integers(-8, 8, size=(d_out, d_in)).astype(np.int8)
    kept = rng.random((d_out, d_in // 4, 4)).argsort(axis=2) < rng.integers(0, 3, size=(d_out, d_in // 4, 1))
    ones = kept.reshape(d_out, d_in).astype(np.uint8)
    any_byte = ones * rng.choice(np.array([1, 2, 127, 128, 255], np.uint8), size=(d_out, d_in))
    half = np.where(rng.random((d_out, d_in // 16, 1)) < 0.5, ones.reshape(d_out, -1, 16), any_byte.reshape(d_out, -1, 16)).reshape(d_out, d_in)
    vals, meta = oracle.pack(codes, ones)
    for mask in (ones, any_byte, half):
        v, m = K.slim_pack(to_dev(codes), to_dev(mask))
        assert np.array_equal(v.cpu().numpy(), vals) and np.array_equal(m.cpu().numpy(), meta)


def test_refused_groups_leave_the_others_as_they_are():
    rng = np.random.default_rng(7)
    codes = rng.integers(-8, 8, size=(16, 64)).astype(np.int8)
    mask = np.tile(np.array([1, 0, 1, 0], np.uint8), (16, 16))
    vals, meta = oracle.pack(codes, mask)
    bad_mask, bad_codes = mask.copy(), codes.copy()
    bad_mask[3, 20:24] = 1                    # four kept values
    bad_codes[5, 32] = 9                      # a kept code out of range (and one that is not kept: no matter)
    bad_codes[6, 33] = 100
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    v, m = K.slim_pack(to_dev(bad_codes), to_dev(bad_mask), status=status, check=False)
    torch.cuda.synchronize()
    v, m = v.cpu().numpy(), m.cpu().numpy()
    assert K.read_status(status) != 0
    vals[3, 5] = vals[5, 8] = 0
    meta[3, 2] = (meta[3, 2] & 0x0F) | 0x40
    meta[5, 4] = (meta[5, 4] & 0xF0) | 0x04
    assert np.array_equal(v, vals) and np.array_equal(m, meta)
