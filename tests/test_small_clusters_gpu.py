"""The small-batch kernel on the packed format without adapters, where its clusters and tile heights change, and either side of the lines
between it and the CTA-pair kernel from 33 tokens on."""
import pytest

from paper_2410_09615_b200 import binding as K
from helpers import run_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d_in,d_out,b", [
    (1024, 4096, 16), (2048, 4112, 1), (2304, 4096, 5),          # tiles of 64 rows: clusters of two CTAs, and of four
    (1088, 6400, 16), (5120, 6160, 3), (5376, 6144, 9),          # of 128 rows, with index bytes by cp.async; of two, of four
    (512, 13824, 16), (2112, 11008, 2),                          # layers that fit 128-row tiles only with clusters of two
    (256, 14336, 8), (768, 19200, 16),                           # one CTA a tile; 256-row tiles
])
def test_small_batches_without_adapters(d_in, d_out, b):
    res = run_case(d_in, d_out, 0, b, seed=62)
    assert res["ok"] and res["launches"] == 1, res
    assert K.slim_select_kernel(b, d_out, d_in, 0) == K.KERNEL_DECODE


@pytest.mark.parametrize("d_in,d_out,r,b,kernel", [
    (2048, 4080, 0, 33, K.KERNEL_SMALL), (2048, 4096, 0, 33, K.KERNEL_PREFILL), (2048, 4096, 0, 64, K.KERNEL_PREFILL), (2048, 4096, 0, 32, K.KERNEL_SMALL),
    (5120, 5104, 32, 40, K.KERNEL_SMALL), (5120, 5120, 32, 64, K.KERNEL_PREFILL), (4032, 5120, 32, 64, K.KERNEL_SMALL),
    (4096, 5120, 416, 33, K.KERNEL_SMALL), (4096, 5120, 432, 33, K.KERNEL_PREFILL), (4160, 6160, 256, 64, K.KERNEL_SMALL),
])
def test_lines_from_33_tokens_on(d_in, d_out, r, b, kernel):
    assert K.slim_select_kernel(b, d_out, d_in, r) == kernel
    res = run_case(d_in, d_out, r, b, seed=63)
    assert res["ok"] and res["launches"] == 1, res
