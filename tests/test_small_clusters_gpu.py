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


@pytest.mark.parametrize("d_in,d_out,r,b", [
    (4096, 4096, 832, 9), (4096, 5504, 832, 13), (2048, 3072, 416, 16), (1088, 4096, 832, 8), (8192, 2048, 1040, 16),
])
def test_ranks_of_many_steps_repeat_bit_for_bit(d_in, d_out, r, b):
    """More steps of L than the ring has places, on tiles of 128 and 64 rows: consumers wait for stages again and again, and each of their warps
    has to go on as a whole."""
    import torch
    gen = torch.Generator(device="cuda").manual_seed(d_in + r)
    codes = torch.randint(-8, 8, (d_out, d_in), generator=gen, device="cuda", dtype=torch.int8)
    vals, meta = K.slim_pack(codes, K.slim_mask_top2(codes, None))
    kept, _ = K.slim_unpack(vals, meta)
    rand = lambda *shape, std=1.0: (torch.randn(shape, generator=gen, device="cuda") * std).bfloat16()
    X, L, R, s = rand(b, d_in), rand(d_out, r, std=0.02), rand(r, d_in, std=0.02), 0.004
    want = X.double() @ (kept.double() * s).T + (X.double() @ R.double().T) @ L.double().T
    ws = K.new_workspace(b, d_out, d_in, r)
    first = None
    for _ in range(40):
        outs = [K.slim_linear_fwd(X, vals, meta, s, L, R, workspace=ws) for _ in range(10)]
        torch.cuda.synchronize()
        first = outs[0] if first is None else first
        assert all(torch.equal(Y.view(torch.int16), first.view(torch.int16)) for Y in outs)
    err = first.double() - want
    # bf16 results (2^-9 of the value) of a T rounded to bf16 once
    assert err.norm() <= 1e-2 * want.norm() and bool((err.abs() <= 1e-2 * want.abs() + 1e-2 * want.pow(2).mean().sqrt()).all())
