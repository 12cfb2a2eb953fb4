"""Sizes whose numbers of items or words leave 32 bits or a fixed region."""
import pytest
import torch

from paper_2410_09615_b200 import binding as K, inputs, parity

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def room():
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < 40 << 30:
        pytest.skip("needs 40 GB of free device memory")
    yield
    torch.cuda.empty_cache()


def test_adapter_expansion_beyond_four_gigabytes_of_codes():
    rows, cols = 1_440_000_000, 6                     # three bytes a row, read one by one: 2^32 and 25 million
    g = torch.Generator(device="cuda").manual_seed(5)
    codes = torch.full((rows, cols // 2), 0x21, dtype=torch.uint8, device="cuda")
    codes[-1000:] = torch.randint(0, 256, (1000, cols // 2), dtype=torch.uint8, device="cuda", generator=g)
    scales = torch.ones((rows, 1), dtype=torch.bfloat16, device="cuda")
    scales[-1000:] = torch.rand((1000, 1), device="cuda", generator=g).bfloat16()
    out = K.slim_unpack_adapter(codes, scales)
    tail = codes[-1000:].int()
    want = torch.stack([((tail & 15) ^ 8) - 8, ((tail >> 4) ^ 8) - 8], -1).reshape(1000, cols)
    assert torch.equal(out[-1000:], (want.float() * scales[-1000:].float()).bfloat16())
    for at in (0, rows // 2, rows - 2000):
        assert torch.equal(out[at], torch.tensor([1, 2, 1, 2, 1, 2], dtype=torch.bfloat16, device="cuda"))


@pytest.mark.parametrize("kernel", [K.KERNEL_AUTO, K.KERNEL_PREFILL_PAIR])
def test_more_tokens_than_the_pair_kernel_has_words_for(kernel):
    d_in, d_out, r, b = 64, 256, 16, 31744 * 256 + 700
    g = torch.Generator(device="cuda").manual_seed(6)
    ly = inputs.make_layer(d_in, d_out, r, 1, 6)
    vals, meta = K.slim_pack(torch.from_numpy(ly.codes).cuda(), torch.from_numpy(ly.mask).cuda())
    L, R = K.bf16_from_bits(ly.L), K.bf16_from_bits(ly.R)
    X = torch.randn((b, d_in), device="cuda", generator=g, dtype=torch.bfloat16)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    Y = K.slim_linear_fwd(X, vals, meta, ly.s, L, R, status=status, kernel=kernel)
    assert K.read_status(status) == 0
    half = (b // 2 + 255) // 256 * 256
    for at in (0, half - 150, b - 300):
        ref = K.slim_linear_fwd(X[at:at + 300], vals, meta, ly.s, L, R, kernel=K.KERNEL_SIMPLE)
        res = parity.compare(inputs.bf16_bits_to_f64(K.bits_from_bf16(Y[at:at + 300])), inputs.bf16_bits_to_f64(K.bits_from_bf16(ref)))
        assert res["ok"], (at, res)
