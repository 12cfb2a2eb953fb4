"""Sizes whose numbers of items or words leave 32 bits or a fixed region."""
import pytest
import torch

from paper_2410_09615_b200 import binding as K

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
