"""What a warp learns from a barrier through one of its lanes is ordered for the others too, and tensor memory is stored over only behind
the fence that follows the wait for the MMAs that read it."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2410_09615_b200", "csrc")
TEXT = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "fwd_prefill.cu")).read())


def test_an_answer_handed_over_by_a_shuffle_is_followed_by_a_warp_barrier():
    shuffles = [m.end() for m in re.finditer(r"__shfl_sync\([^;]*\banswer\b[^;]*;", TEXT)]
    assert shuffles
    for at in shuffles:
        assert re.match(r"\s*__syncwarp\(\);", TEXT[at:]), TEXT[at:at + 80]


def test_tensor_memory_is_stored_over_behind_the_fence():
    stores = [m.start() for m in re.finditer(r"asm volatile\(\"tcgen05\.st\.sync\.aligned\.32x32b\.x[24]\.b32", TEXT)]
    assert len(stores) == 2                          # the index words, before the expanded weights where those go there too
    for at in stores:
        wait = max(TEXT.rfind("mbar_wait(&empty[", 0, at), TEXT.rfind("mbar_wait_all(&pk_full[", 0, at))
        assert "fence_after_sync();" in TEXT[wait:at]
