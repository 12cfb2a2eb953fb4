"""Every entry point of the compiled call path gives the interpreter to other threads while it is inside the library: a stand-in for
the library's function returns only when another thread has run (or, with an error, after a second)."""
import ctypes
import subprocess
import threading
import time

import pytest
import torch

from paper_2410_09615_b200 import binding as K

pytestmark = pytest.mark.gpu

STAND_IN = """
#include <time.h>
volatile int go = 0;
int stall(void) {
    struct timespec nap = {0, 1000000};
    for (int i = 0; i < 1000; ++i) {
        if (go) return 0;
        nanosleep(&nap, 0);
    }
    return 6;
}
"""
NAMES = ["slim_linear_fwd_ex", "slim_linear_fwd_tiled", "slim_linear_fwd_q", "slim_tiled_bytes", "slim_strerror", "slim_pack", "slim_quant",
         "slim_quant_workspace_bytes", "slim_mask_top2", "slim_pack_adapter"]
STALLED = ["slim_linear_fwd_ex", "slim_linear_fwd_tiled", "slim_linear_fwd_q", "slim_pack", "slim_quant", "slim_mask_top2", "slim_pack_adapter"]


def test_other_threads_run_during_a_call(tmp_path):
    src, so = tmp_path / "stall.c", tmp_path / "stall.so"
    src.write_text(STAND_IN)
    subprocess.run(["gcc", "-O1", "-shared", "-fPIC", str(src), "-o", str(so)], check=True)
    lib = ctypes.CDLL(str(so))
    go = ctypes.c_int.in_dll(lib, "go")
    addr = lambda f: ctypes.cast(f, ctypes.c_void_p).value
    own = [addr(getattr(K.lib(), n)) for n in NAMES]
    u8 = lambda *s: torch.zeros(s, dtype=torch.uint8, device="cuda")
    bf = lambda *s: torch.zeros(s, dtype=torch.bfloat16, device="cuda")
    i8, f32 = torch.zeros((16, 256), dtype=torch.int8, device="cuda"), torch.zeros((16, 256), device="cuda")
    calls = {
        "linear_fwd": lambda: K.slim_linear_fwd(bf(1, 256), u8(16, 64), u8(16, 32), 1.0, None, None, workspace=u8(256)),
        "linear_fwd_tiled": lambda: K.slim_linear_fwd_tiled(bf(1, 256), u8(K.slim_tiled_bytes(16, 256)), 16, 1.0, None, None, workspace=u8(256)),
        "linear_fwd_q": lambda: K.slim_linear_fwd_q(bf(1, 256), u8(16, 64), u8(16, 32), 1.0, u8(16, 8), bf(16, 1), u8(16, 128), bf(16, 2), workspace=u8(256)),
        "pack": lambda: K.slim_pack(i8, u8(16, 256), check=False),
        "quant": lambda: K.slim_quant(f32),
        "mask_top2": lambda: K.slim_mask_top2(i8),
        "pack_adapter": lambda: K.slim_pack_adapter(bf(16, 64)),
    }
    native = K.native()
    try:
        native.bind(K.SlimError, *[addr(lib.stall) if n in STALLED else a for n, a in zip(NAMES, own)])
        for name, call in calls.items():
            go.value = 0
            other = threading.Thread(target=lambda: (time.sleep(0.02), setattr(go, "value", 1)))
            other.start()
            try:
                call()                                    # raises where the other thread could not run
            except K.SlimError as e:
                pytest.fail(f"{name} kept the interpreter: {e}")
            finally:
                other.join()
    finally:
        native.bind(K.SlimError, *own)
