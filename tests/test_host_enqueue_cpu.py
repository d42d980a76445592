"""What the library's host code enqueues, against a CUDA runtime without a device (tests/fake_cuda.py)."""
import ctypes as C
import threading

import pytest

from paper_2510_20707_b200 import binding

ONE = C.c_void_p(256)      # an aligned pointer that is not null; nothing looks behind it

@pytest.mark.parametrize("entry", ["layer", "scores", "static", "similarity"])
def test_a_thread_may_make_its_first_cuda_call_here(fake_cuda, entry):
    # no call of the runtime has bound the device's context to the thread yet, and the driver's function that encodes
    # tensor maps wants one
    lib, rc = fake_cuda.lib, []
    p = binding.Params(kv_heads=4, gqa_ratio=4, budget=64).c()
    head = (ONE, ONE, ONE, None, 1, 900, C.byref(p))
    call = dict(
        layer=lambda: lib.mixkv_compress_layer(*head, ONE, 1 << 30, None, ONE, ONE, ONE, *[None] * 6),
        scores=lambda: lib.mixkv_scores(*head, ONE, 1 << 30, ONE, *[None] * 6),
        static=lambda: lib.mixkv_scores_static(*head, ONE, *[None] * 6),
        similarity=lambda: lib.mixkv_similarity_map(ONE, 4, 900, 128, 16, ONE, 1 << 30, ONE, None, None))[entry]
    for _ in range(2):      # (what a device is asked once has been asked by the second)
        t = threading.Thread(target=lambda: rc.append(call()))
        t.start()
        t.join()
    assert rc == [0, 0]
