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


def test_calls_on_the_static_scratch_enqueue_one_after_the_other(fake_cuda):
    # Every call on a device works in the same scratch array: when two threads call, on one stream even, the kernels
    # of one call must not come between those of another (its second pass would read the other's partial results).
    fake_cuda.reset(pause_us=2000)
    p = binding.Params(kv_heads=4, gqa_ratio=4, budget=64, pool_mode=1).c()
    failed = []

    def caller(i):
        fake_cuda.runtime.fake_caller(i)
        for k in range(4):
            f = fake_cuda.lib.mixkv_scores_static if k % 2 else fake_cuda.lib.mixkv_internal_scores
            head = (ONE, ONE, ONE, None, C.c_int32(1), C.c_int32(900 + i), C.byref(p))
            own = () if k % 2 else (C.c_int(1), None, C.c_size_t(0))
            failed.append(f(*head, *own, ONE, None, None, None, None, None, None))

    threads = [threading.Thread(target=caller, args=(i,)) for i in range(3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert failed == [0] * 12
    calls = fake_cuda.launches()
    kernels = ["k_pass1", "k_pass2", "k_poolsum", "k_mixpool"]
    assert [x.kernel for x in calls] == kernels * 12
    assert all(len({x.caller for x in calls[i:i + 4]}) == 1 for i in range(0, 48, 4)), [x.caller for x in calls]
