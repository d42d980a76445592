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


@pytest.mark.parametrize("adaptive,P", [(1, 900), (1, 20000), (1, 30000), (0, 30000), (0, 50000)])
def test_a_device_that_holds_no_cluster_gets_none(fake_cuda, adaptive, P):
    # (a part of a device may have no group of SMs that is large enough): the call takes the kernels that need none
    fake_cuda.reset(device=3, resident={n: 0 for n in range(2, 9)})
    p = binding.Params(kv_heads=4, gqa_ratio=4, budget=64, budget_mode=adaptive).c()
    rc = fake_cuda.lib.mixkv_compress_layer(ONE, ONE, ONE, None, 1, P + 32, C.byref(p), ONE, 1 << 30, None, ONE, ONE, ONE,
                                            *[None] * 6)
    assert rc == 0
    calls = fake_cuda.launches()
    assert all(x.cluster == 1 for x in calls), calls
    unfused = adaptive or P > 40960
    assert [x.kernel for x in calls] == ["k_pass1", "k_pass2"] + ["k_mixpool"] * unfused + ["k_budget"] * adaptive + ["k_tail"]


@pytest.mark.parametrize("sequences,heads,P,shape", [
    (15, 8, 700, (1024, 8)), (17, 8, 700, None), (17, 8, 9000, (512, 8)), (36, 4, 700, (512, 4)), (36, 4, 20000, (1024, 4)),
    (60, 4, 9000, (512, 4)), (31, 8, 9000, None)])
def test_adaptive_budgets_take_clusters_that_are_resident(fake_cuda, sequences, heads, P, shape):
    fake_cuda.reset(device=4, resident={3: 45, 4: 33, 5: 26, 6: 22, 7: 15, 8: 15})
    p = binding.Params(kv_heads=heads, gqa_ratio=4, budget=64, budget_mode=1).c()
    rc = fake_cuda.lib.mixkv_compress_layers(ONE, ONE, ONE, sequences, C.c_int64(0), C.c_int64(0), None, 1, P + 32,
                                             C.byref(p), ONE, 1 << 40, None, ONE, ONE, ONE, *[None] * 7, 0)
    assert rc == 0
    calls = fake_cuda.launches()[2:]
    if shape:
        assert [x[1:] for x in calls] == [(sequences * heads, *shape, "k_tail")]
    else:
        assert [x.kernel for x in calls] == ["k_mixpool", "k_budget", "k_tail"]


@pytest.mark.parametrize("device,error", [(-1, 0), (5, 209), (5, 2)])
def test_questions_that_fail_leave_no_error_behind(fake_cuda, device, error):
    # no device, no image for the device, no memory: shape queries answer all the same, and the next check of the last
    # error, in the caller's own code, must not find theirs
    fake_cuda.reset(device=device, query_error=error)
    lib, c = fake_cuda.lib, C.byref
    fixed, adaptive = (binding.Params(kv_heads=4, gqa_ratio=4, budget=64, budget_mode=m).c() for m in (0, 1))
    assert lib.mixkv_launches_for(c(fixed), 1, 1, 60000) > 0 and lib.mixkv_launches_for(c(adaptive), 1, 1, 9000) > 0
    assert lib.mixkv_stage_name_for(c(fixed), 1, 1, 60000, 0) == b"pass1"
    assert fake_cuda.last_error() == 0
    size = C.c_size_t()
    assert lib.mixkv_workspace_size(c(fixed), 1, 60000, 60000, c(size)) == 0
    cc = C.c_int32()
    assert lib.mixkv_device_check(c(cc)) == (-4 if device < 0 else 0)
    assert fake_cuda.last_error() == 0


def test_a_cluster_that_cannot_be_asked_for_is_not_launched(fake_cuda):
    # what the runtime answers with an error is no cluster at all, and is asked again the next time
    p = binding.Params(kv_heads=4, gqa_ratio=4, budget=64, budget_mode=1).c()
    call = lambda: fake_cuda.lib.mixkv_compress_layer(ONE, ONE, ONE, None, 1, 20032, C.byref(p), ONE, 1 << 30, None, ONE,
                                                      ONE, ONE, *[None] * 6)
    fake_cuda.reset(device=6)
    assert call() == 0 and fake_cuda.launches()[-1].cluster == 4
    fake_cuda.reset(device=7, ask_error=912)
    assert call() == 0 and all(x.cluster == 1 for x in fake_cuda.launches()) and fake_cuda.last_error() == 0
    fake_cuda.reset(device=7)
    assert call() == 0 and fake_cuda.launches()[-1].cluster == 4


def test_an_older_error_is_not_taken_for_a_launch_that_failed(fake_cuda):
    fake_cuda.reset()
    fake_cuda.runtime.cudaSetDevice(99)     # an error of the caller's own, not looked at yet
    assert fake_cuda.last_error() != 0
    assert fake_cuda.lib.mixkv_selftest_bounded_wait(ONE, None, None) == 0


@pytest.mark.parametrize("batch,H,P,budget,tail", [
    (1, 16, 512, 1, 1), (1, 16, 513, 2, 1), (15, 9, 4100, 8, 1), (16, 8, 4100, 4, 1), (30, 8, 4100, 4, 1), (33, 8, 4100, 4, 1),
    (34, 8, 4100, 2, 1), (31, 8, 2100, 4, 1), (60, 8, 1030, 2, 1), (61, 8, 1030, 2, 1), (64, 8, 1030, 2, 1),
    (19, 9, 16384, 4, 1), (40, 8, 13000, 2, 1), (1, 8, 60000, 8, 8),
    (1, 8, 1024, 0, 8), (1, 8, 1025, 0, 8), (15, 8, 4100, 0, 8), (19, 8, 16384, 0, 8)])
def test_adaptive_selection_takes_the_clusters_its_gpu_tests_name(fake_cuda, batch, H, P, budget, tail):
    # test_gpu_parity.py: sizes at which the selection is compared with the oracle, by the number of CTAs that share a
    # sequence in the budget kernel (0: the tail kernel shares the budgets out)
    fake_cuda.reset(device=8, resident={3: 45, 4: 33, 5: 26, 6: 22, 7: 15, 8: 15})
    p = binding.Params(kv_heads=H, gqa_ratio=1, window=16, budget=116, budget_mode=1).c()
    cu = (C.c_int32 * (batch + 1))(*[b * (P + 16) for b in range(batch + 1)])
    rc = fake_cuda.lib.mixkv_select(ONE, cu if batch > 1 else None, batch, P + 16, C.byref(p), ONE, 1 << 40, ONE, ONE, ONE,
                                    None, None)
    assert rc == 0
    calls = [(x.kernel, x.cluster) for x in fake_cuda.launches()]
    assert calls == [("k_budget", budget)] * (budget > 0) + [("k_tail", tail)]
