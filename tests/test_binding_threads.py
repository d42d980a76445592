"""The binding gives up the interpreter lock while a call is in the library: a launch can wait for the GPU, and
what it waits for may be a callback or another thread that needs the interpreter.  The library is replaced by one
whose entry points wait until another Python thread lets them go (two seconds at most)."""
import os
import subprocess
import sys
import threading

import pytest

from paper_2510_20707_b200 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

LIBRARY = r"""
#include <stdatomic.h>
#include <stddef.h>
#include <time.h>
static atomic_int inside, let_go;
int entered(void) { return atomic_load(&inside); }
void release(void) { atomic_store(&let_go, 1); }
static int wait_for_release(void) {
  atomic_store(&inside, 1);
  const struct timespec ms = {0, 1000000};
  int k = 0;
  while (!atomic_load(&let_go) && k++ < 2000) nanosleep(&ms, NULL);
  const int ok = atomic_load(&let_go);
  atomic_store(&inside, 0);
  atomic_store(&let_go, 0);
  return ok ? 0 : -4;
}
int mixkv_internal_scores() { return wait_for_release(); }
int mixkv_internal_select() { return wait_for_release(); }
int mixkv_compress_layer_traced() { return wait_for_release(); }
int mixkv_compress_layers() { return wait_for_release(); }
int mixkv_compress_layers_budgeted() { return wait_for_release(); }
int mixkv_similarity_map() { return wait_for_release(); }
int mixkv_decode_attention() { return wait_for_release(); }
int mixkv_workspace_size_layers(const void* p, int n, int b, long long t, int m, size_t* bytes) {
  return *bytes = 256, 0;
}
int mixkv_similarity_workspace_size(int h, int L, int b, size_t* bytes) { return *bytes = 256, 0; }
"""

PROGRAM = r"""
import ctypes, sys, threading, time, types
import torch
from paper_2510_20707_b200 import binding
device, fake = sys.argv[1:]
lib = ctypes.CDLL(fake)
binding.load_library()
binding.LIB_PATH = fake            # what the native module is bound to
H, L, W, B = 2, 64, 16, 32
p = binding.Params(kv_heads=H, gqa_ratio=1, window=W, budget=B)
t = lambda *shape, dtype=torch.bfloat16: torch.zeros(shape, dtype=dtype, device=device)
i32 = torch.int32
K, Q = t(1, H, L, 128), t(1, 1, H, W, 128)
# "cpu": only the calls that need no new tensor; nothing looks at the stream or at the memory
stream = types.SimpleNamespace(cuda_stream=0) if device == "cpu" else None
ws = t(256, dtype=torch.uint8)
out = dict(K_out=t(1, H * B, 128), V_out=t(1, H * B, 128), out_row_offsets=t(1, H + 1, dtype=i32), status=t(1, dtype=i32))
one = dict(out, **{k: out[k][0] for k in ("K_out", "V_out", "out_row_offsets")})
kw = dict(workspace=ws, stream=stream)
calls = dict(
    layer=lambda: binding.compress_layer(K[0], K[0], Q[0], p, out=one, **kw),
    layers=lambda: binding.compress_layers(K, K, Q, p, out=out, **kw),
    budgeted=lambda: binding.compress_layers(K, K, Q, p, out=out, head_budgets=t(1, H, dtype=i32), **kw))
if device != "cpu":
    calls.update(
        scores=lambda: binding.scores(K[0], K[0], Q[0], p), static=lambda: binding.scores_static(K[0], K[0], Q[0], p),
        select=lambda: binding.select(t(H, L - W, dtype=torch.float32), p),
        new_outputs=lambda: binding.compress_layer(K[0], K[0], Q[0], p),
        similarity=lambda: binding.similarity_map(K[0], 4),
        decode=lambda: binding.decode_attention(K[0], K[0], t(H, 2, dtype=i32), t(H, 1, 1, 128), 1, 1, 4))
for name, call in calls.items():
    def watch():
        end = time.monotonic() + 10
        while not lib.entered() and time.monotonic() < end: time.sleep(0.001)
        lib.release()
    th = threading.Thread(target=watch)
    th.start()
    try:
        call()
    except binding.MixKVError as e:
        sys.exit(f"{name}: no other thread ran during the call ({e})")
    th.join()
print("ok", len(calls))
"""


@pytest.mark.parametrize("device,n", [("cpu", 3), pytest.param("cuda", 9, marks=pytest.mark.gpu)])
def test_other_threads_run_while_a_call_is_in_the_library(device, n, tmp_path):
    build.build()
    src, lib = tmp_path / "waiting.c", tmp_path / "libwaiting.so"
    src.write_text(LIBRARY)
    subprocess.run(["gcc", "-std=gnu11", "-O1", "-shared", "-fPIC", "-w", "-o", str(lib), str(src)], check=True)
    r = subprocess.run([sys.executable, "-c", PROGRAM, device, str(lib)], cwd=ROOT, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == f"ok {n}", r.stdout + r.stderr


@pytest.mark.gpu
def test_calls_from_several_threads():
    # four threads with a stream and a workspace each, through one-layer, adaptive, decode and map calls at the same
    # time (what the library keeps per device is shared): every result has the bits of a call made alone
    import torch
    from paper_2510_20707_b200 import binding
    gen = torch.Generator(device="cuda").manual_seed(1)
    rand = lambda *shape: torch.randn(shape, generator=gen, device="cuda").bfloat16()
    K, V, Q = rand(4, 3000, 128), rand(4, 3000, 128), rand(1, 16, 32, 128)
    cache, q = rand(1, 4 * 300, 128), rand(1, 1, 16, 128)
    offs = (torch.arange(5, dtype=torch.int32, device="cuda") * 300).view(1, 5)
    params = [binding.Params(kv_heads=4, gqa_ratio=4, budget=128, budget_mode=m) for m in (0, 1)]
    size = max(binding.workspace_size(p, 1, 3000, 3000) for p in params)

    def work(ws):
        out = [binding.compress_layer(K, V, Q, p, workspace=ws) for p in params]
        res = [o[k] for o in out for k in ("s_comp", "idx_offsets", "out_row_offsets")]
        res += [o["idx"][:4 * 96] for o in out] + [out[0]["K_out"], out[0]["V_out"]]
        s = binding.scores(K, V, Q, params[0], workspace=ws)
        return res + [s["s_comp"], binding.select(s["s_comp"], params[0], workspace=ws)["idx"],
                      binding.decode_attention(cache, cache, offs, q, 4, 4, 300), *binding.similarity_map(K, 16)]

    new = lambda: torch.empty(size, dtype=torch.uint8, device="cuda")
    ref = work(new())
    torch.cuda.synchronize()
    found = []

    def thread():
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                ws = new()
                for _ in range(20):
                    got = work(ws)
                    stream.synchronize()
                    found.append(all(torch.equal(a, b) for a, b in zip(got, ref, strict=True)))
        except Exception as e:      # (a thread's exception would not fail the test)
            found.append(e)

    threads = [threading.Thread(target=thread) for _ in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert found == [True] * 80, found


@pytest.mark.gpu
def test_what_a_call_allocates_belongs_to_its_stream():
    # a workspace of the call's own is given back when the call returns: it may only be handed out again in the order
    # of the stream its kernels run on, whatever the current stream is
    import torch
    from paper_2510_20707_b200 import binding
    K, Q = torch.randn((4, 20000, 128), device="cuda").bfloat16(), torch.randn((1, 16, 32, 128), device="cuda").bfloat16()
    p = binding.Params(kv_heads=4, gqa_ratio=4, budget=128)
    need = binding.workspace_size(p, 1, 20000, 20000)
    ref = binding.scores(K, K, Q, p)["s_comp"]
    torch.cuda.synchronize()
    offs, q = torch.tensor([[0, 20000]], dtype=torch.int32, device="cuda"), torch.zeros((1, 1, 4, 128), device="cuda").bfloat16()
    for call in (lambda s: binding.scores(K, K, Q, p, stream=s), lambda s: binding.compress_layer(K, K, Q, p, stream=s),
                 lambda s: binding.select(ref, p, stream=s), lambda s: binding.similarity_map(K, 4, stream=s),
                 lambda s: binding.compress_layers(K[None], K[None], Q[None], p, stream=s),
                 lambda s: binding.decode_attention(K[:1], K[:1], offs, q, 1, 4, 20000, stream=s)):
        torch.cuda.empty_cache()
        side = torch.cuda.Stream()
        before = sum(seg["total_size"] for seg in torch.cuda.memory_snapshot() if seg["stream"] == 0)
        out = call(side)
        assert torch.cuda.current_stream() != side
        own = sum(seg["total_size"] for seg in torch.cuda.memory_snapshot() if seg["stream"] == side.cuda_stream)
        assert own > 0 and sum(seg["total_size"] for seg in torch.cuda.memory_snapshot() if seg["stream"] == 0) == before
        side.synchronize()
        if isinstance(out, dict) and "s_comp" in out:
            assert torch.equal(out["s_comp"].view_as(ref), ref) and own >= need
        del out


@pytest.mark.gpu
def test_the_first_cuda_call_of_a_thread():
    # a thread that has made no other CUDA call has no context bound to it, and a call that allocates nothing does not
    # get one from the allocator either
    import torch
    from paper_2510_20707_b200 import binding
    K, Q = torch.randn((4, 1000, 128), device="cuda").bfloat16(), torch.randn((1, 16, 32, 128), device="cuda").bfloat16()
    p = binding.Params(kv_heads=4, gqa_ratio=4, budget=96)
    ws = torch.empty(binding.workspace_size(p, 1, 1000, 1000), dtype=torch.uint8, device="cuda")
    out = binding.compress_layer(K, K, Q, p, workspace=ws, want_aux=False)
    s = binding.scores(K, K, Q, p)["s_comp"]
    offs, q = torch.tensor([[0, 1000]], dtype=torch.int32, device="cuda"), torch.zeros((1, 1, 4, 128), device="cuda").bfloat16()
    calls = [lambda: binding.compress_layer(K, K, Q, p, workspace=ws, out=out),
             lambda: binding.scores(K, K, Q, p, workspace=ws), lambda: binding.scores_static(K, K, Q, p),
             lambda: binding.select(s, p, workspace=ws), lambda: binding.similarity_map(K, 16),
             lambda: binding.decode_attention(K[:1], K[:1], offs, q, 1, 4, 1000)]
    found = []

    def thread(call):
        try:
            call()
            found.append(True)
        except Exception as e:
            found.append(e)

    for call in calls:
        call()                  # what is looked up once per device has been
        t = threading.Thread(target=thread, args=(call,))
        t.start()
        t.join()
    torch.cuda.synchronize()
    assert found == [True] * len(calls), found


@pytest.mark.gpu
def test_two_threads_on_one_stream():
    # two threads, a problem each, all calls on one stream: those that work in the library's own scratch array, and
    # those with a workspace per thread, give the bits of calls made alone
    import torch
    from paper_2510_20707_b200 import binding
    gen = torch.Generator(device="cuda").manual_seed(2)
    rand = lambda *shape: torch.randn(shape, generator=gen, device="cuda").bfloat16()
    stream = torch.cuda.Stream()
    problems, found = [], []
    for L, H, G in ((3000, 4, 4), (7001, 2, 7)):
        p = binding.Params(kv_heads=H, gqa_ratio=G, budget=96)
        ws = torch.empty(binding.workspace_size(p, 1, L, L), dtype=torch.uint8, device="cuda")
        K, V, Q = rand(H, L, 128), rand(H, L, 128), rand(1, H * G, 32, 128)
        ref = binding.scores(K, V, Q, p)
        problems.append((K, V, Q, p, ws, ref))
    torch.cuda.synchronize()
    start = threading.Barrier(2)

    def thread(K, V, Q, p, ws, ref):
        try:
            start.wait()
            for _ in range(10):
                outs = []
                for _ in range(10):
                    outs += [binding.scores_static(K, V, Q, p, stream=stream),
                             binding.scores(K, V, Q, p, workspace=ws, stream=stream)]
                stream.synchronize()
                found.extend(all(torch.equal(o[k], ref[k]) for k in ("s_comp", "s_ex", "s_div", "rbar")) for o in outs)
        except Exception as e:
            found.append(e)

    threads = [threading.Thread(target=thread, args=p) for p in problems]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert found == [True] * 400, found
