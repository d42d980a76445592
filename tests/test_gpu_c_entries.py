"""The public C entry points, called with plain pointers as include/mixkv.h declares them.  The Python binding takes
others for some of them (csrc/internal_api.h: the status word is cleared by the call), so they are run here to a
result: bit for bit that of the binding, whose results are checked against the oracle elsewhere."""
import ctypes as C

import pytest
import torch

from paper_2510_20707_b200 import binding, synth
from parity import params_pair, to_dev

pytestmark = pytest.mark.gpu


def problem(mode=0, batch=2):
    wl = synth.small_workload(H=3, G=2, W=16, seq_lens=(1500, 333)[:batch], pool_kernel=7, budget=64, seed=91)
    x = synth.make_layer(wl, 0, "calibrated")
    _, pg = params_pair(wl, budget_mode=mode)
    cu = [int(c) for c in wl.cu_seqlens]
    arr = (C.c_int32 * len(cu))(*cu) if batch > 1 else None
    ws = torch.empty(binding.workspace_size(pg, batch, cu[-1], max(wl.seq_lens)), dtype=torch.uint8, device="cuda")
    return [to_dev(x[k]) for k in ("K", "V", "Q")], pg, cu if batch > 1 else None, arr, batch, cu[-1], ws


def stream():
    return torch.cuda.current_stream().cuda_stream


def like(t):
    return torch.full_like(t, 3)


@pytest.mark.parametrize("static", [False, True])
@pytest.mark.parametrize("batch", [1, 2])
def test_scores(static, batch):
    (K, V, Q), pg, cu, arr, batch, L, ws = problem(batch=batch)
    ref = binding.scores(K, V, Q, pg, cu_seqlens=cu)
    got = {k: like(ref[k]) for k in ("s_comp", "s_ex", "s_div", "rbar")}
    status, lib, pc = torch.full((1,), 7, dtype=torch.int32, device="cuda"), binding.load_library(), pg.c()
    outs = [got[k].data_ptr() for k in ("s_comp", "s_ex", "s_div", "rbar")] + [None, status.data_ptr(), stream()]
    head = [K.data_ptr(), V.data_ptr(), Q.data_ptr(), arr, batch, L, C.byref(pc)]
    rc = (lib.mixkv_scores_static(*head, *outs) if static else
          lib.mixkv_scores(*head, ws.data_ptr(), ws.numel(), *outs))
    assert rc == 0
    for k, t in got.items():
        assert torch.equal(t, ref[k]), k
    assert int(status.item()) == 7          # the caller's word is written on an error only
    # the optional outputs left out
    s = like(ref["s_comp"])
    outs = [s.data_ptr(), None, None, None, None, None, stream()]
    assert 0 == (lib.mixkv_scores_static(*head, *outs) if static else
                 lib.mixkv_scores(*head, ws.data_ptr(), ws.numel(), *outs))
    assert torch.equal(s, ref["s_comp"])


@pytest.mark.parametrize("mode", [0, 1])
def test_select(mode):
    (K, V, Q), pg, cu, arr, batch, L, ws = problem(mode)
    s = binding.scores(K, V, Q, pg, cu_seqlens=cu)["s_comp"]
    ref = binding.select(s, pg, cu_seqlens=cu)
    got = {k: like(ref[k]) for k in ("idx", "counts", "idx_offsets", "status")}
    pc = pg.c()
    assert 0 == binding.load_library().mixkv_select(
        s.data_ptr(), arr, batch, L, C.byref(pc), ws.data_ptr(), ws.numel(),
        *[got[k].data_ptr() for k in ("idx", "counts", "idx_offsets", "status")], stream())
    n = int(ref["idx_offsets"][-1])
    assert torch.equal(got["idx"][:n], ref["idx"][:n]) and (got["idx"][n:] == 3).all()
    assert torch.equal(got["counts"], ref["counts"]) and torch.equal(got["idx_offsets"], ref["idx_offsets"])
    assert int(got["status"].item()) == 3   # accepted and never written


@pytest.mark.parametrize("mode", [0, 1])
def test_compress_layer(mode):
    (K, V, Q), pg, cu, arr, batch, L, ws = problem(mode)
    ref = binding.compress_layer(K, V, Q, pg, cu_seqlens=cu)
    names = ("K_out", "V_out", "out_row_offsets", "idx", "counts", "idx_offsets", "s_comp")
    got, pc, lib = {k: like(ref[k]) for k in names}, pg.c(), binding.load_library()
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    for aux in (True, False):               # without them they are kept in the workspace
        if not aux:
            got.update({k: like(ref[k]) for k in names[:3]})
        assert 0 == lib.mixkv_compress_layer(
            K.data_ptr(), V.data_ptr(), Q.data_ptr(), arr, batch, L, C.byref(pc), ws.data_ptr(), ws.numel(), None,
            *[got[k].data_ptr() for k in names[:3]], *[got[k].data_ptr() if aux else None for k in names[3:]],
            status.data_ptr(), stream())
        rows, n = int(ref["out_row_offsets"][-1]), int(ref["idx_offsets"][-1])
        for k in names:
            m = {"K_out": rows, "V_out": rows, "idx": n}.get(k, len(ref[k]))
            assert torch.equal(got[k][:m], ref[k][:m]), k
        assert int(status.item()) == 0
