"""GPU parity of mixkv_decode_attention (one query token over the compact cache) against the
plain fp64 definition.  The compact caches fed to the kernel are built by the CPU oracle."""
import numpy as np
import pytest
import torch

import oracle
from oracle import decode_plain
from paper_2510_20707_b200 import binding, synth
from parity import params_pair

pytestmark = pytest.mark.gpu
RTOL, ATOL = 2e-4, 2e-5   # fp32 accumulation of exact bf16 products, weights carried as two bf16


def bits_to_dev(a):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.int16)).cuda().view(torch.bfloat16)


def run(wl, n_layers, **kw):
    po, _ = params_pair(wl, **kw)
    H, G, B = wl.kv_heads, wl.gqa_ratio, po.budget
    cu = wl.cu_seqlens
    rows_cap = wl.batch * H * B
    Kc = np.zeros((n_layers, rows_cap, 128), np.uint16)
    Vc = np.zeros_like(Kc)
    offs = np.zeros((n_layers, wl.batch * H + 1), np.int32)
    rng = np.random.default_rng(wl.seed)
    q = synth.f32_to_bf16_bits(rng.standard_normal((n_layers, wl.batch, H * G, 128)).astype(np.float32))
    refs = []
    for l in range(n_layers):
        x = synth.make_layer(wl, l, "calibrated")
        c = oracle.compress_layer(x["K"], x["V"], x["Q"], po, cu=None if wl.batch == 1 else cu)
        n = c["K_out"].shape[0]
        Kc[l, :n], Vc[l, :n], offs[l] = c["K_out"], c["V_out"], c["out_row_offsets"]
        refs.append(decode_plain.decode_attention(c["K_out"], c["V_out"], c["out_row_offsets"], q[l], H, G))
    most = int(np.diff(offs, axis=1).max())      # adaptive budgets may give a head more than B rows
    out = binding.decode_attention(bits_to_dev(Kc), bits_to_dev(Vc), torch.from_numpy(offs).cuda(),
                                   bits_to_dev(q), H, G, max_rows=most)
    torch.cuda.synchronize()
    got = out.cpu().numpy()
    for l in range(n_layers):
        assert np.allclose(got[l], refs[l], rtol=RTOL, atol=ATOL), f"layer {l}"
    return got


def test_fixed_budget_cache_gqa7():
    wl = synth.small_workload(H=4, G=7, W=32, seq_lens=(2048,), pool_kernel=7, budget=128, seed=71,
                              centroids=16)
    run(wl, 3)


def test_ragged_adaptive_cache():
    wl = synth.small_workload(H=3, G=4, W=16, seq_lens=(900, 200, 1500), pool_kernel=5, budget=96,
                              seed=72, centroids=8)
    run(synth.with_budget(wl, 96, budget_mode=1), 2)


@pytest.mark.parametrize("rows,G", [((4096, 1000, 4096, 37), 7), ((20000, 513), 4), ((256, 257), 16)])
def test_long_rows_split_over_a_cluster(rows, G):
    # heads with thousands of rows (a large budget, or a cache that was not compressed): the rows
    # of a head are dealt out 16 at a time over the warps of a cluster, each with a running
    # softmax; two layers, ragged heads (row counts that are no multiple of 16), G on both sides
    # of 8 (the second half of the 16 head slots), a sharp row so that the running reference moves
    H, NL = len(rows), 2
    rng = np.random.default_rng(sum(rows))
    cap = int(sum(rows))
    K = rng.standard_normal((NL, cap, 128)).astype(np.float32)
    V = rng.standard_normal((NL, cap, 128)).astype(np.float32)
    q = rng.standard_normal((NL, 1, H * G, 128)).astype(np.float32)
    K[0, rows[0] - 3] = 6.0 * q[0, 0, 0]          # one key far above the rest, late in head 0
    Kb, Vb, qb = (synth.f32_to_bf16_bits(a) for a in (K, V, q))
    offs = np.tile(np.concatenate([[0], np.cumsum(rows)]).astype(np.int32), (NL, 1))
    out = binding.decode_attention(bits_to_dev(Kb), bits_to_dev(Vb), torch.from_numpy(offs).cuda(),
                                   bits_to_dev(qb), H, G, max_rows=max(rows)).cpu().numpy()
    for l in range(NL):
        ref = decode_plain.decode_attention(Kb[l], Vb[l], offs[l], qb[l], H, G)
        assert np.allclose(out[l], ref, rtol=RTOL, atol=ATOL), f"layer {l}"


@pytest.mark.parametrize("G", [1, 8, 9, 13])
def test_step_edges_and_head_counts(G):
    # heads of 1, 15, 16, 17 and 33 rows (below, at and past one 16-row step) for group sizes at
    # the edges of the 8 + 8 head slots of a tile
    rows, NL = (1, 15, 16, 17, 33), 2
    H = len(rows)
    rng = np.random.default_rng(100 + G)
    cap = int(sum(rows))
    Kb, Vb, qb = (synth.f32_to_bf16_bits(rng.standard_normal(sh).astype(np.float32))
                  for sh in ((NL, cap, 128), (NL, cap, 128), (NL, 1, H * G, 128)))
    offs = np.tile(np.concatenate([[0], np.cumsum(rows)]).astype(np.int32), (NL, 1))
    out = binding.decode_attention(bits_to_dev(Kb), bits_to_dev(Vb), torch.from_numpy(offs).cuda(),
                                   bits_to_dev(qb), H, G, max_rows=max(rows)).cpu().numpy()
    for l in range(NL):
        ref = decode_plain.decode_attention(Kb[l], Vb[l], offs[l], qb[l], H, G)
        assert np.allclose(out[l], ref, rtol=RTOL, atol=ATOL), f"layer {l}"


@pytest.mark.parametrize("NL,batch,H,G,lo,hi", [
    (4, 16, 8, 7, 0, 40),          # 512 units: empty heads, fewer rows than the warps of a CTA take
    (3, 13, 9, 16, 1, 300),        # wide heads, a unit count that no number of CTAs divides
    (28, 3, 4, 1, 120, 140),       # steps of all eight warps and one more
    (1, 15, 1, 4, 1500, 1600), (1, 16, 1, 9, 1500, 1600), (2, 4, 4, 7, 1, 900),   # few units, a CTA alone on its SM
    (8, 7, 4, 7, 0, 200), (2, 37, 4, 16, 1, 130), (1, 149, 1, 7, 1, 120),   # one wave of two CTAs per SM
    (7, 7, 1, 7, 500, 700), (3, 19, 1, 12, 1, 500), (1, 143, 1, 4, 100, 200),   # one more than fits at 8, 7 and 3 CTAs
    (10, 13, 4, 7, 1, 1020)])      # a second wave that is short: two CTAs per unit
def test_more_units_than_one_wave(NL, batch, H, G, lo, hi):
    rng = np.random.default_rng(NL * batch)
    counts = rng.integers(lo, hi + 1, (NL, batch * H))
    counts[0, 0], counts[-1, -1] = lo, hi
    cap = int(counts.sum(1).max())
    K = synth.f32_to_bf16_bits(rng.standard_normal((NL, cap, 128)).astype(np.float32))
    V = synth.f32_to_bf16_bits(rng.standard_normal((NL, cap, 128)).astype(np.float32))
    q = synth.f32_to_bf16_bits(rng.standard_normal((NL, batch, H * G, 128)).astype(np.float32))
    offs = np.concatenate([np.zeros((NL, 1), np.int64), counts.cumsum(1)], 1).astype(np.int32)
    dev = [torch.from_numpy(x.view(np.int16)).cuda().view(torch.bfloat16) for x in (K, V, q)]
    out = binding.decode_attention(dev[0], dev[1], torch.from_numpy(offs).cuda(), dev[2], H, G, hi)
    again = binding.decode_attention(dev[0], dev[1], torch.from_numpy(offs).cuda(), dev[2], H, G, hi)
    torch.cuda.synchronize()
    assert torch.equal(out, again)
    k, v, qq = (synth.bf16_bits_to_f32(x).astype(np.float64) for x in (K, V, q))
    got = out.cpu().numpy()
    for l in range(NL):
        for u in range(batch * H):
            a, e = offs[l, u], offs[l, u + 1]
            rows = got[l, u // H, (u % H) * G:(u % H + 1) * G]
            if a == e:
                assert (rows == 0).all()
                continue
            s = qq[l, u // H, (u % H) * G:(u % H + 1) * G] @ k[l, a:e].T / np.sqrt(128.0)
            p = np.exp(s - s.max(1, keepdims=True))
            assert np.allclose(rows, p @ v[l, a:e] / p.sum(1, keepdims=True), rtol=2e-4, atol=2e-5), (l, u)


@pytest.mark.parametrize("units,rows,G,ragged", [
    (224, 1280, 7, False), (296, 1265, 16, False), (296, 1300, 4, True), (223, 1281, 9, True), (296, 1264, 4, True),
    (237, 1280, 7, False), (237, 1281, 9, True), (236, 1281, 9, True)])
def test_two_units_per_sm_in_a_cache_of_their_size(units, rows, G, ragged):
    # the cache has room for max_rows rows of every head: from 80 steps and 237 units (1.6 per SM) on one slot pair per
    # warp in flight, else three, whether the heads are of one length or not (none, one, a step and one, all rows among them)
    rng = np.random.default_rng(units + rows)
    counts = rng.integers(0, rows + 1, units) if ragged else np.full(units, rows)
    if ragged:
        counts[:6] = 0, 1, 16, 17, rows - 1, rows
    gen = torch.Generator(device="cuda").manual_seed(rows)
    K, V = (torch.randn((1, units * rows, 128), generator=gen, device="cuda").bfloat16() for _ in range(2))
    q = torch.randn((1, units, G, 128), generator=gen, device="cuda").bfloat16()
    offs = np.concatenate([[0], counts.cumsum()]).astype(np.int32)
    call = lambda: binding.decode_attention(K, V, torch.from_numpy(offs[None]).cuda(), q, 1, G, rows)
    out = call()
    assert torch.equal(out, call())
    Kd, Vd, qd = K[0].double(), V[0].double(), q[0].double()
    for u in range(units):
        a, e = offs[u], offs[u + 1]
        want = torch.softmax(qd[u] @ Kd[a:e].T / np.sqrt(128.0), 1) @ Vd[a:e]     # (no rows: zeros)
        assert torch.allclose(out[0, u].double(), want, rtol=RTOL, atol=ATOL), u


def test_repeated_calls_are_bit_identical():
    # the steps of a head go to fixed warps and the partial results are merged in a fixed order
    # (warps through shared memory, CTAs through distributed shared memory): twenty calls on the
    # same cache give the same bits
    rows, NL, G = (3000, 517, 2048), 3, 7
    H = len(rows)
    rng = np.random.default_rng(7)
    cap = int(sum(rows))
    Kb, Vb, qb = (synth.f32_to_bf16_bits(rng.standard_normal(sh).astype(np.float32))
                  for sh in ((NL, cap, 128), (NL, cap, 128), (NL, 1, H * G, 128)))
    offs = torch.from_numpy(np.tile(np.concatenate([[0], np.cumsum(rows)]).astype(np.int32), (NL, 1))).cuda()
    K, V, q = bits_to_dev(Kb), bits_to_dev(Vb), bits_to_dev(qb)
    first = binding.decode_attention(K, V, offs, q, H, G, max_rows=max(rows))
    for _ in range(20):
        again = binding.decode_attention(K, V, offs, q, H, G, max_rows=max(rows))
        assert torch.equal(first, again)


def test_capture_of_shapes_that_did_not_run_before():
    # a call outside capture is asked for once per entry point: what another shape needs (its kernel's shared memory,
    # the clusters a device holds) may be looked up while a capture is going on
    def problem(units, rows, G):
        offs = (torch.arange(units + 1, dtype=torch.int32, device="cuda") * rows).view(1, -1)
        gen = torch.Generator(device="cuda").manual_seed(units)
        K, V = (torch.randn((1, units * rows, 128), generator=gen, device="cuda").bfloat16() for _ in range(2))
        q = torch.randn((1, units, G, 128), generator=gen, device="cuda").bfloat16()
        return K, V, offs, q, 1, G, rows
    binding.decode_attention(*problem(4, 100, 4))
    for units, rows, G in ((20, 700, 4), (20, 700, 12), (48, 600, 9), (250, 200, 4), (296, 2100, 3), (250, 200, 11)):
        x = problem(units, rows, G)
        graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.graph(graph, stream=side):
            out = binding.decode_attention(*x)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, binding.decode_attention(*x)), (units, rows, G)


def test_empty_head_short_rows_and_bad_arguments():
    H, G = 2, 2
    rng = np.random.default_rng(3)
    K = synth.f32_to_bf16_bits(rng.standard_normal((1, 40, 128)).astype(np.float32))
    V = synth.f32_to_bf16_bits(rng.standard_normal((1, 40, 128)).astype(np.float32))
    q = synth.f32_to_bf16_bits(rng.standard_normal((1, 1, H * G, 128)).astype(np.float32))
    offs = np.array([[0, 0, 33]], np.int32)          # head 0 keeps nothing, head 1 keeps 33 rows
    out = binding.decode_attention(bits_to_dev(K), bits_to_dev(V), torch.from_numpy(offs).cuda(),
                                   bits_to_dev(q), H, G, max_rows=64).cpu().numpy()
    ref = decode_plain.decode_attention(K[0], V[0], offs[0], q[0], H, G)
    assert np.array_equal(out[0, 0, :G], np.zeros((G, 128)))
    assert np.allclose(out[0], ref, rtol=RTOL, atol=ATOL)
    with pytest.raises(binding.MixKVError):
        binding.decode_attention(bits_to_dev(K), bits_to_dev(V), torch.from_numpy(offs).cuda(),
                                 bits_to_dev(q), H, G, max_rows=0)
