"""GPU parity of the redundancy analysis map (mixkv_similarity_map) against the plain pairwise
definition in oracle/similarity_plain.py."""
import numpy as np
import pytest
import torch

from oracle import similarity_plain
from paper_2510_20707_b200 import binding, synth

pytestmark = pytest.mark.gpu
ATOL, RTOL = 2e-5, 2e-4   # fp32 sums of up to `block` unit rows and 128-term dot products


def run(X_bits, block):
    X = torch.from_numpy(X_bits.view(np.int16)).cuda().view(torch.bfloat16)
    cells, mean = binding.similarity_map(X, block)
    torch.cuda.synchronize()
    ref_cells, ref_mean = similarity_plain.block_cosine_map(X_bits, block)
    assert np.allclose(cells.cpu().numpy(), ref_cells, rtol=RTOL, atol=ATOL)
    assert np.allclose(mean.cpu().numpy(), ref_mean, rtol=RTOL, atol=ATOL)
    return cells, mean


@pytest.mark.parametrize("H,L,block", [(3, 1000, 64), (2, 40, 1), (1, 1, 8), (2, 129, 128),
                                       (4, 777, 100), (2, 3000, 700)])
def test_random_rows_with_shared_component(H, L, block):
    rng = np.random.default_rng(L)
    X = rng.standard_normal((H, L, 128)) + 1.3 * rng.standard_normal((H, 1, 128))
    if L > 10:
        X[0, 5] = 0.0                       # a zero row has cosine 0 with everything
    run(synth.f32_to_bf16_bits(X.astype(np.float32)), block)


@pytest.mark.parametrize("H,L,block", [(2, 1000, 16), (1, 700, 4), (3, 300, 2), (2, 257, 1),
                                       (1, 130, 8), (2, 2049, 16), (1, 128, 1), (2, 391, 4)])
def test_small_maps_and_blocks(H, L, block):
    # blocks of which a warp takes whole ones (1, 2, 4, 8, 16 rows): ragged last tile and last block, a zero
    # row, diagonal cells without the i == j pairs
    rng = np.random.default_rng(1000 * block + L)
    X = rng.standard_normal((H, L, 128)) + 0.8 * rng.standard_normal((H, 1, 128))
    X[0, 3] = 0.0
    cells, _ = run(synth.f32_to_bf16_bits(X.astype(np.float32)), block)
    c = cells.cpu().numpy()
    # mirrored tiles are the same numbers; inside a diagonal tile (i, j) and (j, i) are summed in
    # a different order
    assert np.allclose(c, c.transpose(0, 2, 1), rtol=0, atol=1e-6)
    if block == 1:
        assert (np.diagonal(c, axis1=1, axis2=2) == 0).all()


@pytest.mark.parametrize("H,L,block", [
    (2, 331, 3), (1, 997, 31), (2, 1000, 32), (1, 1101, 33), (2, 2049, 255), (1, 1030, 257),   # steps of 32 rows
    (1, 4500, 513), (1, 5000, 4096), (1, 300, 512),                 # a cluster of CTAs per block, one block
    (1, 127, 1), (1, 129, 1), (3, 770, 6), (1, 4112, 16), (2, 2054, 2), (13, 1290, 10)])   # map edges, many heads
def test_block_and_tile_edges(H, L, block):
    rng = np.random.default_rng(7 * block + L)
    X = rng.standard_normal((H, L, 128)) + 0.9 * rng.standard_normal((H, 1, 128))
    X[0, L // 2] = 0.0
    X[0, L - 1] = 0.0
    cells, _ = run(synth.f32_to_bf16_bits(X.astype(np.float32)), block)
    assert torch.allclose(cells, cells.transpose(1, 2), rtol=0, atol=1e-6)


@pytest.mark.parametrize("L,block", [(8192, 1), (32768, 16)])
def test_full_size_sampled(L, block):
    # The map of the keys of two heads at full size.  The pairwise oracle needs the L x L
    # matrix in fp64, so it checks sampled 128-row tiles: a cell depends only on the rows of its
    # two blocks, and the oracle run on the rows of tiles a and b gives the cells of (a, a),
    # (a, b), (b, a), (b, b).  The whole map is checked for symmetry and range, its mean against
    # Eq. 4 from the oracle's key geometry.
    import oracle
    wl = synth.replace(synth.CONFIGS["C3"], seq_lens=(L,), vision_tokens=(L - 256,),
                       frame_tokens=(L - 256) // 32)
    K = synth.make_layer(wl, 3, "calibrated")["K"][:2]
    X = torch.from_numpy(K.view(np.int16)).cuda().view(torch.bfloat16)
    cells, mean = binding.similarity_map(X, block)
    torch.cuda.synchronize()
    nT, per = L // 128, 128 // block
    for h in range(2):
        for a, b in ((0, 1), (5, nT - 1), (nT // 2, nT // 2 + 7), (nT - 2, nT - 1)):
            rows = np.concatenate([np.arange(a * 128, a * 128 + 128), np.arange(b * 128, b * 128 + 128)])
            ref, _ = similarity_plain.block_cosine_map(K[h:h + 1, rows], block)
            ia, ib = slice(a * per, a * per + per), slice(b * per, b * per + per)
            got = torch.cat([torch.cat([cells[h, ia, ia], cells[h, ia, ib]], 1),
                             torch.cat([cells[h, ib, ia], cells[h, ib, ib]], 1)], 0).cpu().numpy()
            assert np.allclose(got, ref[0], rtol=RTOL, atol=ATOL), (h, a, b)
        assert torch.allclose(cells[h], cells[h].T, rtol=0, atol=1e-6)
        assert float(cells[h].abs().max()) <= 1.0 + 1e-4
    rbar = np.array([oracle.key_geometry(K[h])[1] for h in range(2)])
    assert np.allclose(mean.cpu().numpy(), rbar, rtol=RTOL, atol=ATOL)


@pytest.mark.parametrize("H,L,block", [(2, 2899, 1), (1, 8195, 2), (1, 8704, 1), (1, 17408, 2), (2, 2827, 1)])
def test_large_maps_in_dealt_runs(H, L, block):
    # maps whose tiles are dealt to the CTAs in runs: of one where rows split sectors (67 MB), of one and of two where
    # they do not (303 MB), and the last below that line; in fp64 with the identity that similarity_plain is pinned to
    # (the mean of a cell is the product of the sums of unit rows), the whole map
    gen = torch.Generator(device="cuda").manual_seed(L)
    X = (torch.randn((H, L, 128), generator=gen, device="cuda") + 0.9 *
         torch.randn((H, 1, 128), generator=gen, device="cuda")).bfloat16()
    cells, mean = binding.similarity_map(X, block)
    for h in range(H):
        u = X[h].double()
        u = u / u.norm(dim=1, keepdim=True)
        T = -(-L // block)
        sums = torch.zeros((T * block, 128), dtype=torch.float64, device="cuda")
        sums[:L] = u
        sums = sums.view(T, block, 128).sum(1)
        n = torch.full((T,), float(block), dtype=torch.float64, device="cuda")
        n[-1] = L - (T - 1) * block
        ref = (sums @ sums.T) / (n[:, None] * n[None, :])
        pairs = n * (n - 1)
        ref.diagonal().copy_(torch.where(pairs > 0, ((sums * sums).sum(1) - n) / pairs.clamp(min=1), 0.0))
        assert torch.allclose(cells[h].double(), ref, rtol=RTOL, atol=ATOL)
        total = u.sum(0)
        assert abs(float(mean[h]) - float((total @ total - L) / (L * (L - 1.0)))) <= ATOL + RTOL * abs(float(mean[h]))


@pytest.mark.parametrize("H,L,block", [(2, 1500, 2), (2, 1301, 3), (1, 4096, 16), (2, 3003, 17), (1, 4000, 31), (1, 20000, 256),
                                       (1, 15001, 700), (1, 40000, 4096)])
def test_maps_keep_the_bits_of_their_sums(H, L, block):
    # Against 64 bits, tighter than what a single part of the sums, or one product of parts less, would pass: with exact
    # accumulation those leave 1.7e-5 and more.  The bound: eight steps of the largest product truncated to fp32 2^-23 each,
    # 9.5e-7, the parts and the product left out 2 x 2^-23 and 2^-22, the norms of two rows 2 x 2^-22, the sums 2^-23 each.
    gen = torch.Generator(device="cuda").manual_seed(L)
    X = (torch.randn((H, L, 128), generator=gen, device="cuda") + 1.3 *
         torch.randn((H, 1, 128), generator=gen, device="cuda")).bfloat16()
    cells, _ = binding.similarity_map(X, block)
    T = -(-L // block)
    for h in range(H):
        u = X[h].double()
        u = u / u.norm(dim=1, keepdim=True)
        sums = torch.zeros((T * block, 128), dtype=torch.float64, device="cuda")
        sums[:L] = u
        sums = sums.view(T, block, 128).sum(1)
        n = torch.full((T,), float(block), dtype=torch.float64, device="cuda")
        n[-1] = L - (T - 1) * block
        ref = (sums @ sums.T) / (n[:, None] * n[None, :])
        pairs = n * (n - 1)
        ref.diagonal().copy_(torch.where(pairs > 0, ((sums * sums).sum(1) - n) / pairs.clamp(min=1), 0.0))
        assert float((cells[h].double() - ref).norm()) <= 2e-6 * float(ref.norm())


def test_keys_and_values_of_a_c2_layer():
    wl = synth.CONFIGS["C2"]
    x = synth.make_layer(wl, 7, "calibrated")
    cells, mean = run(x["K"], 128)
    # vision keys are built around shared centroids and a shared offset: redundant, as in the paper
    assert float(mean.min()) > 0.2
    run(x["V"], 256)


@pytest.mark.parametrize("L,block", [(256, 1), (2048, 16), (32768, 256)])
def test_map_on_a_four_byte_boundary(L, block):
    # fp32 outputs need 4-byte alignment only: a map that is a slice of a larger buffer gets the same bits as an
    # aligned one, and nothing around it is written (maps of 256, 128 and 128 cells a side: rows of whole 16 bytes)
    import ctypes as C
    gen = torch.Generator(device="cuda").manual_seed(L)
    X = torch.randn((2, L, 128), generator=gen, device="cuda").bfloat16()
    ref, mean = binding.similarity_map(X, block)
    lib, need = binding.load_library(), C.c_size_t(0)
    assert lib.mixkv_similarity_workspace_size(2, L, block, C.byref(need)) == 0
    ws = torch.empty(need.value, dtype=torch.uint8, device="cuda")
    for skip in (1, 2, 3):
        buf = torch.full((ref.numel() + 8,), 7.0, device="cuda")
        m = torch.zeros(2, device="cuda")
        rc = lib.mixkv_similarity_map(X.data_ptr(), 2, L, 128, block, ws.data_ptr(), ws.numel(),
                                      buf.data_ptr() + 4 * skip, m.data_ptr(),
                                      torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        assert rc == 0 and torch.equal(buf[skip:skip + ref.numel()].view_as(ref), ref) and torch.equal(m, mean)
        assert (buf[:skip] == 7).all() and (buf[skip + ref.numel():] == 7).all()


def test_rejects_bad_arguments():
    X = torch.zeros((1, 16, 64), dtype=torch.bfloat16, device="cuda")
    with pytest.raises(binding.MixKVError):
        binding.similarity_map(X, 4)        # head_dim must be 128
