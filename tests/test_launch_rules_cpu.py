"""The rules that split a call's work over clusters of CTAs (csrc/internal_api.h), without a device: whatever number
of clusters a device holds at once, no rule asks for more, which would cost a second wave."""
import ctypes as C
import os
import re

import pytest

from paper_2510_20707_b200 import binding, build

# resident clusters of 1 .. 8 CTAs with one CTA per SM and with three: a B200 with 148 SMs, then chips whose SMs fall
# into other groups, and one with fewer of them
B200 = (148, (148, 74, 45, 33, 26, 22, 15, 15), (444, 222, 142, 104, 82, 71, 56, 48))
CHIPS = [B200, (148, (148, 70, 40, 28, 22, 18, 12, 11), (444, 210, 130, 90, 70, 60, 45, 40)),
         (132, (132, 66, 40, 30, 22, 20, 15, 14), (396, 198, 126, 93, 72, 62, 50, 42)),
         (64, (64, 32, 20, 16, 10, 8, 8, 4), (192, 96, 60, 48, 34, 28, 24, 16))]


@pytest.fixture(scope="module")
def lib():
    build.build()
    return binding.load_library()


def array(limits):
    return (C.c_int32 * 9)(0, *limits)


def decode(lib, chip, units, rows, even=1):
    sms, alone, shared = chip
    ctas, depth = C.c_int32(), C.c_int32()
    lib.mixkv_internal_decode_shape(C.c_int64(units), rows, even, sms, array(shared), array(alone), C.byref(ctas),
                                    C.byref(depth))
    return ctas.value, depth.value


@pytest.mark.parametrize("chip", CHIPS)
def test_no_more_clusters_than_are_resident(lib, chip):
    sms, alone, shared = chip
    for units in list(range(1, 700)) + [896, 1184, 5000]:
        for rows in (1, 17, 300, 512, 1500, 3500, 20000):
            for even in (0, 1):
                S, depth = decode(lib, chip, units, rows, even)
                assert 1 <= S <= 8 and depth in (1, 2, 3, 4)
                halves = S == 2 and 1.1 <= units / (3 * sms) <= 1.5      # evens out a second wave on purpose
                assert S == 1 or halves or units <= (alone if depth == 4 else shared)[S - 1], (units, rows, S, depth)
        for P in (100, 4097, 9000, 33000, 140000):
            cs = lib.mixkv_internal_tail_clusters(C.c_int64(units), P, sms, array(alone))
            assert cs in (1, 2, 4, 8) and (cs == 1 or units <= alone[cs - 1]), (units, P, cs)
            cs = lib.mixkv_internal_budget_clusters(units, C.c_int64(8 * P), array(alone))
            assert cs in (1, 2, 4, 8) and (cs == 1 or units <= alone[cs - 1]), (units, P, cs)


@pytest.mark.parametrize("units,rows,even,want", [
    (4, 512, 1, (8, 2)), (15, 1500, 1, (8, 4)), (16, 1500, 1, (8, 2)), (16, 8000, 1, (6, 4)), (17, 1500, 1, (6, 4)),
    (28, 2500, 0, (8, 2)), (49, 1500, 1, (7, 2)), (896, 512, 0, (1, 2)), (256, 1264, 1, (1, 3)), (256, 1265, 1, (1, 1)), (256, 3400, 0, (1, 3)),
    (236, 3400, 1, (1, 3)), (237, 3400, 1, (1, 1)), (296, 8000, 1, (1, 1)), (297, 3400, 1, (1, 2)), (560, 2500, 0, (2, 2)), (12, 60, 1, (1, 2))])
def test_decode_shapes_as_measured(lib, units, rows, even, want):
    assert decode(lib, B200, units, rows, even) == want


def test_tail_and_budget_clusters_as_measured(lib):
    sms, alone, _ = B200
    tail = lambda units, P: lib.mixkv_internal_tail_clusters(C.c_int64(units), P, sms, array(alone))
    assert [tail(14, 30000), tail(15, 30000), tail(29, 12000), tail(30, 12000), tail(73, 9000), tail(74, 9000),
            tail(4, 4096)] == [8, 4, 4, 2, 2, 1, 1]
    budget = lambda pairs, keys: lib.mixkv_internal_budget_clusters(pairs, C.c_int64(keys), array(alone))
    assert [budget(1, 8192), budget(15, 60000), budget(16, 60000), budget(33, 60000), budget(34, 60000),
            budget(74, 60000), budget(75, 60000), budget(74, 8193)] == [1, 8, 4, 4, 2, 2, 1, 2]


def test_adaptive_budgets_in_the_tail_as_measured(lib):
    sms, alone, _ = B200
    paired = tuple(2 * n for n in alone)
    threads = lambda sequences, heads, P, alone=alone, paired=paired: lib.mixkv_internal_adapt_threads(
        C.c_int64(sequences), heads, P, array(alone), array(paired))
    assert [threads(15, 8, 700), threads(16, 8, 700), threads(16, 8, 8192), threads(16, 8, 8193), threads(30, 8, 8193),
            threads(31, 8, 8193)] == [1024, 0, 0, 512, 512, 0]
    assert [threads(33, 4, 9000), threads(34, 4, 9000), threads(66, 4, 700), threads(67, 4, 700)] == [1024, 512, 512, 0]
    # from some 17600 keys on two CTAs do not share an SM any more
    assert [threads(34, 4, 17000), threads(34, 4, 18000), threads(16, 8, 18000)] == [512, 1024, 1024]
    # a device, or a part of one, that holds no such cluster
    none = (148, 74) + (0,) * 6
    assert [threads(1, 2, 700, none, none), threads(1, 4, 700, none, none), threads(1, 4, 20000, none, none)] == [1024, 0, 0]


def test_maps_are_dealt_out_by_what_l2_holds(lib):
    run = lambda heads, T, parts, whole, l2=132644864: lib.mixkv_internal_gram_run(heads, T, parts, whole, C.c_int64(l2))
    assert [run(4, 2035, 2, 0), run(4, 2036, 2, 0), run(4, 2036, 3, 0)] == [0, 1, 1]
    assert [run(4, 4312, 2, 1), run(4, 4320, 2, 1), run(4, 4320, 3, 1), run(4, 2048, 3, 1)] == [0, 1, 2, 0]
    # half the cache: the same at half the size; a map past 32 bits of bytes
    assert [run(2, 2036, 2, 0, 132644864 // 2), run(2, 4320, 3, 1, 132644864 // 2), run(8, 65535, 2, 0)] == [1, 2, 1]


@pytest.mark.parametrize("sms", [148, 7])
@pytest.mark.parametrize("heads,per_head", [(1, 1), (1, 300), (4, 8), (4, 47), (4, 256), (8, 24), (8, 235), (37, 5), (74, 3),
                                            (148, 2), (149, 2), (112, 32), (5, 148), (64, 1)])
def test_every_tile_has_one_cta(lib, heads, per_head, sms):
    tiles = heads * per_head
    first, owner = (C.c_int32 * (sms + 1))(), (C.c_int32 * tiles)()
    for uniform in (per_head, 0):
        g = lib.mixkv_internal_split_tiles(tiles, uniform, sms, first, owner)
        assert 1 <= g <= min(tiles, sms) and first[0] == 0 and first[g] == tiles
        shares = [first[c + 1] - first[c] for c in range(g)]
        assert min(shares) >= 1 and sum(shares) == tiles
        assert list(owner) == [c for c in range(g) for _ in range(shares[c])]
        even = -(-tiles // min(tiles, sms))
        apart = all(first[c] // per_head == (first[c + 1] - 1) // per_head for c in range(g))   # no CTA on two heads
        assert max(shares) <= even + (1 if uniform and apart else 0)
        if uniform and heads <= sms and -(-per_head // min(per_head, sms // heads)) <= even + 1:
            assert apart


def pass2_segments(lib, lens, heads, layers, window, sms=148):
    """Tiles of the segments of every CTA of pass 2, in the order in which it takes them (the last one first)."""
    per_head = [-(-(n - window) // 128) for n in lens]
    runs = [t for _ in range(layers) for t in per_head for _ in range(heads)]
    tiles, uniform = sum(runs), per_head[0] if len(set(per_head)) == 1 else 0
    first, owner = (C.c_int32 * (sms + 1))(), (C.c_int32 * tiles)()
    g = lib.mixkv_internal_split_tiles(tiles, uniform, sms, first, owner)
    of_cta, t = [[] for _ in range(g)], 0
    for n in runs:
        for c in sorted(set(owner[t:t + n])):
            of_cta[c].append(sum(o == c for o in owner[t:t + n]))
        t += n
    return [segs[::-1] for segs in of_cta]


@pytest.mark.parametrize("lens,heads,layers,window", [
    ((4096,), 4, 28, 32), ((3001, 1777, 6143), 4, 28, 32), ((2100, 130, 1900, 160, 97), 4, 12, 32), ((130, 1030), 8, 12, 16)])
def test_segments_of_one_tile_have_statistics_of_their_own(lib, lens, heads, layers, window):
    # A segment of one tile is one pair's of the epilogue.  The other pair comes to its statistics with nothing in between
    # that waits for its first warp, which may still be reading those of the segment before; only the barrier of the
    # segment in between orders that read ahead of the writes of the one after.  So neighbours never share words.
    segments = pass2_segments(lib, lens, heads, layers, window)
    assert any(1 in of_cta[1:] for of_cta in segments)
    for s in range(max(len(of_cta) for of_cta in segments)):
        tables = {(k, wg): lib.mixkv_internal_stats_table(k, wg) for k in (s, s + 1) for wg in (0, 1)}
        assert sorted(tables.values()) == [0, 1, 2, 3]


def pass2_spare(lib, lens, heads, layers, window, sms=148):
    """Whether pass 2 folds normalisers in its spare warp, and whether any of its CTAs has a second head."""
    tiles = [[-(-(n - w) // 128) for n in lens] for w in (0, window)]
    total = [layers * heads * sum(t) for t in tiles]
    uniform = [t[0] if len(set(t)) == 1 else 0 for t in tiles]
    spare = lib.mixkv_internal_pass2_spare(total[0], uniform[0], total[1], uniform[1], layers * heads * len(lens),
                                           max(tiles[0]), sms)
    return bool(spare), any(len(of_cta) > 1 for of_cta in pass2_segments(lib, lens, heads, layers, window, sms))


@pytest.mark.parametrize("lens,heads,layers,window,spare", [
    ((500,), 4, 1, 32, 0), ((500,), 8, 1, 32, 0), ((1024,), 4, 10, 32, 0), ((900,), 4, 28, 32, 0), ((2000,) * 5, 8, 1, 32, 0),
    ((768,), 4, 25, 32, 0), ((97, 130, 160), 4, 8, 32, 0), ((16384,), 1, 1, 32, 0), ((700,), 1, 1, 32, 0),   # no second head
    ((4096,), 4, 28, 32, 1), ((3001, 1777, 6143), 4, 28, 32, 1), ((700, 650, 800, 900), 4, 28, 32, 1), ((130, 1030), 8, 12, 16, 1),
    ((32768, 20000, 9000), 4, 1, 32, 0)])                       # second heads, but in too many segments for one warp
def test_the_spare_warp_folds_for_second_heads_only(lib, lens, heads, layers, window, spare):
    got, second = pass2_spare(lib, lens, heads, layers, window)
    assert got == bool(spare) and (second or not got)


@pytest.mark.parametrize("sms", [148, 132, 16])
def test_the_spare_warp_folds_for_some_cta(lib, sms):
    for heads in (1, 2, 4, 8):
        for layers in (1, 2, 5, 14, 28):
            for lens in ((33,), (161,), (500,), (1024,), (4096,), (300, 300), (300, 301, 40), (2000, 130, 97, 1500), (900,) * 6):
                got, second = pass2_spare(lib, lens, heads, layers, 32, sms)
                assert second or not got, (sms, heads, layers, lens)


def test_nobody_arrives_twice_ahead_of_a_reader():
    # Bounded waits end at once after an abort, named barriers do not.  A role that arrives at one without waiting could come
    # to it again ahead of the reader's first time; two such arrivals complete it, and the reader waits at its last one for
    # good.  So there are none but in pairs: the reader of the one arrives at the other, at which the writer waits first.
    source = open(os.path.join(os.path.dirname(build.__file__), "csrc", "pass_tc.cu")).read()
    calls = re.findall(r"named_bar_(arrive|sync)\(([^,]+),", source)
    assert [bar for kind, bar in calls if kind == "arrive"] == ["6 + blk", "8 + blk"]
    assert [(kind, bar) for kind, bar in calls if "blk" in bar] == [   # the writer's, then the reader's
        ("sync", "8 + blk"), ("arrive", "6 + blk"), ("sync", "6 + blk"), ("arrive", "8 + blk")]


NAN = 0xffffffff   # key of the NaN that arithmetic on the device gives


@pytest.mark.parametrize("lo", [1, 0x400001ff, 0x42f00dad, 0x7fffffff, 0x80000000, 0xbe123456, 0xbf800001, 0xff800000, NAN])
@pytest.mark.parametrize("hi", [0x42f00dad, 0xbf800001, 0xbf900000, 0xff800000, 0xffc00000, NAN])
def test_a_search_counts_nothing_but_keys_there_are(lib, lo, hi):
    # Whatever the smallest and the largest key, NaNs among them: 2048 bins, the key looked for in every round's range, and
    # no range past the largest key or, over 2^32, at the keys below all others, where the budget kernel's padding is.
    if lo > hi:
        return
    base, span, shift = (C.c_uint32 * 3)(), (C.c_uint32 * 3)(), (C.c_int32 * 3)()
    for key in sorted({lo, hi, max(lo, hi - 1), (lo + hi) // 2, lo + (hi - lo) // 2048 * 2047}):
        n = lib.mixkv_internal_search_rounds(C.c_uint32(lo), C.c_uint32(hi), C.c_uint32(key), base, span, shift)
        assert 1 <= n <= 3 and shift[n - 1] == 0
        for r in range(n):
            assert lo <= base[r] <= key <= base[r] + span[r] <= hi, (r, hex(key), hex(base[r]), hex(span[r]))
            assert span[r] >> shift[r] < 2048
