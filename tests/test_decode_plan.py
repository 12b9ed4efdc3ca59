"""How a decode step, the rows of a fold and an attention launch are cut into CTAs (host arithmetic, no GPU): splits that fill the GPU
where a few heads meet many rows, no empty split inside a single cluster, and merge scratch that holds every plan."""
import pytest

from paper_2605_09877_b200 import kvm

SMS = 148


@pytest.mark.parametrize("B,Hq,Hkv,d", [(1, 1, 1, 128), (1, 8, 1, 128), (1, 8, 1, 64), (1, 4, 2, 128), (1, 8, 8, 128), (1, 32, 8, 128),
                                        (1, 16, 16, 128), (2, 8, 8, 64), (1, 64, 8, 128), (1, 72, 9, 128)])
@pytest.mark.parametrize("rows", [50000, 131072, 1 << 22])
def test_few_heads_over_many_rows_use_most_of_the_gpu(B, Hq, Hkv, d, rows):
    heads, splits, clusters = kvm.decode_plan(B, Hq, Hkv, d, rows)
    assert B * Hq // heads * splits * clusters >= 0.7 * SMS, (heads, splits, clusters)


def test_short_states_and_many_heads_stay_in_one_cluster():
    for B, Hq, Hkv, d, rows in [(1, 1, 1, 128, 700), (1, 32, 8, 128, 800), (1, 32, 32, 128, 700), (1, 8, 8, 128, 1300), (64, 32, 32, 128, 4500),
                                (8, 32, 32, 128, 60000), (2, 8, 8, 64, 4400)]:
        assert kvm.decode_plan(B, Hq, Hkv, d, rows)[2] == 1


def test_plans_over_the_range():
    """Every split of a single cluster has rows (the last ones of several clusters may have none: they merge as nothing), a
    CTA's share of several clusters lies in one head, and all their CTAs have a place in the fixed scratch."""
    for d in (64, 128):
        for G in (1, 2, 3, 4, 6, 8, 12, 16, 32):
            for units in (1, 2, 3, 5, 8, 15, 24, 31, 48, 100, 148, 500, 2048):
                for n in list(range(1, 400, 7)) + [511, 512, 513, 1000, 1325, 2049, 4097, 6400, 10000, 50001, 131072, 1000003, 1 << 23]:
                    heads, splits, clusters = kvm.decode_plan(units, G, 1, d, n)
                    assert G % heads == 0 and heads in (1, 2, 4, 8) and 1 <= splits <= 8 and 1 <= clusters <= 64
                    rows1 = 32 * (256 // d)
                    per = -(-(-(-n // (splits * clusters))) // rows1) * rows1
                    if clusters == 1:
                        assert (splits - 1) * per < n
                    else:
                        assert heads <= 4 and splits == 8 and units * G // heads * splits * clusters <= 48 * 8
                        assert d % (heads * d // splits) == 0


def test_steps_that_fetch_ahead_cover_their_rows():
    """The warps of the cluster cover every row, in one pass or two, and a CTA takes one head, or two of the same group."""
    for d in (64, 128):
        rows1 = 256 // d
        for G in (1, 2, 3, 4, 6, 8):
            for units in (1, 2, 7, 8, 12, 16, 17, 31, 33, 53, 90, 148, 296, 300):
                for n in list(range(1, 200, 13)) + [256, 257, 500, 800, 1023, 1024, 1025, 1500, 2048, 2049, 3000, 4096, 4097]:
                    splits, heads, rpw = kvm.decode_ahead(units, G, 1, d, n)
                    if splits == 0:
                        assert (heads, rpw) == (0, 0)
                        continue
                    assert 1 <= splits <= 8 and heads == (2 if G % 2 == 0 else 1) and rpw % rows1 == 0
                    assert rpw * 8 * splits >= n and rpw <= 2 * 8 * rows1


@pytest.mark.parametrize("Hq,Hkv,d,n,splits", [
    # few rows: no more splits than hold them, also for 8 to 16 groups of heads
    (16, 16, 128, 40, 1), (12, 12, 64, 80, 1), (8, 8, 128, 128, 1), (16, 16, 128, 129, 8), (24, 4, 128, 60, 1), (24, 4, 128, 200, 2),
    (32, 8, 64, 250, 1), (32, 8, 128, 400, 8), (17, 17, 128, 400, 4),
    # clusters that would fill the GPU to the last one are the loop's
    (53, 53, 128, 630, 5), (54, 54, 128, 630, 0), (56, 56, 64, 1260, 0), (36, 36, 128, 890, 7), (37, 37, 128, 890, 0), (32, 32, 128, 1020, 8),
    (33, 33, 128, 1020, 0), (60, 30, 128, 1010, 8), (64, 32, 128, 1010, 0), (64, 32, 64, 2020, 8), (64, 16, 128, 1010, 8), (72, 36, 128, 880, 0),
    # two passes
    (32, 32, 128, 1500, 8), (33, 33, 128, 1500, 0), (40, 20, 128, 1300, 8), (40, 20, 128, 1400, 0), (40, 20, 128, 1500, 0), (40, 20, 128, 1600, 8), (48, 8, 128, 1500, 0), (64, 32, 128, 2000, 0),
    (64, 8, 128, 2000, 8), (64, 16, 64, 4000, 8), (1, 1, 128, 2048, 8), (1, 1, 128, 2049, 0)])
def test_steps_that_fetch_ahead_where_that_is_the_faster_kernel(Hq, Hkv, d, n, splits):
    assert kvm.decode_ahead(1, Hq, Hkv, d, n)[0] == splits


def test_key_splits_of_the_attention_have_keys_and_a_place_in_the_scratch():
    """37 * 8 partial results of a tile, 2 * 37 tickets, and a split has a key tile of the state or the window."""
    for heads in list(range(1, 300)) + [500, 2048]:
        for n in (1, 128, 256):
            tiles = heads * ((n + 127) // 128)
            for d in (64, 128):
                for m in (0, 64, 128, 256, 300, 512, 1000, 1152, 1280, 1500, 2048, 2304, 2560, 4096, 50000):
                    whole, splits = kvm.attention_plan(1, heads, heads, d, n, m, decides=m % 3 != 0)
                    rest = tiles - whole
                    assert 1 <= splits <= 8 and 0 <= whole <= tiles
                    if splits > 1:
                        assert 0 < rest <= 2 * 37 and rest * splits <= 37 * 8 and splits <= (m + 127) // 128 + 1
                    else:
                        assert rest == 0


@pytest.mark.parametrize("Hq,Hkv,d,C,m,splits", [
    (16, 16, 128, 256, 512, 1), (16, 16, 128, 256, 1152, 2), (16, 4, 128, 256, 4096, 3), (19, 19, 128, 256, 1280, 2), (24, 6, 128, 256, 1280, 2),
    # folds as wide beside them: two splits only take SMs from those, up to more rows
    (20, 20, 128, 256, 1536, 1), (20, 20, 128, 256, 1792, 2), (24, 24, 128, 256, 1792, 1), (24, 24, 128, 192, 2048, 2), (27, 27, 128, 192, 2560, 1),
    (48, 48, 128, 64, 1536, 1), (54, 54, 128, 128, 2688, 1), (54, 54, 128, 128, 2816, 2), (24, 24, 64, 256, 1408, 1), (24, 24, 64, 256, 1536, 2),
    (54, 54, 64, 128, 1792, 1), (54, 54, 64, 64, 2048, 2), (40, 40, 64, 128, 1280, 2), (48, 24, 128, 128, 1536, 2)])
def test_key_splits_beside_folds(Hq, Hkv, d, C, m, splits):
    assert kvm.attention_plan(1, Hq, Hkv, d, C, m) == (0 if splits > 1 else Hq * ((C + 127) // 128), splits)
    assert kvm.attention_plan(1, Hq, Hkv, d, C, m, decides=False)[1] == (2 if m >= 1152 and splits == 1 else splits)


def test_states_without_stored_keys_take_four_rows_per_warp():
    """Only that kernel recomputes the keys, and its CTAs cover the rows of a block."""
    for units in (1, 16, 31, 32, 63, 64, 100, 148, 149, 200, 255, 256, 257, 2048):
        for d in (64, 128):
            for C in (8, 64, 128, 136, 256):
                for serial in (False, True):
                    per_warp, ctas = kvm.apply_plan(units, d, C, serial)
                    assert per_warp in (1, 4) and 1 <= ctas <= (C + 7) // 8
                    assert per_warp == 4 or ctas == (C + 7) // 8
                    if (serial or units >= 256) and C * units >= 8192:
                        assert per_warp == 4


@pytest.mark.parametrize("units,d,C,serial,rows", [
    (72, 128, 256, False, 1), (96, 128, 256, False, 1), (127, 128, 136, False, 1), (148, 128, 256, False, 1), (255, 128, 256, False, 1), (32, 128, 256, True, 4),
    (256, 128, 32, False, 4), (256, 128, 24, False, 1), (31, 64, 256, False, 1), (32, 64, 256, False, 4), (37, 64, 256, False, 4), (38, 64, 256, False, 1),
    (48, 64, 256, False, 1), (49, 64, 256, False, 4), (56, 64, 160, False, 4), (60, 64, 136, False, 1), (67, 64, 136, False, 1), (68, 64, 136, False, 4),
    (47, 64, 128, False, 1), (48, 64, 128, False, 4), (96, 64, 64, False, 4), (95, 64, 64, False, 1)])
def test_rows_per_warp_of_the_apply_kernel(units, d, C, serial, rows):
    assert kvm.apply_plan(units, d, C, serial)[0] == rows


@pytest.mark.parametrize("units,d,C,group,rows", [(34, 64, 256, 1, 4), (34, 64, 256, 2, 1), (37, 64, 256, 8, 1), (48, 64, 256, 8, 1), (49, 64, 256, 8, 4), (68, 64, 136, 8, 4), (48, 64, 128, 2, 4)])
def test_rows_per_warp_beside_the_attention_of_several_heads(units, d, C, group, rows):
    assert kvm.apply_plan(units, d, C, group=group)[0] == rows


def test_plan_refuses_what_a_state_refuses():
    for bad in [(0, 1, 1, 64, 10), (1, 3, 2, 64, 10), (1, 2, 2, 96, 10), (1, 2, 2, 64, 0)]:
        with pytest.raises(kvm.KVMError):
            kvm.decode_plan(*bad)


def test_the_other_plans_refuse_what_a_state_refuses():
    for bad in [(0, 1, 1, 64, 10), (1, 3, 2, 64, 10), (1, 2, 2, 96, 10), (1, 2, 2, 64, 0)]:
        with pytest.raises(kvm.KVMError):
            kvm.decode_ahead(*bad)
    for bad in [(0, 64, 64), (1, 96, 64), (1, 64, 60), (1, 64, 264)]:
        with pytest.raises(kvm.KVMError):
            kvm.apply_plan(*bad)
    for bad in [(0, 1, 1, 64, 1, 1), (1, 3, 2, 64, 1, 1), (1, 1, 1, 96, 1, 1), (1, 1, 1, 64, 0, 1), (1, 1, 1, 64, 257, 1), (1, 1, 1, 64, 1, -1)]:
        with pytest.raises(kvm.KVMError):
            kvm.attention_plan(*bad)
