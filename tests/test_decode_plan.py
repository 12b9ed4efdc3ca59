"""How a decode step is cut into CTAs (host arithmetic, no GPU): splits that fill the GPU where a few heads meet many rows,
no empty split inside a single cluster, and merge scratch that holds every plan."""
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


def test_plan_refuses_what_a_state_refuses():
    for bad in [(0, 1, 1, 64, 10), (1, 3, 2, 64, 10), (1, 2, 2, 96, 10), (1, 2, 2, 64, 0)]:
        with pytest.raises(kvm.KVMError):
            kvm.decode_plan(*bad)
