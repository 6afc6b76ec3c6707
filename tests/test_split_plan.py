"""How the linear layer decides to split a reduction over a cluster, on the host: no more clusters than run at a time, none where
none fits."""
import random

import paper_2206_15014_b200 as nm

B200 = (74, 33, 14)
FORMATS = [(2, 4, 8), (4, 4, 8), (2, 4, 4), (1, 4, 8), (4, 8, 4), (1, 8, 8), (4, 4, 4)]


def _shapes():
    rng = random.Random(3)
    for _ in range(400):
        yield (rng.choice((1, 7, 64, 128, 384, 700, 1500)), rng.randint(1, 3000), 128 * rng.randint(1, 64)) + rng.choice(FORMATS)


def test_small_problems_are_split():
    assert nm.nm_split_plan(1, 1024, 8192, 2, 4, 8, B200) // 1000 == 8
    assert nm.nm_split_plan(384, 1024, 4096, 2, 4, 8, B200) == 4096
    assert nm.nm_split_plan(384, 3072, 1024, 2, 4, 8, B200) == 0
    assert nm.nm_split_plan(16384, 1024, 4096, 2, 4, 8, B200) == 0


def test_nothing_is_split_where_no_cluster_fits():
    assert all(nm.nm_split_plan(*s, (0, 0, 0)) == 0 for s in _shapes())


def test_a_cluster_size_that_does_not_fit_is_not_taken():
    taken = [nm.nm_split_plan(*s, (74, 33, 0)) for s in _shapes()]
    assert {p // 1000 for p in taken} == {0, 2, 4}


def test_no_second_round_of_clusters():
    seen = 0
    for tokens, out, k, n, m, bits in _shapes():
        for fits in (B200, (10, 5, 2), (1, 1, 1)):
            plan = nm.nm_split_plan(tokens, out, k, n, m, bits, fits)
            if plan:
                splits, width = divmod(plan, 1000)
                clusters = -(-out // 128) * -(-tokens // width)
                assert clusters <= fits[(2, 4, 8).index(splits)] and clusters * splits <= 148 and k // 128 >= splits
                seen += 1
    assert seen > 100


def test_refusals():
    for bad in ((-1, 128, 128, 2, 4, 8), (4, 128, 100, 2, 4, 8), (4, 128, 128, 3, 4, 8), (4, 128, 16384, 2, 4, 8)):
        try:
            nm.nm_split_plan(*bad, B200)
        except nm.NmError as e:
            assert e.code == nm.nm_int_linear_check(*bad)
        else:
            raise AssertionError(bad)
    assert nm.nm_split_plan(0, 128, 1024, 2, 4, 8, B200) == 0
