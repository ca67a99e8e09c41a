"""Where stage 2b sets its bits, and when stage 3 runs its first cut, starts its bounds from near tokens, keeps visits as lists and selects few from many: host arithmetic on the sizes, no
device."""
import os
import subprocess

import pytest


@pytest.fixture(scope="module")
def routes(tmp_path_factory):
    from paper_2608_23553_b200 import build
    build.build()
    native = os.path.join(os.path.dirname(os.path.abspath(__file__)), "native")
    tmp = tmp_path_factory.mktemp("rule")
    obj, exe = str(tmp / "stage3_rules.o"), str(tmp / "stage3_rules")
    subprocess.check_call([build.NVCC] + build.FLAGS + ["-c", os.path.join(native, "stage3_rules.cu"), "-o", obj])
    objs = [os.path.join(build.OBJ, n) for n in ("g2_gather.o", "g3_filter.o", "g3_batch_scan.o", "g3_centroid_interaction.o",
                                                  "g3_partial.o")]
    subprocess.check_call(["g++", "-no-pie", "-o", exe, obj, os.path.join(native, "fake_cudart.cpp")] + objs +
                          ["-Wl,--unresolved-symbols=ignore-all"])

    def routes(K, N, length, B, nq, P, n_prune, distinct=None, max_len=None, max_candidates=0, longest=0):
        line = "%d %d %d %d %d %d %d %d %d %d %d" % (K, N, N * length, N * (distinct or length), max_len or 2 * length, B, nq,
                                                     P, n_prune, max_candidates, longest or 2 * N * length // K)
        out = subprocess.run([exe], input=line, capture_output=True, text=True, check=True).stdout.split()
        return [x == "1" for x in out[:4]] + [("L2", "shared", "ranges")[int(out[4])], int(out[5])]
    return routes


@pytest.fixture(scope="module")
def rule(routes):
    return lambda *a, **kw: routes(*a, **kw)[0]


@pytest.fixture(scope="module")
def lists(routes):
    return lambda *a, **kw: routes(*a, **kw)[1]


@pytest.fixture(scope="module")
def near_first(routes):
    return lambda *a, **kw: routes(*a, **kw)[2]


@pytest.fixture(scope="module")
def few(routes):
    return lambda *a, **kw: routes(*a, **kw)[3]


@pytest.fixture(scope="module")
def gather(routes):
    return lambda *a, **kw: routes(*a, **kw)[4]


@pytest.mark.parametrize("K,N,length,B,nq,P,n_prune", [(262_144, 1_279_581, 128, 19, 40, 2, 1_235), (51_588, 357_950, 114, 31, 120, 2, 251),
                                                        (107_614, 1_572_938, 30, 14, 32, 22, 1_315), (65_536, 500_000, 120, 40, 32, 4, 1_024)])
def test_tables_of_the_queries_looked_up_at_once_stay_in_l2(routes, K, N, length, B, nq, P, n_prune):
    rows = 32 if nq <= 32 else 64 if nq <= 64 else 128
    blocks = routes(K, N, length, B, nq, P, n_prune)[5]
    assert 4 * 148 / blocks * K * rows <= 1.1 * (16 << 20) or blocks >= 4 * 148       # four blocks per SM


def test_bits_are_set_in_shared_memory_where_words_are_set_often(gather):
    # 10,000 documents of 40 tokens, 313 words: 12 times each are 3,756 entries
    assert [gather(1_000, 10_000, 40, B, 1, 10, 100) for B in (1, 37, 38, 74, 200)] == ["shared"] * 2 + ["ranges"] * 3
    assert [gather(1_000, 10_000, 40, 4, 1, P, 100) for P in (9, 10)] == ["L2", "shared"]
    # 65,536 entries a query: sixteen blocks up to half the SMs
    assert [gather(1_000, 10_000, 40, B, 32, 6, 100) for B in (37, 38, 74, 75, 148)] == ["shared"] * 3 + ["ranges"] * 2
    # bitmaps of 96 KB, and of nine ranges
    assert gather(1_000, 24 * 1024 * 32, 100, 1, 32, 8, 100) == "shared" and gather(1_000, 24 * 1024 * 32 + 1, 100, 1, 32, 8, 100) == "L2"
    assert gather(65_536, 14_417_920, 40, 256, 32, 4, 100) == "ranges" and gather(65_536, 14_417_921, 40, 256, 32, 4, 100) == "L2"


def test_what_the_candidates_hold_counts_and_not_the_room_for_them(rule):
    # one query, one probe per token, 8.8 million documents of 68 tokens: 73,000 candidates, whatever the capacity
    assert not rule(262_144, 8_800_000, 68, 1, 32, 1, 1_024)
    assert not rule(262_144, 8_800_000, 68, 1, 32, 1, 1_024, max_candidates=80_000)
    assert not rule(262_144, 4_000_000, 69, 64, 32, 1, 1_024)
    # half a million documents: one query not, two and more
    assert [rule(65_536, 500_000, 120, B, 32, 4, 1_024) for B in (1, 2, 8, 256)] == [False, True, True, True]
    assert rule(262_144, 8_800_000, 68, 256, 32, 4, 4_096)
    # a capacity below the expected candidates is what is scanned
    assert rule(65_536, 500_000, 120, 4, 32, 4, 1_024) and not rule(65_536, 500_000, 120, 4, 32, 4, 1_024, max_candidates=20_000)
    # documents of few distinct centroids are found by fewer probes
    assert not rule(65_536, 500_000, 120, 2, 32, 4, 1_024, distinct=30)
    # 10,000 documents: one query not, a batch
    assert not rule(1_024, 10_000, 64, 1, 32, 4, 256) and rule(1_024, 10_000, 64, 64, 32, 4, 256)


def test_other_query_lengths_and_what_the_cut_cannot_hold(rule):
    assert rule(16_411, 123_457, 80, 1, 21, 6, 777) and not rule(16_411, 123_457, 80, 1, 21, 1, 777)
    assert rule(32_768, 200_000, 100, 1, 100, 4, 1_024)
    # nothing to cut: most candidates survive the pruning anyway
    assert not rule(6_000, 24_000, 35, 256, 32, 1, 5_900)
    # the numbers of 266,240 centroids still fit a block, documents of 32,000 tokens a sum
    args = (8_800_000, 68, 256, 32, 4, 4_096)
    assert rule(266_240, *args) and not rule(266_241, *args)
    assert rule(262_144, *args, max_len=32_000) and not rule(262_144, *args, max_len=32_001)
    # token positions of 31 bits
    assert not rule(262_144, 8_800_000, 245, 256, 32, 4, 4_096)


def test_visits_are_kept_as_lists_while_candidates_have_few(lists):
    mid = (65_536, 500_000, 120, 256, 32)
    assert lists(*mid, 4, 1_024) and lists(*mid, 16, 1_024) and not lists(*mid, 32, 1_024)
    assert not lists(65_536, 500_000, 120, 16, 32, 4, 1_024)              # few queries
    # documents that repeat their centroids: as few visits, but of fewer candidates
    assert lists(*mid, 4, 1_024, distinct=40) and not lists(*mid, 4, 1_024, distinct=12)
    assert not lists(*mid, 4, 1_024, longest=60_000)                     # as large as the table
    # a third of the table, 8 bytes a node and a head: 24 (128 x 1,000 + m) <= 128 m, and 24 (32 x 500 + m) <= 32 m
    assert [lists(*mid, 4, 1_024, longest=1_000, max_candidates=m) for m in (29_538, 29_539)] == [False, True]
    assert [lists(*mid[:4], 8, 4, 1_024, longest=500, max_candidates=m) for m in (47_999, 48_000)] == [False, True]


def test_bounds_start_with_near_tokens_where_that_decides(near_first):
    mid = (65_536, 500_000, 120)
    assert near_first(*mid, 64, 32, 4, 1_024) and near_first(*mid, 64, 40, 4, 1_024) and near_first(*mid, 64, 64, 4, 1_024)
    assert not near_first(*mid, 64, 32, 4, 1_023)                        # few documents
    # short queries: every length below 32, in a batch scanned together and by query
    assert not any(near_first(*mid, B, nq, 8, 2_048) for nq in (8, 16, 21, 28, 31) for B in (64, 256))
    # documents too short for the query (1.6 x 50 = 80 tokens of weight: 0.4)
    assert not near_first(65_536, 500_000, 50, 64, 32, 8, 2_048) and near_first(65_536, 500_000, 51, 64, 32, 8, 2_048)
    # 6-bit codes from the exact table, a query at a time
    assert not near_first(262_144, 8_800_000, 68, 256, 40, 4, 4_096) and near_first(262_144, 8_800_000, 68, 256, 32, 4, 4_096)


def test_few_are_selected_from_many_where_the_lists_are_long_and_the_wanted_few(few):
    mid = (65_536, 500_000, 120, 256, 32)
    assert few(*mid, 4, 1_024) and few(*mid, 4, 4_096) and few(262_144, 8_800_000, 68, 256, 32, 4, 4_096)
    # short lists, whatever is wanted: 8,184 documents, or 16,384 candidates to be expected of many more
    assert not few(275, 8_184, 30, 140, 32, 7, 133) and not few(275, 16_383, 30, 140, 32, 7, 133) and few(275, 16_384, 30, 140, 32, 7, 133)
    assert [few(65_536, n, 120, 64, 32, 4, 100) for n in (78_000, 79_000)] == [False, True]
    # more than a list of 16,384 has room for, and longer lists with more wanted than that
    assert not few(81_311, 1_240_245, 65, 6, 64, 17, 9_439)
    assert [few(64, 100_000, 4, 64, 8, 16, w) for w in (4_800, 5_800)] == [True, False]
    assert [few(64, n, 4, 64, 8, 16, 1_024) for n in (5_500_000, 5_900_000)] == [True, False]
    # a capacity below the smallest list
    assert not few(*mid, 4, 1_024, max_candidates=16_383) and few(*mid, 4, 1_024, max_candidates=16_384)
