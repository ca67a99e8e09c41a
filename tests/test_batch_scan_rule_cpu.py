"""When the first cut scans a batch at a time: host arithmetic on the sizes, no device."""
import os
import subprocess

import pytest

from test_gpu_batch_scan import CALLS, CROWDED, tokens_and_entries
from test_gpu_filter import CALLS as CUT_CALLS, REPEATED


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    from paper_2608_23553_b200 import build
    build.build()
    native = os.path.join(os.path.dirname(os.path.abspath(__file__)), "native")
    tmp = tmp_path_factory.mktemp("rule")
    obj, exe = str(tmp / "batch_rules.o"), str(tmp / "batch_rules")
    subprocess.check_call([build.NVCC] + build.FLAGS + ["-c", os.path.join(native, "batch_rules.cu"), "-o", obj])
    objs = [os.path.join(build.OBJ, n) for n in ("g3_batch_scan.o", "g3_filter.o", "g3_centroid_interaction.o", "g3_partial.o")]
    subprocess.check_call(["g++", "-no-pie", "-o", exe, obj, os.path.join(native, "fake_cudart.cpp")] + objs +
                          ["-Wl,--unresolved-symbols=ignore-all"])

    def rule(K, N, T, entries, max_len, B, nq, P, n_prune):
        line = "%d %d %d %d %d %d %d %d %d" % (K, N, T, entries, max_len, B, nq, P, n_prune)
        return subprocess.run([exe], input=line, capture_output=True, text=True, check=True).stdout.strip() == "1"
    return rule


@pytest.mark.parametrize("call", CALLS)
def test_the_calls_of_the_gpu_test_take_it(rule, call):
    D, nq, K, N, lo, hi, B, nprobe, n_prune = call
    T, entries, longest = tokens_and_entries(*call)
    assert rule(K, N, T, entries, longest, B, nq, nprobe, n_prune)


@pytest.mark.parametrize("nq", [20, 32, 64])
def test_so_does_the_call_with_too_many_listed_centroids(rule, nq):
    D, K, N, lo, hi, B, nprobe, n_prune = CROWDED
    assert rule(K, N, 100 * N, 99 * N, hi, B, nq, nprobe, n_prune)


@pytest.mark.parametrize("together,nq,K,N,B,nprobe", REPEATED)
def test_the_calls_that_turn_out_not_to_cut_are_of_both_forms(rule, together, nq, K, N, B, nprobe):
    assert rule(K, N, 40 * N, int(9.8 * N), 50, B, nq, nprobe, 100) == bool(together)


def test_two_calls_of_the_cut_go_by_query(rule):
    forms = []
    for cut, _, _, nq, K, N, lo, hi, B, nprobe, n_prune, _, _ in CUT_CALLS:
        length = (lo + hi) / 2
        forms.append(rule(K, N, N * length, N * K * (1 - (1 - 1 / K) ** length), hi, B, nq, nprobe, n_prune))
    assert forms == 10 * [True] + 2 * [False] + 4 * [False]


def test_other_lengths_have_to_save_what_their_steps_cost(rule):
    # documents of 40 tokens that are all candidates: 8 queries save 0.91 token cycles for each token, 3 million in all
    assert [rule(700, n, 40 * n, 39 * n, 60, 8, 21, 8, 100) for n in (81_000, 84_000)] == [False, True]
    assert [rule(700, 80_000, 3_200_000, 3_120_000, 60, 8, nq, 8, 100) for nq in (21, 32, 47, 64)] == [False, True, False, True]


def test_where_it_stops(rule):
    mid = (65_536, 500_000, 60_000_000, 59_945_000, 200)
    assert rule(*mid, 256, 32, 4, 1_024) and not rule(*mid, 16, 32, 4, 1_024)      # 20 % of the documents: a large batch
    assert rule(*mid, 16, 32, 32, 16_384) and not rule(*mid, 4, 32, 32, 16_384)    # 87 %: a small one
    large = (262_144, 8_800_000, 598_000_000, 597_900_000, 180)
    assert not rule(*large, 256, 32, 4, 4_096) and not rule(*large, 256, 32, 32, 16_384)   # 64 MB of codes
    assert rule(*mid[:4], 1_040, 256, 32, 4, 1_024) and not rule(*mid[:4], 1_041, 256, 32, 4, 1_024)   # 16-bit sums
