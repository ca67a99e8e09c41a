"""What token lists add to the workspace of a search: host arithmetic on the sizes, no device."""
import os
import subprocess

import pytest


@pytest.fixture(scope="module")
def sizes(tmp_path_factory):
    from paper_2608_23553_b200 import build
    build.build()
    native = os.path.join(os.path.dirname(os.path.abspath(__file__)), "native")
    tmp = tmp_path_factory.mktemp("sizes")
    obj, exe = str(tmp / "workspace_sizes.o"), str(tmp / "workspace_sizes")
    subprocess.check_call([build.NVCC] + build.FLAGS + ["-c", os.path.join(native, "workspace_sizes.cu"), "-o", obj])
    names = ("api", "g1_score_table", "g2_gather", "g2_probe", "g3_batch_scan", "g3_centroid_interaction", "g3_filter", "g3_partial", "g7_graph")
    objs = [os.path.join(build.OBJ, n + ".o") for n in names]
    subprocess.check_call(["g++", "-no-pie", "-o", exe, obj, os.path.join(native, "fake_cudart.cpp")] + objs + ["-Wl,--unresolved-symbols=ignore-all"])

    def sizes(K, N, length, B, nq, P, n_prune, max_candidates=0):
        line = "%d %d %d %d %d %d %d %d %d" % (K, N, N * length, B, nq, P, n_prune, max_candidates, 2 * N * length // K)
        return [int(x) for x in subprocess.run([exe], input=line, capture_output=True, text=True, check=True).stdout.split()]
    return sizes


@pytest.mark.parametrize("call", [
    (65_536, 500_000, 120, 256, 32, 4, 1_024),               # visit lists
    (65_536, 500_000, 120, 256, 32, 4, 1_024, 160_000),
    (65_536, 500_000, 120, 1, 32, 4, 1_024),                 # a table of maxima
    (1_024, 10_000, 64, 16, 21, 4, 256),                     # ... of a call without any cut
    (262_144, 8_800_000, 68, 64, 32, 4, 4_096, 500_000),
])
def test_scores_of_retrieved_tokens_share_their_place(sizes, call):
    """No call prunes both ways, so the larger of the two scratch areas is what a workspace has to hold."""
    without, with_lists, scores, ranks = sizes(*call)
    maxc = call[7] if len(call) > 7 else call[1]
    bounds = 4 * call[3] * maxc                              # lower, upper bounds and contenders, ranges of candidates or contenders
    shared = 7 * bounds if call[4] in (32, 64) else 0
    assert with_lists - without <= max(scores - shared, 0) + ranks + 1_024
