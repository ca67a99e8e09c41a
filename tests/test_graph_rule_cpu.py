"""How many warps the graph search gives a token: host arithmetic on the sizes, no device."""
import os
import subprocess

import pytest


@pytest.fixture(scope="module")
def warps(tmp_path_factory):
    from paper_2608_23553_b200 import build
    build.build()
    native = os.path.join(os.path.dirname(os.path.abspath(__file__)), "native")
    tmp = tmp_path_factory.mktemp("rule")
    obj, exe = str(tmp / "graph_rules.o"), str(tmp / "graph_rules")
    subprocess.check_call([build.NVCC] + build.FLAGS + ["-c", os.path.join(native, "graph_rules.cu"), "-o", obj])
    subprocess.check_call(["g++", "-no-pie", "-o", exe, obj, os.path.join(native, "fake_cudart.cpp"), os.path.join(build.OBJ, "g7_graph.o"),
                           "-Wl,--unresolved-symbols=ignore-all"])

    def warps(K, tokens):
        return int(subprocess.run([exe], input="%d %d" % (K, tokens), capture_output=True, text=True, check=True).stdout)
    return warps


def test_two_warps_only_where_an_sm_holds_more_of_their_blocks(warps):
    small = (1_000, 65_536)
    assert [warps(K, n) for K in small for n in (1, 32, 1_184, 1_185, 2_368, 8_192)] == 2 * [4, 4, 4, 2, 2, 2]
    # 13 blocks of two warps beside 8 of four: in between and in the end
    assert [warps(131_072, n) for n in (1_184, 1_185, 1_924, 1_925, 4_096, 8_192)] == [4, 2, 2, 4, 4, 2]
    # the visited sets leave room for as many of one kind as of the other
    assert all(warps(K, n) == 4 for K in (262_144, 524_288, 1_048_576) for n in (32, 1_536, 8_192, 65_536))
    # visited sets in global memory
    assert warps(2_000_000, 1_184) == 4 and warps(2_000_000, 8_192) == 2
