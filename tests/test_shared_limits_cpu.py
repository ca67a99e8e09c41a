"""Kernels that take more than 48 KB of shared memory are allowed the same amount by every call (host code against a fake CUDA
runtime, no device)."""
import os
import subprocess


def test_every_call_allows_a_kernel_the_same(tmp_path):
    from paper_2608_23553_b200 import build
    build.build()
    native = os.path.join(os.path.dirname(os.path.abspath(__file__)), "native")
    obj, exe = str(tmp_path / "shared_limits.o"), str(tmp_path / "shared_limits")
    subprocess.check_call([build.NVCC] + build.FLAGS + ["-c", os.path.join(native, "shared_limits.cu"), "-o", obj])
    names = ("api", "g1_score_table", "g2_gather", "g2_probe", "g3_batch_scan", "g3_centroid_interaction", "g3_filter", "g3_partial", "g5_topk", "g7_graph")
    objs = [os.path.join(build.OBJ, n + ".o") for n in names]
    subprocess.check_call(["g++", "-no-pie", "-o", exe, obj, os.path.join(native, "fake_cudart.cpp")] + objs + ["-Wl,--unresolved-symbols=ignore-all"])
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
