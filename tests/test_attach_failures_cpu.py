"""An attachment of 1-bit codes that fails half-way leaves no index with one copy of two (host code against a fake CUDA
runtime, no device)."""
import os
import subprocess


def test_a_failed_attachment_leaves_the_index_as_it_was(tmp_path):
    from paper_2608_23553_b200 import build
    build.build()
    native = os.path.join(os.path.dirname(os.path.abspath(__file__)), "native")
    obj, exe = str(tmp_path / "attach_failures.o"), str(tmp_path / "attach_failures")
    subprocess.check_call([build.NVCC] + build.FLAGS + ["-c", os.path.join(native, "attach_failures.cu"), "-o", obj])
    objs = [os.path.join(build.OBJ, n) for n in ("api.o", "index_build.o", "rabitq.o")]
    # the other objects are never called: their symbols may stay open
    subprocess.check_call(["g++", "-no-pie", "-o", exe, obj, os.path.join(native, "fake_cudart.cpp")] + objs + ["-Wl,--unresolved-symbols=ignore-all"])
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
