"""A device snapshot is read in place only where the context's own device can
read it: memory of another GPU, or memory the runtime does not know, is copied
first, as cudaMemcpy reaches it from anywhere.  No GPU is needed (or used): the
library's host object runs against a runtime of host memory
(restore_route_host.cu)."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))

WANT = {"own": "direct", "managed": "direct", "other": "staged", "pinned": "staged", "unknown": "staged",
        "refused": "staged"}


def test_memory_of_another_device_is_staged(tmp_path):
    from paper_1011_0917_gb300 import build
    obj = os.path.join(build.BUILD, "pic_capi.o")
    build.build(force=not os.path.exists(obj))
    src, main, runtime, exe = os.path.join(HERE, "restore_route_host.cu"), *(
        str(tmp_path / n) for n in ("main.o", "runtime.o", "route"))
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    subprocess.run([build.nvcc(), *build._flags("restore_route_host.cu"), "-c", src, "-o", main], check=True)
    subprocess.run(["g++", "-std=c++17", "-I", cuda, "-x", "c++", "-c", src, "-o", runtime], check=True)
    # (the kernels' launches that a restore does not reach stay unresolved)
    subprocess.run(["g++", main, runtime, obj, "-o", exe, "-Wl,--unresolved-symbols=ignore-all", "-no-pie"], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split("\n")
    got = {tuple(line.split()[:2]): line.split()[2] for line in out if line}
    assert got == {(p, k): v for p in "01" for k, v in WANT.items()}
