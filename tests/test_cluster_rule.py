"""The coarsest-grid solver's cluster size follows what the device holds at once (no GPU: the runtime's
answers come from tests/cluster_rule.cpp)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_clusters_are_the_largest_that_run_in_one_wave(tmp_path):
    from paper_1009_0798_gb300 import build
    lib = build.build()
    cuda = os.path.dirname(os.path.dirname(build.NVCC))
    exe = str(tmp_path / "cluster_rule")
    subprocess.run(["g++", "-std=c++17", "-rdynamic", "-I", build.CSRC, "-I", os.path.join(cuda, "include"),
                    os.path.join(ROOT, "tests", "cluster_rule.cpp"), lib, "-o", exe,
                    "-L", os.path.join(cuda, "lib64"), "-lcudart", f"-Wl,-rpath,{os.path.dirname(lib)}",
                    f"-Wl,-rpath,{os.path.join(cuda, 'lib64')}"], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout == "ok\n", r.stdout + r.stderr
