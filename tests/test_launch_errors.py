"""A kernel launch that the CUDA runtime refuses is reported by the call that made it and by no later one.

No GPU: tests/launch_errors.cpp calls the launchers against a runtime whose launches fail.
"""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_failed_launches_are_returned_and_leave_no_error(tmp_path):
    from paper_1009_0798_gb300 import build
    lib = build.build()
    cuda = os.path.dirname(os.path.dirname(build.NVCC))
    exe = str(tmp_path / "launch_errors")
    subprocess.run(["g++", "-std=c++17", "-rdynamic", "-I", build.CSRC, "-I", os.path.join(cuda, "include"),
                    os.path.join(ROOT, "tests", "launch_errors.cpp"), lib, "-o", exe,
                    "-L", os.path.join(cuda, "lib64"), "-lcudart", f"-Wl,-rpath,{os.path.dirname(lib)}",
                    f"-Wl,-rpath,{os.path.join(cuda, 'lib64')}"], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout == "ok\n", r.stdout + r.stderr
