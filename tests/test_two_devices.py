"""Jobs on two devices of one process, without a GPU: librbx over a runtime that keeps, as CUDA does, what a
kernel is allowed (shared memory above 48 KB) by device (fake_cudart.c)."""
import os
import subprocess

from paper_2211_00316_gb300 import build as B

HERE = os.path.dirname(os.path.abspath(__file__))


def test_every_kernel_is_set_up_on_either_device(tmp_path):
    lib = B.build()
    exe = str(tmp_path / "two_devices")
    subprocess.run(["gcc", "-rdynamic", "-I", os.path.join(HERE, "..", "include"), "-o", exe,
                    os.path.join(HERE, "fake_cudart.c"), lib, "-Wl,-rpath," + os.path.dirname(lib),
                    "-Wl,--unresolved-symbols=ignore-in-shared-libs"], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
