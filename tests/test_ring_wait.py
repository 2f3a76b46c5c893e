"""What a tensor-core kernel's roles wait for before their block ends or frees
its tensor memory: the copies and MMAs they still have in flight, each at its
slot and parity. Only a wait that ran out leaves any, which no test brings
about on a GPU; the functions are the kernels' own, compiled for the host."""
import os
import subprocess

from paper_2507_17094_gb300.build import CSRC

HERE = os.path.dirname(os.path.abspath(__file__))


def test_nothing_is_left_in_flight(tmp_path):
    exe = str(tmp_path / "ring_wait")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I" + CSRC, os.path.join(HERE, "ring_wait.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr


def test_every_role_waits_once_one_gave_up():
    """Each kernel that starts tensor-map copies and MMAs ends so before it
    frees its tensor memory."""
    for f in ("mlp.cu", "knn.cu"):
        with open(os.path.join(CSRC, f)) as fh:
            end = fh.read().split("__syncthreads_or(!ok)")
        assert len(end) == 2, f
        drain = end[1].split("tcgen05.dealloc")[0]
        for role in ("wait_last_uses(it, ", "wait_last_use(issued, ", "__syncthreads();"):
            assert role in drain, (f, role)
