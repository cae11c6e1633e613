"""Clients that wait for their results have their requests started at once while
slots are free: no request is held back for others to join."""
import os
import subprocess

import pytest

from paper_2511_02742_gb300 import build, synth

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.parametrize("clients", [2, 4])
def test_clients_that_wait(hough, tmp_path, clients):
    """Native clients, since the interpreter's own time between two requests
    would hide a wait.  Held, the median request was launched after 58 and 47
    us; not held it waits for the worker to hand over the one before: 3 and 10."""
    lib = build.build()
    cuda = os.path.dirname(os.path.dirname(build.nvcc()))
    exe = tmp_path / "two_clients"
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", os.path.join(build.ROOT, "include"),
                    "-I", os.path.join(cuda, "include"), os.path.join(HERE, "c", "two_clients.cpp"),
                    "-o", str(exe), "-L", os.path.dirname(lib), "-lhough",
                    "-L", os.path.join(cuda, "lib64"), "-lcudart", "-lpthread",
                    "-Wl,-rpath," + os.path.dirname(lib) + ":" + os.path.join(cuda, "lib64")],
                   check=True)
    geometry = tmp_path / "geometry.bin"
    geometry.write_bytes(bytes(hough.make_geometry(synth.GEOMETRY)))
    r = subprocess.run([str(exe), str(geometry), str(clients), "1000"], check=True, timeout=120,
                       capture_output=True, text=True)
    assert int(r.stdout) < 30_000, r.stdout
