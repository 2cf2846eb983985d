"""Device code whose results hang on its barriers, on the CPU: the threads run as fibers in several orders
(tests/simt), and every order has to give the bits of the serial computation."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1903_12522_gb300", "csrc")


@pytest.mark.parametrize("name", ["coarsest", "cluster_total"])
def test_every_order_of_the_threads_gives_the_same(name, tmp_path):
    exe = tmp_path / name
    src = os.path.join(HERE, "simt", name + ".cpp")
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-I", CSRC, src, "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr[-2000:]
    lines = out.stdout.strip().splitlines()
    assert lines and all(line.endswith(": 0") for line in lines), [q for q in lines if not q.endswith(": 0")][:10]
