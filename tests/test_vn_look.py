"""The trials that the stability search looks ahead at are those that its bisection can come to read:
none is solved in vain, none is missing."""
import ctypes
import itertools
import os
import shutil
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_nodes_are_the_ones_a_bisection_reads(tmp_path):
    (tmp_path / "h.cpp").write_text('#include "lbm_internal.h"\nextern "C" int looks() { return lbmh::kVnLooks; }\n'
                                    'extern "C" int node(int q) { return lbmh::vn_look_node(q); }\n')
    r = subprocess.run([shutil.which("g++") or "g++", "-std=c++17", "-shared", "-fPIC", "-I",
                        os.path.join(ROOT, "paper_2303_08163_gb300", "csrc"), "-I",
                        os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include"),
                        str(tmp_path / "h.cpp"), "-o", str(tmp_path / "h.so")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    lib = ctypes.CDLL(str(tmp_path / "h.so"))
    n = lib.looks()
    nodes = [lib.node(q) for q in range(n)]
    read = set()
    # the search goes on below the swept trial while what it looked at was unstable
    for stable, depth in itertools.product((0, 1), range(n // 2)):
        node = 2 + stable
        for _ in range(depth):
            node = 2 * node
        read.add(node)
    assert len(set(nodes)) == n and set(nodes) == read
    # after a stable swept trial the second half, after an unstable one the first
    assert nodes[0] == 2 and nodes[n // 2] == 3
    assert all(nodes[q + 1] == 2 * nodes[q] for q in range(n - 1) if q + 1 != n // 2)
