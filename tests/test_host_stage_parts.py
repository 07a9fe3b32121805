"""The stage kernel's parts of a block along z (csrc/stage_parts.hpp), built with g++ behind a small C
shim: every part of every count the rule may choose replayed on the asynchronous-copy groups that the
kernel commits and waits for.  No GPU is needed."""
import ctypes as C
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_1912_05371_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    out = str(tmp_path_factory.mktemp("hostparts") / "libhostparts.so")
    subprocess.run([gxx, "-O1", "-std=c++17", "-fPIC", "-shared", "-I", CSRC,
                    os.path.join(HERE, "host", "stage_parts_shim.cpp"), "-o", out], check=True)
    L = C.CDLL(out)
    L.hp_z_parts.argtypes = [C.c_longlong, C.c_int, C.c_int, C.c_longlong, C.c_longlong]
    return L


def replay(lib, z0, z1, M):
    """The part z0 .. z1 - 1 as the kernel walks it: groups of copies in the order of their commits, a
    wait that leaves the newest group pending, and in iteration z the reads of plane z's halos and, from
    M - 2 on, of the planes beyond the upper face.  Returns the reads whose copies had not arrived."""
    groups, arrived, early = [], set(), []

    def wait():
        while len(groups) > 1:
            arrived.update(groups.pop(0))

    first = {"upper"} if lib.hp_upper_in_prologue(z0, M) else set()
    groups.append(first | {("halo", z0)})
    groups.append({("halo", z0 + 1)} if z0 + 1 < z1 else set())
    wait()
    for z in range(z0, z1):
        g = {"upper"} if lib.hp_upper_in_loop(z, z0, z1, M) else set()
        if z + 2 < z1:
            g.add(("halo", z + 2))
        groups.append(g)
        if z + 1 < z1:
            wait()
        if z + 3 > M and "upper" not in arrived:
            early.append((z, "upper"))
        if ("halo", z) not in arrived:
            early.append((z, "halo"))
    return early


@pytest.mark.parametrize("Bs", [9, 17, 33])
def test_copies_arrive_before_they_are_read(lib, Bs):
    M = Bs - 1
    assert replay(lib, 0, Bs, M) == []                      # a block in one part
    for nz in range(2, Bs // 2 + 1):
        edges = [lib.hp_part_begin(k, nz, Bs) for k in range(nz + 1)]
        assert edges[0] == 0 and edges[-1] == Bs and all(b - a >= 2 for a, b in zip(edges, edges[1:]))
        for z0, z1 in zip(edges, edges[1:]):
            assert replay(lib, z0, z1, M) == [], (Bs, nz, z0, z1)


def test_the_rule_reaches_parts_that_start_three_planes_below_the_top(lib):
    """The parts whose upper planes are wanted in their second iteration occur: five parts of a 17^3
    block (FP32: 304 resident CTAs, a start of five planes; FP64: 152 and one) and nine of a 33^3 block."""
    assert {lib.hp_z_parts(n, 1, 17, 304, 5) for n in range(51, 61)} == {5}
    assert {lib.hp_z_parts(n, 1, 17, 152, 1) for n in range(26, 31)} == {5}
    assert lib.hp_z_parts(6, 5, 33, 304, 5) == 9
    assert lib.hp_part_begin(4, 5, 17) == 13 and lib.hp_part_begin(8, 9, 33) == 29
    assert lib.hp_z_parts(100000, 1, 17, 304, 5) == 1
