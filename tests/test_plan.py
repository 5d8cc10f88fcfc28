"""The planner of the walkers' launches (csrc/wl_plan.h), on the host: what it does for a
GPU with a GB300's limits, without one."""
import ctypes
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
PLAN_H = os.path.join(os.path.dirname(HERE), "paper_1302_2320_gb300", "csrc", "wl_plan.h")

LATTICE = {"square": 0, "triangular": 1, "cubic": 2, "square_p2": 3, "square_open": 4}
Z = {"square": 4, "triangular": 6, "cubic": 6, "square_p2": 4, "square_open": 4}
SMS = 152


class Gpu(ctypes.Structure):
    _fields_ = [(n, ctypes.c_int) for n in ("sms", "per_block", "per_sm", "reserved")]


class Key(ctypes.Structure):
    _fields_ = [("lattice", ctypes.c_int), ("S", ctypes.c_int), ("det", ctypes.c_bool), ("idx16", ctypes.c_bool),
                ("L", ctypes.c_int), ("N", ctypes.c_int), ("pstride", ctypes.c_int), ("max_bins", ctypes.c_int),
                ("lines", ctypes.c_int), ("lone", ctypes.c_bool)]


class Slot(ctypes.Structure):
    _fields_ = [(n, ctypes.c_int) for n in ("bytes", "off_perm", "off_sites", "off_win", "off_rec", "win", "owner_mask")] + [
        ("stage_sites", ctypes.c_bool), ("stage_perm", ctypes.c_bool), ("lone", ctypes.c_int)]


class Shape(ctypes.Structure):
    _fields_ = [("grid", ctypes.c_uint), ("block", ctypes.c_uint), ("smem", ctypes.c_size_t), ("slot", Slot)]


@pytest.fixture(scope="module")
def planner():
    src = os.path.join(HERE, "helpers", "plan_shapes.cpp")
    out = os.path.join(HERE, "helpers", "_build", "libplan_shapes.so")
    if not os.path.exists(out) or os.path.getmtime(out) < max(os.path.getmtime(src), os.path.getmtime(PLAN_H)):
        if shutil.which("g++") is None:
            pytest.skip("g++ not available")
        os.makedirs(os.path.dirname(out), exist_ok=True)
        subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", src, "-o", out], check=True, capture_output=True)
    lib = ctypes.CDLL(out)

    def plan(lattice, L, lines, S=32, lone=True, reserved=1024, per_sm=233472, max_lone=10, max_batch=20, **more):
        """The shape for `lines` lines, or None if none fits."""
        N = L ** 3 if lattice == "cubic" else L * L
        open_ = lattice == "square_open"
        NB = 2 * L * (L - 1) if open_ else N * Z[lattice] // 2
        idx16 = N <= 65536
        isz = 2 if idx16 else 4
        k = Key(LATTICE[lattice], S, True, idx16, L, N, (N * isz + 15) // 16 * 16 // isz,
                min(Z[lattice] * (N // 2), NB) // (1 if open_ else 2) + 1, lines, lone, **more)
        g = Gpu(SMS, per_sm - reserved, per_sm, reserved)
        s = Shape()
        rc = lib.plan_shapes(ctypes.byref(k), ctypes.byref(g), max_lone, max_batch, ctypes.byref(s))
        assert rc in (0, 1)
        if rc == 1:
            return None
        assert s.smem <= g.per_block and s.grid >= 1 and s.slot.win >= 1
        return s
    plan.turns = lambda sh, running, moves: lib.turns_of(ctypes.byref(sh), ctypes.c_longlong(running), ctypes.c_longlong(moves))
    return plan


# one lane a walker has the least room: 32 walkers share a block's shared memory
@pytest.mark.parametrize("lattice,L", [("square", 64), ("square", 300), ("square_open", 64), ("triangular", 57),
                                       ("triangular", 58), ("triangular", 128), ("triangular", 300), ("cubic", 14),
                                       ("cubic", 15), ("cubic", 40), ("cubic", 101)])
@pytest.mark.parametrize("S", [1, 2, 4, 8, 16, 32])
def test_every_lane_count_has_a_shape(planner, lattice, L, S):
    for lines in (1, 100, 5000):
        sh = planner(lattice, L, lines, S=S, lone=False)
        assert sh is not None, lines
        # two margins of a run of 8 steps of the largest bin step, and a walk between them
        zb = {"square": 4, "square_open": 8}.get(lattice, 6)
        N = L ** 3 if lattice == "cubic" else L * L
        assert sh.slot.win >= min(Z[lattice] * (N // 2) // 2 + 1, 2 * 8 * (zb + 1) + 32)


def test_a_block_per_line_only_where_shared_memory_starts_at_its_address(planner):
    """Its list entries are addresses past 1024, the share the system keeps of a block."""
    for lattice, L in (("square", 16), ("square_p2", 64), ("triangular", 32), ("cubic", 8), ("square_open", 15)):
        assert planner(lattice, L, 100).slot.lone != 0
        for reserved in (0, 2048):
            sh = planner(lattice, L, 100, reserved=reserved)
            assert sh is not None and sh.slot.lone == 0


def test_turns_are_for_running_lines_without_a_block(planner):
    sh = planner("square_p2", 64, 2049)
    assert sh.slot.lone and 1400 < sh.grid < 2049
    assert planner.turns(sh, 2049, 1 << 20) == 8
    assert planner.turns(sh, 2049, 1 << 15) == 2 and planner.turns(sh, 2049, 5000) == 1
    assert planner.turns(sh, 2049, (1 << 26) + 1) == 1
    assert planner.turns(sh, sh.grid, 1 << 20) == 1             # the others are done
    assert planner.turns(planner("square_p2", 64, 2049, lone=False), 5000, 1 << 20) == 1
