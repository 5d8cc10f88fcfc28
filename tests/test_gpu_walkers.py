"""The two walkers at the edges of their ranges, against the oracle.

A block per line (wl_lone.cuh) and batches of proposed moves (wl_walk.cuh) walk
the same chain; both are compared with the oracle bit for bit, at lattice sizes
where a row or the number of sites crosses a power of two (rows of site codes, 4
bytes a site against one, 16-bit list entries), with checks, slices and budgets
that are no multiple of a block of steps, and with windows smaller than a line.
"""
import ctypes

import numpy as np
import pytest

import oracle
import paper_1302_2320_gb300 as wl
from test_gpu_parity import LAT, assert_line_equal, oracle_lines
from test_zz_no_alloc import Buffers, _fn

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    wl.build()
    oracle.build()


def walk(lattice, L, ells, seed, u, C, budget, **opt):
    h = wl.Handle(lattice, L, seed=seed, check_interval=C, move_budget=budget, **opt)
    h.select_lines(list(ells))
    h.run(u, 0.8)
    return h


# rows of site codes: L and (open) L + 1 at, just below and just above a power of two
@pytest.mark.parametrize("lattice,L", [("square", 3), ("square", 7), ("square", 8), ("square", 9), ("square", 17),
                                       ("triangular", 3), ("triangular", 8), ("triangular", 9),
                                       ("cubic", 3), ("cubic", 5), ("cubic", 8),
                                       ("square_open", 3), ("square_open", 7), ("square_open", 8)])
@pytest.mark.parametrize("tail", [0, 1])
def test_all_lines_of_small_lattices(lattice, L, tail):
    h = wl.Handle(lattice, L, seed=5, check_interval=101, move_budget=30_011, tail=tail, mapping=32)
    h.run(1e-7, 0.8)
    ells = sorted({0, 1, 2, 3, h.N // 4, h.N // 2 - 1, h.N // 2})
    ref = oracle_lines(LAT[lattice], L, ells, 5, 1e-7, 101, 30_011)
    for ell in ells:
        assert_line_equal(h, ell, ref[ell], f"{lattice} {L} tail={tail}")
    h.close()


# 4 bytes a site up to 16384 codes, one byte up to 65536, lists of 16 bits up to
# 65536 sites; beyond, batches with the spins in global memory
@pytest.mark.parametrize("lattice,L", [("square", 128), ("square", 129), ("square", 256), ("square", 257),
                                       ("triangular", 128), ("triangular", 130),
                                       ("cubic", 16), ("cubic", 17), ("cubic", 32), ("cubic", 33),
                                       ("square_open", 126), ("square_open", 127),
                                       ("square_open", 254), ("square_open", 255)])
@pytest.mark.parametrize("tail", [0, 1])
def test_lines_where_the_form_changes(lattice, L, tail):
    N = L ** 3 if lattice == "cubic" else L * L
    ells = [1, 5, 700, N // 2]
    h = walk(lattice, L, ells, 3, 1e-6, 4096, 20_005, tail=tail, mapping=32)
    ref = oracle_lines(LAT[lattice], L, ells, 3, 1e-6, 4096, 20_005)
    for ell in ells:
        assert_line_equal(h, ell, ref[ell], f"{lattice} {L} tail={tail}")
    h.close()


@pytest.mark.parametrize("lattice,L", [("square", 96), ("triangular", 90), ("square_open", 64), ("cubic", 21)])
def test_more_lines_than_resident_blocks(lattice, L):
    """Small windows: each walker has its share of a crowded SM's shared memory."""
    h = wl.Handle(lattice, L, seed=2, check_interval=3000, move_budget=7_777)
    h.run(1e-6, 0.8)
    ells = [0, 1, 2, 33, 400, h.N // 4, h.N // 2]
    ref = oracle_lines(LAT[lattice], L, ells, 2, 1e-6, 3000, 7_777)
    for ell in ells:
        assert_line_equal(h, ell, ref[ell], f"{lattice} {L}")
    h.close()


@pytest.mark.parametrize("slice_ms,budget", [(0, 100_003), (2, 70_001)])
def test_lines_that_take_turns(slice_ms, budget):
    """More lines than resident blocks, with moves enough for several turns of each;
    a time limit ends a slice between the turns."""
    h = wl.Handle("square", 56, seed=3, check_interval=1500, move_budget=budget, slice_ms=slice_ms)
    h.run(1e-6, 0.8)
    ells = [0, 1, 2, 50, 400, 1000, 1567, 1568]
    ref = oracle_lines(LAT["square"], 56, ells, 3, 1e-6, 1500, budget)
    for ell in ells:
        assert_line_equal(h, ell, ref[ell], f"slice_ms={slice_ms}")
    assert h.stats()["moves"] == budget * 1568 or h.stats()["lines_converged"] > 1
    h.close()


@pytest.mark.parametrize("lattice,L,tail", [("square", 10, 1), ("square", 10, 0), ("triangular", 6, 1), ("cubic", 4, 1),
                                            ("square_open", 6, 1), ("square", 130, 1)])
def test_slices_of_odd_lengths(lattice, L, tail):
    """A slice ends anywhere in a block of steps; the pending move is drawn again."""
    ells = [1, 2, 9, 18]
    h = walk(lattice, L, ells, 4, 1e-6, 640, 0, tail=tail, mapping=32, slice_moves=1013)
    for budget in (1, 17, 32, 33, 1300, 9_001):
        h.set_option("move_budget", budget)
        h.run(1e-6, 0.8)
    ref = oracle_lines(LAT[lattice], L, ells, 4, 1e-6, 640, 9_001)
    for ell in ells:
        assert_line_equal(h, ell, ref[ell], f"{lattice} {L} tail={tail}")
    h.close()


@pytest.mark.parametrize("lattice,L", [("square", 12), ("triangular", 9), ("cubic", 5), ("square_open", 7), ("square", 132)])
def test_production_walks_are_the_same_in_both_forms(lattice, L):
    ells = [1, 4, 20, 24]
    a = walk(lattice, L, ells, 6, 1e-6, 1000, 40_009, deterministic=0, tail=1, mapping=32)
    b = walk(lattice, L, ells, 6, 1e-6, 1000, 40_009, deterministic=0, tail=0, mapping=32)
    for ell in ells:
        x, y = a.line_state(ell), b.line_state(ell)
        for key in x:
            assert np.array_equal(x[key], y[key]), (ell, key)
    a.close()
    b.close()


def test_lines_between_the_selected_ones():
    """Not walked: their list and spins are the initial ones, their status says that
    nothing is left to do, and their part of the surface has no visited bin."""
    h = walk("square", 9, [3, 30], 8, 1e-6, 1000, 5_000)
    ref = oracle_lines(oracle.SQUARE, 9, [3, 30], 8, 1e-6, 1000, 5_000)
    init = oracle_lines(oracle.SQUARE, 9, [4, 29], 8, 1e-6, 1000, 0)
    for ell in (3, 30):
        assert_line_equal(h, ell, ref[ell])
    for ell in (4, 29):
        got = h.line_state(ell)
        assert list(got["sc"]) == [0, 0, 0, 0, 0, 0, 1, 0]
        for key in ("perm", "spins", "lng", "hist", "visited"):
            assert np.array_equal(got[key], getattr(init[ell], key)), (ell, key)
    h.assemble()
    surf, offs = h.get_surface()                    # from the first selected line on
    for ell in (3, 30):
        assert np.isfinite(surf[offs[ell - 3]:offs[ell - 2]]).any()
    for ell in (4, 29):
        assert np.isneginf(surf[offs[ell - 3]:offs[ell - 2]]).all()
    h.close()


@pytest.mark.parametrize("lattice,L,first,n", [("square", 9, 0, 41), ("triangular", 8, 5, 9), ("cubic", 17, 2000, 3)])
def test_noalloc_with_the_shape_left_to_the_library(lattice, L, first, n):
    import torch
    f = _fn()
    buf = Buffers(lattice, L, first, n)
    for call, budget in enumerate((1_003, 9_001)):
        rc = f(wl.LATTICES[lattice], L, first, n, 3, 1, 1e-6, 0.8, 500, budget, 0, 1 if call == 0 else 0,
               *buf.ptrs(), buf.stream)
        assert rc in (wl.WL_OK, wl.WL_ENOTCONVERGED), wl.wl_last_error()
        torch.cuda.synchronize()
    ells = range(first, first + n)
    ref = oracle_lines(LAT[lattice], L, ells, 3, 1e-6, 500, 9_001)
    for i, ell in enumerate(ells):
        got = buf.line(i)
        assert np.array_equal(got["sc"], ref[ell].sc), ell
        for key in ("perm", "spins", "lng", "hist", "visited"):
            assert np.array_equal(got[key], getattr(ref[ell], key)), (ell, key)


def test_noalloc_refuses_a_state_that_is_none_of_the_line():
    """Two equal list entries: found before the walk, on the line that has them."""
    import torch
    f = _fn()
    buf = Buffers("square", 8, 4, 3)
    args = (wl.WL_SQUARE, 8, 4, 3, 3, 1, 1e-6, 0.8, 500)
    assert f(*args, 1000, 0, 1, *buf.ptrs(), buf.stream) == wl.WL_ENOTCONVERGED
    torch.cuda.synchronize()
    buf.perm[buf.P + 1] = buf.perm[buf.P].item()
    rc = f(*args, 2000, 0, 0, *buf.ptrs(), buf.stream)
    torch.cuda.synchronize()
    assert rc not in (wl.WL_OK, wl.WL_ENOTCONVERGED)
    assert buf.line(1)["sc"][6] == 3 and buf.line(0)["sc"][6] != 3


@pytest.mark.parametrize("lattice,L,z", [("square", 4, 4), ("triangular", 6, 6), ("square", 12, 4)])
def test_thermo_sums_from_hot_to_cold(lattice, L, z):
    """Line sums that a field weighs by many orders of magnitude; a single line's
    share, one temperature alone, and the whole grid give the same."""
    h = wl.Handle(lattice, L, seed=2, check_interval=1000, move_budget=100_000)
    h.run(1e-6, 0.8)
    h.assemble()
    surf, offs = h.get_surface()
    T = np.array([0.05, 0.4, 1.0, 2.269, 50.0, 1e4])
    H = np.array([-20.0, -0.5, 0.0, 1e-3, 3.0])
    got = h.thermo(T, H)
    ref = oracle.thermo(h.N, h.N * z // 2, offs, surf, T, H)
    # sums of up to N^2 positive terms in FP64, each exp good to a few ulp of its
    # argument (up to 20 N / 0.05): 1e-9, as for the other grids; C and chi are
    # differences of squares of such sums
    assert np.allclose(got[..., :2], ref[..., :2], rtol=1e-9, atol=1e-12)
    for i in range(len(T)):
        assert np.array_equal(h.thermo(T[i:i + 1], H), got[i:i + 1])
    h.close()


def _set_line(buf, i, lattice, L, up, entries):
    """Line i of the caller's buffers: the spins up at `up`, its k, the list `entries`
    followed by the sites that are down."""
    N = buf.N
    spins = np.zeros(N, dtype=np.uint8)
    spins[list(up)] = 1
    g = spins.reshape(L, L).astype(int)
    k = int((g != np.roll(g, 1, 0)).sum() + (g != np.roll(g, 1, 1)).sum())
    words = np.zeros(buf.W, dtype=np.uint32)
    np.bitwise_or.at(words, np.arange(N) >> 5, spins.astype(np.uint32) << (np.arange(N, dtype=np.uint32) & 31))
    down = np.flatnonzero(spins == 0)
    perm = np.concatenate([np.array(entries), down]).astype(np.int64)
    wide = buf.perm.element_size() == 4
    perm = perm.astype(np.uint32).view(np.int32) if wide else perm.astype(np.uint16).view(np.int16)
    import torch
    buf.perm[i * buf.P:i * buf.P + N] = torch.from_numpy(perm).to(buf.perm.device)
    buf.spins[i * buf.W:(i + 1) * buf.W] = torch.from_numpy(words.view(np.int32)).to(buf.spins.device)
    buf.state[i * 9] = k


@pytest.mark.parametrize("L,mapping", [(8, 0), (8, 8), (260, 0), (700, 0)])
def test_noalloc_refuses_equal_entries_whose_sums_are_right(L, mapping):
    """The sites 0, 4, 5 twice in the place of 0, 1, 2, 4, 5, 6: as many up spins, the
    same sum and the same sum of squares, and no line's list."""
    import torch
    f = _fn()
    up, twice = [0, 1, 2, 4, 5, 6], [0, 4, 5, 0, 4, 5]
    assert sum(up) == sum(twice) and sum(x * x for x in up) == sum(x * x for x in twice)
    buf = Buffers("square", L, 6, 2)
    args = (wl.WL_SQUARE, L, 6, 2, 3, 1, 1e-6, 0.8, 500)
    assert f(*args, 0, mapping, 1, *buf.ptrs(), buf.stream) == wl.WL_ENOTCONVERGED
    torch.cuda.synchronize()
    _set_line(buf, 0, "square", L, up, up)                      # a line's state: walked
    assert f(*args, 300, mapping, 0, *buf.ptrs(), buf.stream) == wl.WL_ENOTCONVERGED
    torch.cuda.synchronize()
    assert buf.line(0)["sc"][1] == 300 and sorted(buf.line(0)["perm"]) == list(range(L * L))
    _set_line(buf, 0, "square", L, up, twice)
    assert f(*args, 600, mapping, 0, *buf.ptrs(), buf.stream) not in (wl.WL_OK, wl.WL_ENOTCONVERGED)
    torch.cuda.synchronize()
    assert buf.line(0)["sc"][6] == 3 and buf.line(0)["sc"][1] == 300


def test_noalloc_refuses_a_running_line_without_up_spins():
    """l = 0 has no move and is done from the start; a state that has it running is none."""
    import torch
    f = _fn()
    buf = Buffers("square", 8, 0, 2)
    args = (wl.WL_SQUARE, 8, 0, 2, 3, 1, 1e-6, 0.8, 500)
    assert f(*args, 0, 0, 1, *buf.ptrs(), buf.stream) == wl.WL_ENOTCONVERGED
    torch.cuda.synchronize()
    buf.state[2] = 10**6                                       # ln f = 1 in units of ln f_min
    buf.state[6] = 0
    assert f(*args, 300, 0, 0, *buf.ptrs(), buf.stream) not in (wl.WL_OK, wl.WL_ENOTCONVERGED)
    torch.cuda.synchronize()
    assert buf.line(0)["sc"][6] == 3 and buf.line(0)["sc"][1] == 0


# one lane a walker, with more sites than 32 walkers' windows of 384 bins leave room for
@pytest.mark.parametrize("lattice,L", [("triangular", 58), ("cubic", 15), ("triangular", 128)])
@pytest.mark.parametrize("form", [0, 1])
def test_one_lane_with_six_neighbours(lattice, L, form):
    N = L ** 3 if lattice == "cubic" else L * L
    ells = [1, 40, N // 2]
    h = walk(lattice, L, ells, 5, 1e-6, 300, 2_001, mapping=1, form=form)
    ref = oracle_lines(LAT[lattice], L, ells, 5, 1e-6, 300, 2_001)
    for ell in ells:
        assert_line_equal(h, ell, ref[ell], f"{lattice} {L} form={form}")
    h.close()


def test_noalloc_with_one_lane_and_six_neighbours():
    import torch
    f = _fn()
    buf = Buffers("cubic", 15, 1200, 3)
    assert f(wl.WL_SIMPLE_CUBIC, 15, 1200, 3, 5, 1, 1e-6, 0.8, 300, 2_001, 1, 1, *buf.ptrs(), buf.stream) == wl.WL_ENOTCONVERGED
    torch.cuda.synchronize()
    ref = oracle_lines(oracle.CUBIC, 15, range(1200, 1203), 5, 1e-6, 300, 2_001)
    for i in range(3):
        got = buf.line(i)
        for key in ("perm", "spins", "lng", "hist", "visited"):
            assert np.array_equal(got[key], getattr(ref[1200 + i], key)), (i, key)
