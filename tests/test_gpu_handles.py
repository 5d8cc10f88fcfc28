"""A handle that is kept: options that change between its walks.

Every walk is a function of its lattice, options and seed alone, so a handle that
has walked before gives what a fresh one gives, and an option set between two
walks holds for the second.
"""
import numpy as np
import pytest

import paper_1302_2320_gb300 as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    wl.build()


def _assert_same(a, b, ells, what):
    for ell in ells:
        x, y = a.line_state(ell), b.line_state(ell)
        for key in x:
            assert np.array_equal(x[key], y[key]), (what, ell, key)


@pytest.mark.parametrize("lattice,L,mapping", [("square", 8, 0), ("triangular", 6, 32), ("square", 8, 8)])
@pytest.mark.parametrize("first", [0, 1])
def test_both_acceptance_rules_on_one_handle(lattice, L, mapping, first):
    opt = dict(seed=3, check_interval=500, move_budget=30_000, mapping=mapping)
    kept = wl.Handle(lattice, L, deterministic=first, **opt)
    kept.run(1e-6, 0.8)
    kept.reset()
    kept.set_option("deterministic", 1 - first)
    kept.run(1e-6, 0.8)
    fresh = wl.Handle(lattice, L, deterministic=1 - first, **opt)
    fresh.run(1e-6, 0.8)
    _assert_same(kept, fresh, range(1, kept.lines, 5), f"deterministic {first} then {1 - first}")


def test_a_shorter_time_limit_of_a_slice_holds_from_the_next_walk_on():
    """2^18 moves a line take 15 ms or more: one slice of 10 s, and many of 1 ms (two
    launches a slice, two for the initialisation)."""
    h = wl.Handle("square", 16, seed=2, check_interval=1000, move_budget=1 << 18, slice_moves=1 << 40, slice_ms=10_000)
    h.run(1e-6, 0.8)
    assert h.stats()["launches"] == 4
    h.reset()
    h.set_option("slice_ms", 1)
    h.run(1e-6, 0.8)
    assert h.stats()["launches"] >= 2 + 2 * 4


@pytest.mark.parametrize("L,tail", [(64, 1), (96, 0)])
def test_slices_that_end_by_time_take_every_line_along(L, tail):
    """More lines than walkers at once and no budget that ends a line's slice: after some
    60 slices no line that still walks has a fraction of another's moves."""
    h = wl.Handle("square", L, seed=5, check_interval=1000, move_budget=1 << 40, slice_moves=1 << 40, slice_ms=4,
                  timeout_ms=240, tail=tail, mapping=32)
    assert h.run(1e-6, 0.8, allow=(wl.WL_ETIMEOUT,)) == wl.WL_ETIMEOUT
    states = [h.line_state(ell)["sc"] for ell in range(64, h.lines, h.lines // 64)]
    moves = [int(sc[1]) for sc in states if sc[6] == 0]
    assert len(moves) > 48
    assert min(moves) * 3 > max(moves), (min(moves), max(moves))
    h.close()


def test_workspace_of_thermodynamics_is_counted_and_within_the_budget():
    """A small one stays with the handle and shows in device_bytes, unless the budget has
    no room for it; a large one is given back.  The values do not depend on it."""
    need = wl.wl_required_bytes(wl.LATTICES["square"], 16)
    T, H = np.linspace(1.0, 5.0, 600), np.linspace(0.0, 2.0, 200)       # 5.8 MB of results
    got = {}
    for name, budget in (("free", 0), ("tight", need)):
        h = wl.Handle("square", 16, seed=2, check_interval=1000, move_budget=20_000, hbm_budget=budget)
        h.run(1e-6, 0.8)
        h.assemble()
        assert h.get_option("device_bytes") == need
        large = h.thermo(T, H)
        assert h.get_option("device_bytes") == need
        small = h.thermo(T[:3], H[:2])
        held = h.get_option("device_bytes") - need
        assert held == 0 if name == "tight" else 0 < held <= 4 << 20
        assert np.array_equal(small, large[:3, :2]) and np.isfinite(large).all()
        got[name] = small
        h.close()
    assert np.array_equal(got["free"], got["tight"])


@pytest.mark.parametrize("opt,expect", [({}, 1), ({"mapping": 32}, 1), ({"mapping": 8}, 0), ({"tail": 0}, 0),
                                        ({"form": 1}, 0)])
def test_the_library_names_the_walker_that_ran(opt, expect):
    h = wl.Handle("square", 16, seed=2, check_interval=1000, move_budget=5_000, **opt)
    h.run(1e-6, 0.8)
    assert h.get_option("block_per_line") == expect
    h.close()
