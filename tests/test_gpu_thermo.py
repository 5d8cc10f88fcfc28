"""All six outputs of the thermodynamics from hot to cold and through strong fields,
against sums in long double about the mean.

Tolerances.  A weight exp(x) has the relative error of its argument, |x| <= (N_B + |H| N) / T
+ N ln 2, times a few units of 2^-53: below 1e-10 on these grids, and 1e-9 covers the sums.
The library leaves out bins below e^-46 of their line's likeliest: to C they would add at most
bins * e^-46 * (2 N_B / T)^2 / N < 1e-11, to chi bins * e^-46 * N / T < 1e-14.
"""
import numpy as np
import pytest

import paper_1302_2320_gb300 as wl

pytestmark = pytest.mark.gpu

T = np.array([0.05, 0.4, 1.0, 2.269, 50.0, 1e4])
H = np.array([-20.0, -0.5, 0.0, 1e-3, 3.0])


@pytest.fixture(scope="module", autouse=True)
def _built():
    wl.build()


def _reference(h, surf, offs):
    N, NB, step = h.N, h.NB, h.get_option("k_step")
    lg, bond, M = [], [], []
    for ell in range(h.lines):
        g = surf[offs[ell]:offs[ell + 1]].astype(np.longdouble)
        b = np.arange(g.size)
        for m in {2 * ell - N, N - 2 * ell}:                 # the line and its mirror
            ok = np.isfinite(g)
            lg.append(g[ok])
            bond.append((2 * step * b - NB)[ok].astype(np.longdouble))
            M.append(np.full(ok.sum(), m, dtype=np.longdouble))
    lg, bond, M = np.concatenate(lg), np.concatenate(bond), np.concatenate(M)
    out = np.zeros((T.size, H.size, 6), dtype=np.longdouble)
    for a, t in enumerate(T.astype(np.longdouble)):
        for c, f in enumerate(H.astype(np.longdouble)):
            E = bond - f * M
            x = lg - E / t
            w = np.exp(x - x.max())
            z = w.sum()
            w /= z
            e, m = (w * E).sum(), (w * M).sum()
            out[a, c] = [(x.max() + np.log(z)) / N, e / N, (w * (E - e) ** 2).sum() / t ** 2 / N,
                         m / N, (w * abs(M)).sum() / N, (w * (M - m) ** 2).sum() / t / N]
    return out


@pytest.mark.parametrize("lattice,L", [("square", 4), ("square", 12), ("triangular", 6), ("cubic", 4), ("square_open", 7)])
def test_all_moments_from_hot_to_cold(lattice, L):
    h = wl.Handle(lattice, L, seed=2, check_interval=1000, move_budget=100_000)
    h.run(1e-6, 0.8)
    h.assemble()
    got = h.thermo(T, H)
    ref = _reference(h, *h.get_surface())
    names = ("ln Z", "E", "C", "M", "|M|", "chi")
    for q, name in enumerate(names):
        assert np.allclose(got[..., q], ref[..., q].astype(float), rtol=1e-9, atol=1e-11), (
            name, float(abs(got[..., q] - ref[..., q]).max()))
    h.close()
