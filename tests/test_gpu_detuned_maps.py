"""Gradient and LDOS beside strongly detuned atoms (a removed atom as the limit of a
large on-site energy), where c0 and c3 do not follow from the rows of z - H at c1
and c2: on every column of an interior cell, at the first and the last column's
partners, alone and as neighbours, with the bond inside a checkpoint segment and
between two.  Against the oracle's two-sided recursion with the closed-form leads;
tolerances as the other gradient and LDOS tests, 1e-10 in binary64, 1e-8 in
double-float, 1e-9 for digit-sliced binary64: of the largest gradient entry (at
least 1), of the largest LDOS."""
import numpy as np
import pytest

import workloads
from oracle import gradient as ograd
from oracle import ldos as oldos
from oracle import modes

pytestmark = pytest.mark.gpu
T_HOP = -2.7
TOL = {0: 1e-10, 1: 1e-8, 2: 1e-8, 3: 1e-9}
PLACES = {"c1": [(3, 1)], "c2": [(3, 2)], "c1c2": [(3, 1), (3, 2)], "c2c3": [(2, 2), (2, 3)],
          "c3c0": [(3, 3), (4, 0)], "c2 and next c1": [(2, 2), (3, 1)], "first c1": [(0, 1)],
          "last c2": [(-1, 2)], "both ends": [(0, 1), (-1, 2), (0, 0), (-1, 3)]}


def check(rgflib, N, L, eps, prec, strides):
    rib = rgflib.Ribbon(N, L, T_HOP, onsite=eps)
    Es = np.array([0.31, -0.87])
    sig = [modes.self_energies(N, E, 1e-8, T_HOP) for E in Es]
    grad = [ograd.two_sided(N, L, E, 1e-8, 1e-8, T_HOP, eps, sig=s)[1] for E, s in zip(Es, sig)]
    ldos = [oldos.ldos(N, L, E, 1e-8, 1e-8, T_HOP, eps, sig=s) for E, s in zip(Es, sig)]
    for stride in strides:
        T, g, st = rgflib.conductance_grad([rib] * 2, Es, 1e-8, 1e-8, prec, ckpt_stride=stride)
        assert (st == 0).all()
        T, r, st = rgflib.ldos([rib] * 2, Es, 1e-8, 1e-8, prec, ckpt_stride=stride)
        assert (st == 0).all()
        for c, E in enumerate(Es):
            err = np.abs(g[c] - grad[c]).max()
            assert err < TOL[prec] * max(1.0, np.abs(grad[c]).max()), ("gradient", stride, E, err)
            err = np.abs(r[c] - ldos[c]).max()
            assert err < TOL[prec] * np.abs(ldos[c]).max(), ("ldos", stride, E, err)


@pytest.mark.parametrize("prec", [0, 1, 2, 3])
@pytest.mark.parametrize("V", [12.0, -1e3, 1e6, -1e8])
@pytest.mark.parametrize("place", list(PLACES))
def test_detuned_atoms(rgflib, place, V, prec):
    N, L = 21, 6
    eps = workloads.anderson_onsite(N, L, 0.6, 5)
    for cell, col in PLACES[place]:
        eps[cell, 4 * 3 + col] = V
    check(rgflib, N, L, eps, prec, (1, 2, 4))


@pytest.mark.parametrize("prec", [0, 1, 2, 3])
@pytest.mark.parametrize("N,L", [(2, 1), (3, 2), (8, 1), (11, 5), (33, 4), (66, 3)])
def test_detuned_atoms_anywhere(rgflib, N, L, prec):
    eps = workloads.anderson_onsite(N, L, 0.3, 900 + N)
    u = workloads.uniform01(950 + N, np.arange(L * 2 * N, dtype=np.uint64)).reshape(L, 2 * N)
    eps[u < 0.05] += 40.0
    eps[u > 0.95] -= 2e4
    check(rgflib, N, L, eps, prec, (1, 0))


@pytest.mark.parametrize("prec", [0, 2])
def test_rows_on_both_sides_of_the_limit(rgflib, prec):
    # |z - eps| of single atoms from 1.5 to 2.5 |t|: no step between the two routes
    N, L = 14, 5
    eps = workloads.anderson_onsite(N, L, 0.2, 3)
    for cell, x in enumerate((1.5, 1.95, 2.0, 2.05, 2.5)):
        eps[cell, 4 * 2 + 1 + (cell & 1)] = 2.7 * x
    check(rgflib, N, L, eps, prec, (2,))
