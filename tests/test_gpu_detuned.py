"""Atoms shut off by a large on-site energy (the limit of a removed atom), alone
and as both atoms of one row, in every pair of columns that a step of the
recursion joins: T against the oracle in every precision, with two and three
domains.  Steps that hold products of two columns' diagonals must give way
before such a row makes the others look singular.  Tolerances as the other
parity tests: 1e-9 in binary64, 1e-7 in double-float."""
import numpy as np
import pytest

import workloads
from oracle import rgf as orgf

pytestmark = pytest.mark.gpu
N, L, T_HOP = 21, 7, -2.7
TOL = {0: 1e-9, 1: 1e-7, 2: 1e-7, 3: 1e-9}
ATOMS = {"c0c1": [(4, 0), (4, 1)], "c1c2": [(3, 1), (3, 2)], "c2c3": [(2, 2), (2, 3)],
         "c3c0": [(3, 3), (4, 0)], "c1": [(3, 1)], "c2": [(3, 2)],
         "c0..c3": [(3, 0), (3, 1), (3, 2), (3, 3)]}


def detuned(atoms, V, row=3):
    eps = workloads.anderson_onsite(N, L, 0.6, 5)
    for cell, col in ATOMS[atoms]:
        eps[cell, 4 * row + col] = V
    return eps


@pytest.mark.parametrize("prec", [0, 1, 2, 3])
@pytest.mark.parametrize("V", [100.0, -200.0, 1e6, -1e7, 1e8, 1e10])
@pytest.mark.parametrize("atoms", list(ATOMS))
def test_detuned_rows_vs_oracle(rgflib, atoms, V, prec):
    eps = detuned(atoms, V)
    rib = rgflib.Ribbon(N, L, T_HOP, onsite=eps)
    Es = np.array([0.05, 0.31, -0.87])
    ref = np.array([orgf.transmission(N, L, e, 1e-8, 1e-8, T_HOP, eps) for e in Es])
    for ndom in (2, 3):
        rgflib.set_domains(ndom)
        try:
            T, st = rgflib.conductance([rib] * len(Es), Es, 1e-8, 1e-8, prec, check=False)
        finally:
            rgflib.set_domains(2)
        assert (st == 0).all(), (ndom, st)
        assert np.abs(T - ref).max() < TOL[prec], (ndom, np.abs(T - ref))
