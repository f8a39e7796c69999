"""Cell steps of the column recursion (four columns in one inverse) against the
oracle where they can go wrong: widths whose even and odd rows hold equal and
unequal numbers of atoms, the narrowest and the first with more than one
32-column chunk, removed atoms anywhere (identity rows of A, of T, dimers with
one atom), lengths that leave one to four columns after the last cell step, and
energies at the dimers' own levels (near +-t), where the pair steps take over.
Tolerances as the other parity tests: 1e-9 in binary64, 1e-7 in double-float."""
import numpy as np
import pytest

import workloads
from oracle import rgf as orgf

pytestmark = pytest.mark.gpu
T_HOP = -2.7
TOL = {0: 1e-9, 1: 1e-7, 2: 1e-7, 3: 1e-9}


@pytest.mark.parametrize("prec", [0, 1, 2, 3])
@pytest.mark.parametrize("N,L,p", [(2, 6, 0.0), (3, 5, 0.0), (7, 4, 0.1), (8, 7, 0.1), (33, 5, 0.05),
                                   (65, 6, 0.02), (66, 5, 0.0)])
def test_cell_steps_vs_oracle(rgflib, N, L, p, prec):
    eps = workloads.anderson_onsite(N, L, 0.3, 100 + N)
    u = workloads.uniform01(200 + N, np.arange(L * 2 * N, dtype=np.uint64)).reshape(L, 2 * N)
    rem = (u < p).astype(np.uint8)
    rem[0] = rem[-1] = 0
    rib = rgflib.Ribbon(N, L, T_HOP, onsite=eps, removed=rem if p else None)
    Es = np.array([-1.9, -0.6, 0.003, 0.21, 0.9, 2.6, 2.72])
    ref = np.array([orgf.transmission(N, L, e, 1e-8, 1e-8, T_HOP, eps, rem) for e in Es])
    T, st = rgflib.conductance([rib] * len(Es), Es, 1e-8, 1e-8, prec)
    assert (st == 0).all()
    assert np.abs(T - ref).max() < TOL[prec], np.abs(T - ref)
    with_domains(rgflib, rib, Es, ref, prec)


def with_domains(rgflib, rib, Es, ref, prec):
    rgflib.set_domains(3)
    try:
        T, st = rgflib.conductance([rib] * len(Es), Es, 1e-8, 1e-8, prec)
    finally:
        rgflib.set_domains(2)
    assert (st == 0).all()
    assert np.abs(T - ref).max() < TOL[prec], np.abs(T - ref)


@pytest.mark.parametrize("prec", [0, 2])
def test_isolated_atoms_of_the_dimer_columns(rgflib, prec):
    # an atom of c or d whose partner is removed, with its on-site energy at E:
    # alone it would be 1 / (E - eps); the step gives way to the pairs
    N, L, E = 10, 6, 0.31
    eps = workloads.anderson_onsite(N, L, 0.1, 5)
    rem = np.zeros((L, 2 * N), dtype=np.uint8)
    rem[2, 4 * 1 + 0] = 1
    eps[2, 4 * 1 + 1] = E + 1e-3
    rem[3, 4 * 2 + 3] = 1
    eps[3, 4 * 2 + 2] = E - 1e-3
    rib = rgflib.Ribbon(N, L, T_HOP, onsite=eps, removed=rem)
    ref = orgf.transmission(N, L, E, 1e-8, 1e-8, T_HOP, eps, rem)
    T, st = rgflib.conductance([rib], np.array([E]), 1e-8, 1e-8, prec)
    assert st[0] == 0 and abs(T[0] - ref) < TOL[prec]
