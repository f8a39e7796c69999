"""Gradient where the atoms of c3 and of the next cell's c0 have lost their partners
in their rows (c2 of one cell and c1 of the next removed over a run of rows), with
those atoms raised by a potential step: their rows of z - H follow from one another
by a factor of (z - eps) / t a row, which must not amplify rounding.  Runs of one to
24 atoms, steps of 0 to 1000 eV, a run from the edge of the ribbon, and known rows
that never meet; the bond within a checkpoint segment and between two.  Against
the oracle, with the leads of the closed form of their modes (the decimated ones
of N = 50 at 0.31 eV are off by 4e-11, which moves the gradient by 1e-10); tolerances as the other gradient tests: 1e-10 in binary64, 1e-8 in
double-float, 1e-9 for digit-sliced binary64, of the largest entry (at least 1)."""
import numpy as np
import pytest

import workloads
from oracle import gradient as ograd
from oracle import modes

pytestmark = pytest.mark.gpu
N, L, T_HOP = 50, 4, -2.7
TOL = {0: 1e-10, 1: 1e-8, 2: 1e-8, 3: 1e-9}


def orphan_rows(rows, U, cell=1):
    """On-site energies and removals that leave those rows of the bond between
    `cell` and the next without partners, raised by U."""
    eps = workloads.anderson_onsite(N, L, 0.6, 7)
    rem = np.zeros((L, 2 * N), dtype=np.uint8)
    for r in rows:
        n, col = (cell, 2) if r & 1 else (cell + 1, 1)
        rem[n, 4 * (r // 2) + col] = 1
        eps[n, 4 * (r // 2) + (3 if r & 1 else 0)] += U
    return eps, rem


def check(rgflib, eps, rem, prec, strides=(1, 2, 4)):
    rib = rgflib.Ribbon(N, L, T_HOP, onsite=eps, removed=rem)
    Es = np.array([0.31, -0.87])
    refs = [ograd.two_sided(N, L, E, 1e-8, 1e-8, T_HOP, eps, rem, sig=modes.self_energies(N, E, 1e-8, T_HOP))[1]
            for E in Es]
    for stride in strides:
        T, g, st = rgflib.conductance_grad([rib] * 2, Es, 1e-8, 1e-8, prec, ckpt_stride=stride)
        assert (st == 0).all()
        for c, ref in enumerate(refs):
            err = np.abs(g[c] - ref).max()
            assert err < TOL[prec] * max(1.0, np.abs(ref).max()), (stride, Es[c], err)


@pytest.mark.parametrize("prec", [0, 1, 2, 3])
@pytest.mark.parametrize("U", [0.0, 2.7, 9.0, -20.0, 1000.0])
@pytest.mark.parametrize("first,run", [(10, 1), (10, 3), (11, 4), (10, 8), (9, 16), (10, 24), (0, 12), (30, 20)])
def test_runs_of_orphans(rgflib, first, run, U, prec):
    check(rgflib, *orphan_rows(range(first, first + run), U), prec, strides=(1, 2) if run > 3 else (2,))


@pytest.mark.parametrize("prec", [0, 2])
@pytest.mark.parametrize("U", [0.0, 12.0])
def test_known_rows_that_never_meet(rgflib, prec, U):
    # segments cut out of the rows in which orphans and known rows alternate, with
    # orphans at both ends
    eps, rem = orphan_rows([11, 13, 15, 31, 33], U)
    for r in (10, 16, 30, 34):
        n, col = (1, 3) if r & 1 else (2, 0)
        rem[n, 4 * (r // 2) + col] = 1
    check(rgflib, eps, rem, prec)


@pytest.mark.parametrize("prec", [0, 2])
def test_runs_at_every_bond(rgflib, prec):
    eps, rem = orphan_rows(range(12, 24), 15.0, 0)
    for cell in (1, 2):
        e2, r2 = orphan_rows(range(20 - 4 * cell, 34), -15.0, cell)
        eps, rem = np.where(r2 | (np.abs(e2) > 5), e2, eps), rem | r2
    check(rgflib, eps, rem, prec)
