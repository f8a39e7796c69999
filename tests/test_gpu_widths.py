"""Column sizes at the edges of the inverse's panels and of the products' tiles,
against the oracle: 16 / 17 (one entry per thread up to 16, one panel or two),
18, 32 / 33 (the 32-column passes and the row groups of a warp), 64 / 65, and
128 / 129 (two tensor tiles, two groups of inner entries).  Rough edges make the
columns of one ribbon differ.  Tolerances as the other parity tests: 1e-9 in
binary64, 1e-7 in double-float."""
import numpy as np
import pytest

import workloads
from oracle import rgf as orgf

pytestmark = pytest.mark.gpu
T_HOP = -2.7
TOL = {0: 1e-9, 1: 1e-7, 2: 1e-7, 3: 1e-9}


@pytest.mark.parametrize("prec", [0, 1, 2, 3])
@pytest.mark.parametrize("N", [30, 32, 33, 35, 64, 66, 129, 256, 257])
def test_widths_vs_oracle(rgflib, N, prec):
    L = 4
    eps = workloads.anderson_onsite(N, L, 0.2, 300 + N)
    rem = workloads.edge_removed(N, L, 0.1, 400 + N)
    rib = rgflib.Ribbon(N, L, T_HOP, onsite=eps, removed=rem)
    Es = np.array([-0.63, 0.27])
    ref = np.array([orgf.transmission(N, L, e, 1e-8, 1e-8, T_HOP, eps, rem) for e in Es])
    T, st = rgflib.conductance([rib] * 2, Es, 1e-8, 1e-8, prec)
    assert (st == 0).all()
    assert np.abs(T - ref).max() < TOL[prec], np.abs(T - ref)
