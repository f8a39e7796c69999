"""Gradient and LDOS of the four-column recursions against the oracle where they
can go wrong: the shortest ribbons (no cell between the two cuts, one, two), the
narrowest ones, even and odd widths, removed atoms anywhere (the end cells
included: their columns meet the leads), and checkpoint strides that do not
divide the length.  Tolerances as the other gradient and LDOS tests: 1e-10 in
binary64, 1e-8 in double-float, 1e-9 for digit-sliced binary64, of the largest
entry (at least 1)."""
import numpy as np
import pytest

import workloads
from oracle import gradient as ograd
from oracle import ldos as oldos

pytestmark = pytest.mark.gpu
T_HOP = -2.7
TOL = {0: 1e-10, 1: 1e-8, 2: 1e-8, 3: 1e-9}


def ribbon(rgflib, N, L, p):
    eps = workloads.anderson_onsite(N, L, 0.3, 500 + 10 * N + L)
    u = workloads.uniform01(600 + N, np.arange(L * 2 * N, dtype=np.uint64)).reshape(L, 2 * N)
    rem = (u < p).astype(np.uint8)
    return rgflib.Ribbon(N, L, T_HOP, onsite=eps, removed=rem if p else None), eps, rem


CASES = [(2, 1, 0.0), (3, 1, 0.0), (2, 2, 0.0), (3, 3, 0.0), (8, 1, 0.1), (7, 2, 0.1), (10, 3, 0.1),
         (9, 5, 0.08), (36, 3, 0.03), (65, 2, 0.0)]


@pytest.mark.parametrize("prec", [0, 1, 2, 3])
@pytest.mark.parametrize("N,L,p", CASES)
def test_gradient_vs_oracle(rgflib, N, L, p, prec):
    rib, eps, rem = ribbon(rgflib, N, L, p)
    Es = np.array([-0.87, 0.31])
    for stride in (1, 2, 0):
        T, g, st = rgflib.conductance_grad([rib] * 2, Es, 1e-8, 1e-8, prec, ckpt_stride=stride)
        assert (st == 0).all()
        for c, E in enumerate(Es):
            ref = ograd.closed_form(N, L, E, 1e-8, 1e-8, T_HOP, eps, rem if p else None)
            err = np.abs(g[c] - ref).max()
            assert err < TOL[prec] * max(1.0, np.abs(ref).max()), (stride, E, err)


@pytest.mark.parametrize("prec", [0, 1, 2, 3])
@pytest.mark.parametrize("N,L,p", CASES)
def test_ldos_vs_oracle(rgflib, N, L, p, prec):
    rib, eps, rem = ribbon(rgflib, N, L, p)
    Es = np.array([-0.87, 0.31])
    for stride in (1, 2, 0):
        T, rho, st = rgflib.ldos([rib] * 2, Es, 1e-8, 1e-8, prec, ckpt_stride=stride)
        assert (st == 0).all()
        for c, E in enumerate(Es):
            ref = oldos.ldos(N, L, E, 1e-8, 1e-8, T_HOP, eps, rem)
            err = np.abs(rho[c] - ref).max()
            assert err < TOL[prec] * max(1.0, np.abs(ref).max()), (stride, E, err)
