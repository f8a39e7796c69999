"""Panel widths of the inverse in RGF_FP64_TC on both sides of the one up to which
the rank-b update stays on the FP64 pipe, at column sizes below, at and past a
panel and with a last panel of one column, against RGF_FP64 of the same panels
(the same arithmetic there but for the products of a step) and the oracle;
tolerance 1e-9 as the other binary64 tests."""
import numpy as np
import pytest

import workloads
from oracle import modes
from oracle import rgf as orgf

pytestmark = pytest.mark.gpu
T_HOP = -2.7


@pytest.mark.parametrize("panel", [2, 4, 8])
@pytest.mark.parametrize("pairs", [0, 1])
@pytest.mark.parametrize("N", [3, 8, 9, 34, 66, 259])
def test_panels_of_binary64_tensor_core_inverse(rgflib, N, pairs, panel):
    L = 4
    eps = workloads.anderson_onsite(N, L, 0.2, 700 + N)
    rib = rgflib.Ribbon(N, L, T_HOP, onsite=eps)
    Es = np.array([-0.63, 0.27])
    ref = np.array([orgf.transmission(N, L, e, 1e-8, 1e-8, T_HOP, eps, sig=modes.self_energies(N, e, 1e-8, T_HOP))
                    for e in Es])
    entry = [dict(K_max=1 << 20, engine=rgflib.RGF_ENGINE_TENSOR, panel=panel, pairs=pairs)]
    for prec in (rgflib.RGF_FP64, rgflib.RGF_FP64_TC):
        rgflib.set_tuning(prec, entry)
        try:
            T, st = rgflib.conductance([rib] * 2, Es, 1e-8, 1e-8, prec)
        finally:
            rgflib.set_tuning(prec, [])
        assert (st == 0).all() and np.abs(T - ref).max() < 1e-9, (prec, np.abs(T - ref))
