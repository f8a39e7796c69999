"""The widest ribbon whose columns the tensor-core layout holds (N = 2012, 1006
orbitals a column: panels of 2, eight tiles of rows and groups of inner entries,
nearly all of a block's shared memory): both tensor-core precisions against binary64
on the pipes, tolerances as for the other wide ribbons (1e-7 in double-float, 1e-9
in binary64).  The layout's limit itself is checked when the library is compiled."""
import numpy as np
import pytest

import workloads
from oracle import bands

pytestmark = pytest.mark.gpu


@pytest.mark.slow
def test_widest_tensor_core_ribbon(rgflib):
    N, L, E = 2012, 2, np.array([0.083])
    rib = rgflib.Ribbon(N, L, -2.7, onsite=workloads.anderson_onsite(N, L, 0.1, 2012),
                        removed=workloads.edge_removed(N, L, 0.05, 2013))
    T = {}
    for prec in (0, 2, 3):
        T[prec], st = rgflib.conductance([rib], E, 1e-8, 1e-8, prec)
        assert st[0] == 0
    assert -1e-9 <= T[0][0] <= bands.channels_closed_form(N, E[0]) + 1e-9
    assert abs(T[2][0] - T[0][0]) < 1e-7 and abs(T[3][0] - T[0][0]) < 1e-9
