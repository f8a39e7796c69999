"""A lead that does not converge, in the calls that return maps: the chain gets
RGF_ENOCONV, T = NaN and a map of zeros in the gradient and in the LDOS, with and
without removed atoms (the LDOS of the two comes from different kernels), and a
chain of the same call whose lead converges is not touched by it.  The failure is
made on the host (iteration cap of the decimation)."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu
N, L, T_HOP = 11, 3, -2.7


@pytest.fixture
def cap(rgflib):
    yield lambda n: rgflib.set_lead_controls(n, 1e-10)
    rgflib.set_lead_controls(200, 1e-10)      # the defaults


def ribbons(rgflib):
    eps = workloads.anderson_onsite(N, L, 0.2, 1)
    rem = np.zeros((L, 2 * N), dtype=np.uint8)
    rem[1, 5] = 1
    return [rgflib.Ribbon(N, L, T_HOP, onsite=eps), rgflib.Ribbon(N, L, T_HOP, onsite=eps, removed=rem)]


@pytest.mark.parametrize("prec", [0, 1, 2, 3])
@pytest.mark.parametrize("call", ["conductance_grad", "ldos"])
def test_failed_lead_is_reported(rgflib, cap, call, prec):
    f, ribs = getattr(rgflib, call), ribbons(rgflib)
    E = np.array([0.2, 0.2])
    cap(1)
    for order in (ribs, ribs[::-1]):
        T, out, st = f(order, E, precision=prec, check=False)
        assert (st == rgflib.RGF_ENOCONV).all() and np.isnan(T).all() and (out == 0.0).all()


@pytest.mark.parametrize("call", ["conductance_grad", "ldos"])
def test_good_chains_beside_a_failed_lead(rgflib, cap, call):
    # far outside the bands the decimation needs a few steps, inside about 30:
    # a cap between the two fails one lead of the call
    f, ribs = getattr(rgflib, call), ribbons(rgflib)
    E = np.array([9.5, 0.2, 9.5, 0.2])
    four = [ribs[0], ribs[0], ribs[1], ribs[1]]
    T0, out0, st0 = f(four, E)
    assert (st0 == 0).all()
    _, it = rgflib.lead_selfenergy(N, E[:2], 1e-8, 0)
    assert 0 < it[0] < it[1]
    cap(int(it[0]) + 1)
    T, out, st = f(four, E, check=False)
    assert list(st) == [0, rgflib.RGF_ENOCONV] * 2
    for c in (0, 2):
        assert T[c] == T0[c] and np.array_equal(out[c], out0[c])
        assert np.isnan(T[c + 1]) and (out[c + 1] == 0.0).all()
