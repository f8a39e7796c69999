"""Accuracy of the LDOS of ordinary disordered ribbons away from E = 0 in double-float:
the blocks it is read from may not lose digits against a column-by-column sweep. The
geometric mean over 16 chains of the largest error, relative to the largest LDOS of the
chain, stays below 64 units of the working precision (2^-48; a column-wise sweep has
about 30, the form that adds G_c1c2 W^T gl to gl about 150)."""
import numpy as np
import pytest

from oracle import ldos as oldos
from oracle import modes

pytestmark = pytest.mark.gpu
T_HOP = -2.7


@pytest.mark.parametrize("prec", [1, 2])
def test_mean_error_in_double_float(rgflib, prec):
    err = []
    for s in range(16):
        rng = np.random.default_rng(4000 + s)
        N, L = int(rng.integers(30, 60)), int(rng.integers(3, 8))
        eps, E = rng.uniform(-0.2, 0.2, (L, 2 * N)), float(rng.uniform(0.3, 1.2) * rng.choice([-1, 1]))
        ref = oldos.ldos(N, L, E, 1e-8, 1e-8, T_HOP, eps, sig=modes.self_energies(N, E, 1e-8, T_HOP))
        _, rho, st = rgflib.ldos([rgflib.Ribbon(N, L, T_HOP, onsite=eps)], np.array([E]), 1e-8, 1e-8, prec)
        assert st[0] == 0
        err.append(np.abs(rho[0] - ref).max() / np.abs(ref).max())
    assert np.exp(np.log(err).mean()) < 64 * 2.0 ** -48, err
