"""The tensor-core contractions of a step on their own, in double-float and binary64:
C = op(A) B and the rank-b update of the inverse, at the edges of their tiles (128
rows, 32 and 16 columns a pass, 8 inner entries a chunk, 128 a group, panels of 1 to
16), entry by entry against extended precision.

Bounds per real part, k the inner entries, a and b the largest entries of the row of
A and the column of B.  An operand is within 0.52 2^-55 of its scale (below 2 a) and
the digit levels left out below 6.1 2^-56 of the scales' product, over 2 k real
terms: together below 2^-49.9 k a b.  Binary64 adds its rounding, 2^-53 of a sum of at
most 2 k a b for each group of 128 and their sum; double-float at most four units of
2^-48 of it."""
import ctypes as C
import os
import shutil
import subprocess
from pathlib import Path

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
HERE = Path(__file__).resolve().parent
PKG = HERE.parent / "paper_1107_5300_gb300"


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    import torch  # noqa: F401  (the CUDA runtime's context)
    from paper_1107_5300_gb300.build import ARCH, FLAGS, nvcc
    out = tmp_path_factory.mktemp("dense") / "dense_check.so"
    subprocess.run([nvcc(), *ARCH, *FLAGS, "-shared", "-o", str(out), str(HERE / "kernels" / "dense_check.cu"),
                    "-lcudart"], check=True)
    so = C.CDLL(str(out))
    so.check_product.argtypes = [C.c_int] * 5 + [C.c_void_p, C.c_int] * 3
    so.check_update.argtypes = [C.c_int] * 3 + [C.c_void_p] * 3 + [C.c_int] * 4
    return so


def pack(a, f64):
    """(what the kernel reads, 16 bytes an entry; the values it stands for in extended precision)"""
    import torch
    if f64:
        raw, val = a.view(np.float64), a.astype(np.clongdouble)
    else:
        x = a.view(np.float64).reshape(*a.shape, 2)
        hi = x.astype(np.float32)
        lo = (x - hi).astype(np.float32)
        raw = np.stack([hi, lo], -1)
        v = hi.astype(np.longdouble) + lo
        val = v[..., 0] + 1j * v[..., 1]
    return torch.from_numpy(np.ascontiguousarray(raw)).cuda(), val


def unpack(t, shape, f64):
    x = t.cpu().numpy()
    if f64:
        v = x.reshape(*shape, 2).astype(np.longdouble)
    else:
        x = x.reshape(*shape, 2, 2).astype(np.longdouble)
        v = x[..., 0] + x[..., 1]
    return v[..., 0] + 1j * v[..., 1]


def random(rng, shape, wide):
    a = rng.standard_normal(shape) + 1j * rng.standard_normal(shape)
    if wide:                                    # entries of one row over 20 decades, zeros, exact powers of two
        a *= 10.0 ** rng.uniform(-20, 0, shape)
        a[rng.random(shape) < 0.1] = 0.0
        a[rng.random(shape) < 0.1] = 0.5
    return a


def amax(v, axis):
    return np.maximum(np.abs(v.real), np.abs(v.imag)).max(axis=axis)


def unit(f64, groups=1):
    return 2.0 ** -49.9 + 2 * ((groups + 1) * 2.0 ** -53 if f64 else 4 * groups * 2.0 ** -48)


def worst(d, bound):
    return float((np.maximum(np.abs(d.real), np.abs(d.imag)) / np.maximum(bound, 1e-300)).max())


@pytest.mark.parametrize("f64", [0, 1])
@pytest.mark.parametrize("wide", [0, 1])
@pytest.mark.parametrize("ta,m,n,k", [(0, 1, 1, 1), (0, 33, 17, 9), (1, 31, 128, 16), (0, 32, 129, 17), (0, 64, 127, 128),
                                      (1, 65, 16, 129), (0, 7, 131, 250), (0, 246, 123, 123)])
def test_product(lib, ta, m, n, k, wide, f64):
    import torch
    rng = np.random.default_rng(m + 1000 * n + k)
    lda, ldb, ldc = (m if ta else k) + 3, n + 1, n + 2
    a, b = random(rng, (k if ta else m, lda), wide), random(rng, (k, ldb), wide)
    ra, va = pack(a, f64)
    rb, vb = pack(b, f64)
    rc = torch.zeros(m * ldc * 2 if f64 else m * ldc * 4, dtype=torch.float64 if f64 else torch.float32, device="cuda")
    torch.cuda.synchronize()
    assert lib.check_product(f64, ta, m, n, k, ra.data_ptr(), lda, rb.data_ptr(), ldb, rc.data_ptr(), ldc) == 0
    va, vb = (va[:, :m].T if ta else va[:, :k]), vb[:, :n]
    got = unpack(rc, (m, ldc), f64)
    assert (got[:, n:] == 0).all()
    bound = unit(f64, -(-k // 128)) * k * np.outer(amax(va, 1), amax(vb, 0))
    assert worst(got[:, :n] - va @ vb, bound) < 1.0


@pytest.mark.parametrize("f64", [0, 1])
@pytest.mark.parametrize("bb", [1, 2, 7, 8, 9, 15, 16])
@pytest.mark.parametrize("M,N", [(1, 17), (127, 1), (128, 15), (128, 16), (33, 112), (64, 33)])
def test_rank_update(lib, bb, M, N, f64):
    rng = np.random.default_rng(bb + 100 * M + N)
    for r0, j0 in ((0, 0), (3, N // 2)):
        K = max(r0 + M, N + bb, j0 + bb)
        c, x, w = random(rng, (bb, K), 0), random(rng, (bb, K), 0), random(rng, (K, K), 0)
        (rc, vc), (rx, vx), (rw, vw) = pack(c, f64), pack(x, f64), pack(w, f64)
        assert lib.check_update(f64, K, bb, rc.data_ptr(), rx.data_ptr(), rw.data_ptr(), r0, M, j0, N) == 0
        got = unpack(rw, (K, K), f64)
        cols = [l if l < j0 else l + bb for l in range(N)]
        ref, bound = vw.copy(), np.zeros((K, K))
        rows = slice(r0, r0 + M)
        ref[cols, rows] -= (vx[:, cols].T @ vc[:, rows])
        bound[cols, rows] = unit(f64) * bb * np.outer(amax(vx[:, cols], 0), amax(vc[:, rows], 0))
        bound[cols, rows] += (2.0 ** -52 if f64 else 2.0 ** -46) * np.abs(vw[cols, rows])
        untouched = np.ones((K, K), bool)
        untouched[np.ix_(cols, range(r0, r0 + M))] = False
        assert np.array_equal(got[untouched], vw[untouched])
        assert worst((got - ref)[cols, rows], bound[cols, rows]) < 1.0
