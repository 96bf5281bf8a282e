"""The tensor-core Schur products (kkt_oz.cuh) on the device against exact
rational arithmetic, at the edges of their 16 x 8 x 16 tiles, with zero rows
and rows that keep their doubles."""
import ctypes
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def probe():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    out = os.path.join(HERE, "_build")
    os.makedirs(out, exist_ok=True)
    so = os.path.join(out, "liboz_probe.so")
    subprocess.check_call([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-shared",
                           "-Xcompiler", "-fPIC", "-o", so, os.path.join(HERE, "csrc", "oz_probe.cu")])
    L = ctypes.CDLL(so)
    vp, i = ctypes.c_void_p, ctypes.c_int
    L.oz_probe.argtypes = [vp, i, i, i, vp, i, vp]

    def run(Z, T):
        rows, n = Z.shape
        z, t = torch.from_numpy(Z).cuda(), torch.from_numpy(T).cuda()
        f = torch.zeros(rows, dtype=torch.int32, device="cuda")
        assert L.oz_probe(z.data_ptr(), n, rows, n, t.data_ptr(), rows, f.data_ptr()) == 0
        return t.cpu().numpy(), f.cpu().numpy()
    return run


@pytest.mark.parametrize("rows,n", [(1, 1), (7, 5), (8, 16), (16, 17), (17, 31), (24, 32), (33, 33), (40, 48)])
def test_products_exact_up_to_one_rounding(probe, rows, n):
    """|T' - (T - sum)| <= 2^-53 (|sum| + |T'|) + n 2^-57.9 2^(fa + fb) (the bound
    of test_oz_cpu.py and the subtraction's rounding)."""
    rng = np.random.default_rng(100 * rows + n)
    Z = rng.normal(size=(rows, n)) * 10.0 ** rng.uniform(-3, 3, size=(rows, 1))
    Z[:, n // 2:] *= 1e-3
    if rows > 3:
        Z[2] = 0.0
        Z[3] = -(256.0 / 511.0)  # largest digits everywhere
    T = rng.normal(size=(rows, rows))
    out, f = probe(Z.copy(), T.copy())
    for a in range(rows):
        for b in range(a + 1):
            s = sum((Fraction(float(x)) * Fraction(float(y)) for x, y in zip(Z[a], Z[b])), Fraction(0))
            err = abs(Fraction(float(out[a, b])) - (Fraction(float(T[a, b])) - s))
            bound = (abs(s) + abs(Fraction(float(out[a, b])))) / 2**53 + \
                n * Fraction(2.0 ** -57.9) * Fraction(2) ** (int(f[a]) + int(f[b]))
            assert err <= bound, (a, b, float(err), float(bound))
    iu = np.triu_indices(rows, 1)
    np.testing.assert_array_equal(out[iu], T[iu])  # the upper triangle is not touched


def test_rows_outside_the_split_take_fp64(probe):
    """Infinities, NaN and extreme scales: the FP64 products, and no effect on
    the other rows."""
    rng = np.random.default_rng(9)
    rows, n = 20, 12
    Z = rng.normal(size=(rows, n))
    ref, _ = probe(Z.copy(), np.zeros((rows, rows)))
    W = Z.copy()
    W[5, 3], W[9, 0], W[13] = np.nan, np.inf, Z[13] * 1e160
    out, f = probe(W.copy(), np.zeros((rows, rows)))
    assert (f[[5, 9, 13]] == 1 << 20).all() and (np.delete(f, [5, 9, 13]) < 401).all()
    keep = [r for r in range(rows) if r not in (5, 9, 13)]
    low = np.tril(np.ones((rows, rows), bool))
    m = np.ix_(keep, keep)
    np.testing.assert_array_equal(out[m][low[m]], ref[m][low[m]])
    assert np.isnan(out[5, :6]).all() and np.isnan(out[6:, 5]).all()
    assert not np.isfinite(out[9, :5]).any()
    x = -(W[13] @ W[0])
    assert abs(out[13, 0] - x) <= n * 2.0 ** -52 * float(np.abs(W[13]) @ np.abs(W[0]))
