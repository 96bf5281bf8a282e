"""The blocked pivot sweep of the FP64 CTA tasks: its integer reciprocal against
exact values, and factor blocks against the oracle at the edges of its blocks
of eight columns (whole, partial, more rows than lanes), with and without
fill-in rows and arrow, and at scales where the reciprocal, the panel products
and the Schur products leave their fast paths."""
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
def kkt():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2511_00946_gb300 as k
    return k


def dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()


def system(N, n, m):
    """I + perturbations: couplings and arrow of 2-norm at most 1/8 (Frobenius),
    so that block Gershgorin bounds the eigenvalues by [1/2, 3/2] (the corner
    grows with N |G|^2)."""
    rng = np.random.default_rng(10 * n + m)

    def small(*shape):
        A = rng.normal(size=shape)
        return A / (8 * np.sqrt((A ** 2).sum(axis=(-2, -1), keepdims=True))) if A.size else A

    S = small(N, n, n)
    D = np.eye(n) + S + S.transpose(0, 2, 1)
    return D, small(N - 1, n, n), small(N, m, n) / np.sqrt(N), np.eye(m)


def test_pivot_reciprocal(kkt):
    """At most 0.52 units in the last place: half a unit from the rounding, and
    the 62-bit value is off by at most 3 2^-62 (three truncations)."""
    import torch
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    out = os.path.join(HERE, "_build")
    os.makedirs(out, exist_ok=True)
    so = os.path.join(out, "librcp_probe.so")
    subprocess.check_call([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-shared", "-Xcompiler", "-fPIC",
                           "-o", so, os.path.join(HERE, "csrc", "rcp_probe.cu")])
    L = ctypes.CDLL(so)
    L.rcp_probe.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_longlong]
    rng = np.random.default_rng(1)
    m = np.concatenate([1.0 + np.arange(4096) / 4096, rng.uniform(1, 2, 20000), [np.nextafter(2, 1), np.nextafter(1, 2)]])
    d = np.concatenate([m, m[:4096] * 2.0 ** rng.integers(-500, 1016, 4096),
                        [0.0, -1.0, np.nan, np.inf, -np.inf, 5e-324, 1e-160, 1.7e308]])
    x = dev(d)
    r, ok = torch.empty_like(x), torch.empty_like(x)
    assert L.rcp_probe(x.data_ptr(), r.data_ptr(), ok.data_ptr(), x.numel()) == 0
    r, ok = r.cpu().numpy(), ok.cpu().numpy()
    assert ok[:-8].all() and not ok[-8:].any()
    for a, b in zip(d[:-8], r[:-8]):
        exact = 1 / Fraction(float(a))
        assert abs(Fraction(float(b)) - exact) <= Fraction(52, 100) * Fraction(float(np.spacing(float(b))))


@pytest.mark.parametrize("scale", [0, 1014, -1000])
@pytest.mark.parametrize("N,n,m,P", [(3, 1, 0, 1), (9, 2, 1, 3), (9, 6, 2, 3), (7, 8, 4, 2), (7, 15, 0, 2), (5, 16, 15, 1)])
def test_small_factor_blocks(kkt, orc, N, n, m, P, scale):
    """As test_factor_blocks, one warp per task."""
    D, E, G, R = system(N, n, m)
    Fo = orc.par_factor(D, E, G, R, P=P)
    s, h = 2.0 ** scale, 2.0 ** (scale // 2)
    hd = kkt.kkt_create(N, n, m, P)
    try:
        kkt.kkt_factor(hd, dev(D * s), dev(E * s), dev(G * s) if m else None, dev(R * s) if m else None)
        F = kkt.kkt_get_factor(hd, N, n, m)
        assert kkt.kkt_get_info(hd)["status"] == 0
    finally:
        kkt.kkt_destroy(hd)
    for k in ("Ld", "Le", "Lw", "Lh", "Lg", "Lr"):
        if F[k].size:
            np.testing.assert_allclose(F[k] / h, Fo[k], rtol=0, atol=1e-13 * max(1.0, np.abs(Fo[k]).max()), err_msg=k)


@pytest.mark.parametrize("scale", [0, 1014, -1000])
@pytest.mark.parametrize("N,n,m,P", [(5, 17, 0, 1), (7, 23, 3, 2), (5, 24, 15, 1), (9, 25, 2, 3), (7, 31, 1, 2),
                                     (7, 32, 8, 2), (5, 33, 0, 2), (7, 40, 5, 2), (5, 41, 4, 1), (5, 48, 15, 2)])
def test_factor_blocks(kkt, orc, N, n, m, P, scale):
    """A well-conditioned Psi (below) scaled by 2^scale (its factor by the
    square root): blocks within 1e-13 of the oracle's, one CTA per task and pairs
    alike. Perturbation of a Cholesky factor: the backward error of either side,
    at most (n + 1) 2^-53 of the scale per level, times the condition number."""
    D, E, G, R = system(N, n, m)
    Fo = orc.par_factor(D, E, G, R, P=P)
    s, h = 2.0 ** scale, 2.0 ** (scale // 2)
    outs = []
    for pairing in (kkt.KKT_PAIR_OFF, kkt.KKT_PAIR_ON):
        hd = kkt.kkt_create(N, n, m, P)
        try:
            kkt.kkt_set_pairing(hd, pairing)
            kkt.kkt_factor(hd, dev(D * s), dev(E * s), dev(G * s) if m else None, dev(R * s) if m else None)
            F = kkt.kkt_get_factor(hd, N, n, m)
            assert kkt.kkt_get_info(hd)["status"] == 0
        finally:
            kkt.kkt_destroy(hd)
        for k in ("Ld", "Le", "Lw", "Lh", "Lg", "Lr"):
            if F[k].size:
                np.testing.assert_allclose(F[k] / h, Fo[k], rtol=0, atol=1e-13 * max(1.0, np.abs(Fo[k]).max()),
                                           err_msg=f"{k} pairing {pairing}")
        outs.append(F)
    for k in outs[0]:
        np.testing.assert_array_equal(outs[0][k], outs[1][k])


def test_breakdown_in_every_block(kkt):
    """A pivot that is not positive in any block of eight columns is reported at
    its stage."""
    N, n, m = 4, 41, 2
    D, E, G, R = system(N, n, m)
    for c in (0, 7, 8, 20, 33, 40):
        B = D.copy()
        B[2, c, c] = -1e3
        h = kkt.kkt_create(N, n, m, 1)
        try:
            kkt.kkt_factor(h, dev(B), dev(E), dev(G), dev(R))
            info = kkt.kkt_get_info(h)
            assert info["status"] == kkt.KKT_ERR_NOT_SPD and info["stage"] == 2 and info["level"] == 1, (c, info)
        finally:
            kkt.kkt_destroy(h)


@pytest.mark.parametrize("n,m", [(17, 0), (20, 3), (32, 8)])
def test_many_systems_and_one(kkt, orc, n, m):
    """More systems than the chip holds tasks of 256 threads (their launches then
    use 128): every system's factor is bitwise that of the persistent schedule and
    of a handle of its own, and the oracle's within the tolerance above."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    N, count, P = 5, 4 * sms + 1, 2
    systems = [system(N, n, m) for _ in range(2)]
    for a in systems[1]:
        a *= 0.75
    pick = [systems[i % 2] for i in range(count)]
    args = [dev(np.concatenate([s[k].ravel() for s in pick])) if k < 2 or m else None for k in range(4)]
    got = []
    for persistent in (False, True):
        h = kkt.kkt_batch_create([N] * count, [n] * count, [m] * count, [P] * count)
        try:
            kkt.kkt_set_persistent(h, persistent)
            kkt.kkt_factor(h, *args)
            got.append({s: kkt.kkt_get_factor(h, N, n, m, s) for s in (0, 1, count - 2, count - 1)})
            assert kkt.kkt_get_info(h)["status"] == 0
        finally:
            kkt.kkt_destroy(h)
    for i in (0, 1):
        D, E, G, R = systems[i]
        h = kkt.kkt_create(N, n, m, P)
        try:
            kkt.kkt_set_pairing(h, kkt.KKT_PAIR_OFF)
            kkt.kkt_factor(h, dev(D), dev(E), dev(G) if m else None, dev(R) if m else None)
            one = kkt.kkt_get_factor(h, N, n, m)
        finally:
            kkt.kkt_destroy(h)
        Fo = orc.par_factor(D, E, G, R, P=P)
        for k in one:
            for g in got:
                for s, F in g.items():
                    if s % 2 == i:
                        np.testing.assert_array_equal(F[k], one[k], err_msg=f"{k} system {s}")
            if k in Fo and one[k].size:
                np.testing.assert_allclose(one[k], Fo[k], rtol=0, atol=1e-13 * max(1.0, np.abs(Fo[k]).max()))


@pytest.mark.parametrize("N,n,m,P", [(7, 17, 1, 2), (9, 31, 0, 3), (9, 32, 8, 3), (7, 33, 2, 2), (9, 45, 5, 2), (7, 48, 15, 1)])
def test_substitution_columns(kkt, orc, N, n, m, P):
    """One to seventeen right-hand sides (a warp takes one or two columns, warps
    without one do the copies): every column is bitwise that of a solve of its own
    and within 1e-13 of the dense solution."""
    D, E, G, R = system(N, n, m)
    b = np.random.default_rng(n).normal(size=(N * n + m, 17))
    h = kkt.kkt_create(N, n, m, P)
    try:
        kkt.kkt_factor(h, dev(D), dev(E), dev(G) if m else None, dev(R) if m else None)
        one = []
        for c in range(17):
            x = dev(b[:, c])
            kkt.kkt_solve(h, x)
            one.append(x.cpu().numpy())
        one = np.stack(one, axis=1)
        for nrhs in (2, 7, 8, 9, 16, 17):
            x = dev(b[:, :nrhs])
            kkt.kkt_solve(h, x)
            # (a plan of one level solves a single column by another kernel)
            if P > 1:
                np.testing.assert_array_equal(x.cpu().numpy(), one[:, :nrhs])
            np.testing.assert_allclose(x.cpu().numpy(), one[:, :nrhs], rtol=0, atol=1e-13 * np.abs(one).max())
    finally:
        kkt.kkt_destroy(h)
    A = orc.assemble_dense(D, E, G, R)
    np.testing.assert_allclose(one, np.linalg.solve(A, b), rtol=0, atol=1e-13 * np.abs(one).max())
