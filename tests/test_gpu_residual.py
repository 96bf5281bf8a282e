"""The refinement's residual kernel at the edges of its work split: tasks of
eight stages, their rows in groups of 32. The handle holds the factor of one
matrix and refines with another, so that the residual is large: eta of the
first sweep against the definition, and the second sweep's solution, which
every row of the residual enters, against the dense one."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


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


def system(N, n, m, seed):
    """Eigenvalues in about [1/2, 2] (blocks of small norm around the identity)."""
    rng = np.random.default_rng(seed)

    def small(*shape):
        A = rng.normal(size=shape)
        return A / (8 * np.sqrt((A ** 2).sum(axis=(-2, -1), keepdims=True))) if A.size else A

    S = small(N, n, n)
    return np.eye(n) + S + S.transpose(0, 2, 1), small(N - 1, n, n), small(N, m, n) / np.sqrt(N), np.eye(m)


def dense(D, E, G, R):
    N, n, m = D.shape[0], D.shape[1], R.shape[0]
    A = np.zeros((N * n + m, N * n + m))
    for j in range(N):
        s = slice(j * n, (j + 1) * n)
        A[s, s] = D[j]
        if j + 1 < N:
            t = slice((j + 1) * n, (j + 2) * n)
            A[t, s], A[s, t] = E[j], E[j].T
        if m:
            A[N * n:, s], A[s, N * n:] = G[j], G[j].T
    if m:
        A[N * n:, N * n:] = R
    return A


@pytest.mark.parametrize("N,n,m,nrhs", [(1, 1, 0, 1), (1, 33, 3, 1), (7, 6, 4, 2), (8, 16, 5, 1), (9, 12, 8, 3),
                                        (17, 32, 9, 1), (16, 24, 0, 1), (9, 45, 16, 17), (25, 48, 4, 1)])
def test_residual(kkt, N, n, m, nrhs):
    """eta within 1e-5 (its row sums are formed in FP32, each addend at most 2^-20
    low) and the solution within 1e-12: errors of at most (3 n + m) 2^-53 per
    product and solve at a condition number of about 4."""
    A, B = system(N, n, m, 1), system(N, n, m, 2)
    dA, dB = dense(*A), dense(*B)
    b = np.random.default_rng(3).normal(size=(N * n + m, nrhs))
    x1 = np.linalg.solve(dA, b)
    x2 = x1 + np.linalg.solve(dA, b - dB @ x1)
    blocks = lambda S: [dev(v) if v.size else None for v in S]
    h = kkt.kkt_create(N, n, m, 1)
    try:
        kkt.kkt_factor(h, *blocks(A))
        got = []
        for sweeps in (1, 2):
            x = dev(np.zeros_like(b))
            kkt.kkt_solve_refined(h, *blocks(B), dev(b), x, sweeps=sweeps, tol=-1.0)
            got.append(x.cpu().numpy())
            if sweeps == 1:
                eta = float(kkt.kkt_refine_eta(h, 0)[0])
    finally:
        kkt.kkt_destroy(h)
    last = slice(nrhs - 1 - (nrhs - 1) % 16, nrhs)  # eta is that of the last chunk of 16 right-hand sides
    ref = np.abs(b - dB @ x1)[:, last].max() / (np.abs(dB).sum(axis=1).max() * np.abs(x1)[:, last].max() +
                                                np.abs(b)[:, last].max())
    assert abs(eta - ref) <= 1e-5 * ref
    np.testing.assert_allclose(got[0], x1, rtol=0, atol=1e-12 * np.abs(x1).max())
    np.testing.assert_allclose(got[1], x2, rtol=0, atol=1e-12 * np.abs(x2).max())
