"""kkt_solve_noalloc on the block sizes that a handle runs one warp per task: one
warp up to n = 5, a CTA from n = 6 on, whole and partial blocks of eight columns,
with and without arrow and fill-in rows, against the dense solution; and a pivot
that is not positive."""
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


def system(N, n, m):
    """I + perturbations: couplings and arrow of 2-norm at most 1/8, so that the
    eigenvalues lie in [1/2, 3/2]."""
    rng = np.random.default_rng([N, n, m])

    def small(*shape):
        A = rng.normal(size=shape)
        return A / (8 * np.sqrt((A ** 2).sum(axis=(-2, -1), keepdims=True))) if A.size else A

    S = small(N, n, n)
    return np.eye(n) + S + S.transpose(0, 2, 1), small(N - 1, n, n), small(N, m, n) / np.sqrt(N), np.eye(m)


def args(sys, m):
    return [dev(a) if k < 2 or m else None for k, a in enumerate(sys)]


@pytest.mark.parametrize("N,P", [(4, 1), (23, 4)])
@pytest.mark.parametrize("n,m", [(1, 0), (5, 2), (5, 16), (6, 0), (6, 16), (7, 3), (8, 0), (8, 16), (9, 1), (15, 2), (16, 0),
                                 (16, 16)])
def test_against_the_dense_solution(kkt, orc, N, P, n, m):
    """Within 1e-13 of the largest entry: backward errors of a few n 2^-53 at a
    condition of 3; the same bits twice."""
    A = system(N, n, m)
    b = np.random.default_rng(n + m).normal(size=(N * n + m, 2))
    xs = []
    for _ in range(2):
        x = dev(b)
        kkt.kkt_solve_noalloc(N, n, m, P, *args(A, m), x)
        xs.append(x.cpu().numpy())
    ref = np.linalg.solve(orc.assemble_dense(*A), b)
    np.testing.assert_allclose(xs[0], ref, rtol=0, atol=1e-13 * np.abs(ref).max())
    np.testing.assert_array_equal(xs[0], xs[1])


@pytest.mark.parametrize("n", [5, 6, 12])
def test_breakdown_is_reported(kkt, n):
    import torch
    N, m = 6, 2
    D, E, G, R = system(N, n, m)
    for c in (0, n - 1):
        B = D.copy()
        B[3, c, c] = -1e3
        info = torch.zeros(4, dtype=torch.int32, device="cuda")
        kkt.kkt_solve_noalloc(N, n, m, 1, *args((B, E, G, R), m), dev(np.ones(N * n + m)), info=info)
        assert info.tolist() == [kkt.KKT_ERR_NOT_SPD, 0, 3, 1]
