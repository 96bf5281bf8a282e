"""Variables in different units. With S a diagonal of powers of two, the Cholesky
factor of S Psi S is S L and the solution for S b is S^-1 x, both exactly: every
rounding of the elimination, of its digit products and of the substitutions
scales with the row and column it belongs to. So every layout has to return the
unscaled answer's bits, S drawn per variable within 2^+-30."""
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


def system(N, n, m, seed=0):
    """I + perturbations: couplings and arrow of 2-norm at most 1/8, so that the
    eigenvalues lie in [1/2, 3/2]."""
    rng = np.random.default_rng([N, n, m, seed])

    def small(*shape):
        A = rng.normal(size=shape)
        return A / (8 * np.sqrt((A ** 2).sum(axis=(-2, -1), keepdims=True))) if A.size else A

    S = small(N, n, n)
    D = np.eye(n) + S + S.transpose(0, 2, 1)
    return D, small(N - 1, n, n), small(N, m, n) / np.sqrt(N), np.eye(m)


def scaled(sys, s, sg):
    """S Psi S: s (N, n) for the stages, sg (m,) for the arrow."""
    D, E, G, R = sys
    return (s[:, :, None] * D * s[:, None, :], s[1:, :, None] * E * s[:-1, None, :],
            sg[None, :, None] * G * s[:, None, :], sg[:, None] * R * sg[None, :])


def units(N, n, m, seed=1):
    rng = np.random.default_rng([seed, N, n, m])
    return 2.0 ** rng.integers(-30, 31, (N, n)), 2.0 ** rng.integers(-30, 31, m)


def args(sys, m):
    return [dev(a) if k < 2 or m else None for k, a in enumerate(sys)]


@pytest.mark.parametrize("N,n,m,P", [(7, 16, 3, 2), (5, 17, 0, 1), (9, 20, 2, 3), (7, 32, 8, 2), (5, 33, 1, 1),
                                     (9, 45, 5, 3), (7, 48, 15, 2)])
def test_factor_and_solutions_of_one_system(kkt, N, n, m, P):
    """One CTA per task, pairs, and caller-owned memory; factor blocks, several
    right-hand sides and the bordered pass."""
    A = system(N, n, m)
    s, sg = units(N, n, m)
    S = np.concatenate([s.ravel(), sg])
    b = np.random.default_rng(n).normal(size=(N * n + m, 2))
    for pairing in (kkt.KKT_PAIR_OFF, kkt.KKT_PAIR_ON):
        got = []
        for M, c in ((A, b), (scaled(A, s, sg), S[:, None] * b)):
            h = kkt.kkt_create(N, n, m, P)
            try:
                kkt.kkt_set_pairing(h, pairing)
                a = args(M, m)
                x, y, z = dev(c), dev(c[:, 0]), dev(c[:, 0])
                kkt.kkt_factor(h, *a)
                F = kkt.kkt_get_factor(h, N, n, m)
                kkt.kkt_solve(h, x)
                kkt.kkt_factor_solve(h, *a, y)
                kkt.kkt_solve_noalloc(N, n, m, P, *a, z)
                assert kkt.kkt_get_info(h)["status"] == 0
                got.append((F, x.cpu().numpy(), y.cpu().numpy(), z.cpu().numpy()))
            finally:
                kkt.kkt_destroy(h)
        (F, *xs), (Fs, *xss) = got
        for i in range(N):
            np.testing.assert_array_equal(s[i][:, None] * F["Ld"][i], Fs["Ld"][i], err_msg=f"stage {i}")
        for x, xsc in zip(xs, xss):
            sc = S if x.ndim == 1 else S[:, None]
            np.testing.assert_array_equal(sc * xsc, x, err_msg=f"pairing {pairing}")


@pytest.mark.parametrize("N,n,m,levels", [(63, 17, 3, [16, 8, 4, 2, 1]), (63, 32, 8, [16, 8, 4, 2, 1]),
                                          (47, 48, 0, [12, 6, 3, 1])])
def test_solutions_on_clusters(kkt, N, n, m, levels):
    """A plan whose deep levels run on clusters."""
    A = system(N, n, m)
    s, sg = units(N, n, m)
    S = np.concatenate([s.ravel(), sg])
    b = np.random.default_rng(n).normal(size=N * n + m)
    got = []
    for M, c in ((A, b), (scaled(A, s, sg), S * b)):
        h = kkt.kkt_create_plan(N, n, m, levels)
        try:
            assert max(kkt.kkt_factor_ctas_per_task(h, l) for l in range(len(levels))) > 2
            a = args(M, m)
            x, y = dev(c), dev(c)
            kkt.kkt_factor(h, *a)
            kkt.kkt_solve(h, x)
            kkt.kkt_factor_solve(h, *a, y)
            assert kkt.kkt_get_info(h)["status"] == 0
            got.append((x.cpu().numpy(), y.cpu().numpy()))
        finally:
            kkt.kkt_destroy(h)
    for x, xs in zip(*got):
        np.testing.assert_array_equal(S * xs, x)


@pytest.mark.parametrize("persistent", [False, True])
@pytest.mark.parametrize("n,m", [(20, 3), (32, 8)])
def test_solutions_of_a_batch(kkt, n, m, persistent):
    """More systems than the chip holds tasks of 256 threads; every other one scaled."""
    import torch
    count, N, P = 4 * torch.cuda.get_device_properties(0).multi_processor_count + 2, 5, 2
    A = system(N, n, m)
    s, sg = units(N, n, m)
    S = np.concatenate([s.ravel(), sg])
    pick = [A, scaled(A, s, sg)]
    b = np.random.default_rng(n).normal(size=N * n + m)
    a = [dev(np.concatenate([pick[i % 2][k].ravel() for i in range(count)])) for k in range(4)]
    x = dev(np.concatenate([b if i % 2 == 0 else S * b for i in range(count)]))
    h = kkt.kkt_batch_create([N] * count, [n] * count, [m] * count, [P] * count)
    try:
        kkt.kkt_set_persistent(h, persistent)
        kkt.kkt_factor(h, *a)
        kkt.kkt_solve(h, x)
        assert kkt.kkt_get_info(h)["status"] == 0
    finally:
        kkt.kkt_destroy(h)
    x = x.cpu().numpy().reshape(count, -1)
    for i in range(count):
        np.testing.assert_array_equal(x[i] if i % 2 == 0 else S * x[i], x[0], err_msg=f"system {i}")


def halves(N, n, m, far, seed=0):
    """Two systems that nothing couples, their variables (and arrow rows) in turn,
    the second one's right-hand side smaller by `far`; both solutions' exact
    values to rounding."""
    D, E, G, R = system(N, n, m, seed)
    own = np.arange(n)[:, None] % 2 == np.arange(n) % 2
    D, E, G = D * own, E * own, G * (np.arange(m)[:, None] % 2 == np.arange(n) % 2)
    rng = np.random.default_rng([2, N, n, m, seed])
    second = np.concatenate([np.tile(np.arange(n) % 2 == 1, N), np.arange(m) % 2 == 1])
    b = rng.normal(size=N * n + m) * np.where(second, far, 1.0)
    return (D, E, G, R), b, second


def check_halves(A, b, second, x, assemble):
    """Each half within 1e-13 of its own largest entry (the tolerance of the
    one-system tests: backward errors of a few n 2^-53 at a condition of 3)."""
    Psi = assemble(*A)
    for part in (second, ~second):
        ref = np.linalg.solve(Psi[np.ix_(part, part)], b[part])
        np.testing.assert_allclose(x[part], ref, rtol=0, atol=1e-13 * np.abs(ref).max())


@pytest.mark.parametrize("far", [1e-8, 1e-20])
@pytest.mark.parametrize("N,n,m,levels", [(9, 12, 2, [3, 1]), (7, 17, 0, [1]), (40, 24, 1, [4, 1]), (40, 32, 8, [1]),
                                          (63, 33, 2, [16, 8, 4, 2, 1]), (63, 48, 14, [16, 8, 4, 2, 1])])
def test_right_hand_side_without_a_common_scale(kkt, orc, N, n, m, levels, far):
    """The bordered pass (kkt_factor_solve) carries the right-hand side as a row of
    the factorization: it has to keep the small half as accurate as the large
    one, in every layout alike."""
    A, b, second = halves(N, n, m, far)
    out = []
    for pairing in (kkt.KKT_PAIR_OFF, kkt.KKT_PAIR_ON, kkt.KKT_PAIR_AUTO):
        h = kkt.kkt_create_plan(N, n, m, levels)
        try:
            kkt.kkt_set_pairing(h, pairing)
            x = dev(b)
            kkt.kkt_factor_solve(h, *args(A, m), x)
            assert kkt.kkt_get_info(h)["status"] == 0
            out.append(x.cpu().numpy())
        finally:
            kkt.kkt_destroy(h)
    check_halves(A, b, second, out[0], orc.assemble_dense)
    for x in out[1:]:
        np.testing.assert_array_equal(x, out[0])


@pytest.mark.parametrize("P", [1, 2])
@pytest.mark.parametrize("n,m", [(17, 2), (32, 8)])
def test_right_hand_sides_of_a_batch(kkt, orc, n, m, P):
    """More systems than the chip holds tasks of 256 threads: as above, and
    bitwise the result of a handle of its own."""
    import torch
    count, N = 4 * torch.cuda.get_device_properties(0).multi_processor_count + 2, 5
    two = [halves(N, n, m, 1e-12, seed) for seed in (0, 1)]
    a = [dev(np.concatenate([two[i % 2][0][k].ravel() for i in range(count)])) for k in range(4)]
    x = dev(np.concatenate([two[i % 2][1] for i in range(count)]))
    h = kkt.kkt_batch_create([N] * count, [n] * count, [m] * count, [P] * count)
    try:
        kkt.kkt_factor_solve(h, *a, x)
        assert kkt.kkt_get_info(h)["status"] == 0
    finally:
        kkt.kkt_destroy(h)
    x = x.cpu().numpy().reshape(count, -1)
    for seed, (A, b, second) in enumerate(two):
        check_halves(A, b, second, x[seed], orc.assemble_dense)
        for i in range(seed, count, 2):
            np.testing.assert_array_equal(x[i], x[seed], err_msg=f"system {i}")
        if P == 1:  # (one system's backward sweep runs in the factor kernel, a batch's in its own)
            continue
        h = kkt.kkt_create(N, n, m, P)
        try:
            y = dev(b)
            kkt.kkt_set_pairing(h, kkt.KKT_PAIR_OFF)
            kkt.kkt_factor_solve(h, *args(A, m), y)
        finally:
            kkt.kkt_destroy(h)
        np.testing.assert_array_equal(x[seed], y.cpu().numpy())


def test_persistent_schedule_of_uneven_blocks(kkt):
    """One-warp and CTA tasks of two levels in one persistent launch of 128-thread
    CTAs (more CTA tasks than the chip holds at 256 threads): bitwise the
    solutions of the launches per level."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    shapes = [(5, 17, 2, 2), (9, 4, 1, 3), (5, 20, 0, 1), (7, 16, 3, 2), (6, 24, 1, 2)]
    pick = [shapes[i % 5] for i in range(10 * sms)]
    sys = {q: system(*q[:3]) for q in shapes}
    a = [dev(np.concatenate([sys[q][k].ravel() for q in pick])) for k in range(4)]
    b = np.random.default_rng(5).normal(size=sum(N * n + m for N, n, m, _ in pick))
    out = []
    for persistent in (False, True):
        h = kkt.kkt_batch_create(*[[q[k] for q in pick] for k in range(4)])
        try:
            kkt.kkt_set_persistent(h, persistent)
            x = dev(b)
            kkt.kkt_factor(h, *a)
            kkt.kkt_solve(h, x)
            assert kkt.kkt_get_info(h)["status"] == 0
            out.append(x.cpu().numpy())
        finally:
            kkt.kkt_destroy(h)
    assert np.isfinite(out[0]).all()
    np.testing.assert_array_equal(out[0], out[1])


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n,m,P", [(17, 2, 1), (32, 0, 2), (33, 3, 1), (41, 1, 2)])
def test_substitutions_of_many_and_few_systems(kkt, n, m, P, precision):
    """More systems than the chip holds CTAs at two per SM: the dense substitution
    kernels, whose every system is bitwise the few systems' of a handle of five."""
    import torch
    many, N = 2 * torch.cuda.get_device_properties(0).multi_processor_count + 5, 7
    sys = [system(N, n, m, seed) for seed in range(5)]
    for nrhs in (1, 3, 9, 16):
        b = np.random.default_rng(nrhs).normal(size=(5, N * n + m, nrhs))
        out = []
        for count in (5, many):
            a = [dev(np.concatenate([sys[i % 5][k].ravel() for i in range(count)])) if k < 2 or m else None for k in range(4)]
            x = dev(np.concatenate([b[i % 5] for i in range(count)]))
            h = kkt.kkt_batch_create([N] * count, [n] * count, [m] * count, [P] * count, precision)
            try:
                kkt.kkt_factor(h, *a)
                if precision == 0:
                    kkt.kkt_solve(h, x)
                else:
                    y = torch.zeros_like(x)
                    kkt.kkt_solve_refined(h, *a, x, y)
                    x = y
                assert kkt.kkt_get_info(h)["status"] == 0
            finally:
                kkt.kkt_destroy(h)
            out.append(x.cpu().numpy().reshape(count, N * n + m, nrhs))
        assert np.isfinite(out[0]).all()
        for i in range(many):
            np.testing.assert_array_equal(out[1][i], out[0][i % 5], err_msg=f"system {i} of {nrhs} columns")
