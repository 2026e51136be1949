"""The Cholesky factor of -sym(M) and its inverse for one block of orbitals (n <= 32), on matrices
handed over exactly: W_j is 1 at one grid point and Psi holds -A / dV there (dV = 1/8), so
M = -A, and xi = W L^{-T} shows the entries of L^{-1} themselves."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def exx():
    import paper_2501_16572_gb300 as m
    m.load()
    assert torch.cuda.is_available()
    return m


def _inverse_factor(exx, A):
    """L^{-1} of A = L L^T as an FP64 plan computes it."""
    n = len(A)
    p = exx.Plan((8, 8, 8), 0.5, (1, 1, 0), 12, exx.EXX_KERNEL_ERFC, 0.106)
    at = 3 * np.arange(n) + 1
    psi, W = np.zeros((n, p.N)), np.zeros((n, p.N))
    psi[:, at] = -8.0 * A
    W[np.arange(n), at] = 1.0
    xi = p.ace_build(torch.from_numpy(psi).cuda(), torch.from_numpy(W).cuda())
    return xi.cpu().numpy()[:, at]


@pytest.mark.parametrize("n", [2, 32, 64])
def test_factor_entries_are_correctly_rounded_quotients(exx, n):
    """Blocks [[p^2, q], [q, 2^60]]: L = [[p, q / p], [., 2^30]] (the second root rounds to 2^30 as
    (q / p)^2 < 2^6), so the inverse's lower entry is -(q / p)(1 / p) 2^-30, two roundings in it."""
    rng = np.random.default_rng(n)
    root = rng.choice([3.0, 7.0, 11.0, 13.0, 19.0, 49.0], n // 2)
    q = np.floor(rng.uniform(0.1, 7.9, n // 2) * root)
    A, X = np.zeros((n, n)), np.zeros((n, n))
    for b in range(n // 2):
        i = 2 * b
        A[i:i + 2, i:i + 2] = [[root[b] ** 2, q[b]], [q[b], 2.0 ** 60]]
        X[i, i], X[i + 1, i + 1] = 1.0 / root[b], 2.0 ** -30
        X[i + 1, i] = -((q[b] / root[b]) * (1.0 / root[b])) * 2.0 ** -30
    got = _inverse_factor(exx, A)
    assert np.array_equal(got, X)


@pytest.mark.parametrize("n", [1, 7, 8, 9, 15, 16, 17, 31, 32, 33])
def test_one_block_sizes(exx, n):
    """Around the widths of the one-block form; A = C C^T + n I is conditioned below 10, so both factors
    agree to n rounding errors of 2.2e-16 times that: 1e-12.  A negative last diagonal entry is
    the pivot reported."""
    rng = np.random.default_rng(n)
    C = rng.standard_normal((n, n))
    A = C @ C.T + n * np.eye(n)
    got = _inverse_factor(exx, A)
    ref = np.linalg.inv(np.linalg.cholesky(A))
    assert np.linalg.norm(got - ref) <= 1e-12 * np.linalg.norm(ref)
    assert not np.triu(got, 1).any()
    A[n - 1, n - 1] = -1.0
    with pytest.raises(exx.ExxError) as e:
        _inverse_factor(exx, A)
    assert e.value.status == exx.EXX_ERR_NOT_POSDEF and e.value.pivot == n - 1


def test_one_block_is_one_launch(exx):
    """Two kernels for M, one for the factor and its inverse, one for xi."""
    p = exx.Plan((8, 8, 8), 0.5, (1, 1, 0), 12, exx.EXX_KERNEL_ERFC, 0.106)
    g = torch.Generator(device="cuda").manual_seed(1)
    psi = torch.randn((32, p.N), dtype=torch.float64, device="cuda", generator=g)
    p.ace_build(psi, -psi)
    assert p.launch_count() == 4
