"""The tensor-core GEMM of the ACE products at the edges of its tiles (128 rows, 96 columns, 32-
and 320-long steps of k, unaligned and padded columns), on inputs whose products it must give
exactly: entries are integers below 2^7 (times a power of two per column), which leaves the
first digit and a half in the second, so that the FP32 combination of the digit levels has
nothing to round and all sums stay far below 2^48.  What is left is the factor dV, held to 48
bits, and one rounding to FP64: 1e-13 per entry."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-13
SIZES = [
    (1, 1, (2, 2, 2), 0),            # one block of k, one row, one column
    (16, 7, (5, 7, 9), 0),           # 315 grid points: one chunk, not a whole one
    (17, 16, (8, 8, 5), 3),          # exactly 320 points, columns 8-byte aligned only
    (33, 97, (7, 23, 2), 1),         # 322 points; two column tiles
    (128, 96, (20, 20, 20), 2),      # whole tiles, 16-byte aligned padded columns
    (129, 193, (21, 19, 17), 0),     # odd column length: alternate columns unaligned
    (321, 40, (24, 24, 24), 0),      # the short contraction crosses a chunk
    (70, 3, (48, 48, 52), 5),        # many k splits
]


@pytest.fixture(scope="module")
def exx():
    import paper_2501_16572_gb300 as m
    m.load()
    assert torch.cuda.is_available()
    return m


def _plan(exx, n):
    p = exx.Plan(n, 0.3, (1, 1, 0), 12, exx.EXX_KERNEL_ERFC, 0.106)
    p.set_precision(exx.EXX_PREC_BF16X7)
    return p


def _ints(m, N, pad, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    buf = torch.randint(-127, 128, (m, N + pad), device="cuda", generator=g).double()
    buf[:, : N // 7] = 0.0
    return buf[:, :N]


def _close(got, ref):
    assert torch.isfinite(got).all()
    assert bool(((got - ref).abs() <= TOL * ref.abs()).all())


@pytest.mark.parametrize("n, nphi, grid, pad", SIZES)
def test_gram_product_is_exact(exx, n, nphi, grid, pad):
    """M = dV Psi^T W: both operands contiguous along k (the grid)."""
    p = _plan(exx, grid)
    psi, W = _ints(n, p.N, pad, n), _ints(n, p.N, pad, n + 1)
    psi *= torch.exp2((torch.arange(n, device="cuda") % 81).double() - 40.0)[:, None]
    M = torch.full((n, n), float("nan"), dtype=torch.float64, device="cuda")
    try:
        p.ace_build(psi, W, M=M)
    except exx.ExxError as e:   # M is written before its factor is found not to exist
        assert e.status == exx.EXX_ERR_NOT_POSDEF
    _close(M.mT, p.dV * (psi @ W.mT))


@pytest.mark.parametrize("n, nphi, grid, pad", SIZES)
def test_ace_apply_is_exact(exx, n, nphi, grid, pad):
    """-dV xi (xi^T Phi) with one grid point per column of Phi: the second product contracts the
    orbitals, its operands contiguous along the grid."""
    p = _plan(exx, grid)
    xi = _ints(n, p.N, pad, n)
    at = (torch.arange(nphi, device="cuda") * 7919) % p.N
    phi = torch.zeros((nphi, p.N + pad), dtype=torch.float64, device="cuda")[:, :p.N]
    scale = torch.exp2((torch.arange(nphi, device="cuda") % 21).double() - 10.0)
    phi[torch.arange(nphi, device="cuda"), at] = scale
    out = torch.full((nphi, p.N + pad), float("nan"), dtype=torch.float64, device="cuda")[:, :p.N]
    p.ace_apply(xi, phi, out)
    _close(out, -p.dV * ((xi[:, at] * scale).mT @ xi))


@pytest.mark.parametrize("n", [5, 97, 130])
def test_ace_build_triangular_product(exx, n):
    """xi = W L^{-T}: column tiles of the triangular factor stop at their last column.  An operand
    entry is rounded within 2^-30 of its row's largest (below 5 standard deviations here), so
    two operands twice in a row stay below 4 * 5 * 2^-30 = 2e-8 of the norm."""
    p = _plan(exx, (16, 15, 14))
    g = torch.Generator(device="cuda").manual_seed(n)
    psi = torch.randn((n, p.N), dtype=torch.float64, device="cuda", generator=g)
    W = -psi * (0.5 + torch.rand((1, p.N), dtype=torch.float64, device="cuda", generator=g))
    xi = p.ace_build(psi, W)
    low = torch.linalg.cholesky(-p.dV * (psi @ W.mT))
    ref = torch.linalg.solve_triangular(low, W, upper=False)
    assert float(torch.linalg.norm(xi - ref) / torch.linalg.norm(ref)) < 2e-8
