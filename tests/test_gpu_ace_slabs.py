"""The ACE products cut into several slabs of rows and of the contraction, as large operands are: the
budget of the digit planes lowered to a few MB, on integer inputs whose products are exact, and
workspaces that do not fit."""
import ctypes

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
MB = 1 << 20


@pytest.fixture(scope="module")
def exx():
    import paper_2501_16572_gb300 as m
    m.load()
    assert torch.cuda.is_available()
    return m


def _plan(exx, n):
    p = exx.Plan(n, 0.5, (1, 1, 0), 12, exx.EXX_KERNEL_ERFC, 0.106)   # dV = 1/8
    p.set_precision(exx.EXX_PREC_BF16X7)
    return p


def _limits(exx, p, budget=0, cap=0):
    f = exx.load().exx_debug_limits
    f.argtypes = [ctypes.c_void_p, ctypes.c_long, ctypes.c_long]
    assert f(p._h, budget, cap) == 0


def _ints(m, N, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randint(-127, 128, (m, N), device="cuda", generator=g).double()


def _gram(exx, p, psi, W):
    M = torch.full((psi.shape[0],) * 2, float("nan"), dtype=torch.float64, device="cuda")
    try:
        p.ace_build(psi, W, M=M)
    except exx.ExxError as e:   # M is written before its factor is found not to exist
        assert e.status == exx.EXX_ERR_NOT_POSDEF
    return M.mT


# 77 chunks, the last of 256 points; 20 MB: slabs of 20, 20, 20 and 17 chunks with k splits;
# 3 MB: two splits; 1 MB: one chunk a slab, each added to D
@pytest.mark.parametrize("n", [3, 20, 130])
@pytest.mark.parametrize("budget", [20 * MB, 3 * MB, MB])
def test_slabs_of_the_contraction(exx, n, budget):
    p = _plan(exx, (32, 32, 24))
    psi, W = _ints(n, p.N, 1), _ints(n, p.N, 2)
    _limits(exx, p, budget)
    assert torch.equal(_gram(exx, p, psi, W), p.dV * (psi @ W.mT))


# -dV xi (xi^T Phi): rows of the second product in slabs, the last one short; 330 orbitals: two chunks
@pytest.mark.parametrize("n, nphi", [(7, 40), (130, 5), (330, 49)])
@pytest.mark.parametrize("budget", [3 * MB, MB // 2])
def test_slabs_of_the_rows(exx, n, nphi, budget):
    p = _plan(exx, (24, 23, 22))
    xi = _ints(n, p.N, 3)
    at = (torch.arange(nphi, device="cuda") * 7919) % p.N
    phi = torch.zeros((nphi, p.N), dtype=torch.float64, device="cuda")
    phi[torch.arange(nphi, device="cuda"), at] = 1.0
    _limits(exx, p, budget)
    assert torch.equal(p.ace_apply(xi, phi), -p.dV * (xi[:, at].mT @ xi))


@pytest.mark.parametrize("n, budget", [(40, MB), (330, 8 * MB), (330, 3 * MB)])
def test_triangular_product_over_slabs(exx, n, budget):
    """xi = W L^{-T} row slab by row slab (and, at 3 MB, chunk by chunk): the same sums."""
    p = _plan(exx, (16, 15, 18))
    g = torch.Generator(device="cuda").manual_seed(n)
    psi = torch.randn((n, p.N), dtype=torch.float64, device="cuda", generator=g)
    W = -psi * (0.5 + torch.rand((1, p.N), dtype=torch.float64, device="cuda", generator=g))
    # M of integers in whole, so that both builds factor the same matrix
    psi = torch.round(16 * psi)
    W = torch.round(16 * W)
    W = W - 100000.0 * psi
    ref = p.ace_build(psi, W)
    _limits(exx, p, budget)
    assert torch.equal(p.ace_build(psi, W), ref)


def test_products_run_in_smaller_slabs_where_memory_is_short(exx):
    p = _plan(exx, (32, 32, 24))
    psi, W = _ints(130, p.N, 1), _ints(130, p.N, 2)
    ref = p.dV * (psi @ W.mT)
    _limits(exx, p, cap=8 * MB)   # one slab takes 80 MB
    assert torch.equal(_gram(exx, p, psi, W), ref)
    _limits(exx, p, cap=1000)
    with pytest.raises(exx.ExxError) as e:
        p.ace_apply(psi, W)
    assert e.value.status == exx.EXX_ERR_OOM
    _limits(exx, p)
    assert torch.equal(_gram(exx, p, psi, W), ref)
