"""The sums of the ACE products are FP64 in every mode: chunks of 320 grid points of very different
size, sums that need 53 bits, the factor dV in full.  Entries are integers below 2^7 times a power
of two per chunk, whose chunk sums the digits give exactly, and every partial sum fits 53 bits, so
any order of FP64 additions gives the same bits."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
CHUNK = 320


@pytest.fixture(scope="module")
def exx():
    import paper_2501_16572_gb300 as m
    m.load()
    assert torch.cuda.is_available()
    return m


def _plan(exx, n, h):
    p = exx.Plan(n, h, (1, 1, 0), 12, exx.EXX_KERNEL_ERFC, 0.106)
    p.set_precision(exx.EXX_PREC_BF16X7)
    return p


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


# 9, 40: narrow and wide tiles; (8, 8, 20): four chunks in one k split; (24, 24, 24): many splits
@pytest.mark.parametrize("n, grid", [(9, (8, 8, 20)), (40, (8, 8, 20)), (130, (10, 8, 24)), (20, (24, 24, 24))], ids=str)
def test_chunk_sums_hold_53_bits(exx, n, grid):
    """Two chunks in full size (below 2^24 together), the others 2^-28 of it: 52 bits."""
    p = _plan(exx, grid, 0.5)
    psi, W = _ints(n, p.N, 1), _ints(n, p.N, 2)
    chunk = torch.arange(p.N, device="cuda") // CHUNK
    psi *= torch.where((chunk == 1) | (chunk == 2), 1.0, 2.0 ** -28)
    ref = p.dV * (psi @ W.mT)   # dV = 1/8
    assert torch.equal(_gram(exx, p, psi, W), ref)


@pytest.mark.parametrize("n, grid", [(9, (8, 8, 20)), (40, (8, 8, 20)), (20, (24, 24, 24))], ids=str)
@pytest.mark.parametrize("small", [-90, -400])
def test_small_chunks_count_beside_large_ones(exx, n, grid, small):
    """Psi is large where W vanishes, W where Psi does; the product comes from the chunks where both
    are small (2^-180 and 2^-800 of the largest products)."""
    p = _plan(exx, grid, 0.5)
    psi, W = _ints(n, p.N, 3), _ints(n, p.N, 4)
    chunk = torch.arange(p.N, device="cuda") // CHUNK
    scale = torch.tensor([1.0, 0.0, 2.0 ** small], dtype=torch.float64, device="cuda")
    psi *= scale[torch.clamp(chunk, max=2)]
    W *= scale[torch.where(chunk < 2, 1 - chunk, 2)]
    ref = p.dV * (psi @ W.mT)
    assert bool((ref != 0).any())
    assert torch.equal(_gram(exx, p, psi, W), ref)


@pytest.mark.parametrize("n, grid", [(9, (8, 8, 20)), (40, (8, 8, 20)), (130, (5, 8, 24))], ids=str)
def test_the_volume_factor_is_a_full_double(exx, n, grid):
    """dV = h^3 times an integer: one rounding, in both products."""
    p = _plan(exx, grid, 0.3)
    psi, W = _ints(n, p.N, 5), _ints(n, p.N, 6)
    dV = 0.3 * 0.3 * 0.3   # as the library forms it
    assert torch.equal(_gram(exx, p, psi, W), dV * (psi @ W.mT))
    at = (torch.arange(n, device="cuda") * 7919) % p.N
    phi = torch.zeros((n, p.N), dtype=torch.float64, device="cuda")
    phi[torch.arange(n, device="cuda"), at] = 1.0
    assert torch.equal(p.ace_apply(psi, phi), -dV * (psi[:, at].mT @ psi))
