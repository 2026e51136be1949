"""The direct forms of the BF16X7 passes against the older forms, which a hand-set tuning still
selects: the same digits, products and roundings, so every bit of the result is the same, at the
edges of their layouts (axis lengths around multiples of 8, 16 and 32, the switches between three,
two and one tile groups, resident and streamed matrices, staged and unstaged slices, unaligned
rows).  The pair blocks are held fixed, so that the sums run in the same order.

The other kernels of the exchange path that take new routes by size: the FP64 passes on even and odd
axes, the complex axis contractions, and the blocked Cholesky with its doubling inverse."""
import ctypes

import numpy as np
import pytest

import oracle
import synth
from tests import pinmath as pm

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def exx():
    import paper_2501_16572_gb300 as m
    m.load()
    assert torch.cuda.is_available()
    return m


GRIDS = [
    ((2, 3, 2), (0, 1, 0)), ((5, 2, 7), (0, 0, 0)),          # fewer points than a unit of 8
    ((16, 16, 16), (1, 1, 0)), ((17, 15, 33), (0, 1, 0)),    # one 16-step, one more
    ((24, 24, 24), (0, 0, 0)), ((31, 33, 48), (1, 0, 0)),
    ((42, 43, 49), (0, 1, 0)),                               # three / two tile groups; z past 48
    ((48, 47, 64), (1, 0, 1)), ((49, 48, 65), (0, 0, 1)),    # z past 64: one group of 512
    ((64, 64, 96), (1, 1, 0)), ((65, 33, 97), (0, 0, 0)),    # z past 96: streamed
    ((72, 72, 144), (1, 1, 0)), ((80, 78, 145), (1, 0, 0)),  # z past 144: digits in shared memory
    ((90, 96, 17), (0, 0, 0)), ((97, 97, 9), (1, 1, 0)),
    ((117, 117, 30), (1, 1, 0)), ((128, 128, 5), (1, 1, 0)),  # slices too wide for staging
    ((110, 100, 20), (0, 1, 0)),                             # two matrices that do not stay resident
    ((20, 20, 208), (1, 1, 0)),
]


@pytest.mark.parametrize("n, bc", GRIDS, ids=lambda v: "x".join(map(str, v)))
def test_direct_forms_keep_every_bit(exx, n, bc):
    g = torch.Generator(device="cuda").manual_seed(sum(n))
    N = n[0] * n[1] * n[2]
    psi = torch.randn((5, N), dtype=torch.float64, device="cuda", generator=g)
    psi *= torch.exp(6 * torch.rand((1, N), dtype=torch.float64, device="cuda", generator=g) - 5)
    f = torch.tensor([2.0, 1.7, 0.3], dtype=torch.float64, device="cuda")
    p = exx.Plan(n, 0.3, bc, 12, exx.EXX_KERNEL_ERFC, 0.106)
    p.set_precision(exx.EXX_PREC_BF16X7)
    p.set_tuning(pairs_per_batch=64, block_orbitals=8)
    new = p.apply(psi[:3], f, psi)
    p.set_tuning(pairs_per_batch=64, block_orbitals=8, z_block=-16, z_buffers=2, pipeline=0)
    old = p.apply(psi[:3], f, psi)
    torch.cuda.synchronize()
    assert torch.isfinite(new).all() and float(new.abs().max()) > 0
    assert torch.equal(new, old)


@pytest.mark.parametrize("n, bc", [((2, 3, 4), (0, 1, 0)), ((5, 33, 2), (1, 0, 0)), ((17, 9, 40), (0, 0, 1)),
                                   ((7, 18, 6), (1, 1, 1))], ids=str)
def test_fp64_folded_passes_match_oracle(exx, n, bc):
    """Sums of at most 40 products four times over: far below 1e-12."""
    s = synth.small_system(n=n, h=0.4, bc=bc, n_orb=4, kernel=1, omega=0.106, seed=5)
    ref = oracle.Plan(s.n, s.h, s.bc, s.fd_order, s.kernel, s.omega).exx_apply(s.psi[:3], s.f[:3], s.psi)
    p = exx.Plan(s.n, s.h, s.bc, s.fd_order, s.kernel, s.omega)
    psi, f = torch.from_numpy(s.psi).cuda(), torch.from_numpy(s.f[:3].copy()).cuda()
    assert pm.rel(p.apply(psi[:3], f, psi).cpu().numpy(), ref) < 1e-12


@pytest.mark.parametrize("n, bc, no, ni", [((2, 3, 4), (1, 1, 0), 1, 1), ((5, 34, 3), (1, 1, 1), 2, 3),
                                           ((33, 4, 6), (0, 1, 1), 3, 2), ((6, 7, 36), (1, 0, 1), 2, 5)], ids=str)
def test_complex_axes_match_fp64(exx, n, bc, no, ni):
    """Against dense complex eigenbases in torch; sums of at most 36 products six times over."""
    theta = [0.7, -1.3, 2.1]
    g = torch.Generator(device="cuda").manual_seed(sum(n))
    N = n[0] * n[1] * n[2]
    z = torch.randn((no + ni, N), dtype=torch.complex128, device="cuda", generator=g)
    occ, phi = z[:no].contiguous(), z[no:].contiguous()
    f = torch.rand(no, dtype=torch.float64, device="cuda", generator=g)
    p = exx.Plan.bloch(n, 0.3, bc, theta, 12, exx.EXX_KERNEL_ERFC, 0.106)
    got = p.apply_complex(occ, f, phi)
    orc = oracle.CPlan(n, 0.3, bc, 12, 1, 0.106, theta=tuple(theta))
    ref = orc.exx_apply(occ.cpu().numpy(), f.cpu().numpy(), phi.cpu().numpy())
    assert pm.rel(got.cpu().numpy(), ref) < 1e-12


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 64, 65, 96, 129, 200])
def test_cholesky_and_doubling_inverse(exx, n):
    """xi = W L^{-T} of an FP64 plan; -M is close to the identity, so rounding stays near 1e-15 n."""
    p = exx.Plan((12, 11, 10), 0.4, (1, 1, 0), 12, exx.EXX_KERNEL_ERFC, 0.106)
    rng = np.random.default_rng(n)
    q, _ = np.linalg.qr(rng.standard_normal((p.N, n)))
    psi = torch.from_numpy(np.ascontiguousarray(q.T) / np.sqrt(p.dV)).cuda()
    W = -psi * (0.8 + 0.4 * torch.rand((1, p.N), dtype=torch.float64, device="cuda"))
    xi = p.ace_build(psi, W)
    low = torch.linalg.cholesky(-p.dV * (psi @ W.mT))
    ref = torch.linalg.solve_triangular(low, W, upper=False)
    assert float(torch.linalg.norm(xi - ref) / torch.linalg.norm(ref)) < 1e-12


def test_a_warp_gives_up_a_wait_as_one(exx):
    """Half of the lanes run out of time, half see the barrier complete: none may go on alone."""
    L = exx.load()
    L.exx_debug_wait_warp.argtypes = [ctypes.POINTER(ctypes.c_uint)]
    on = ctypes.c_uint(1)
    assert L.exx_debug_wait_warp(ctypes.byref(on)) == 0
    assert on.value == 0


def test_complex_axes_by_one_output_or_four(exx):
    """Few pencils take one output a thread, many four: the same sums, so the same bits."""
    n, no, ni = (24, 20, 22), 6, 20
    g = torch.Generator(device="cuda").manual_seed(7)
    N = n[0] * n[1] * n[2]
    z = torch.randn((no + ni, N), dtype=torch.complex128, device="cuda", generator=g)
    f = torch.rand(no, dtype=torch.float64, device="cuda", generator=g)
    p = exx.Plan.bloch(n, 0.3, (1, 1, 0), [0.7, -1.3, 0.0], 12, exx.EXX_KERNEL_ERFC, 0.106)
    out = p.apply_complex(z[:1].contiguous(), f[:1], z[no:].contiguous())
    for j in (0, 7, 19):
        assert torch.equal(p.apply_complex(z[:1].contiguous(), f[:1], z[no + j:no + j + 1].contiguous())[0], out[j])
