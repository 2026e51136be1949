"""The direct forms of the BF16X7 passes over many tiles a group, with an uneven tail, against the
older forms bit for bit: what is carried from one tile to the next (staged input, row maxima cleared
for the next tile, barrier phases, tile counters, operands reused after a drain) in each layout that
has two or three tile groups on an SM."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# 1023 fields: at least 5115 slice tiles and 5115 z tiles for at most 456 groups
@pytest.mark.parametrize("n, bc", [((24, 24, 24), (0, 0, 0)), ((16, 17, 40), (0, 1, 0)), ((42, 43, 49), (0, 1, 0)),
                                   ((48, 47, 64), (1, 0, 1)), ((33, 29, 100), (1, 1, 0)), ((20, 20, 130), (1, 1, 0))],
                         ids=lambda v: "x".join(map(str, v)))
def test_many_tiles_keep_every_bit(n, bc):
    import paper_2501_16572_gb300 as exx
    g = torch.Generator(device="cuda").manual_seed(sum(n))
    N = n[0] * n[1] * n[2]
    psi = torch.randn((64, N), dtype=torch.float64, device="cuda", generator=g)
    psi *= torch.exp(6 * torch.rand((1, N), dtype=torch.float64, device="cuda", generator=g) - 5)
    f = torch.rand(31, dtype=torch.float64, device="cuda", generator=g)
    p = exx.Plan(n, 0.3, bc, 12, exx.EXX_KERNEL_ERFC, 0.106)
    p.set_precision(exx.EXX_PREC_BF16X7)
    p.set_tuning(pairs_per_batch=1024, block_orbitals=8)
    new = p.apply(psi[:31], f, psi[31:])
    p.set_tuning(pairs_per_batch=1024, block_orbitals=8, z_block=-16, z_buffers=2, pipeline=0)
    old = p.apply(psi[:31], f, psi[31:])
    assert torch.isfinite(new).all() and float(new.abs().max()) > 0
    assert torch.equal(new, old)
