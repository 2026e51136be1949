"""Calls on a device too full for their automatic workspaces: a cap stands for the memory that is
left.  The smaller form gives what the same form gives when it is asked for."""
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


def _cap(exx, p, cap):
    f = exx.load().exx_debug_limits
    f.argtypes = [ctypes.c_void_p, ctypes.c_long, ctypes.c_long]
    assert f(p._h, 0, cap) == 0


@pytest.mark.parametrize("prec, cap", [("FP64", 8 * MB), ("BF16X7", 5 * MB), ("BF16X10", 8 * MB)])
@pytest.mark.parametrize("n_occ, n_in, aliased", [(40, 40, True), (16, 16, True), (30, 40, True), (40, 9, False)])
def test_apply_takes_smaller_batches(exx, prec, cap, n_occ, n_in, aliased):
    """24^3 points: 64 fields take 3.5 MB (7 MB in FP64 and BF16X10), the automatic batch up to 1024."""
    g = torch.Generator(device="cuda").manual_seed(n_in)
    psi = torch.randn((max(n_occ, n_in), 24 ** 3), dtype=torch.float64, device="cuda", generator=g)
    f = torch.rand(n_occ, dtype=torch.float64, device="cuda", generator=g)
    phi = psi[:n_in] if aliased else psi[:n_in].clone()

    def plan():
        p = exx.Plan((24, 24, 24), 0.3, (1, 1, 0), 12, exx.EXX_KERNEL_ERFC, 0.106)
        p.set_precision(getattr(exx, "EXX_PREC_" + prec))
        return p
    p, q = plan(), plan()
    _cap(exx, p, cap)
    q.set_batch(64, 0)
    for _ in range(2):
        assert torch.equal(p.apply(psi[:n_occ], f, phi), q.apply(psi[:n_occ], f, phi))
    _cap(exx, p, 1000)   # nothing fits
    p.set_batch(0, 0)
    with pytest.raises(exx.ExxError) as e:
        p.apply(psi[:n_occ], f, phi)
    assert e.value.status == exx.EXX_ERR_OOM
    _cap(exx, p, 0)
    assert torch.isfinite(p.apply(psi[:n_occ], f, phi)).all()


def test_complex_apply_takes_fewer_columns(exx):
    """6 occupied x 20 columns of 24 x 20 x 22 points: 2 MB a column, all of them at once without a cap."""
    n, no, ni = (24, 20, 22), 6, 20
    g = torch.Generator(device="cuda").manual_seed(3)
    z = torch.randn((no + ni, n[0] * n[1] * n[2]), dtype=torch.complex128, device="cuda", generator=g)
    f = torch.rand(no, dtype=torch.float64, device="cuda", generator=g)
    p = exx.Plan.bloch(n, 0.3, (1, 1, 0), [0.7, -1.3, 0.0], 12, exx.EXX_KERNEL_ERFC, 0.106)
    ref = p.apply_complex(z[:no].contiguous(), f, z[no:].contiguous())
    _cap(exx, p, 5 * MB)
    assert torch.equal(p.apply_complex(z[:no].contiguous(), f, z[no:].contiguous()), ref)
    _cap(exx, p, MB)   # less than a column
    with pytest.raises(exx.ExxError) as e:
        p.apply_complex(z[:no].contiguous(), f, z[no:].contiguous())
    assert e.value.status == exx.EXX_ERR_OOM
