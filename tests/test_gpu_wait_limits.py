"""The bounded waits inside the inversion kernels.  With QSI_INV_WAIT_NS = 0 no wait
waits: every index a kernel forms from what a wait was to bring is checked, so the
launch ends, the next synchronize reports QSI_ERR_TIMEOUT, and the context goes on."""
import numpy as np
import pytest

from oracle import rgf
from paper_2601_04904_gb300 import inputs
from paper_2601_04904_gb300.metrics import max_block_rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2601_04904_gb300 import qsi

    c = qsi.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("b", [5, 32, 130, 300, 600])
def test_refined_inversion_without_waits(ctx, monkeypatch, b):
    """One panel (no hand-over), several, every rows-per-thread form: the timeout is
    reported rather than the singular pivots the unfinished data may show."""
    from paper_2601_04904_gb300 import qsi

    n, a = 2, 3
    h, B = inputs.hamiltonian(n, b, a), inputs.lesser_rhs(n, b, a)
    A = ctx.assemble(qsi.to_device(h), 0.3, 1e-3, 0.5)
    Bd = qsi.to_device(B)
    with monkeypatch.context() as m:
        m.setenv("QSI_INV_WAIT_NS", "0")
        f = ctx.factor(A, Bd, qsi.FP64_EMU)
        ctx.selquad(f)
        with pytest.raises(qsi.QsiError, match="FP32 Gauss-Jordan: bounded wait ran out") as e:
            ctx.synchronize()
        f.close()
        assert e.value.status == qsi.ERR_TIMEOUT
    ctx.synchronize()  # cleared
    f = ctx.factor(A, Bd, qsi.FP64_EMU)
    GR, GL = ctx.selquad(f)
    ctx.synchronize()
    f.close()
    oR, oL = rgf.selquad(rgf.assemble_a(h, 0.3, 1e-3, 0.5), B)
    assert max_block_rel_err(qsi.to_host(GR), oR) < 1e-10 and max_block_rel_err(qsi.to_host(GL), oL) < 1e-10


def test_batched_inversion_without_waits(ctx, monkeypatch):
    """A wide batch (as many panels per column CTA as fit)."""
    from paper_2601_04904_gb300 import qsi

    n, b, a, points = 2, 46, 3, 9
    h = qsi.to_device(inputs.hamiltonian(n, b, a))
    E, g = inputs.energy_grid(points)
    B = qsi.to_device({k: np.stack([inputs.lesser_rhs(n, b, a, seed=k2)[k] for k2 in range(points)])
                       for k in qsi.KEYS})
    monkeypatch.setenv("QSI_INV_WAIT_NS", "0")
    ctx.selquad_batched(h, E, 1e-3, g, B, precision=qsi.FP64_EMU)
    with pytest.raises(qsi.QsiError) as e:
        ctx.synchronize()
    assert e.value.status == qsi.ERR_TIMEOUT


@pytest.mark.parametrize("b", [9, 32, 40, 64])
def test_small_fp64_inversion_without_waits(ctx, monkeypatch, b):
    """The cluster form of the IEEE FP64 inversion, one and two row halves: reported by
    the sweeps, and by the allocation-free inversion as info = -1."""
    import ctypes
    import torch
    from paper_2601_04904_gb300 import build, qsi

    n, a = 2, 3
    h, B = inputs.hamiltonian(n, b, a), inputs.lesser_rhs(n, b, a)
    A = ctx.assemble(qsi.to_device(h), 0.3, 1e-3, 0.5)
    Bd = qsi.to_device(B)
    block = torch.from_numpy(np.ascontiguousarray(rgf.assemble_a(h, 0.3, 1e-3, 0.5)["diag"][0])).cuda()
    out, info = torch.empty_like(block), torch.zeros(1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    lib = ctypes.CDLL(build.LIB)

    def inverse():
        assert lib.qsi_block_inverse_noalloc(ctypes.c_void_p(block.data_ptr()), ctypes.c_void_p(out.data_ptr()), b,
                                             None, ctypes.c_void_p(info.data_ptr())) == 0
        torch.cuda.synchronize()
        return int(info.item())

    with monkeypatch.context() as m:
        m.setenv("QSI_INV_WAIT_NS", "0")
        f = ctx.factor(A, Bd, qsi.FP64)
        ctx.selquad(f)
        with pytest.raises(qsi.QsiError, match="FP64 inversion: bounded wait ran out") as e:
            ctx.synchronize()
        f.close()
        assert e.value.status == qsi.ERR_TIMEOUT
        assert inverse() == -1
    assert inverse() == 0
    assert np.abs(out.cpu().numpy() @ block.cpu().numpy() - np.eye(b)).max() < 1e-11
    f = ctx.factor(A, Bd, qsi.FP64)
    GR, GL = ctx.selquad(f)
    ctx.synchronize()
    f.close()
    oR, oL = rgf.selquad(rgf.assemble_a(h, 0.3, 1e-3, 0.5), B)
    assert max_block_rel_err(qsi.to_host(GR), oR) < 1e-10 and max_block_rel_err(qsi.to_host(GL), oL) < 1e-10
