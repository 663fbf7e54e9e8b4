"""Which inverses the refined inversion of the tensor-core precisions accepts:
blocks whose rows have very different scales, on which the Newton residuals are
far from normal and a bound on a product of two residuals bounds neither."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
U = 2.0**-53


@pytest.mark.parametrize("precision", ["fp64_emu", "mixed"])
@pytest.mark.parametrize("b", [8, 16, 48])
@pytest.mark.parametrize("ratio", [1.0, 1e6, 1e9, 1e12])
def test_accepted_inverses_are_accurate(precision, b, ratio):
    """A = D G with G of condition kappa below 20 and D's rows spread over `ratio`:
    the inverse is refused (QSI_ERR_ACCURACY) or every column of it, whose scale D
    sets, has FP64's error: at most 4 b U kappa of its norm (b rounded products of
    relative error U each, through G's condition; 2 U kappa is typical).  Up to a
    spread of 1e6 nothing is refused."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2601_04904_gb300 import qsi

    z = lambda *s: torch.zeros(*s, dtype=torch.complex128, device="cuda")
    ctx = qsi.Context(0)
    for seed in range(30):
        rng = np.random.default_rng(seed)
        g = (rng.standard_normal((b, b)) + 1j * rng.standard_normal((b, b))) / np.sqrt(b) + 2 * np.eye(b)
        d = np.exp(rng.uniform(0.0, np.log(ratio), b)) if ratio > 1 else np.ones(b)
        m = {"diag": torch.from_numpy((d[:, None] * g)[None].copy()).cuda(), "upper": z(0, b, b), "lower": z(0, b, b),
             "arrow_r": z(1, b, 0), "arrow_b": z(1, 0, b), "tip": z(0, 0)}
        f = ctx.factor(m, None, qsi.PRECISIONS[precision])
        X = ctx.selinv(f)["diag"][0]
        try:
            ctx.synchronize()
        except qsi.QsiError as e:
            assert e.status == qsi.ERR_ACCURACY and ratio > 1e6, (seed, str(e))
            continue
        finally:
            f.close()
        ref = np.linalg.inv(g) / d[None, :]
        err = np.linalg.norm(X.cpu().numpy() - ref, axis=0) / np.linalg.norm(ref, axis=0)
        assert err.max() <= 4 * b * U * np.linalg.cond(g), (seed, err.max(), np.linalg.cond(g))
    ctx.close()
