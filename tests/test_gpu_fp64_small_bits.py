"""IEEE FP64 inversion of small blocks: the bits of its stated arithmetic, worked
out in exact rational arithmetic with one rounding per operation."""
from fractions import Fraction as Q

import numpy as np
import pytest


def _fma(a, b, c):
    return float(Q(a) * Q(b) + Q(c))


def _mul(a, b):
    return _fma(a[0], b[0], -(a[1] * b[1])), _fma(a[1], b[0], a[0] * b[1])


def _reciprocal(d):
    """Smith's 1 / d."""
    re = abs(d[0]) >= abs(d[1])
    g, l = (d[0], d[1]) if re else (d[1], d[0])
    r = l / g
    den = _fma(l, r, g)
    u, w = 1.0 / den, r / den
    return (u, -w) if re else (w, -u)


def gauss_jordan(x):
    """In-place Gauss-Jordan with partial pivoting (largest |x|^2, lowest row on
    ties): scaled pivot row, every product rounded before it is subtracted."""
    b = len(x)
    m = [[(float(z.real), float(z.imag)) for z in row] for row in x]
    piv = []
    for c in range(b):
        p = max(range(c, b), key=lambda r: (_fma(m[r][c][0], m[r][c][0], m[r][c][1] * m[r][c][1]), -r))
        piv.append(p)
        m[c], m[p] = m[p], m[c]
        inv = _reciprocal(m[c][c])
        f = [row[c] for row in m]
        m[c] = [_mul((1.0, 0.0) if j == c else m[c][j], inv) for j in range(b)]
        for r in range(b):
            if r != c:
                t = [_mul(f[r], y) for y in m[c]]
                v = [(0.0, 0.0) if j == c else m[r][j] for j in range(b)]
                m[r] = [(v[j][0] - t[j][0], v[j][1] - t[j][1]) for j in range(b)]
    idx = list(range(b))
    for k in reversed(range(b)):
        idx[k], idx[piv[k]] = idx[piv[k]], idx[k]
    return np.array([[complex(*row[idx[j]]) for j in range(b)] for row in m])


def test_the_rational_elimination_inverts():
    rng = np.random.default_rng(0)
    x = rng.standard_normal((6, 6)) + 1j * rng.standard_normal((6, 6))
    assert np.abs(gauss_jordan(x) @ x - np.eye(6)).max() < 1e-13


@pytest.mark.gpu
@pytest.mark.parametrize("b", [1, 2, 7, 8, 9, 17, 33])
def test_small_inverse_bits(b):
    """One and two row halves, one CTA and several, random entries and entries of
    +-1 +- i, whose pivots tie."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2601_04904_gb300 import qsi

    z = lambda *s: torch.zeros(*s, dtype=torch.complex128, device="cuda")
    ctx = qsi.Context(0)
    rng = np.random.default_rng(b)
    signs = lambda: rng.choice([-1.0, 1.0], (b, b))
    for x in (rng.standard_normal((b, b)) + 1j * rng.standard_normal((b, b)),
              signs() + 1j * signs() + 0.25 * rng.integers(0, 2, (b, b))):
        m = {"diag": torch.from_numpy(x[None].copy()).cuda(), "upper": z(0, b, b), "lower": z(0, b, b),
             "arrow_r": z(1, b, 0), "arrow_b": z(1, 0, b), "tip": z(0, 0)}
        f = ctx.factor(m, None, qsi.FP64)
        got = ctx.selinv(f)["diag"][0].cpu().numpy()
        ctx.synchronize()
        f.close()
        assert (got == gauss_jordan(x)).all()
    ctx.close()
