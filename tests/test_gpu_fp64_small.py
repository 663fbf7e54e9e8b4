"""IEEE FP64 products and inversions at small sizes: the edges of the small-tile
product kernel and of the one-cluster block inversion."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (3, 5, 31), (4, 4, 32), (5, 4, 33), (37, 29, 65), (192, 200, 7),
                                   (208, 192, 7), (33, 2, 200)])
def test_product_small_tiles(ctx, m, n, k):
    """4 x 4 tiles up to 152 tiles of 16 x 16 (192 x 200 is the last, 208 x 192 the
    first above), ragged tiles and depth chunks, every op, alpha and beta."""
    import torch

    rng = np.random.default_rng(m + 10 * n + k)
    cn = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)
    for opA in (0, 1):
        for opB in (0, 1):
            for alpha, beta in ((1.0, 0.0), (-1.0, 1.0), (0.5, 0.25 - 2.0j)):
                A, B, C = cn(*((k, m) if opA else (m, k))), cn(*((n, k) if opB else (k, n))), cn(m, n)
                # rows longer than the matrix, the rest NaN
                dA, dB, dev = (torch.full((x.shape[0], x.shape[1] + 3), float("nan"), dtype=torch.complex128,
                                          device="cuda")[:, :x.shape[1]] for x in (A, B, C))
                for d, x in ((dA, A), (dB, B), (dev, C)):
                    d.copy_(torch.from_numpy(x))
                torch.cuda.synchronize()
                ctx.zgemm(dA, dB, dev, opA=opA, opB=opB, alpha=alpha, beta=beta)
                ctx.synchronize()
                ref = alpha * ((A.conj().T if opA else A) @ (B.conj().T if opB else B)) + beta * C
                scale = np.linalg.norm(A) * np.linalg.norm(B) + 3.0 * np.linalg.norm(C)
                assert np.linalg.norm(dev.cpu().numpy() - ref) < 1e-15 * (k + 4) * scale


def _single(qsi, blocks):
    """n = 1 BTA containers of a batch of blocks (one per energy point)."""
    import torch

    b = blocks.shape[-1]
    z = lambda *s: torch.zeros(*s, dtype=torch.complex128, device="cuda")
    return [{"diag": torch.from_numpy(x[None].copy()).cuda(), "upper": z(0, b, b), "lower": z(0, b, b),
             "arrow_r": z(1, b, 0), "arrow_b": z(1, 0, b), "tip": z(0, 0)} for x in blocks]


@pytest.mark.parametrize("b", [1, 7, 8, 9, 31, 32, 33, 57, 63, 64])
def test_small_inverse(ctx, b):
    """One cluster per block: ragged last CTA, one and two row halves, rows needing
    every pivot order (a random permutation times a well-conditioned block)."""
    from paper_2601_04904_gb300 import qsi

    rng = np.random.default_rng(b)
    cn = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)
    blocks = np.stack([cn(b, b) * 0.2 / np.sqrt(b) + np.eye(b)[rng.permutation(b)] for _ in range(3)])
    for m, a in zip(_single(qsi, blocks), blocks):
        f = ctx.factor(m, None, qsi.FP64)
        X = ctx.selinv(f)["diag"][0].cpu().numpy()
        ctx.synchronize()
        f.close()
        assert np.linalg.norm(X - np.linalg.inv(a)) < 1e-13 * np.linalg.norm(X) * np.linalg.cond(a)


@pytest.mark.parametrize("b,col", [(5, 4), (32, 0), (40, 37), (64, 9), (64, 63)])
def test_small_inverse_reports_the_singular_column(ctx, b, col):
    """A zero column is reported with its index, whichever CTA owns it."""
    from paper_2601_04904_gb300 import qsi

    rng = np.random.default_rng(col)
    a = rng.standard_normal((b, b)) + 1j * rng.standard_normal((b, b)) + 4 * np.eye(b)
    a[:, col] = 0
    f = ctx.factor(_single(qsi, a[None])[0], None, qsi.FP64)
    ctx.selinv(f)
    with pytest.raises(qsi.QsiError, match=f"column {col}") as e:
        ctx.synchronize()
    assert e.value.status == qsi.ERR_SINGULAR
    f.close()


@pytest.mark.parametrize("b,points", [(5, 97), (32, 97), (33, 65), (64, 65)])
def test_wide_batches_of_small_blocks_give_the_bits_of_narrow_ones(ctx, b, points):
    """One CTA per block above 96 (b <= 32) or 64 blocks, a cluster per block up to
    there: a batch on either side of the line, the same bits."""
    import torch
    from paper_2601_04904_gb300 import inputs, qsi

    n = 2
    Hd = qsi.to_device(inputs.hamiltonian(n, b, 0))
    E, g = inputs.energy_grid(points)
    B = qsi.batched_zeros(points, n, b, 0)
    B["diag"].copy_(torch.eye(b, dtype=torch.complex128, device="cuda") * 1j)
    torch.cuda.synchronize()
    wide = ctx.selquad_batched(Hd, E, 1e-3, g, B, precision=qsi.FP64)
    half = points // 2 + 1
    narrow = [ctx.selquad_batched(Hd, E[s], 1e-3, g[s], {k: v[s].contiguous() for k, v in B.items()},
                                  precision=qsi.FP64) for s in (slice(0, half), slice(half, points))]
    ctx.synchronize()
    for i in (0, 1):
        for key in qsi.KEYS:
            assert (torch.cat([narrow[0][i][key], narrow[1][i][key]]) == wide[i][key]).all(), key


@pytest.mark.parametrize("b,first", [(64, 0), (64, 7), (64, 31), (33, 31), (16, 7)])
def test_the_first_of_several_singular_columns_is_reported(ctx, b, first):
    """Zero columns on both sides of a boundary between CTAs (and every column after
    the first, whose pivots are no longer finite): always the first one."""
    from paper_2601_04904_gb300 import qsi

    rng = np.random.default_rng(first)
    a = rng.standard_normal((b, b)) + 1j * rng.standard_normal((b, b)) + 4 * np.eye(b)
    a[:, [first, first + 1]] = 0
    m = _single(qsi, a[None])[0]
    for _ in range(30):
        f = ctx.factor(m, None, qsi.FP64)
        with pytest.raises(qsi.QsiError, match=f"column {first}$"):
            ctx.synchronize()
        f.close()


@pytest.mark.parametrize("m,n,k", [(128, 304, 9), (144, 272, 9), (150, 259, 40)])
def test_product_kernels_either_side_of_the_line(ctx, m, n, k):
    """152 tiles of 16 x 16 (128 x 304) take the 4 x 4 tiles, 153 (144 x 272) and more
    the 16 x 16 ones: every op against numpy, nothing written past a row's end, and the
    rows of a product the bits they have in a larger one across the line."""
    import torch

    rng = np.random.default_rng(m + n + k)
    cn = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)

    def product(A, B, C, opA, opB):
        nan = complex(float("nan"), float("nan"))
        full = [torch.full((x.shape[0], x.shape[1] + 3), nan, dtype=torch.complex128, device="cuda") for x in (A, B, C)]
        for d, x in zip(full, (A, B, C)):
            d[:, :x.shape[1]].copy_(torch.from_numpy(x))
        torch.cuda.synchronize()
        dA, dB, dC = (d[:, :x.shape[1]] for d, x in zip(full, (A, B, C)))
        ctx.zgemm(dA, dB, dC, opA=opA, opB=opB, alpha=-1.0, beta=1.0)
        ctx.synchronize()
        assert torch.isnan(full[2][:, C.shape[1]:].real).all() and torch.isnan(full[2][:, C.shape[1]:].imag).all()
        return dC.cpu().numpy()

    for opA in (0, 1):
        for opB in (0, 1):
            A, B, C = cn(*((k, m) if opA else (m, k))), cn(*((n, k) if opB else (k, n))), cn(m, n)
            got = product(A, B, C, opA, opB)
            ref = C - (A.conj().T if opA else A) @ (B.conj().T if opB else B)
            scale = np.linalg.norm(A) * np.linalg.norm(B) + np.linalg.norm(C)
            assert np.linalg.norm(got - ref) < 1e-15 * (k + 4) * scale
            more = cn(*((k, 64) if opA else (64, k)))
            large = product(np.concatenate([A, more], axis=1 if opA else 0), B, np.concatenate([C, cn(64, n)]), opA, opB)
            assert (large[:m] == got).all()
