"""Dense products at the edges of their tiles, in FP64 and double-float: Gram matrices of one block
(its upper triangle, mirrored) and of two, rotations, and Cholesky-QR, whose rotation by a triangular
factor skips column groups; odd basis sizes and leading dimensions."""
import pytest

from tests.gpu_common import need_gpu

pytestmark = pytest.mark.gpu

# columns: 1 .. 6 groups of 16 with remainders, the last that fit one tile, and several tiles
COLUMNS = [1, 15, 17, 33, 49, 65, 81, 96, 97, 113, 200]
BITS = {"CS_FP64": 53, "CS_DF64": 48}  # of an operand; the sums round like their terms



@pytest.mark.parametrize("dense", list(BITS))
@pytest.mark.parametrize("n", COLUMNS)
def test_products_match_fp64(dense, n):
    """Bars: every term and every addition within one unit of the sum of magnitudes."""
    torch, cs = need_gpu()
    ctx = cs.cs_basis_init(8.0, 10, 15, 20, 12, 24)
    assert ctx.d % 2 == 1 and ctx.d % 64 != 0
    cs.cs_set_dense_precision(ctx, getattr(cs, dense))
    gen = torch.Generator(device="cuda").manual_seed(n)
    eps = 2.0 ** -BITS[dense]

    def block(k, pad):
        b = torch.zeros((k, ctx.d + pad), dtype=torch.float64, device="cuda")
        b[:, :ctx.d] = torch.randn((k, ctx.d), generator=gen, dtype=torch.float64, device="cuda")
        b[:, :ctx.d] *= 10.0 ** torch.empty((k, 1), dtype=torch.float64,
                                            device="cuda").uniform_(-6, 6, generator=gen)
        return b

    A, B = block(n, 3), block(max(1, n - 7), 1)
    a, b = A[:, :ctx.d], B[:, :ctx.d]
    C = torch.full((n, n + 2), 5.0, dtype=torch.float64, device="cuda")
    cs.cs_dense_gram(ctx, A, A, C)
    assert torch.all((C[:, :n] - a @ a.T).abs() <= (ctx.d + 8) * eps * (a.abs() @ a.abs().T))
    assert torch.all(C[:, n:] == 5.0)
    if n <= 96:  # one tile: the lower triangle is the upper one's image
        assert torch.equal(C[:, :n], C[:, :n].T)
    C = torch.full((B.shape[0], n), 5.0, dtype=torch.float64, device="cuda")
    cs.cs_dense_gram(ctx, A, B, C)
    assert torch.all((C - b @ a.T).abs() <= (ctx.d + 8) * eps * (b.abs() @ a.abs().T))
    m = max(1, n - 3)
    Q = torch.randn((m, n + 1), generator=gen, dtype=torch.float64, device="cuda")
    out = torch.full((m, ctx.d + 2), 5.0, dtype=torch.float64, device="cuda")
    cs.cs_dense_rotate(ctx, A, Q, out)
    q = Q[:, :n]
    assert torch.all((out[:, :ctx.d] - q @ a).abs() <= (n + 8) * eps * (q.abs() @ a.abs()))
    assert torch.all(out[:, ctx.d:] == 5.0)


@pytest.mark.parametrize("dense", list(BITS))
@pytest.mark.parametrize("n", COLUMNS)
def test_cholqr_orthonormalises(dense, n):
    """X = Q R: Q orthonormal, R = Q^T X upper triangular with Q R = X, to the Gram matrix's bar."""
    torch, cs = need_gpu()
    ctx = cs.cs_basis_init(8.0, 10, 15, 20, 12, 24)
    cs.cs_set_dense_precision(ctx, getattr(cs, dense))
    gen = torch.Generator(device="cuda").manual_seed(100 + n)
    X = torch.zeros((n, ctx.d + 5), dtype=torch.float64, device="cuda")
    X[:, :ctx.d] = torch.randn((n, ctx.d), generator=gen, dtype=torch.float64, device="cuda")
    x0 = X[:, :ctx.d].clone()
    cs.cs_cholqr(ctx, X)
    q = X[:, :ctx.d]
    unit = 4 * (ctx.d + 8) * 2.0 ** -BITS[dense]
    eye = torch.eye(n, dtype=torch.float64, device="cuda")
    assert float((q @ q.T - eye).abs().max()) <= unit
    R = q @ x0.T  # R[i, j] = q_i . x_j
    norm = float(x0.norm(dim=1).max())
    assert float(R.tril(-1).abs().max()) <= unit * norm
    assert float((R.T @ q - x0).norm(dim=1).max()) <= unit * norm
    assert torch.all(X[:, ctx.d:] == 0.0)
