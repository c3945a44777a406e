"""Rayleigh-Ritz on blocks whose projected matrix has repeated eigenvalues: with no potential the
basis functions of one (l, n) share their level, and the block mixes several whole multiplets by
an orthogonal matrix. The Ritz values are the levels, the vectors stay orthonormal and nothing is
NaN, in every dense precision and with H X in FP64 and FP32."""
import numpy as np
import pytest

from tests.gpu_common import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dense", ["CS_FP64", "CS_DF64", "CS_FP64_SLICED"])
@pytest.mark.parametrize("rr", ["CS_FP64", "CS_FP32"])
@pytest.mark.parametrize("seed", [1, 2, 3])
def test_ritz_values_of_mixed_multiplets(dense, rr, seed):
    torch, cs = need_gpu()
    lmax, nmax = 6, 8
    ctx = cs.cs_basis_init(8.0, lmax, nmax, 20, 14, 28)
    cs.cs_set_potential(ctx, torch.zeros(20 * 14 * 28, dtype=torch.float64, device="cuda"))
    cs.cs_set_dense_precision(ctx, getattr(cs, dense))
    cs.cs_set_rr_precision(ctx, getattr(cs, rr))
    half = cs.cs_kinetic(ctx)
    cols = [(l * l + l + m) * nmax + n for l, n in ((0, 0), (1, 0), (2, 0), (2, 1), (4, 0))
            for m in range(-l, l + 1)]
    k = len(cols)
    q = np.linalg.qr(np.random.default_rng(seed).standard_normal((k, k)))[0]
    X = torch.zeros((k, ctx.d), dtype=torch.float64, device="cuda")
    X[:, cols] = torch.tensor(q, device="cuda")
    theta = torch.empty(k, dtype=torch.float64, device="cuda")
    resid = torch.empty_like(theta)
    cs.cs_rayleigh_ritz(ctx, X, theta, resid)
    want = np.sort(half[cols])
    # H X: FP64 (or FP32) roundings of 1/2 Lambda x, summed over the block's width
    tol = (1e-13 if rr == "CS_FP64" else 4e-7) * want[-1] * np.sqrt(k)
    assert np.max(np.abs(theta.cpu().numpy() - want)) <= tol
    off = (X @ X.T - torch.eye(k, dtype=torch.float64, device="cuda")).abs().max()
    assert float(off) <= 1e-11
    assert float(resid.max()) <= 10 * tol
