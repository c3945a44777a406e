"""Rayleigh-Ritz on projected matrices whose levels lie 1e-5 to 1e-4 of the range apart: close enough
that the FP32 inverse iterations leave vectors that overlap, too far apart for the Gram-Schmidt of
its clusters. With no potential H is diagonal, and projectors on single basis functions move their
levels to the wanted ones; the block mixes them by an orthogonal matrix."""
import numpy as np
import pytest

from tests.gpu_common import need_gpu

pytestmark = pytest.mark.gpu


def _levels(kind, k, rng):
    """k ascending levels in [1, 10]."""
    gap = {"pairs": 1.5e-5, "tens": 1.2e-5, "tens_wide": 3e-5}.get(kind)
    if kind == "random":  # gaps spread over 1e-5 .. 1e-4 of the range, a few large ones
        gaps = 10.0 * 10.0 ** rng.uniform(-5, -4, k)
        gaps[:: k // 8] = 1.0
        lv = 1.0 + np.cumsum(gaps)
        return lv * (10.0 / lv[-1]) if lv[-1] > 10.0 else lv
    m = 2 if kind == "pairs" else 10
    base = np.linspace(1.0, 9.9, (k + m - 1) // m)
    return np.sort((base[:, None] + 10.0 * gap * np.arange(m)[None, :]).ravel()[:k])


@pytest.mark.parametrize("kind", ["pairs", "tens", "tens_wide", "random"])
@pytest.mark.parametrize("k", [80, 112])
@pytest.mark.parametrize("dense", ["CS_FP64", "CS_FP64_SLICED"])
def test_close_levels_keep_orthonormal_vectors(kind, k, dense):
    """Bars, in units of 2^-53: the sums of k products round to about k each (orthogonality), and
    the products with H of norm 10 likewise (values, residuals); 8 of that for the chain of Gram
    matrix, eigenvectors and rotation."""
    torch, cs = need_gpu()
    ctx = cs.cs_basis_init(8.0, 6, 8, 20, 14, 28)
    cs.cs_set_potential(ctx, torch.zeros(20 * 14 * 28, dtype=torch.float64, device="cuda"))
    cs.cs_set_dense_precision(ctx, getattr(cs, dense))
    rng = np.random.default_rng(k + len(kind))
    want = _levels(kind, k, rng)
    cols = np.arange(k) * 3 % ctx.d
    half = cs.cs_kinetic(ctx)
    P = torch.zeros((k, ctx.d), dtype=torch.float64, device="cuda")
    P[torch.arange(k), torch.tensor(cols)] = 1.0
    cs.cs_set_projectors(ctx, P, want - half[cols])
    q = np.linalg.qr(rng.standard_normal((k, k)))[0]
    X = torch.zeros((k, ctx.d), dtype=torch.float64, device="cuda")
    X[:, torch.tensor(cols)] = torch.tensor(q, device="cuda")
    theta = torch.empty(k, dtype=torch.float64, device="cuda")
    resid = torch.empty_like(theta)
    cs.cs_rayleigh_ritz(ctx, X, theta, resid)
    unit = 8.0 * k * 2.0 ** -53
    off = (X @ X.T - torch.eye(k, dtype=torch.float64, device="cuda")).abs().max()
    err = np.max(np.abs(theta.cpu().numpy() - want))
    # the largest kinetic energy is cancelled by its projector: its rounding stays
    scale = max(10.0, float(half[cols].max()))
    print(f"close {kind} {k} {dense}: orth {float(off):.1e} ({unit:.1e}) theta {err:.1e} "
          f"resid {float(resid.max()):.1e} ({unit * scale:.1e})")
    assert float(off) <= unit
    assert err <= unit * scale and float(resid.max()) <= unit * scale
