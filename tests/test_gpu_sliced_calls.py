"""The calls that reach the slice products through the double-float and residual-form paths: their
FP64 and double-float forms take the same products, so they return the same bits; and the FP64 form
agrees with the FMA kernels."""
import pytest

import workloads as W
from tests.gpu_common import make_ctx, need_gpu, register, rel_errors, to_dev, to_host

pytestmark = pytest.mark.gpu

CLOSE = 64 * 2.0 ** -53  # both forms' rounding per H.X (test_gpu_sliced_hx.py)
W1 = W.small_cluster(lmax=24, nmax=6, n_r=40, n_theta=30, n_phi=60, n_s=20)  # 15.0M rows L^2
register(W1)


def _setup(monkeypatch, projectors):
    torch, cs = need_gpu()
    monkeypatch.delenv("CS_ANGULAR_KERNEL", raising=False)
    ctx = make_ctx(W1)
    cs.cs_set_dense_precision(ctx, cs.CS_FP64_SLICED)
    gen = torch.Generator(device="cuda").manual_seed(9)
    if projectors:
        P = torch.randn((7, ctx.d), generator=gen, dtype=torch.float64, device="cuda")
        cs.cs_set_projectors(ctx, P / ctx.d ** 0.5, [1.0, -2.0, 3.0, 0.5, -0.1, 4.0, -3.0])
    return torch, cs, ctx, to_dev(W1.x_block(), ld=ctx.d + 3)


def _both(torch, cs, monkeypatch, run):
    """run(precision) in FP64 and double-float by the slices, then in FP64 by the FMA kernels."""
    a, b = run(cs.CS_FP64), run(cs.CS_DF64)
    monkeypatch.setenv("CS_ANGULAR_KERNEL", "fma")
    ref = run(cs.CS_FP64)
    monkeypatch.delenv("CS_ANGULAR_KERNEL")
    return a, b, ref


@pytest.mark.parametrize("projectors", [False, True])
def test_apply(projectors, monkeypatch):
    torch, cs, ctx, X = _setup(monkeypatch, projectors)

    def run(prec):
        out = torch.full_like(X, 3.0)
        cs.cs_apply_H(ctx, X, out, prec)
        return out

    a, b, ref = _both(torch, cs, monkeypatch, run)
    assert torch.equal(a, b) and torch.all(a[:, ctx.d:] == 3.0)
    fro, col = rel_errors(to_host(a, ctx.d), to_host(ref, ctx.d))
    assert 0 < fro <= CLOSE and col <= CLOSE, (fro, col)
    assert cs.cs_device_error(ctx) == 0


@pytest.mark.parametrize("residual_form", [False, True])
def test_filter(residual_form, monkeypatch):
    torch, cs, ctx, X = _setup(monkeypatch, False)
    hi = float(cs.cs_kinetic(ctx).max()) + 1.0
    HX = torch.zeros_like(X)
    cs.cs_apply_H(ctx, X, HX, cs.CS_FP64)
    theta = torch.linspace(-8.0, hi, W1.n_s, dtype=torch.float64, device="cuda")

    def run(prec):
        Y = X.clone()
        if residual_form:
            cs.cs_cheb_filter_ritz(ctx, Y, HX, theta, 5, 2.0, hi, -8.0, prec)
        else:
            cs.cs_cheb_filter(ctx, Y, 5, 2.0, hi, -8.0, prec)
        return Y

    a, b, ref = _both(torch, cs, monkeypatch, run)
    assert torch.equal(a, b)
    fro, col = rel_errors(to_host(a, ctx.d), to_host(ref, ctx.d))
    assert 0 < fro <= 16 * CLOSE and col <= 16 * CLOSE, (fro, col)  # five products, amplified
    assert cs.cs_device_error(ctx) == 0


@pytest.mark.parametrize("projectors", [False, True])
def test_rayleigh_ritz(projectors, monkeypatch):
    torch, cs, ctx, X = _setup(monkeypatch, projectors)
    cs.cs_cholqr(ctx, X)
    out = []
    for prec in (cs.CS_FP64, cs.CS_DF64):
        cs.cs_set_rr_precision(ctx, prec)
        Y, HY = X.clone(), torch.zeros_like(X)
        theta = torch.empty(W1.n_s, dtype=torch.float64, device="cuda")
        resid = torch.empty_like(theta)
        cs.cs_rayleigh_ritz(ctx, Y, theta, resid, HY)
        out.append((Y, HY, theta, resid))
    assert all(torch.equal(a, b) for a, b in zip(*out))
