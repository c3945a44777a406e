"""FP64 H.X from slice products on the tensor cores: against the FP64 oracle, and against the
FP64 kernels on the FMA pipe, at the edges of its tiles; non-finite and zero operands."""
import numpy as np
import pytest

import workloads as W
from tests.gpu_common import make_ctx, need_gpu, oracle_H, register, rel_errors, to_dev, to_host

pytestmark = pytest.mark.gpu

# two roundings per contraction of either form, each below 2^-53 of the row's norm times a modest
# constant: the two agree to 64 units of 2^-53
CLOSE = 64 * 2.0 ** -53

# name: lmax, nmax, n_r, n_theta, n_phi, n_s. Edges: n_phi 2 lmax + 2 and no multiple of four, odd
# n_theta; 16 / 17 modes per class (lmax 31 / 32); K of 32, 64 and 128 with a remainder;
# 129 states (two blocks); 64 quarter angles and theta pairs
EDGES = {
    "min_phi": (5, 7, 19, 13, 12, 40),
    "odd_theta": (9, 16, 33, 23, 42, 17),
    "modes16": (31, 12, 25, 33, 66, 7),
    "modes17": (32, 12, 25, 64, 128, 5),
    "radial_129": (6, 65, 129, 15, 28, 3),
    "two_blocks": (8, 17, 20, 19, 36, 129),
    "largest": (62, 9, 21, 127, 254, 2),
}


def _work(case):
    lmax, nmax, n_r, n_theta, n_phi, n_s = EDGES[case]
    w = W.small_cluster(lmax=lmax, nmax=nmax, n_r=n_r, n_theta=n_theta, n_phi=n_phi, n_s=n_s)
    register(w)
    return w


def _fma(monkeypatch, cs, call):
    monkeypatch.setenv("CS_ANGULAR_KERNEL", "fma")
    call()
    monkeypatch.delenv("CS_ANGULAR_KERNEL")


@pytest.mark.parametrize("case", list(EDGES))
def test_sliced_hx_matches_fma_kernels(case, monkeypatch):
    torch, cs = need_gpu()
    monkeypatch.delenv("CS_ANGULAR_KERNEL", raising=False)
    w = _work(case)
    ctx = make_ctx(w)
    X = to_dev(w.x_block(), ld=ctx.d + 3)
    a, b = torch.zeros_like(X), torch.zeros_like(X)
    n0 = cs.cs_launch_count(ctx)
    cs.cs_apply_H(ctx, X, a, cs.CS_FP64)
    assert cs.cs_launch_count(ctx) - n0 > 3  # not the three FMA kernels
    _fma(monkeypatch, cs, lambda: cs.cs_apply_H(ctx, X, b, cs.CS_FP64))
    fro, col = rel_errors(to_host(a, ctx.d), to_host(b, ctx.d))
    print(f"sliced against FMA {case}: fro {fro:.2e} col {col:.2e}")
    assert fro <= CLOSE and col <= CLOSE, (fro, col)
    assert torch.all(a[:, ctx.d:] == 0)
    if case == "largest":  # double-float calls of this size take the same products
        cs.cs_apply_H(ctx, X, b, cs.CS_DF64)
        assert torch.equal(a, b)
    assert cs.cs_device_error(ctx) == 0


@pytest.mark.parametrize("case", ["min_phi", "odd_theta", "two_blocks"])
def test_sliced_hx_matches_oracle(case, monkeypatch):
    torch, cs = need_gpu()
    monkeypatch.delenv("CS_ANGULAR_KERNEL", raising=False)
    w = _work(case)
    ctx = make_ctx(w)
    X = w.x_block()
    Xd = to_dev(X)
    out = torch.zeros_like(Xd)
    cs.cs_apply_H(ctx, Xd, out, cs.CS_FP64)
    fro, col = rel_errors(to_host(out, ctx.d), oracle_H(w.name).apply(X))
    assert fro <= 1e-11 and col <= 1e-11, (fro, col)


def test_sliced_filter_takes_the_recurrence(monkeypatch):
    torch, cs = need_gpu()
    monkeypatch.delenv("CS_ANGULAR_KERNEL", raising=False)
    w = _work("odd_theta")
    ctx = make_ctx(w)
    X = to_dev(w.x_block())
    a, b = X.clone(), X.clone()
    hi = float(cs.cs_kinetic(ctx).max()) + 1.0
    cs.cs_cheb_filter(ctx, a, 5, 2.0, hi, -8.0, cs.CS_FP64)
    _fma(monkeypatch, cs, lambda: cs.cs_cheb_filter(ctx, b, 5, 2.0, hi, -8.0, cs.CS_FP64))
    fro, col = rel_errors(to_host(a, ctx.d), to_host(b, ctx.d))
    assert fro <= 16 * CLOSE and col <= 16 * CLOSE, (fro, col)  # five products, amplified


def test_sliced_hx_zero_and_non_finite_operands(monkeypatch):
    """A zero column stays zero; a NaN or an infinity fills its own column and no other; a
    potential of zeros leaves the kinetic term; a NaN in the potential reaches every column."""
    torch, cs = need_gpu()
    monkeypatch.delenv("CS_ANGULAR_KERNEL", raising=False)
    w = _work("odd_theta")
    ctx = make_ctx(w)
    X = to_dev(w.x_block())
    clean = torch.zeros_like(X)
    cs.cs_apply_H(ctx, X, clean, cs.CS_FP64)
    Y = X.clone()
    Y[1] = 0.0
    Y[3, 5] = float("nan")
    Y[4, ctx.d - 1] = float("inf")
    out = torch.zeros_like(X)
    cs.cs_apply_H(ctx, Y, out, cs.CS_FP64)
    assert torch.all(out[1] == 0)
    assert torch.isnan(out[3]).all() and not torch.isfinite(out[4]).any()
    keep = [i for i in range(w.n_s) if i not in (1, 3, 4)]
    assert torch.equal(out[keep], clean[keep])
    v = torch.zeros(ctx.n_r * ctx.n_theta * ctx.n_phi, dtype=torch.float64, device=X.device)
    cs.cs_set_potential(ctx, v)
    cs.cs_apply_H(ctx, X, out, cs.CS_FP64)
    half = torch.as_tensor(cs.cs_kinetic(ctx), device=X.device)
    assert torch.equal(out[:, :ctx.d], X[:, :ctx.d] * half)
    v[7] = float("nan")
    cs.cs_set_potential(ctx, v)
    cs.cs_apply_H(ctx, X, out, cs.CS_FP64)
    assert torch.isnan(out[:, :ctx.d]).all()


@pytest.mark.parametrize("scale", [1e-280, 1e-150, 1e150, 1e280])
def test_sliced_hx_scales(scale, monkeypatch):
    """H (s X) = s H X at both ends of the FP64 range, with states of unequal magnitude."""
    torch, cs = need_gpu()
    monkeypatch.delenv("CS_ANGULAR_KERNEL", raising=False)
    w = _work("odd_theta")
    ctx = make_ctx(w)
    X = w.x_block()
    out, ref = (torch.zeros((w.n_s, ctx.d), dtype=torch.float64, device="cuda:0") for _ in "ab")
    cs.cs_apply_H(ctx, to_dev(X), ref, cs.CS_FP64)
    cs.cs_apply_H(ctx, to_dev(X * scale), out, cs.CS_FP64)
    fro, _ = rel_errors(to_host(out, ctx.d) / scale, to_host(ref, ctx.d))
    assert np.isfinite(fro) and fro <= CLOSE, fro


@pytest.mark.parametrize("case", list(EDGES))
def test_sliced_transforms_and_density_match_fma_kernels(case, monkeypatch):
    """The transforms, the density (in blocks of states) and the Hartree potential (one state)
    through the same passes; rows of zeros in the grid functions."""
    torch, cs = need_gpu()
    monkeypatch.delenv("CS_ANGULAR_KERNEL", raising=False)
    w = _work(case)
    ctx = make_ctx(w)
    X = to_dev(w.x_block(), ld=ctx.d + 1)
    shape = (w.n_s, ctx.n_r, ctx.n_theta, ctx.n_phi)
    gen = torch.Generator(device="cuda").manual_seed(5)
    g = torch.randn(shape, dtype=torch.float64, device="cuda", generator=gen)
    g[:, 1, 2] = 0.0
    g[0] = 0.0
    occ = torch.rand(w.n_s, dtype=torch.float64, device="cuda", generator=gen)

    def run():
        coef = torch.zeros_like(X)
        cs.cs_forward_transform(ctx, g, coef)
        f = torch.zeros(shape, dtype=torch.float64, device="cuda")
        cs.cs_inverse_transform(ctx, X, f)
        rho, vh = torch.zeros_like(f[0]), torch.zeros_like(f[0])
        cs.cs_density(ctx, X, occ, rho)
        cs.cs_hartree(ctx, rho, vh)
        return coef, f, rho, vh

    got = run()
    monkeypatch.setenv("CS_ANGULAR_KERNEL", "fma")
    ref = run()
    assert torch.all(got[0][0] == 0)
    for name, a, b in zip(("forward", "inverse", "density", "hartree"), got, ref):
        rel = float((a - b).norm() / b.norm())
        print(f"sliced {name} {case}: {rel:.2e}")
        assert rel <= CLOSE, (name, rel)
    assert cs.cs_device_error(ctx) == 0
