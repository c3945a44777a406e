"""Workspaces of the FP64 slice products: their intermediates lie over slots that are not in use
beside them, every call stays inside the bytes that the queries give, and what lies under them is
rebuilt before it is read."""
import pytest

import workloads as W
from tests.gpu_common import make_ctx, need_gpu, register, to_dev

pytestmark = pytest.mark.gpu

MIB = 1 << 20


def test_intermediates_lie_over_slots_not_in_use():
    torch, cs = need_gpu()
    ctx = cs.cs_basis_init(14.0, 30, 48, 96, 60, 120)
    plain = cs.cs_workspace_bytes(ctx, 80, cs.CS_FP64)
    cs.cs_set_dense_precision(ctx, cs.CS_FP64_SLICED)
    # the operands of the slice-product Gram matrices are smaller than the intermediates
    assert cs.cs_workspace_bytes(ctx, 80, cs.CS_FP64) == plain
    cs.cs_set_dense_precision(ctx, cs.CS_FP64)
    # an FP32 block more, but none of it beside the intermediates
    assert cs.cs_workspace_bytes(ctx, 80, cs.CS_FP32) == plain
    # the SCF calls: the transforms' workspace and 16 grid functions, or in their place G and the
    # intermediates (Legendre sums, four class sums per quarter angle, scales) of 32 states
    grid = ctx.n_r * ctx.n_theta * ctx.n_phi
    base = cs.cs_workspace_bytes(ctx, 16, cs.CS_FP64) + 16 * 8 * grid
    node = 8 * (2 * 30 * 61 + 60 * 4 * 31) + 12 * 60 + 4
    density = 32 * 96 * (8 * 31 ** 2 + node + 4)
    assert cs.cs_scf_workspace_bytes(ctx) <= max(base, density) + 8 * MIB


@pytest.mark.parametrize("lmax", [9, 36])  # fused and three-pass angular blocks
@pytest.mark.parametrize("dense", ["CS_FP64", "CS_FP64_SLICED"])
def test_calls_stay_inside_their_workspace(lmax, dense, monkeypatch):
    torch, cs = need_gpu()
    monkeypatch.delenv("CS_ANGULAR_KERNEL", raising=False)
    n_theta = (lmax + 4) // 2 * 2
    w = W.small_cluster(lmax=lmax, nmax=9, n_r=22, n_theta=n_theta, n_phi=2 * n_theta + 4, n_s=21)
    register(w)
    ctx = make_ctx(w)
    cs.cs_set_dense_precision(ctx, getattr(cs, dense))
    gen = torch.Generator(device="cuda").manual_seed(3)
    P = torch.randn((5, ctx.d), generator=gen, dtype=torch.float64, device="cuda") / ctx.d ** 0.5
    cs.cs_set_projectors(ctx, P, [0.5, -1.0, 2.0, 0.1, -0.3])
    X0 = to_dev(w.x_block())
    v0 = torch.randn(ctx.d, generator=gen, dtype=torch.float64, device="cuda")
    n_s = w.n_s

    def chain(prec, n, work):
        """Lanczos, Cholesky-QR, Rayleigh-Ritz and two filters with one workspace."""
        X = X0[:n].clone()
        th = torch.empty(n, dtype=torch.float64, device="cuda")
        r = torch.empty_like(th)
        HX = torch.empty_like(X)
        b, lo = cs.cs_lanczos_bound(ctx, v0, 8, work)
        cs.cs_cholqr(ctx, X, work)
        cs.cs_rayleigh_ritz(ctx, X, th, r, HX, work)
        Y = X.clone()
        cs.cs_cheb_filter(ctx, Y, 4, 0.5 * (lo + b), b + 1.0, lo - 1.0, cs.CS_FP64, work)
        cs.cs_chfsi_step_ritz(ctx, X, HX, 4, 0.5 * (lo + b), b + 1.0, lo - 1.0, th, r, prec, work)
        return X, HX, th, r, Y

    for prec in (cs.CS_FP64, cs.CS_FP32, cs.CS_MIXED_BF16):
        nbytes = cs.cs_workspace_bytes(ctx, n_s, prec)
        buf = torch.full((nbytes + 4 * MIB,), 0xAB, dtype=torch.uint8, device="cuda")
        # what an earlier call left behind must not matter: NaN patterns, then zeros
        outs = []
        for fill in (0xFF, 0):
            buf[:nbytes] = fill
            outs.append(chain(prec, n_s, buf[:nbytes]))
        assert all(torch.equal(a, b) for a, b in zip(*outs))
        assert torch.all(buf[nbytes:] == 0xAB)
        # smaller blocks in the same workspace
        small = chain(prec, 5, buf[:nbytes])
        own = torch.zeros(cs.cs_workspace_bytes(ctx, 5, prec), dtype=torch.uint8, device="cuda")
        assert all(torch.equal(a, b) for a, b in zip(small, chain(prec, 5, own)))
        assert torch.all(buf[nbytes:] == 0xAB)
    nbytes = cs.cs_scf_workspace_bytes(ctx)
    buf = torch.full((nbytes + 4 * MIB,), 0xAB, dtype=torch.uint8, device="cuda")
    occ = torch.rand(n_s, generator=gen, dtype=torch.float64, device="cuda")
    grid = ctx.n_r * ctx.n_theta * ctx.n_phi
    rho = [torch.empty(grid, dtype=torch.float64, device="cuda") for _ in "ab"]
    vh = [torch.empty_like(rho[0]) for _ in "ab"]
    for i, fill in enumerate((0xFF, 0)):
        buf[:nbytes] = fill
        cs.cs_density(ctx, X0, occ, rho[i], buf[:nbytes])
        cs.cs_hartree(ctx, rho[i], vh[i], buf[:nbytes])
    assert torch.equal(*rho) and torch.equal(*vh)
    assert torch.all(buf[nbytes:] == 0xAB)
    assert cs.cs_device_error(ctx) == 0
