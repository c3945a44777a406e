"""Mixed H.X and filter on blocks without 16-byte alignment: the radial analysis then passes through
shared memory or stores word by word, by size. Every form rounds alike, so that an odd leading
dimension returns the bits of an aligned block."""
import pytest

from tests.gpu_common import need_gpu

pytestmark = pytest.mark.gpu

# lmax, nmax, n_r, n_theta, n_phi, n_s. nmax <= 4; one partial tile per l; several tiles per l;
# more than one tile per SM; 112 functions per l (the last that one pass through shared memory
# takes) and more (two passes), with few and with many live columns
SHAPES = [(2, 4, 9, 5, 8, 5), (6, 16, 24, 16, 28, 1), (6, 16, 24, 16, 28, 33),
          (12, 32, 40, 26, 52, 20), (16, 20, 32, 34, 68, 80), (5, 112, 120, 12, 24, 9),
          (5, 116, 130, 12, 24, 2), (8, 116, 130, 18, 36, 64), (4, 240, 250, 10, 20, 3)]


@pytest.mark.parametrize("shape", SHAPES, ids=str)
def test_unaligned_blocks_return_the_aligned_bits(shape):
    torch, cs = need_gpu()
    lmax, nmax, n_r, n_theta, n_phi, n_s = shape
    ctx = cs.cs_basis_init(9.0, lmax, nmax, n_r, n_theta, n_phi)
    gen = torch.Generator(device="cuda").manual_seed(11)
    v = -torch.rand(n_r * n_theta * n_phi, generator=gen, dtype=torch.float64, device="cuda")
    cs.cs_set_potential(ctx, v)
    X = torch.randn((n_s, ctx.d), generator=gen, dtype=torch.float32, device="cuda")
    hi = float(cs.cs_kinetic(ctx).max()) + 1.0

    def run(ld):
        B = torch.zeros((n_s, ld), dtype=torch.float32, device="cuda")
        B[:, :ctx.d] = X
        out = torch.full_like(B, 7.0)
        cs.cs_apply_H(ctx, B, out, cs.CS_MIXED_BF16)
        assert torch.all(out[:, ctx.d:] == 7.0)
        cs.cs_cheb_filter(ctx, B, 3, 1.0, hi, -2.0, cs.CS_MIXED_BF16)
        assert torch.all(B[:, ctx.d:] == 0.0)
        return out[:, :ctx.d].clone(), B[:, :ctx.d].clone()

    aligned = run(ctx.d + (-ctx.d) % 4)
    for pad in (1, 3):
        got = run(ctx.d + (-ctx.d) % 4 + pad)
        assert all(torch.equal(a, b) for a, b in zip(got, aligned))
    # projectors add their block to the epilogue
    P = torch.randn((3, ctx.d), generator=gen, dtype=torch.float64, device="cuda") / ctx.d ** 0.5
    cs.cs_set_projectors(ctx, P, [0.5, -1.0, 2.0])
    aligned = run(ctx.d + (-ctx.d) % 4)
    got = run(ctx.d + (-ctx.d) % 4 + 1)
    assert all(torch.equal(a, b) for a, b in zip(got, aligned))
    assert cs.cs_device_error(ctx) == 0
