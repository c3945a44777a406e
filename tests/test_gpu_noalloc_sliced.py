"""cs_apply_H_noalloc returns the bits of cs_apply_H also for FP64 blocks that take the slice
products: the library's array then holds G and a part of the radial nodes at a time."""
import pytest

import workloads as W
from tests.gpu_common import make_ctx, need_gpu, register, to_dev

pytestmark = pytest.mark.gpu

# lmax, nmax, n_r, n_theta, n_phi, n_s: all states and nodes at once; G above half the array (two
# passes of 75 states, one or several nodes at a time); the basis limits, one state per pass
CASES = {"small": (6, 8, 20, 14, 28, 16), "odd_theta": (9, 16, 33, 23, 42, 17),
         "two_passes": (20, 6, 48, 24, 44, 150), "one_state": (62, 5, 300, 64, 128, 3)}


@pytest.mark.parametrize("case", list(CASES))
def test_noalloc_returns_the_bits_of_apply(case, monkeypatch):
    torch, cs = need_gpu()
    monkeypatch.delenv("CS_ANGULAR_KERNEL", raising=False)
    lmax, nmax, n_r, n_theta, n_phi, n_s = CASES[case]
    w = W.small_cluster(lmax=lmax, nmax=nmax, n_r=n_r, n_theta=n_theta, n_phi=n_phi, n_s=n_s)
    register(w)
    ctx = make_ctx(w)
    X = to_dev(w.x_block(), ld=ctx.d + 3)
    ref, got = torch.zeros_like(X), torch.zeros_like(X)
    n0 = cs.cs_launch_count(ctx)
    cs.cs_apply_H(ctx, X, ref, cs.CS_FP64)
    assert cs.cs_launch_count(ctx) - n0 > 3  # the slice products
    for _ in range(2):  # the second call finds the first one's contents in the array
        got.zero_()
        cs.cs_apply_H_noalloc(ctx, X, got, cs.CS_FP64)
        assert torch.equal(got, ref)
    assert cs.cs_device_error(ctx) == 0
