"""CS_ANGULAR_KERNEL: which values keep the FP64-class calls on the FMA kernels. A value that chooses
among FP32 or mixed kernels, or an empty one, leaves the FP64 and double-float calls alone."""
import pytest

import workloads as W
from tests.gpu_common import make_ctx, need_gpu, register, to_dev

pytestmark = pytest.mark.gpu

W1 = W.small_cluster(lmax=24, nmax=6, n_r=40, n_theta=30, n_phi=60, n_s=20)  # 15.0M rows L^2
register(W1)

FMA_FP64 = {"stream": True, "rp": True, "rp2": True, "fma": True, "wide": False, "gm": False,
            "gm1": False, "tc": False, "": False}


@pytest.mark.parametrize("value", list(FMA_FP64))
def test_only_values_that_name_an_fma_kernel_switch_the_slices_off(value, monkeypatch):
    torch, cs = need_gpu()
    ctx = make_ctx(W1)
    X = to_dev(W1.x_block())

    def launches(prec):
        out = torch.zeros_like(X)
        n0 = cs.cs_launch_count(ctx)
        cs.cs_apply_H(ctx, X, out, prec)
        return cs.cs_launch_count(ctx) - n0, out

    monkeypatch.delenv("CS_ANGULAR_KERNEL", raising=False)
    n_slices, ref = launches(cs.CS_FP64)
    assert n_slices > 3
    monkeypatch.setenv("CS_ANGULAR_KERNEL", value)
    n64, a = launches(cs.CS_FP64)
    ndf, b = launches(cs.CS_DF64)
    assert (n64 == 3) == FMA_FP64[value] and (n64 == n_slices) != FMA_FP64[value]
    # the double-float call converts in and out around its own kernels
    assert (ndf == n_slices and torch.equal(b, ref)) != (FMA_FP64[value] or value == "wide")
    assert torch.equal(a, ref) or FMA_FP64[value]


def test_profile_tells_the_slice_products_apart(monkeypatch):
    torch, cs = need_gpu()
    ctx = make_ctx(W1)
    X = to_dev(W1.x_block())
    out = torch.zeros_like(X)
    names = cs.profile_class_names()

    def profile(prec):
        cs.cs_profile_begin(ctx)
        cs.cs_apply_H(ctx, X, out, prec)
        ms, n = cs.cs_profile_end(ctx)
        sms, sn = cs.cs_profile_sliced(ctx)
        assert all(0.0 <= b <= a for a, b in zip(ms, sms)) and len(names) == len(sn) == len(n)
        return [{k: v for k, v in zip(names, x) if v} for x in (n, sn)]

    monkeypatch.delenv("CS_ANGULAR_KERNEL", raising=False)
    fams = ("radial_synth", "angular", "radial_anal")
    assert profile(cs.CS_FP64) == [dict.fromkeys(fams, 1)] * 2
    assert profile(cs.CS_DF64) == [{f + "_df64": 1 for f in fams}] * 2
    monkeypatch.setenv("CS_ANGULAR_KERNEL", "fma")
    assert profile(cs.CS_FP64) == [dict.fromkeys(fams, 1), {}]
