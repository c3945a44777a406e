"""The double-float phi pass keeps its table as values or as broadcast pairs, by the CTAs that shared
memory leaves: both against the row-stream kernel, on grids on either side of the rule."""
import pytest

import workloads as W
from tests.gpu_common import make_ctx, need_gpu, register, rel_errors, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_phi", [124, 148, 180, 240])  # values up to 148, pairs above
def test_double_float_phi_tables(n_phi, monkeypatch):
    torch, cs = need_gpu()
    monkeypatch.delenv("CS_ANGULAR_KERNEL", raising=False)
    # at most 7.8M rows x L^2: below the slice products; 34 states: a second, ragged block
    w = W.small_cluster(lmax=60, nmax=3, n_r=1 + 3 * (n_phi == 124), n_theta=62, n_phi=n_phi,
                        n_s=5 if n_phi == 124 else 34 if n_phi == 180 else 3)
    register(w)
    ctx = make_ctx(w)
    X = to_dev(w.x_block(), ld=ctx.d + 3)
    a, b = torch.zeros_like(X), torch.zeros_like(X)
    cs.cs_apply_H(ctx, X, a, cs.CS_DF64)
    monkeypatch.setenv("CS_ANGULAR_KERNEL", "stream")
    cs.cs_apply_H(ctx, X, b, cs.CS_DF64)
    fro, col = rel_errors(to_host(a, ctx.d), to_host(b, ctx.d))
    assert 0 < fro <= 1e-12 and col <= 1e-12, (fro, col)  # the double-float level
    assert torch.all(a[:, ctx.d:] == 0.0)
