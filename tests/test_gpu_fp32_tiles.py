"""FP32 H.X at the edges of the register-blocked angular kernel's 8-row tiles: quarter angles and
mode classes that end inside a tile, blocks of one row, odd n_theta, a ragged last state tile."""
import pytest

import workloads as W
from tests.gpu_common import make_ctx, need_gpu, oracle_H, register, rel_errors, to_dev, to_host

pytestmark = pytest.mark.gpu

# lmax, nmax, n_r, n_theta, n_phi, n_s: padded quarter angles 4, 12, 20, 28, 32; even / odd modes
# per class 4/4, 8/4, 12/8, 16/12, 16/16 (padded to four)
EDGES = {
    "one_tile": (2, 4, 9, 5, 8, 3),
    "q12_m8_4": (8, 6, 13, 11, 36, 9),
    "q20_m12_8": (16, 5, 11, 20, 78, 17),
    "q28_m16_12": (24, 5, 9, 31, 108, 8),
    "q32_m16_16": (30, 4, 7, 33, 124, 5),
}


@pytest.mark.parametrize("case", list(EDGES))
def test_fp32_tile_edges(case):
    """Bars: those of every FP32 H.X against the oracle, 2e-5 and ten times that per column."""
    torch, cs = need_gpu()
    lmax, nmax, n_r, n_theta, n_phi, n_s = EDGES[case]
    w = W.small_cluster(lmax=lmax, nmax=nmax, n_r=n_r, n_theta=n_theta, n_phi=n_phi, n_s=n_s)
    register(w)
    ctx = make_ctx(w)
    X = w.x_block().astype("float32").astype("float64")
    Xd = to_dev(X, ld=ctx.d + 4, dtype=torch.float32)
    a = torch.zeros_like(Xd)
    cs.cs_apply_H(ctx, Xd, a, cs.CS_FP32)
    fro, col = rel_errors(to_host(a, ctx.d), oracle_H(w.name).apply(X))
    print(f"FP32 tiles {case}: fro {fro:.2e} col {col:.2e}")
    assert fro <= 2e-5 and col <= 2e-4, (fro, col)
