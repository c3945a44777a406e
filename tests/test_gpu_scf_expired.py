"""Device waits that expire in the density of an SCF step: the step reports CS_ERR_TIMEOUT, mixes
nothing and can be repeated. A stand-in for the launch leaves the error word and an invalid density
behind (tests/native/expired_density.cu); no wait expires on the GPU."""
import os
import shutil
import subprocess
import sys

import pytest

from tests.gpu_common import need_gpu

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import ctypes, sys
fake = ctypes.CDLL(sys.argv[1], mode=ctypes.RTLD_GLOBAL)
sys.path.insert(0, sys.argv[2])
import numpy as np, torch
import paper_1404_3773_gb300 as cs
import workloads as W

n_s = 16  # 20 x 14 x 16 rows: the density takes the slice products
ctx = cs.cs_basis_init(8.0, 6, 8, 20, 14, 28)
xyz = torch.tensor(cs.grid_points(ctx), device="cuda")
r2 = ((xyz - torch.tensor([0.3, -0.2, 0.4], device="cuda", dtype=torch.float64)) ** 2).sum(1)
v_ext = (-4.0 * torch.special.erf(r2.sqrt()) / r2.sqrt()).contiguous()
rho0 = (4.0 * (2 * np.pi) ** -1.5 * torch.exp(-r2 / 2)).contiguous()
v0 = torch.tensor(W.gaussian(17, ctx.d), device="cuda")
p = cs.ScfParams(n_s=n_s, n_want=6, degree=10, filter_prec=cs.CS_FP64, n_electrons=4.0, kT=1e-2,
                 beta=0.3, history=4, first_tol=1e-8, first_max_iter=60, lanczos_k=10, e_ion=0.0)
expire = ctypes.c_int.in_dll(fake, "expire_density")

def loop(fail_at):
    S = cs.cs_scf_create(ctx, p, v_ext, rho0, v0)
    X = torch.tensor(W.gaussian_block(31, ctx.d, n_s).T.copy(), device="cuda")
    theta = torch.empty(n_s, dtype=torch.float64, device="cuda")
    resid = torch.empty_like(theta)
    out = []
    while len(out) < 3:
        if len(out) + 1 == fail_at:
            expire.value = 1
            try:
                cs.cs_scf_step(S, X, theta, resid)
                raise SystemExit("the expired wait was not reported")
            except cs.CsError as e:
                assert "CS_ERR_TIMEOUT" in str(e), e
            assert expire.value == 0 and cs.cs_device_error(ctx) == 0
            fail_at = 0
        rep = cs.cs_scf_step(S, X, theta, resid)
        out.append((rep["iteration"], rep["energy"], rep["max_resid"]))
    S.close()
    return out

ref = loop(0)
assert ctypes.c_int.in_dll(fake, "density_calls").value == 3
for fail_at in (1, 2):
    got = loop(fail_at)
    assert [i for i, _, _ in got] == [1, 2, 3], got
    # the repeated step filters its block once more, so that the energies differ by less than the
    # residuals of both runs allow (first order, four electrons, three steps)
    r = 12.0 * max(x[2] for x in ref + got) + 1e-9
    assert all(abs(a - b) <= r for (_, a, _), (_, b, _) in zip(got, ref)), (got, ref)

# a density whose wait expired, then the integrals over it
rho = torch.ones(xyz.shape[0], dtype=torch.float64, device="cuda")
occ = torch.ones(n_s, dtype=torch.float64, device="cuda")
X = torch.tensor(W.gaussian_block(31, ctx.d, n_s).T.copy(), device="cuda")
expire.value = 1
cs.cs_density(ctx, X, occ, rho)
try:
    cs.cs_grid_integrals(ctx, [rho], [None])
    raise SystemExit("cs_grid_integrals did not report the expired wait")
except cs.CsError as e:
    assert "CS_ERR_TIMEOUT" in str(e), e
cs.cs_density(ctx, X, occ, rho)
assert np.isfinite(cs.cs_grid_integrals(ctx, [rho], [None])).all()
print("reported")
"""


def test_expired_wait_in_the_density_is_reported(tmp_path):
    need_gpu()
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    fake = str(tmp_path / "expired_density.so")
    subprocess.run([nvcc, "-O1", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-cudart", "shared",
                    "-gencode", "arch=compute_103a,code=sm_103a", "-o", fake,
                    os.path.join(ROOT, "tests", "native", "expired_density.cu"), "-ldl"],
                   check=True, capture_output=True, timeout=300)
    env = dict(os.environ, CLUSTERSPEC_LIB=os.path.join(ROOT, "paper_1404_3773_gb300",
                                                        "libclusterspec.so"))
    r = subprocess.run([sys.executable, "-c", CHILD, fake, ROOT], capture_output=True, text=True,
                       timeout=300, env=env, cwd=ROOT)
    assert r.returncode == 0 and "reported" in r.stdout, r.stdout[-2000:] + r.stderr[-3000:]
