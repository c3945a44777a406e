"""Host checks of the slice-product kernels (csrc/sliced_hx.cu)."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "paper_1404_3773_gb300", "csrc", "sliced_hx.cu")

# what no kernel of a chain writes: set-up tables, W V of the potential, weights, occupations
CONSTANT = {"a.fexp", "a.rexp", "wv", "ewv", "wkj", "occ", "w"}


def _code():
    with open(SRC) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_chain_data_is_read_with_ordinary_loads():
    """A kernel launched early (griddepcontrol) is resident while its predecessor still writes, so
    what the chain writes may not be read through the read-only path, nor through a __restrict__
    pointer, whose loads the compiler may move above the wait."""
    code = _code()
    for arg in re.findall(r"__ldg\(\s*([A-Za-z_.]+)", code):
        assert arg in CONSTANT, f"__ldg({arg})"
    # in the pointwise pass `w` is a row of W V
    assert "const long long* w = wv + gr * Np;" in code
    early = 0
    for params, body in re.findall(r"__global__[^;{]*?\bk_sl\w*\(([^)]*)\)\s*\{(.*?)\n\}", code, re.S):
        if "pdl_wait()" not in body:
            continue
        early += 1
        assert body.index("pdl_wait()") >= body.index("pdl_trigger()")
        for name in re.findall(r"__restrict__\s+(\w+)", params):
            assert name in CONSTANT, f"__restrict__ {name}"
    assert early == 6  # k_sl, pointwise, fold, grid, density, gexp


def test_images_and_mmas_settle_after_an_expired_wait(tmp_path):
    """Whichever wait of whichever step expires, a CTA leaves with no bulk copy into its shared
    memory and no MMA on its tensor memory still open. A host program on modelled barriers."""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    # the kernel takes its slots, parities and last waits from the checked header
    code = _code()
    for use in ("image_slot(issued)", "image_slot(step)", "image_parity(step)", "mma_parity(step)",
                "settle_images("):
        assert use in code, use
    with open(os.path.join(os.path.dirname(SRC), "angular_wide.cu")) as f:
        phi = f.read().split("k_phi_tc(WaArgs a) {")[1].split("\nvoid residency")[0]
    for use in ("mbar_wait(bar_mma, given_up(ph_mma));\n    mbar_wait(bar_f, ph_f);",
                "ph_f = given_up(ph_f);\n      return false;", "mbar_wait(bar_tab, 0);\n"):
        assert use in phi, use
    src = os.path.join(os.path.dirname(__file__), "native", "image_ring_check.cu")
    exe = str(tmp_path / "image_ring_check")
    subprocess.run([nvcc, "-O2", "-std=c++17", "-o", exe, src], check=True, capture_output=True,
                   timeout=300)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout[-2000:]
