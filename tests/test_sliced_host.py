"""Host checks of the slice-product kernels (csrc/sliced_hx.cu)."""
import os
import re

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
