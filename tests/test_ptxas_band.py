"""Register and spill budget of the kernels of a band-limited mixed frame, as
test_ptxas_budget.py's: the coarse sums run eight 64-thread CTAs per SM (128
registers), the interpolation four of 256 threads (64, for which it spills a
little: measured faster than two CTAs without), the one-launch sort one of
1024 (64); none of the others spills.
"""
import os
import re
import shutil

import pytest

from paper_2208_10939_gb300 import _build
from test_ptxas_budget import _ptxas_report

pytestmark = pytest.mark.slow

# (translation unit, demangled-name regex, register limit or None, spilled bytes)
BUDGET = [
    ("band.cu", r"synth_band_kernel\(", 128, 0),
    ("band.cu", r"band_expand_kernel\(", 64, 160),
    ("band.cu", r"band_(plan|ref|small|lists|items|fill|reduce)_kernel\(", None, 0),
    ("visibility.cu", r"(visibility(_single|_far)?|compact_\w+)_kernel\(", None, 0),
    ("scene_bvh.cu", r"cluster_sort_kernel\(", 64, 0),
    ("scene_bvh.cu", r"(build_facets|leaf_levels|lbvh_\w+)_kernel\(", None, 0),
]


@pytest.fixture(scope="module")
def reports(tmp_path_factory):
    if shutil.which("c++filt") is None:
        pytest.skip("c++filt not available")
    try:
        _build.nvcc()
    except RuntimeError as e:
        pytest.skip(str(e))
    out = str(tmp_path_factory.mktemp("ptxas"))
    return {u: _ptxas_report(os.path.join(_build.CSRC, u), out) for u in sorted({b[0] for b in BUDGET})}


@pytest.mark.parametrize("unit,pattern,reg_limit,spilled", BUDGET, ids=[b[1] for b in BUDGET])
def test_band_frame_kernels_fit_their_budget(reports, unit, pattern, reg_limit, spilled):
    found = {n: v for n, v in reports[unit].items() if re.search(pattern, n)}
    assert found, f"no entry function matching {pattern} in {unit}"
    for name, (regs, st, ld) in found.items():
        assert max(st, ld) <= spilled, f"{name}: {st} bytes spill stores, {ld} loads"
        if reg_limit is not None:
            assert regs <= reg_limit, f"{name}: {regs} registers > {reg_limit}"
