"""What the launch rules take for granted about the compiled GEMM kernels, from the compiler's own report."""
import os
import re

import pytest

from paper_2503_23367_b200 import build as fv_build


def test_builds_for_few_rows_fit_two_ctas_per_sm():
    """The launcher's rule for up to 48 rows counts two CTAs per SM; the compiler's own report has to bear it out."""
    fv_build.build()
    report = os.path.join(fv_build.BUILD, "gemm_cluster.ptxas.txt")
    if not os.path.exists(report):
        pytest.skip("built elsewhere")
    text = open(report).read()
    found = re.findall(r"gemm_cluster_kernelILi128ELi(\d)ELi(32|64)E.*?Used (\d+) registers", text, flags=re.S)
    builds = {(int(s), int(rows)): int(regs) for s, rows, regs in found}
    assert set(builds) == {(s, rows) for s in (2, 4, 8) for rows in (32, 64)}
    for key, regs in builds.items():
        per_warp = -(-regs * 32 // 256) * 256                    # registers are handed out to a warp 256 at a time
        assert 2 * 6 * per_warp <= 65536, (key, regs)
