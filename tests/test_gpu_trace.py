"""The clock traces print the kernel that ran, under its own slot map: every stamp a title's kernel is said to make is there, and the
steps of one role come in order."""
import re
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("what, kernels", [("small_m", ["rotate_quant_kernel", "w4a4_narrow_kernel"]), ("w4a4", ["w4a4_gemm_kernel"]),
                                           ("nvfp4", ["nvfp4_gemm_kernel"]), ("w4a8", ["w4a8_pair_kernel"]), ("w4a8_single", ["w4a8_gemm_kernel"])])
def test_trace(what, kernels):
    r = subprocess.run([sys.executable, "-m", "paper_2605_16732_b200.trace", "--what", what], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    titles = [line for line in r.stdout.splitlines() if not line.startswith(" ")]
    assert [t.split(",")[0] for t in titles] == kernels
    rows = [[int(v) for v in re.split(r"\s{2,}", line.strip())[1].split()] for line in r.stdout.splitlines() if line.startswith(" ")]
    assert len(rows) >= 4 * len(kernels)
    for row in rows:
        assert row == sorted(row) and row[0] >= 0 and row[-1] < 10 ** 7, r.stdout
