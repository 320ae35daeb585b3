"""The rotation kernel's 128 x 128 plan in CTA pairs (256 tokens x 128 columns per pair): a second CTA with one row or none, ragged columns,
two chunks per tile (groups of 64) and one (groups of 128), every epilogue it serves; against the oracle."""
import pytest

import test_gpu_asym
import test_gpu_parity
import test_gpu_w4a8
from paper_2605_16732_b200 import binding as dq
from paper_2605_16732_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("run, M, K, r, G", [
    (test_gpu_parity._run_case, 129, 448, 32, 64),   # 3.5 column tiles
    (test_gpu_parity._run_case, 257, 640, 128, 128),
    (test_gpu_parity._run_case, 384, 64, 16, 64),    # one k-block
    (test_gpu_asym._run_case, 300, 704, 32, 64),
    (test_gpu_w4a8._run_case, 257, 576, 32, 64),
])
def test_parity(run, M, K, r, G):
    dq.dirotq_set_rotation_tile(1)
    try:
        run(synth.LayerSpec(K=K, N=160, r=r, G=G, model=synth.PIXART, seed=K + M, calib_tokens=512), M=M)
    finally:
        dq.dirotq_set_rotation_tile(0)
