"""The grouped INT4 second kernel for few token rows (128 x 64 tiles, one hand-over per 128 codes): an odd number of groups (the last k-block
has one), a single k-block, ragged rows and columns, several tiles per CTA; against the oracle."""
import pytest

import test_gpu_parity
from paper_2605_16732_b200 import binding as dq
from paper_2605_16732_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("knob", [64, 66])  # one CTA per tile; the reduction split over a cluster where it applies
@pytest.mark.parametrize("M, K, N, r, G", [
    (1, 512, 80, 64, 64),      # 7 groups
    (129, 128, 144, 32, 64),   # 96 codes: one k-block
    (257, 640, 400, 128, 128),  # 4 groups of 128, two rank-r chunks
    (1500, 320, 1200, 16, 64),  # 5 groups (the last one partly padding); 228 tiles
])
def test_parity(knob, M, K, N, r, G):
    dq.dirotq_set_gemm_tile(knob)
    try:
        spec = synth.LayerSpec(K=K, N=N, r=r, G=G, model=synth.PIXART, seed=K + M, calib_tokens=512)
        test_gpu_parity._run_case(spec, M=M, check_rot=False)
    finally:
        dq.dirotq_set_gemm_tile(0)
