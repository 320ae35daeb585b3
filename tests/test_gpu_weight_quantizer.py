"""The residual weight's quantizer, alone: with the identity as rotation the fold is exact, so codes and scales equal the oracle's without exception, at
ragged last groups and column blocks, with exact ties, groups of zeros and scales among bf16's smallest numbers."""
import numpy as np
import pytest
import torch

from oracle import dirotq_oracle as orc
from paper_2605_16732_b200 import binding as dq

from parity_utils import bf16_tensor_to_bits

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,N,r,G", [(64, 16, 16, 64), (256, 48, 32, 64), (256, 80, 16, 128), (128, 32, 32, 128), (512, 1040, 64, 64)])
def test_codes_and_scales(K, N, r, G):
    rng = np.random.default_rng(K + N)
    W = rng.standard_normal((K, N)).astype(np.float32)
    W[:, 1] *= np.float32(1e-39)
    W[:, 2] = 0
    W[:, 3] = 0.125 * rng.integers(-14, 15, K) / 2  # scale 1/8: every odd multiple of 1/16 is a tie
    W[r::G, 3] = 0.875
    W[r:r + G, 4] = 0
    lo = orc.prepare_layer(W, np.eye(K), r, G)
    layer = dq.dirotq_prepare_layer(torch.from_numpy(W).cuda(), torch.eye(K, dtype=torch.float64, device="cuda"), r, G)
    wcodes, wscales, _, _ = dq.dirotq_layer_export(layer)
    assert np.array_equal(bf16_tensor_to_bits(wscales), lo["wscales"])
    assert np.array_equal(wcodes.cpu().numpy(), lo["wcodes"])
    layer.close()
