"""Parity of the statistics per channel and per tensor with the oracle where a warp takes runs of pieces: planes around one, two and
many pieces of 512 groups, fewer and more pieces than warps, runs that begin and end inside a channel."""
import numpy as np
import pytest

from paper_2510_11400_b200 import api, synth
from tests.test_gpu_parity import full_parity, gpu_compress, oracle_compress

pytestmark = pytest.mark.gpu

SHAPES = [(7, 5, 2, 130), (3, 61, 20, 20), (40, 130, 4, 66), (5, 3, 32, 64), (9, 7, 4, 513), (2, 3, 64, 64), (6, 11, 4, 1025), (1, 37, 56, 56),
          (3, 2, 200, 140), (700, 11, 4, 72)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("dtype", [synth.F32, synth.BF16])
@pytest.mark.parametrize("mode", [api.FH_SALIENT_CHANNEL, api.FH_SALIENT_TENSOR])
def test_parity_of_runs_of_pieces(shape, dtype, mode):
    for kind in ("spiky_relu", "normal"):
        full_parity(synth.TensorSpec("t", shape, dtype, kind, 81), bits=4, salient_mode=mode)


def test_parity_where_the_rule_does_not_apply():
    spec = synth.TensorSpec("t", (4, 6, 24, 24), synth.F32, "normal", 82)
    x = synth.make(spec).reshape(4, 6, 24, 24)
    x[:, 1] = 0.75           # a constant channel
    x[:, 3] *= np.float32(1e-20)   # a range below the rule's domain
    for mode in (api.FH_SALIENT_CHANNEL, api.FH_SALIENT_TENSOR):
        for data in (x, x * np.float32(1e-20)):
            st_o, buf_o, total_o, _ = oracle_compress(data.reshape(-1), spec.shape, spec.dtype, bits=2, salient_mode=mode)
            st_g, packed, total_g = gpu_compress(data.reshape(-1), spec.shape, spec.dtype, bits=2, salient_mode=mode)
            assert st_o == st_g == api.FH_OK and total_o == total_g
            assert np.array_equal(packed[:total_g].cpu().numpy(), buf_o)
