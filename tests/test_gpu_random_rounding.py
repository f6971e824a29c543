"""Random rounding: codes by a sum of integers.  Parity with the oracle, whose definition is the fraction compared with the draw,
where that could go wrong: ranges near the ends of fp32, values at and around the last code, every kernel that draws."""
import numpy as np
import pytest

from oracle import fho
from paper_2510_11400_b200 import api, synth
from tests.test_gpu_parity import to_dev

pytestmark = pytest.mark.gpu


def _bits(x, dtype):
    """float32 values as the tensor's own type (bf16: bit patterns, truncated)."""
    return x if dtype == synth.F32 else (x.view(np.uint32) >> 16).astype(np.uint16)


@pytest.mark.parametrize("scale", [1e-44, 1e-38, 1e-30, 1.0, 1e30])
@pytest.mark.parametrize("hw,mode", [((7, 7), api.FH_SALIENT_AUTO), ((19, 27), api.FH_SALIENT_AUTO), ((32, 32), api.FH_SALIENT_AUTO),
                                     ((56, 56), api.FH_SALIENT_AUTO), ((37, 35), api.FH_SALIENT_AUTO), ((14, 14), api.FH_SALIENT_OFF),
                                     ((5, 5), api.FH_SALIENT_OFF)])
@pytest.mark.parametrize("dtype", [synth.F32, synth.BF16])
def test_parity_at_the_ends_of_the_range(scale, hw, mode, dtype):
    shape = (2, 9, *hw)
    rng = np.random.default_rng([7, *hw])
    x = rng.uniform(0.0, 1.0, shape).astype(np.float32)
    x[:, 1] = np.round(x[:, 1] * 255.0) / 255.0     # many elements at whole codes, the last one among them
    x[:, 2, :, 1:] = 0.0                            # zeros and a few others
    x[:, 3] = 0.25                                  # constant
    x[:, 4, 0, :3] = (0.0, 1.0, np.nextafter(np.float32(1.0), np.float32(0.0)))
    raw = _bits((x * np.float32(scale)).astype(np.float32), dtype)
    for bits in (2, 4, 8):
        kw = dict(bits=bits, rounding=1, seed=0x0123456789ABCDEF, salient_mode=mode)
        st_o, buf_o, total_o = fho.compress(raw, fho.desc(shape, dtype, tensor_id=11), fho.params(**kw))
        st_g, packed, total_g = api.compress_tensor(to_dev(raw), shape, dtype, api.default_params(**kw), tensor_id=11)
        assert st_o == fho.OK and st_g == api.FH_OK and total_g == total_o
        assert np.array_equal(packed[:total_g].cpu().numpy(), buf_o), (scale, hw, bits)
