"""Which planes fit the block-wise path's shared memory with the Huffman stage: the largest of four shapes and the next one."""
import ctypes as C

import pytest

from paper_2510_11400_b200 import api, synth
from tests.test_gpu_parity import full_parity

LARGEST = [(synth.F32, 225, 225), (synth.F32, 2, 25446), (synth.F32, 12642, 3), (synth.F32, 8, 6369),
           (synth.BF16, 308, 308), (synth.BF16, 2, 47988), (synth.BF16, 19453, 3), (synth.BF16, 8, 12027)]
OK, ARG, UNSUPPORTED = 0, -1, -2


def checked(dtype, h, w):
    """What the schedule runner's own check says of a plane.  Its entries are checked in order and before anything is launched,
    and the second one is never valid, so this neither needs nor touches a GPU: FH_ERR_ARG means that the first one passed."""
    e = (api.fh_sched_entry * 2)()
    e[0].desc = api.fh_tensor_desc(0 if dtype == synth.F32 else 1, 2, 2, h, w, 0)
    e[0].action, e[0].d_dense, e[0].d_restored = 1, 4096, 4096
    e[1].action = 99
    p = api.default_params()
    p.entropy = 1
    return api.lib().fh_run_schedule(e, 2, C.byref(p), 4096, 1 << 40, C.byref(api.fh_sched_report()), None)


@pytest.mark.parametrize("dtype,h,w", LARGEST)
def test_the_largest_planes_are_taken_and_no_larger_ones(dtype, h, w):
    assert checked(dtype, h, w) == ARG
    grown = (h + 1, w + 1) if h == w else (h, w + 1) if w > h else (h + 1, w)
    assert checked(dtype, *grown) == UNSUPPORTED


@pytest.mark.gpu
@pytest.mark.parametrize("dtype,h,w", LARGEST)
def test_parity_of_the_largest_planes(dtype, h, w):
    full_parity(synth.TensorSpec("t", (1, 2, h, w), dtype, "spiky_relu", 61), entropy=1, salient_mode=api.FH_SALIENT_ALL)
