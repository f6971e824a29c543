"""Schedules whose kernels run side by side: inputs that are loaded before the previous kernel has ended, decompress kernels that
do not wait for one another; and buffers that overlap, whose results depend on the order."""
import numpy as np
import pytest

from paper_2510_11400_b200 import api, synth
from tests.test_gpu_parity import to_dev

pytestmark = pytest.mark.gpu

SHAPES = [(4, 16, 56, 56), (2, 64, 7, 7), (3, 20, 112, 112), (16, 64, 14, 14), (1, 7, 33, 17), (8, 64, 32, 32), (64, 64, 4, 4), (2, 12, 149, 149)]


def _alone(items, p):
    """Every item compressed and restored by itself, in its own buffers."""
    import torch
    packed, restored = [], []
    for it in items:
        dst = torch.zeros(api.compressed_bytes(it.desc, p, 1), dtype=torch.uint8, device="cuda")
        out2, st, out = torch.zeros(2, dtype=torch.int64, device="cuda"), torch.zeros(1, dtype=torch.int64, device="cuda"), torch.empty_like(it.dense)
        assert api.fh_compress(it.desc, p, it.dense, dst, out2) == api.FH_OK
        torch.cuda.synchronize()
        n, status = out2.tolist()
        assert status == api.FH_OK and api.fh_decompress(dst, n, it.desc, out, st) == api.FH_OK
        torch.cuda.synchronize()
        assert int(st.item()) == api.FH_OK
        packed.append(dst[:n])
        restored.append(out)
    return packed, restored


def _items(dtype, count):
    import torch
    items = []
    for i in range(count):
        shape = SHAPES[i % len(SHAPES)]
        kind = ("spiky_relu", "normal", "relu")[i % 3]
        x = to_dev(synth.make(synth.TensorSpec("s", shape, dtype, kind, 900 + i)))
        items.append(api.SchedItem(api.desc(shape, api.FH_F32 if dtype == synth.F32 else api.FH_BF16, tensor_id=i), api.FH_COMPRESS, x,
                                   torch.empty_like(x)))
    return items


@pytest.mark.parametrize("dtype", [synth.F32, synth.BF16])
@pytest.mark.parametrize("kw", [dict(bits=4), dict(bits=2, entropy=1), dict(bits=8, rounding=1, seed=3),
                                dict(bits=4, salient_mode=api.FH_SALIENT_CHANNEL), dict(bits=4, salient_mode=api.FH_SALIENT_OFF)])
def test_containers_and_restored_tensors_are_those_of_calls_alone(dtype, kw):
    import torch
    p = api.default_params(**kw)
    items = _items(dtype, 19)
    packed, restored = _alone(items, p)
    arena = torch.zeros(sum((api.compressed_bytes(i.desc, p, 1) + 255) & ~255 for i in items), dtype=torch.uint8, device="cuda")
    for _ in range(5):
        arena.zero_()
        for i in items:
            i.restored.zero_()
        torch.cuda.synchronize()
        rep = api.fh_run_schedule(items, p, arena)
        assert rep.status == api.FH_OK and rep.total_packed_bytes == sum(b.numel() for b in packed)
        at = 0
        for it, b, r in zip(items, packed, restored):
            assert torch.equal(arena[at:at + b.numel()], b) and torch.equal(it.restored, r)
            at += (b.numel() + 255) & ~255


def test_buffers_that_overlap_keep_the_order():
    """Restored in reverse order: of two items that share a buffer, the one listed first is restored last."""
    import torch
    p = api.default_params(bits=4)
    items = _items(synth.F32, 17)
    _, restored = _alone(items, p)
    items[16].restored = items[0].restored = items[8].restored      # (the same shape)
    items[3].restored = items[3].dense                             # in place
    arena = torch.zeros(sum((api.compressed_bytes(i.desc, p, 1) + 255) & ~255 for i in items), dtype=torch.uint8, device="cuda")
    rep = api.fh_run_schedule(items, p, arena)
    assert rep.status == api.FH_OK
    assert all(torch.equal(items[i].restored, restored[i]) for i in range(17) if i not in (8, 16))
    assert not np.array_equal(restored[0].cpu().numpy(), restored[8].cpu().numpy())
