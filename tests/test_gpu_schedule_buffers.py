"""Schedules whose buffers overlap one another or the arena come to what the same calls do one at a time: a tensor that lies where an
earlier container is written, tensors restored over a container, over one another in part, over an input, in place."""
import numpy as np
import pytest

from paper_2510_11400_b200 import api, synth
from tests.test_gpu_parity import to_dev

pytestmark = pytest.mark.gpu

# (restored in reverse order; the second one is the larger, so that it is still at work when the first one's turn comes)
SHAPES = [(1, 64, 14, 14), (1, 60, 112, 112), (4, 64, 14, 14), (8, 64, 32, 32), (2, 61, 7, 7)]
PARAMS = dict(bits=8)


def esize(dtype):
    return 4 if dtype == synth.F32 else 2


def a256(n):
    return (n + 255) & ~255


class Buffers:
    """One piece of device memory with the arena at its start, then the inputs, then the restored tensors."""

    def __init__(self, dtype, shapes):
        import torch
        self.dtype, self.shapes = dtype, shapes
        self.sizes = [int(np.prod(s)) * esize(dtype) for s in shapes]
        self.descs = [api.desc(s, api.FH_F32 if dtype == synth.F32 else api.FH_BF16, tensor_id=i) for i, s in enumerate(shapes)]
        worst = [a256(api.compressed_bytes(d, api.default_params(**PARAMS), 1)) for d in self.descs]
        self.arena_bytes = sum(worst)
        at = self.arena_bytes
        self.inputs, self.outputs = [], []
        for places in (self.inputs, self.outputs):
            for n in self.sizes:
                places.append(at)
                at += a256(n)
        self.pool = torch.zeros(at, dtype=torch.uint8, device="cuda")

    def part(self, place, i):
        import torch
        return self.pool[place:place + self.sizes[i]].view(torch.float32 if self.dtype == synth.F32 else torch.int16)

    def fill(self, i, values):
        x = to_dev(values)
        self.part(self.inputs[i], i).copy_(x.view(self.part(self.inputs[i], i).dtype).flatten())

    def items(self):
        return [api.SchedItem(d, api.FH_COMPRESS, self.part(self.inputs[i], i), self.part(self.outputs[i], i)) for i, d in enumerate(self.descs)]


def one_at_a_time(items, p, arena):
    import torch
    out2, st = torch.zeros(2, dtype=torch.int64, device="cuda"), torch.zeros(1, dtype=torch.int64, device="cuda")
    at, places = 0, []
    for it in items:
        assert api.fh_compress(it.desc, p, it.dense, arena[at:], out2) == api.FH_OK
        torch.cuda.synchronize()
        n, status = out2.tolist()
        assert status == api.FH_OK
        places.append((at, n))
        at += a256(n)
    for it, (place, n) in reversed(list(zip(items, places))):
        assert api.fh_decompress(arena[place:], arena.numel() - place, it.desc, it.restored, st) == api.FH_OK
        torch.cuda.synchronize()
        assert int(st.item()) == api.FH_OK
    return sum(n for _, n in places)


def container(shapes, i, dtype):
    """Where container i starts when all planes of those before it are normal."""
    p = api.default_params(**PARAMS)
    return sum(a256(api.compressed_bytes(api.desc(s, api.FH_F32 if dtype == synth.F32 else api.FH_BF16), p)) for s in shapes[:i])


def lay_out(case, dtype):
    """Buffers with the case's overlap and values in them."""
    shapes = list(SHAPES)
    if case == "input where an earlier container is written":
        shapes[0], shapes[1] = shapes[1], shapes[0]
    b = Buffers(dtype, shapes)
    for i, s in enumerate(shapes):
        b.fill(i, synth.make(synth.TensorSpec("b", s, dtype, "normal", 700 + i)))
    if case == "input where an earlier container is written":
        # the first tensor's planes are constant, so their codes are zero; the second tensor lies among them, with other values before
        b.part(b.inputs[0], 0).fill_(1)
        place = 64 + 16 * 60 + 40 * 12544
        b.inputs[1] = place
        b.fill(1, synth.make(synth.TensorSpec("b", shapes[1], dtype, "normal", 701)))
        assert place + b.sizes[1] <= 64 + 16 * 60 + 60 * 12544 <= container(shapes, 1, dtype)
    elif case == "restored over a container":
        b.outputs[0] = container(shapes, 1, dtype)      # container 1 has been restored by then
    elif case == "restored in part over one another":
        b.outputs[0] = b.outputs[1] + b.sizes[1] - b.sizes[0] // 2 & ~15
        b.outputs[2] = b.outputs[1] - b.sizes[2] // 2 & ~15
    elif case == "restored over an input":
        b.outputs[0] = b.inputs[1]
    elif case == "restored in place":
        b.outputs = list(b.inputs)
    return b


@pytest.mark.parametrize("dtype", [synth.F32, synth.BF16])
@pytest.mark.parametrize("case", ["apart", "input where an earlier container is written", "restored over a container",
                                  "restored in part over one another", "restored over an input", "restored in place"])
def test_overlapping_buffers(case, dtype):
    import torch
    p = api.default_params(**PARAMS)
    alone = lay_out(case, dtype)
    packed = one_at_a_time(alone.items(), p, alone.pool[:alone.arena_bytes])
    torch.cuda.synchronize()
    for _ in range(3):
        b = lay_out(case, dtype)
        torch.cuda.synchronize()
        rep = api.fh_run_schedule(b.items(), p, b.pool[:b.arena_bytes])
        assert rep.status == api.FH_OK and rep.total_packed_bytes == packed
        torch.cuda.synchronize()
        assert torch.equal(b.pool, alone.pool)


def test_a_schedule_on_several_streams_and_with_one_entry():
    """Side streams belong to the stream's scratch: schedules on streams of the caller's, one after the other and again after a
    shutdown; one entry and two need none or one of them."""
    import torch
    p = api.default_params(**PARAMS)
    alone = lay_out("apart", synth.F32)
    one_at_a_time(alone.items(), p, alone.pool[:alone.arena_bytes])
    streams = [torch.cuda.Stream() for _ in range(3)] + [None]
    for stream in streams + streams:
        for count in (5, 1, 2):
            b = lay_out("apart", synth.F32)
            torch.cuda.synchronize()
            rep = api.fh_run_schedule(b.items()[:count], p, b.pool[:b.arena_bytes], stream=stream)
            torch.cuda.synchronize()
            assert rep.status == api.FH_OK
            for i in range(count):
                assert torch.equal(b.part(b.outputs[i], i), alone.part(alone.outputs[i], i))
        if stream is None:
            api.shutdown()
