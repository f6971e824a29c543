"""Workloads of the activation codec, for timing: what a training engine asks of it, through the Python binding.

A case is one pass over a list of saved activations, as a training step makes it: `forward` compresses every tensor in
order, `backward` restores every tensor in reverse order from containers that are at hand, `step` does both, and
`schedule` hands the list to fh_run_schedule.  `shapes` lists the tensors (n x c x h x w), `kind` says how their values
are distributed (the recipes of the package's synth module, drawn on the GPU), the other fields are the codec's
parameters.  Every container and every restored tensor comes back whole.
"""
from __future__ import annotations

import math

import torch

from paper_2510_11400_b200 import api

SCOPES = {"auto": api.FH_SALIENT_AUTO, "off": api.FH_SALIENT_OFF, "channel": api.FH_SALIENT_CHANNEL,
          "tensor": api.FH_SALIENT_TENSOR}


def _resnet18(batch):
    """Saved activations of a ResNet-18-shaped CNN at 224 x 224."""
    return [(batch, 64, 112, 112)] + [(batch, 64, 56, 56)] * 4 + [(batch, 128, 28, 28)] * 4 + \
        [(batch, 256, 14, 14)] * 4 + [(batch, 512, 7, 7)] * 4


def _mobilenetv2(batch):
    """Expanded depthwise tensors of a MobileNetV2-shaped CNN at 224 x 224."""
    return [(batch, 96, 112, 112), (batch, 144, 56, 56), (batch, 192, 28, 28), (batch, 384, 14, 14), (batch, 960, 7, 7)]


def _cifar(batch):
    """Twenty saved activations of a ResNet-18-shaped CNN on 32 x 32 input; the schedule compresses every other one."""
    return [(batch, 64, 32, 32)] * 5 + [(batch, 128, 16, 16)] * 5 + [(batch, 256, 8, 8)] * 5 + [(batch, 512, 4, 4)] * 5


def _case(op, shapes, dtype, kind, bits, scope="auto", rounding=0, entropy=0, name=None):
    c = {} if name is None else {"name": name}
    c.update(op=op, shapes=",".join("x".join(map(str, s)) for s in shapes), dtype=dtype, kind=kind, bits=bits,
             scope=scope, rounding=rounding, entropy=entropy)
    return c


def listed():
    return [
        # One small tensor there and back: the latency of a single call in each direction.
        _case("step", [(32, 16, 32, 32)], "f32", "relu", 2, name="small_tensor_step"),
        # The forward and the backward pass of the headline workload: planes from 112 x 112 down to 7 x 7, half of
        # the tensors post-ReLU, half pre-activation.
        _case("forward", _resnet18(64), "f32", "mixed", 4, name="resnet18_b64_forward"),
        _case("backward", _resnet18(64), "f32", "mixed", 4, name="resnet18_b64_backward"),
        # A whole step in bf16 with rare large values: independent per element, and clustered in every eighth channel
        # (those channels' planes take the block-wise path).
        _case("step", _mobilenetv2(128), "bf16", "laplace_iid", 2, name="mobilenetv2_b128_bf16_step"),
        _case("step", _mobilenetv2(128), "bf16", "laplace_ch", 2, name="mobilenetv2_b128_bf16_outliers"),
        # Large single tensors, one direction each: the memory-bound end.
        _case("forward", [(4096, 64, 32, 32)], "f32", "relu", 2, name="single_1gib_f32_forward"),
        _case("backward", [(8192, 64, 32, 32)], "bf16", "relu", 8, name="single_1gib_bf16_backward"),
        # One training step handed over as a schedule, report read on the host.
        _case("schedule", _cifar(128), "f32", "relu", 2, name="cifar_b128_schedule"),
        # Feature maps whose sides are no multiples of anything: planes that start off the 16-byte grid.
        _case("step", [(8, 64, 149, 149), (8, 61, 73, 73), (8, 192, 35, 35), (8, 256, 27, 27), (8, 61, 33, 17), (8, 768, 17, 17),
                       (8, 383, 13, 13)], "f32", "mixed", 8, name="odd_sizes_step"),
        # The codec's options: random rounding, three-sigma statistics per channel over the batch, Huffman stage.
        _case("forward", _resnet18(64), "f32", "mixed", 2, rounding=1, name="random_rounding_forward"),
        _case("forward", _mobilenetv2(32), "bf16", "laplace_ch", 4, scope="channel", name="channel_scope_forward"),
        _case("step", _resnet18(8), "f32", "spiky", 4, entropy=1, name="huffman_step"),
    ]


def _elems(shapes):
    return sum(math.prod(s) for s in shapes)


def _log_int(rng, lo, hi):
    return max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    dtype = rng.choice(["f32", "bf16"])
    bits = rng.choice([2, 4, 8])
    op = rng.choice(["forward", "backward", "step"])
    what = rng.choice(["network", "network", "single", "single", "odd", "odd", "schedule", "option"])
    if what == "network":
        net, most = rng.choice([(_resnet18, 64), (_mobilenetv2, 128)])
        b = _log_int(rng, 1, most if op != "step" or dtype == "bf16" else most // 2)
        kind = rng.choice(["mixed", "mixed", "laplace_iid", "laplace_ch"])
        return _case(op, net(b), dtype, kind, bits, scope=rng.choice(["auto", "auto", "auto", "off"]))
    if what == "single":
        h, w = _log_int(rng, 4, 128), _log_int(rng, 4, 128)
        planes = max(1, _log_int(rng, 1 << 18, 1 << 27) // (h * w))
        c = min(planes, rng.choice([16, 24, 61, 64, 128]))
        return _case(op, [(max(1, planes // c), c, h, w)], dtype, rng.choice(["relu", "normal", "laplace_iid"]), bits)
    if what == "odd":
        shapes = []
        for _ in range(rng.randint(3, 7)):
            h = _log_int(rng, 5, 150)
            w = h if rng.random() < 0.7 else _log_int(rng, 5, 150)
            shapes.append((_log_int(rng, 1, 16), min(rng.randrange(17, 800, 2), max(1, (1 << 21) // (h * w))), h, w))
        return _case(op, shapes, dtype, rng.choice(["mixed", "normal", "laplace_iid"]), bits)
    if what == "schedule":
        return _case("schedule", _cifar(_log_int(rng, 1, 160)), dtype, rng.choice(["relu", "mixed"]), bits)
    net, most = rng.choice([(_resnet18, 32), (_mobilenetv2, 32)])
    option = rng.choice([{"rounding": 1}, {"scope": "channel"}, {"scope": "tensor"}, {"entropy": 1}])
    b = _log_int(rng, 1, most if "entropy" not in option else 8)
    return _case(op, net(b), dtype, rng.choice(["mixed", "laplace_ch"]), bits, **option)


def _shapes(case):
    return [tuple(int(v) for v in s.split("x")) for s in case["shapes"].split(",")]


def _marked(case):
    """Positions of the tensors that go through the codec."""
    k = len(_shapes(case))
    return [i for i in range(k) if case["op"] != "schedule" or i % 2 == 0]


def _values(gen, shape, kind, i):
    """float32 values of one tensor: see the package's synth module for what each recipe stands for."""
    n, c, h, w = shape

    def normal(*s):
        return torch.randn(s, generator=gen, device="cuda")

    def uniform(*s):
        return torch.rand(s, generator=gen, device="cuda")

    if kind == "relu" or (kind in ("mixed", "spiky") and i % 2 == 0):
        x = normal(*shape).relu_()
    elif kind in ("normal", "mixed", "spiky"):
        x = normal(*shape)
    else:
        x = torch.empty(shape, device="cuda").exponential_(generator=gen)
        x.mul_((uniform(*shape) < 0.5).float().mul_(2).sub_(1))
        hit, at = (0.01, slice(None)) if kind == "laplace_iid" else (0.08, slice(0, None, 8))
        part = x[:, at]
        u = uniform(*part.shape)
        part.masked_fill_(u < hit, 50.0)
        part.masked_fill_(u < hit / 2, -50.0)
    if kind == "spiky":
        part = x[:, ::16]
        s = tuple(part.shape)
        spikes = torch.where(uniform(*s) < 0.06, 6.0 + normal(*s).abs(), torch.zeros((), device="cuda"))
        spikes[..., :max(1, w // 4)] = normal(n, s[1], h, max(1, w // 4)).relu_()
        part.copy_(spikes)
    return x


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    shapes, f32 = _shapes(case), case["dtype"] == "f32"
    p = api.default_params(bits=case["bits"], salient_mode=SCOPES[case["scope"]], rounding=case["rounding"], seed=20251011,
                           entropy=case["entropy"])
    descs = [api.desc(s, api.FH_F32 if f32 else api.FH_BF16, tensor_id=i) for i, s in enumerate(shapes)]
    dense = [_values(gen, s, case["kind"], i).to(torch.float32 if f32 else torch.bfloat16) for i, s in enumerate(shapes)]
    caps = [api.compressed_bytes(d, p, 1) for d in descs]
    state = {"op": case["op"], "p": p, "descs": descs, "dense": dense}
    if case["op"] == "schedule":
        marked = set(_marked(case))
        restored = [torch.empty_like(t) if i in marked else t for i, t in enumerate(dense)]
        state["items"] = [api.SchedItem(d, api.FH_COMPRESS if i in marked else api.FH_KEEP, t, r)
                          for i, (d, t, r) in enumerate(zip(descs, dense, restored))]
        state["restored"] = [restored[i] for i in sorted(marked)]
        state["arena"] = torch.zeros(sum((caps[i] + 255) & ~255 for i in marked), dtype=torch.uint8, device="cuda")
        return state
    k = len(shapes)
    state["packed"] = [torch.zeros(c, dtype=torch.uint8, device="cuda") for c in caps]
    state["sizes"] = torch.zeros(k, 2, dtype=torch.int64, device="cuda")    # container bytes, status
    state["out2"] = list(state["sizes"])
    state["nbytes"] = caps
    if case["op"] != "forward":
        state["status"] = torch.zeros(k, 1, dtype=torch.int64, device="cuda")
        state["statuses"] = list(state["status"])
        state["restored"] = [torch.empty_like(t) for t in dense]
    if case["op"] == "backward":    # the containers that the forward pass left; the dense tensors are gone by then
        _forward(state)
        state["nbytes"] = [int(v) for v in state["sizes"][:, 0].tolist()]
        state["dense"] = None
    return state


def _forward(s):
    p = s["p"]
    for d, x, dst, out2 in zip(s["descs"], s["dense"], s["packed"], s["out2"]):
        rc = api.fh_compress(d, p, x, dst, out2)
        if rc != api.FH_OK:
            raise api.FhError(rc, "fh_compress")


def _backward(s):
    for d, src, nbytes, dst, status in zip(reversed(s["descs"]), reversed(s["packed"]), reversed(s["nbytes"]),
                                           reversed(s["restored"]), reversed(s["statuses"])):
        rc = api.fh_decompress(src, nbytes, d, dst, status)
        if rc != api.FH_OK:
            raise api.FhError(rc, "fh_decompress")


def run(state):
    if state["op"] == "schedule":
        rep = api.fh_run_schedule(state["items"], state["p"], state["arena"])
        return {"restored": state["restored"], "arena": state["arena"], "packed_bytes": int(rep.total_packed_bytes),
                "peak_bytes": int(rep.peak_packed_bytes), "status": int(rep.status)}
    out = {}
    if state["op"] != "backward":
        _forward(state)
        out.update(packed=state["packed"], sizes=state["sizes"])
    if state["op"] != "forward":
        _backward(state)
        out.update(restored=state["restored"], status=state["status"])
    return out


def work(case):
    """Dense bytes once and container bytes once, for each direction.  The container is counted with every plane
    normal (header, plane table, codes); outlier-rich planes make it larger.  All arithmetic is on the way."""
    shapes, esize = _shapes(case), 4 if case["dtype"] == "f32" else 2
    total = 0
    for i in _marked(case):
        n, c, h, w = shapes[i]
        slot = (4 * -(-h * w * case["bits"] // 32) + 15) // 16 * 16
        total += n * c * h * w * esize + 64 + n * c * (16 + slot)
    return {"bytes": total * (1 if case["op"] in ("forward", "backward") else 2), "flops": 0}


def tolerance(case):
    """The container's bytes are a function of the input, and each restored value is one correctly rounded result."""
    return "exact"
