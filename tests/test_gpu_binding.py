"""The marshalling of the hot calls (csrc/native_binding.cpp): what it refuses, and with which exception, is what the
library's own checks and torch's allocations give; what a call is asked for decides what runs."""
from collections import UserDict

import numpy as np
import pytest
import torch

from paper_2604_07853_b200 import binding, build, inputs
from util import bits_to_torch, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    build.build()
    c = binding.Context(0)
    yield c
    assert c.poll() == 0
    c.close()


@pytest.fixture(scope="module")
def layer():
    return inputs.moe_case(6, 5, h=256, i=128, e=4, k=2)


def _io(c):
    return bits_to_torch(c.x), to_dev(c.ids), to_dev(c.weights)


class Parts:
    """A sequence that makes its items on request and keeps none of them."""

    def __init__(self, items):
        self.items = items

    def __len__(self):
        return len(self.items)

    def __getitem__(self, i):
        return self.items[i].clone()


def test_four_bit_format_is_the_one_of_the_method(ctx, layer):
    """The method called says which format runs, whatever the weights' tuples hold besides the parts it takes: without
    zero points the integer layer raises and launches nothing, and the e2m1 layer looks at the first two parts only, with
    and without the debug dumps."""
    io = _io(layer)
    masters = [bits_to_torch(w) for w in (layer.w13, layer.w2)]
    w4, fp4 = ([q(w) for w in masters] for q in (ctx.quantize_weight_w4, ctx.quantize_weight_fp4))
    launches = ctx.launch_count()
    for pair in ((fp4[0], fp4[1]), (w4[0], fp4[1]), (fp4[0], w4[1])):
        with pytest.raises(IndexError):
            ctx.moe_fwd_w4a16(*io, *pair)
    assert ctx.launch_count() == launches
    for pair in ((fp4[0], fp4[1]), ((*fp4[0], None), (*fp4[1], None)), (fp4[0], w4[1]), (w4[0], fp4[1]), (w4[0], w4[1])):
        got = ctx.moe_fwd_fp4a16(*io, *pair).clone()
        assert torch.equal(got, ctx.moe_fwd_fp4a16(*io, *pair, debug=True)[0])
    assert torch.equal(ctx.moe_fwd_w4a16(*io, *w4).clone(), ctx.moe_fwd_w4a16(*io, *w4, debug=True)[0])


def test_parts_are_kept_while_the_call_runs(ctx, layer):
    """The parts of a weight may come from any sequence, also one that hands out new tensors."""
    io = _io(layer)
    w = [ctx.quantize_weight_fp4(bits_to_torch(w)) for w in (layer.w13, layer.w2)]
    want = ctx.moe_fwd_fp4a16(*io, *w).clone()
    assert torch.equal(ctx.moe_fwd_fp4a16(*io, *(list(p) for p in w)), want)
    assert torch.equal(ctx.moe_fwd_fp4a16(*io, *(Parts(p) for p in w)), want)



def test_out_of_memory_is_torchs_error(ctx):
    """Two tebibytes of output: the allocation's own error type, which programs catch to retry with less."""
    x = torch.zeros((1 << 20, 128), dtype=torch.bfloat16, device="cuda")
    wc = torch.zeros((1 << 20, 128), dtype=torch.uint8, device="cuda")
    ws = torch.zeros((1 << 13, 1), dtype=torch.float32, device="cuda")
    with pytest.raises(torch.OutOfMemoryError):
        ctx.linear_fwd(x, wc, ws)



def test_closed_context_is_refused_by_the_library(layer):
    c = binding.Context(0)
    w = c.quantize_weight(bits_to_torch(layer.w13[0]))
    x = bits_to_torch(layer.x)
    c.close()
    for call in (lambda: c.linear_fwd(x, *w), lambda: c.quantize_act(x), lambda: c.linear_fwd_q(*w, *w)):
        with pytest.raises(binding.QarlError) as e:
            call()
        assert e.value.status == -1



def test_publish_takes_buffers_it_is_given(ctx, layer):
    """quantize_weight makes the outputs it is not given, quantize_weight_publish makes none."""
    w = bits_to_torch(layer.w13)
    codes, scales = ctx.quantize_weight(w)
    pub = [torch.zeros_like(t) for t in (codes, scales)]
    for own in ((None, scales), (codes, None), (None, None)):
        with pytest.raises(binding.QarlError) as e:
            ctx.quantize_weight_publish(w, *own, *pub)
        assert e.value.status == -1
    with pytest.raises(binding.QarlError):
        ctx.quantize_weight_publish(w, codes, scales, pub[0], None)
    got = ctx.quantize_weight_publish(w, codes, scales, *pub)
    assert got[0] is codes and got[1] is scales
    assert torch.equal(pub[0], codes) and torch.equal(pub[1], scales)



def test_shapes_and_containers_the_calls_take(ctx, layer):
    """Ids with trailing dimensions of one, a router weight with a dimension in between, any mapping as the loss's `out`;
    a save dict has to hold both tensors."""
    x, ids, wts = _io(layer)
    q = [t for w in (layer.w13, layer.w2) for t in ctx.quantize_weight(bits_to_torch(w))]
    want = ctx.moe_fwd(x, ids, wts, *q).clone()
    assert torch.equal(ctx.moe_fwd(x, ids.unsqueeze(2), wts.unsqueeze(2), *q), want)
    gate_up = torch.empty((layer.M * layer.k, 2 * layer.I), dtype=torch.bfloat16, device="cuda")
    with pytest.raises((AttributeError, TypeError)):
        ctx.moe_fwd(x, ids, wts, *q, save={"gate_up": gate_up, "h": None})
    with pytest.raises(KeyError):
        ctx.moe_fwd(x, ids, wts, *q, save={"gate_up": gate_up})
    wr = torch.randn((8, 256), device="cuda").to(torch.bfloat16)
    for a, b in zip(ctx.router_fwd(x, wr, 2), ctx.router_fwd(x, wr.unsqueeze(1), 2)):
        assert torch.equal(a, b)
    lp = torch.linspace(-1.0, -0.5, 40, device="cuda")
    offsets = torch.tensor([0, 10, 40], device="cuda")
    adv = torch.tensor([1.0, -1.0], device="cuda")
    first = ctx.tbpo_loss(lp + 1e-3, lp, lp, offsets, adv)
    again = UserDict({k: torch.zeros_like(v) for k, v in first.items()})
    assert ctx.tbpo_loss(lp + 1e-3, lp, lp, offsets, adv, out=again) is again
    assert all(torch.equal(again[k], first[k]) for k in first)



def test_flags_without_a_truth_value_raise(ctx, layer):
    x = bits_to_torch(layer.x)
    w = ctx.quantize_weight(bits_to_torch(layer.w13[0]))
    with pytest.raises(ValueError):
        ctx.linear_fwd(x, *w, want_f32=np.ones(2))
