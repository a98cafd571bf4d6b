"""Failure detection without a GPU fault: a device-side wait that nothing satisfies gives up at
its limit, the kernel returns, the error is reported through the status word and the context keeps
working.  (The pipeline waits of the GEMM use the same bounded wait with a 2 s limit.)"""
import time

import numpy as np
import pytest
import torch

from paper_2604_07853_b200 import binding, build, inputs
from util import bits_to_torch

pytestmark = pytest.mark.gpu


def test_expired_wait_is_reported_and_context_survives():
    build.build()
    ctx = binding.Context(0)
    case = inputs.linear_case(3, 8, 128, 128)
    wc, ws = ctx.quantize_weight(bits_to_torch(case.w))
    before = ctx.linear_fwd(bits_to_torch(case.x), wc, ws).clone()
    assert ctx.poll() == 0
    t0 = time.perf_counter()
    ctx.harness_wait_selftest(limit_ns=2_000_000)          # 2 ms
    assert ctx.poll() == -7                                # QARL_ERR_DEVICE_TIMEOUT, then cleared
    assert time.perf_counter() - t0 < 1.0
    assert ctx.poll() == 0
    after = ctx.linear_fwd(bits_to_torch(case.x), wc, ws)  # the context is still usable
    assert torch.equal(before, after) and ctx.poll() == 0
    ctx.harness_wait_selftest(limit_ns=1000)
    with pytest.raises(binding.QarlError) as ei:
        ctx.check_device_status()
    assert ei.value.status == -7
    ctx.close()


@pytest.mark.parametrize("stop_after", [0, 1, 5])
def test_gemm_pipeline_wait_expires_and_context_survives(stop_after):
    """The FP8 GEMM's own abort protocol: the TMA producer stops arming stages (a host-set test
    switch), so the MMA role waits on a stage that nothing fills; its bounded wait (1 ms here)
    runs out, the CTA aborts, drains and frees its TMEM, the kernel returns, the status word says
    QARL_ERR_DEVICE_TIMEOUT, and the next call with the normal settings gives the reference bytes."""
    build.build()
    ctx = binding.Context(0)
    case = inputs.linear_case(5, 300, 384, 1024)           # 3 row tiles x 2 column tiles x 8 K-blocks
    wc, ws = ctx.quantize_weight(bits_to_torch(case.w))
    x = bits_to_torch(case.x)
    ref = ctx.linear_fwd(x, wc, ws).clone()
    assert ctx.poll() == 0
    ctx.harness_set_wait_limit_ns(1_000_000)
    ctx.harness_stop_producer_after(stop_after)
    t0 = time.perf_counter()
    ctx.linear_fwd(x, wc, ws)
    assert ctx.poll() == -7
    assert time.perf_counter() - t0 < 1.0
    ctx.harness_stop_producer_after(-1)
    ctx.harness_set_wait_limit_ns(0)
    assert ctx.poll() == 0
    for _ in range(2):
        assert torch.equal(ctx.linear_fwd(x, wc, ws), ref) and ctx.poll() == 0
    # the same through the grouped (MoE) kernels
    c = inputs.moe_case(2, 96, h=512, i=256, e=8, k=2)
    w13c, w13s = ctx.quantize_weight(bits_to_torch(c.w13))
    w2c, w2s = ctx.quantize_weight(bits_to_torch(c.w2))
    args = (bits_to_torch(c.x), torch.from_numpy(c.ids).cuda(), torch.from_numpy(c.weights).cuda(), w13c, w13s, w2c, w2s)
    ref_moe = ctx.moe_fwd(*args).clone()
    ctx.harness_set_wait_limit_ns(1_000_000)
    ctx.harness_stop_producer_after(min(stop_after, 2))     # a gate_up tile of this shape has 4 stages
    ctx.moe_fwd(*args)
    assert ctx.poll() == -7
    ctx.harness_stop_producer_after(-1)
    ctx.harness_set_wait_limit_ns(0)
    assert torch.equal(ctx.moe_fwd(*args), ref_moe) and ctx.poll() == 0
    ctx.close()


def _gives_up(ctx, stop_after, call):
    """`call` with producers that stop: the status says so within the second, nothing else happens; then it is normal again."""
    ref = [t.clone() for t in call()]
    assert ctx.poll() == 0
    ctx.harness_set_wait_limit_ns(1_000_000)
    ctx.harness_stop_producer_after(stop_after)
    t0 = time.perf_counter()
    call()
    assert ctx.poll() == -7
    assert time.perf_counter() - t0 < 1.0
    ctx.harness_stop_producer_after(-1)
    ctx.harness_set_wait_limit_ns(0)
    assert ctx.poll() == 0
    for _ in range(2):
        out = call()
        assert all(torch.equal(a.view(torch.uint8), b.view(torch.uint8)) for a, b in zip(out, ref)) and ctx.poll() == 0


@pytest.fixture
def ctx():
    build.build()
    c = binding.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("stop_after", [0, 1, 5])
@pytest.mark.parametrize("m,columns", [(300, 64), (300, 128), (300, 256), (8, 0)])
def test_every_dense_form_gives_up(ctx, m, columns, stop_after):
    """The dense FP8 call with tiles of 64, 128 and 256 columns, and (8 rows, choice by size) the form that quantizes its
    rows itself."""
    case = inputs.linear_case(5, m, 384, 1024)              # 8 K-blocks
    w = ctx.quantize_weight(bits_to_torch(case.w))
    x = bits_to_torch(case.x)
    ctx.harness_set_dense_columns(columns)
    _gives_up(ctx, stop_after, lambda: [ctx.linear_fwd(x, *w)])


def _unaligned(t):
    """The same values one element further on in memory."""
    buf = torch.empty(t.numel() + 1, dtype=t.dtype, device="cuda")
    buf[1:] = t.reshape(-1)
    return buf[1:].view(t.shape)


@pytest.mark.parametrize("stop_after", [0, 1, 3])
@pytest.mark.parametrize("m", [8, 40, 200])                 # tiles of 32, 64 and 128 token rows
@pytest.mark.parametrize("aligned", [True, False])
def test_four_bit_gemm_gives_up(ctx, m, aligned, stop_after):
    """The 4-bit GEMM, with the bulk copies of scales and zero points and with its own loads of unaligned ones."""
    case = inputs.linear_case(6, m, 384, 1024)              # 8 quantization groups
    packed, scales, zeros = ctx.quantize_weight_w4(bits_to_torch(case.w))
    if not aligned:
        scales, zeros = _unaligned(scales), _unaligned(zeros)
    x = bits_to_torch(case.x)
    _gives_up(ctx, stop_after, lambda: [ctx.linear_fwd_w4a16(x, packed, scales, zeros)])


@pytest.mark.parametrize("stop_after", [0, 1, 5])
def test_dense_backward_gives_up(ctx, stop_after):
    case = inputs.linear_case(7, 520, 384, 512)
    dy = torch.randn((520, 384), device="cuda").to(torch.bfloat16)
    x, w = bits_to_torch(case.x), bits_to_torch(case.w)
    _gives_up(ctx, stop_after, lambda: [t for t in ctx.linear_bwd(dy, x, w) if t is not None])


@pytest.mark.parametrize("stop_after", [0, 1, 3])          # (the longest contraction is 5 steps)
@pytest.mark.parametrize("dx,dw", [(True, False), (False, True)])
def test_grouped_backward_gives_up(ctx, dx, dw, stop_after):
    """Grouped rows (dX) and the grouped contraction (dW: two accumulators, and a warp that follows every step)."""
    sizes = [300, 0, 17, 70, 1, 130]
    offsets = torch.tensor(np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32), device="cuda")
    g = torch.Generator(device="cuda").manual_seed(1)
    dy, x, w = (torch.randn(s, device="cuda", generator=g).to(torch.bfloat16)
                for s in ((sum(sizes), 512), (sum(sizes), 256), (len(sizes), 512, 256)))
    _gives_up(ctx, stop_after, lambda: [t for t in ctx.grouped_linear_bwd(dy, x, w, offsets, dx=dx, dw=dw) if t is not None])


@pytest.mark.parametrize("form", [2, 3])
@pytest.mark.parametrize("stop_after", [0, 1, 5])
def test_router_pipeline_wait_expires_and_context_survives(stop_after, form):
    """The same for the one-launch routers (2: persistent CTAs, 3: clusters): the TMA producer stops arming stages, the MMA role's bounded
    wait (1 ms here) runs out, the CTA aborts (epilogue warps leave through the abort flag, logits
    stores in flight are waited for, TMEM is freed), the status word says QARL_ERR_DEVICE_TIMEOUT and
    the next call gives the reference bytes."""
    build.build()
    ctx = binding.Context(0)
    ctx.harness_set_router_form(form)
    rng = np.random.default_rng(8)
    x = bits_to_torch(inputs.act_bf16(rng, 300, 512))       # 3 tiles of 8 contraction steps each
    wr = bits_to_torch(inputs.weight_bf16(rng, 64, 512))
    ref = [t.clone() for t in ctx.router_fwd(x, wr, 4)]
    assert ctx.poll() == 0
    ctx.harness_set_wait_limit_ns(1_000_000)
    ctx.harness_stop_producer_after(stop_after)
    t0 = time.perf_counter()
    ctx.router_fwd(x, wr, 4)
    assert ctx.poll() == -7
    assert time.perf_counter() - t0 < 1.0
    ctx.harness_stop_producer_after(-1)
    ctx.harness_set_wait_limit_ns(0)
    assert ctx.poll() == 0
    for _ in range(2):
        out = ctx.router_fwd(x, wr, 4)
        assert all(torch.equal(a.view(torch.int32), b.view(torch.int32)) for a, b in zip(out, ref)) and ctx.poll() == 0
    ctx.close()
