"""The dense FP8 GEMM and the bf16 GEMM of the backward (dense and grouped rows) have a form in which two CTAs share a tile of
256 rows: one MMA over both, each loading half of the tile's columns.  It must give the bytes of the single-CTA form: one input
goes through each, forced by the harness switch, at row counts around the tile's two halves, column counts that leave half
a tile, one step of the contraction, and ragged and empty groups."""
import pytest
import torch

from paper_2604_07853_b200 import binding, build, inputs
from util import bits_to_torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    build.build()
    c = binding.Context(0)
    yield c
    c.close()


def _forced(ctx, path, f):
    ctx.harness_set_gemm_path(path)
    try:
        r = f()
        assert ctx.poll() == 0
        return r
    finally:
        ctx.harness_set_gemm_path(0)


@pytest.mark.parametrize("m,n,k", [(1, 128, 128), (128, 256, 256), (129, 384, 128), (255, 256, 640), (256, 128, 512), (257, 640, 1152),
                                   (385, 256, 896), (2000, 1280, 256), (8192, 2048, 384)])
def test_dense_pair_equals_single(ctx, m, n, k):
    case = inputs.linear_case(900 + m + n + k, m, n, k)
    w = ctx.quantize_weight(bits_to_torch(case.w))
    xq = ctx.quantize_act(bits_to_torch(case.x))

    def run(path, f32):
        r = _forced(ctx, path, lambda: ctx.linear_fwd_q(*xq, *w, want_f32=f32))
        return [t.clone().view(torch.uint8) for t in (r if f32 else (r,))]

    for f32 in (True, False):
        for a, b in zip(run(1, f32), run(3, f32)):
            assert torch.equal(a, b), f32


@pytest.mark.parametrize("stop_after", [0, 1, 5])
def test_pair_gives_up_on_a_wait_and_the_context_survives(ctx, stop_after):
    """Both CTAs' producers stop; the pair's waits run out (1 ms), both leave together, the next call is normal."""
    case = inputs.linear_case(6, 700, 384, 1024)
    w = ctx.quantize_weight(bits_to_torch(case.w))
    xq = ctx.quantize_act(bits_to_torch(case.x))
    ref = _forced(ctx, 3, lambda: ctx.linear_fwd_q(*xq, *w)).clone()
    ctx.harness_set_gemm_path(3)
    ctx.harness_set_wait_limit_ns(1_000_000)
    ctx.harness_stop_producer_after(stop_after)
    try:
        ctx.linear_fwd_q(*xq, *w)
        assert ctx.poll() == -7
    finally:
        ctx.harness_stop_producer_after(-1)
        ctx.harness_set_wait_limit_ns(0)
        ctx.harness_set_gemm_path(0)
    for _ in range(2):
        assert torch.equal(_forced(ctx, 3, lambda: ctx.linear_fwd_q(*xq, *w)), ref)


def _rand(seed, *shape):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.empty(shape, dtype=torch.bfloat16, device="cuda").normal_(0.0, 1.0, generator=g)


def _same(a, b):
    for s, t in zip(a, b):
        if s is not None:
            assert torch.equal(s.view(torch.uint8), t.view(torch.uint8))


@pytest.mark.parametrize("m,n,k", [(1, 8, 8), (64, 128, 128), (127, 256, 256), (129, 520, 264), (300, 1280, 768), (1000, 136, 2048), (257, 2048, 72),
                                   (511, 1024, 640)])
def test_bf16_dense_pair_equals_single(ctx, m, n, k):
    dy, x, w = _rand(1, m, n), _rand(2, m, k), _rand(3, n, k)
    single = _forced(ctx, 1, lambda: ctx.linear_bwd(dy, x, w, want_dx_f32=True))
    _same(single, _forced(ctx, 3, lambda: ctx.linear_bwd(dy, x, w, want_dx_f32=True)))


@pytest.mark.parametrize("sizes", [[0, 1, 63, 64, 65, 0, 200, 128, 16, 15], [700], [0, 0, 5], [256, 257, 255, 512, 48, 49], [3] * 300 + [1000] * 3])
@pytest.mark.parametrize("n,k", [(256, 128), (384, 512)])
def test_bf16_grouped_rows_pair_equals_single(ctx, sizes, n, k):
    off = torch.tensor([0, *torch.tensor(sizes).cumsum(0).tolist()], dtype=torch.int32, device="cuda")
    p = sum(sizes)
    dy, x, w = _rand(4, p, n), _rand(5, p, k), _rand(6, len(sizes), n, k)
    single = _forced(ctx, 1, lambda: ctx.grouped_linear_bwd(dy, x, w, off, want_dx_f32=True, dw=False))
    for _ in range(3):
        _same(single, _forced(ctx, 3, lambda: ctx.grouped_linear_bwd(dy, x, w, off, want_dx_f32=True, dw=False)))


@pytest.mark.parametrize("stop_after", [0, 1, 7])
def test_bf16_pair_gives_up_on_a_wait_and_the_context_survives(ctx, stop_after):
    off = torch.tensor([0, 100, 100, 730, 900], dtype=torch.int32, device="cuda")
    dy, x, w = _rand(7, 900, 512), _rand(8, 900, 256), _rand(9, 4, 512, 256)
    calls = (lambda: ctx.grouped_linear_bwd(dy, x, w, off, dw=False), lambda: ctx.linear_bwd(dy, x, w[0]))
    for call in calls:
        ref = _forced(ctx, 3, call)
        ctx.harness_set_gemm_path(3)
        ctx.harness_set_wait_limit_ns(1_000_000)
        ctx.harness_stop_producer_after(stop_after)
        try:
            call()
            assert ctx.poll() == -7
        finally:
            ctx.harness_stop_producer_after(-1)
            ctx.harness_set_wait_limit_ns(0)
            ctx.harness_set_gemm_path(0)
        for _ in range(2):
            _same(ref, _forced(ctx, 3, call))
