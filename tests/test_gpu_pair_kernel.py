"""The dense FP8 GEMM has a form in which two CTAs share a tile of 256 rows: one MMA over both, each loading half of the tile's
columns.  It must give the bytes of the single-CTA form: one input goes through each, forced by the harness switch, at row
counts around the tile's two halves, column counts that leave half a tile, and one K-block."""
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
