"""The grouping of pairs by expert against the oracle's permutation, bit for bit, around the limits of its forms:
counted pair against pair (at most 256 pairs of a decode-sized layer), histogram in one CTA (2048), one launch of a
cluster of 1, 2, 4 or 8 CTAs with 1, 2, 4 or 8 rounds (65536), three launches beyond.  Expert counts that are not a multiple of a
warp leave a warp half inside the per-expert loops."""
import numpy as np
import pytest
import torch

import oracle
from paper_2604_07853_b200 import binding, build
from util import to_dev

pytestmark = pytest.mark.gpu

GUARD = 64
FILL = -7


@pytest.fixture(scope="module")
def ctx():
    build.build()
    c = binding.Context(0)
    yield c
    assert c.poll() == 0
    c.close()


def _ids(seed, m, k, e):
    """Distinct ids per token, half of the tokens on a quarter of the experts."""
    rng = np.random.default_rng(seed)
    score = rng.random((m, e))
    score[: m // 2, : max(k, e // 4)] += 1.0
    return np.argsort(-score, axis=1, kind="stable")[:, :k].astype(np.int32).copy()


def _expected(ids, e):
    """The permutation of the pairs with good ids; a bad pair has no position (FILL)."""
    flat = ids.reshape(-1)
    good = np.flatnonzero((flat >= 0) & (flat < e))
    off, srt, pos = oracle.permute(flat[good][:, None], e)
    full = np.full(flat.size, FILL, np.int32)
    full[good] = pos
    return off, good[srt].astype(np.int32), full


def _guarded(n, dtype=torch.int32):
    t = torch.full((n + 2 * GUARD,), FILL, dtype=torch.int32, device="cuda").view(dtype)
    return t, t[GUARD:GUARD + n]


def check_dispatch(ctx, ids, e):
    """qarl_moe_dispatch (launch_permute whatever the size) on guarded buffers."""
    m, k = ids.shape
    p, h = m * k, 128
    x = torch.zeros((m, h), dtype=torch.bfloat16, device="cuda")
    wts = torch.arange(p, dtype=torch.float32, device="cuda").reshape(m, k)
    off_all, off = _guarded(e + 1)
    pos_all, pos = _guarded(p)
    codes = torch.empty((p, h), dtype=torch.uint8, device="cuda")
    scales = torch.empty((p, 1), device="cuda")
    sw_all, sw = _guarded(p, torch.float32)
    ws = torch.empty(ctx.lib.qarl_moe_dispatch_workspace_bytes(m, e, k), dtype=torch.uint8, device="cuda")
    dev_ids = to_dev(ids)
    ptr = lambda t: t.data_ptr()  # noqa: E731
    rc = ctx.lib.qarl_moe_dispatch(ctx.h, ptr(x), ptr(dev_ids), ptr(wts), m, h, e, k, ptr(codes), ptr(scales), ptr(sw),
                                   ptr(off), ptr(pos), ptr(ws), ws.numel(), torch.cuda.current_stream().cuda_stream)
    assert rc == 0
    status = ctx.poll()
    want_off, want_srt, want_pos = _expected(ids, e)
    assert np.array_equal(off.cpu().numpy(), want_off)
    assert np.array_equal(pos.cpu().numpy(), want_pos)
    good = want_srt.size
    if good == p:
        assert np.array_equal(sw.cpu().numpy(), want_srt.astype(np.float32))  # the weight of a pair is its id here
    for t in (off_all, pos_all, sw_all.view(torch.int32)):
        assert (t[:GUARD] == FILL).all() and (t[-GUARD:] == FILL).all()
    return status, good == p


@pytest.mark.parametrize("e", [1, 16, 40, 128, 1000])
@pytest.mark.parametrize("p", [1, 255, 256, 257, 1024, 1025, 2048, 2049, 8192, 8193, 16385, 32769, 65536, 65537])
def test_grouping_of_single_choices(ctx, p, e):
    status, all_good = check_dispatch(ctx, _ids(p + e, p, 1, e), e)
    assert all_good and status == 0


@pytest.mark.parametrize("m,k,e", [(37, 7, 40), (300, 7, 40), (1171, 7, 16), (9363, 7, 33)])
def test_grouping_of_several_choices(ctx, m, k, e):
    status, all_good = check_dispatch(ctx, _ids(m, m, k, e), e)
    assert all_good and status == 0


@pytest.mark.parametrize("e", [16, 40, 1000])
@pytest.mark.parametrize("p", [30, 300, 1500, 5000, 20000, 70000])
def test_bad_ids_are_skipped_and_reported(ctx, p, e):
    ids = _ids(p, p, 1, e)
    for at, bad in ((0, e), (p // 3, -1), (p // 2, 1 << 30), (p - 1, -(1 << 31))):
        ids[at, 0] = bad
    status, all_good = check_dispatch(ctx, ids, e)
    assert not all_good and status == -8


@pytest.mark.parametrize("e", [1, 16, 40, 1000])
@pytest.mark.parametrize("p", [1, 255, 256, 257, 2047, 2048])
@pytest.mark.parametrize("bad", [False, True])
def test_grouping_inside_the_decode_sized_layer(ctx, p, e, bad):
    """The decode-sized layer groups in the launch that quantizes (seen through its debug dumps)."""
    ids = _ids(p, p, 1, e)
    if bad:
        ids[p // 2, 0] = e
    x = torch.ones((p, 128), dtype=torch.bfloat16, device="cuda")
    w13 = ctx.quantize_weight(torch.ones((e, 256, 128), dtype=torch.bfloat16, device="cuda"))
    w2 = ctx.quantize_weight(torch.ones((e, 128, 128), dtype=torch.bfloat16, device="cuda"))
    _, d = ctx.moe_fwd(x, to_dev(ids), torch.ones((p, 1), device="cuda"), *w13, *w2, debug=True)
    assert ctx.poll() == (-8 if bad else 0)
    off, srt, _ = _expected(ids, e)
    assert np.array_equal(d["expert_offsets"].cpu().numpy(), off)
    assert np.array_equal(d["sorted_pair"].cpu().numpy()[:srt.size], srt)
