"""A context is ready for steps on any stream when its constructor returns, whatever the default stream is busy with."""
import numpy as np
import pytest
import torch

import tlr_synth as S
from tests.parity import to_np

pytestmark = pytest.mark.gpu

N, D, V = 16, 64, 20000


# A row that is not finite raises a flag in the status word: a clear of the workspace that lands behind the step wipes it.
@pytest.mark.parametrize("fp8", [False, True])
def test_a_new_context_steps_on_a_side_stream_while_the_default_stream_is_busy(pkg, fp8):
    W, scale = S.make_W8(D, V, seed=3, std=0.2) if fp8 else (S.make_W(D, V, seed=3, std=0.2), None)
    W, scale = W.cuda(), None if scale is None else scale.cuda()
    h = S.make_h(N, D, seed=4).h.cuda()
    bad = h.clone()
    bad[3] = float("nan")
    make = lambda: pkg.tlr_create_fp8(D, V, W, scale, N) if fp8 else pkg.tlr_create(D, V, W, N)  # noqa: E731
    out = [torch.zeros(N, dtype=t, device="cuda") for t in (torch.int32, torch.float32, torch.float32, torch.uint8, torch.int32)]
    out.append(torch.zeros(1, dtype=torch.int32, device="cuda"))
    warm = make()
    pkg.tlr_route(warm, h, N, 0.01, *out)
    torch.cuda.synchronize()
    want = [to_np(t).copy() for t in out]
    side = torch.cuda.Stream()
    torch.cuda._sleep(2_000_000_000)                     # a second, about
    ctx = make()
    for rows in (bad, h):
        pkg.tlr_route(ctx, rows, N, 0.01, *out, stream=side)
    side.synchronize()
    assert not torch.cuda.default_stream().query()       # the steps are done and the default stream still is not
    got = [to_np(t) for t in _on(side, out)]
    torch.cuda.synchronize()
    assert pkg.tlr_last_device_status(ctx) == pkg.TLR_DEV_NONFINITE
    count = int(want[5][0])
    for a, b in zip(got[:4] + [got[4][:count], got[5]], want[:4] + [want[4][:count], want[5]]):
        assert np.array_equal(a, b)
    assert pkg.tlr_last_device_status(ctx) == 0          # the read cleared it
    pkg.tlr_route(ctx, bad, N, 0.01, *out, stream=side)
    assert pkg.tlr_last_device_status(ctx) == pkg.TLR_DEV_NONFINITE
    pkg.tlr_destroy(ctx)
    pkg.tlr_destroy(warm)


def _on(stream, tensors):
    with torch.cuda.stream(stream):
        return [t.cpu() for t in tensors]


# The tables of the peers' addresses are on the device, and what came before on the default stream is complete (the block's
# zeros), when the attaching call returns.
def test_an_attached_context_steps_on_a_side_stream(pkg):
    W = S.make_W(D, V, seed=3, std=0.2).cuda()
    h = S.make_h(N, D, seed=4).h.cuda()
    out = [torch.zeros(N, dtype=t, device="cuda") for t in (torch.int32, torch.float32, torch.float32, torch.uint8, torch.int32)]
    out.append(torch.zeros(1, dtype=torch.int32, device="cuda"))
    ctx = pkg.tlr_create(D, V, W, N)
    pkg.tlr_route(ctx, h, N, 0.01, *out)
    torch.cuda.synchronize()
    want = to_np(out[0]).copy()
    block = torch.empty(pkg.tlr_shard_block_bytes(N, 1), dtype=torch.uint8, device="cuda")
    side = torch.cuda.Stream()
    torch.cuda._sleep(100_000_000)
    out[0].fill_(-1)
    block.zero_()
    pkg.tlr_shard_attach(ctx, 0, 1, [block])
    assert torch.cuda.default_stream().query()
    pkg.tlr_shard_push(ctx, h, N, 0, stream=side)
    pkg.tlr_shard_finish_fused(ctx, N, 0.01, *out, stream=side)
    side.synchronize()
    assert pkg.tlr_last_device_status(ctx) == 0
    assert np.array_equal(to_np(out[0]), want)
    pkg.tlr_destroy(ctx)
