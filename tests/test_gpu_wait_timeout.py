"""Failure handling of the projection kernel, without faulting or hanging the GPU.

Every barrier wait in the kernel is bounded.  The test hook makes the W producer issue no
copies, so the consumers' waits run out; the kernel must then raise TLR_DEV_WAIT_TIMEOUT, return
by itself, and leave the context fully usable for the next call."""
import numpy as np
import pytest
import torch

import tlr_synth as S
from tests.parity import to_np

pytestmark = pytest.mark.gpu


# one CTA per worker / a pair of CTAs per worker / two row blocks to a unit, the second of 44 and of all 256 rows
@pytest.mark.parametrize("n,d,V,two", [(48, 128, 40000, False), (300, 128, 40000, False), (300, 712, 105000, True),
                                       (1024, 584, 61000, True)])
def test_wait_runs_out_and_context_survives(pkg, n, d, V, two):
    W = S.make_W(d, V, seed=2, std=0.1)
    hid = S.make_h(n, d, seed=3)
    r = pkg.Router(W.cuda(), max_n=n)
    assert (pkg.tlr_plan_query(r.ctx, n).reserved == 2) == two
    h = hid.h.cuda()

    def run():
        r.route(h, 0.01)
        torch.cuda.synchronize()
        return to_np(r.token[:n]).copy(), to_np(r.conf[:n]).copy(), int(r.routed_count.item())

    good = run()
    assert pkg.tlr_last_device_status(r.ctx) == 0

    pkg.tlr_debug_inject(r.ctx, 1, 200)             # copies dropped, every wait limited to 0.2 s
    t0 = torch.cuda.Event(enable_timing=True); t1 = torch.cuda.Event(enable_timing=True)
    t0.record(); r.route(h, 0.01); t1.record()
    torch.cuda.synchronize()                        # returns: the kernel gave up by itself
    assert t0.elapsed_time(t1) < 5000.0
    assert pkg.tlr_last_device_status(r.ctx) & pkg.TLR_DEV_WAIT_TIMEOUT

    # the host-buffer entry point reports the condition as an error code
    pin = hid.h.pin_memory()
    cnt = torch.zeros(1, dtype=torch.int32).pin_memory()
    with pytest.raises(pkg.TlrError) as e:
        pkg.tlr_route_host(r.ctx, pin, n, 0.01, None, None, None, None, None, cnt)
    assert e.value.code == 7
    pkg.tlr_last_device_status(r.ctx)               # clear

    pkg.tlr_debug_inject(r.ctx, 0, 0)
    again = run()
    assert pkg.tlr_last_device_status(r.ctx) == 0
    assert np.array_equal(good[0], again[0]) and np.array_equal(good[1], again[1]) and good[2] == again[2]
    r.close()


def test_wait_runs_out_on_the_8bit_head(pkg):
    """The same hook on the fp8 decode kernel: the flag is raised, the kernel returns, the context recovers."""
    n, d, V = 24, 128, 40000
    codes, scale = S.make_W8(d, V, seed=2, std=0.1)
    r = pkg.Router(codes.cuda(), max_n=n, wscale=scale.cuda())
    h = S.make_h(n, d, seed=3).h.cuda()

    def run():
        r.route(h, 0.01)
        torch.cuda.synchronize()
        return to_np(r.token[:n]).copy(), to_np(r.conf[:n]).copy(), int(r.routed_count.item())

    good = run()
    assert pkg.tlr_last_device_status(r.ctx) == 0
    pkg.tlr_debug_inject(r.ctx, 1, 200)
    t0 = torch.cuda.Event(enable_timing=True); t1 = torch.cuda.Event(enable_timing=True)
    t0.record(); r.route(h, 0.01); t1.record()
    torch.cuda.synchronize()
    assert t0.elapsed_time(t1) < 5000.0
    assert pkg.tlr_last_device_status(r.ctx) & pkg.TLR_DEV_WAIT_TIMEOUT
    pkg.tlr_debug_inject(r.ctx, 0, 0)
    again = run()
    assert pkg.tlr_last_device_status(r.ctx) == 0
    assert np.array_equal(good[0], again[0]) and np.array_equal(good[1], again[1]) and good[2] == again[2]
    r.close()


# d a multiple of 8, no multiple of 8 (one CTA per worker / a pair), the 8-bit head
@pytest.mark.parametrize("n,d,fp8", [(48, 128, False), (48, 100, False), (300, 101, False), (48, 128, True)])
def test_a_tensor_map_that_cannot_be_encoded_is_an_error(pkg, n, d, fp8):
    V = 4000
    W, scale = S.make_W8(d, V, seed=2, std=0.1) if fp8 else (S.make_W(d, V, seed=2, std=0.1), None)
    h = S.make_h(n, d, seed=3).h.cuda()
    r = pkg.Router(W.cuda(), max_n=n, wscale=None if scale is None else scale.cuda())
    r.route(h, 0.5)
    torch.cuda.synchronize()
    good = to_np(r.token[:n]).copy()
    pkg.tlr_debug_inject(r.ctx, 2)
    for _ in range(2):
        with pytest.raises(pkg.TlrError) as e:
            r.route(h, 0.5)
        assert e.value.code == 4
    torch.cuda.synchronize()
    assert pkg.tlr_last_device_status(r.ctx) == 0
    pkg.tlr_debug_inject(r.ctx, 0)
    r.token.fill_(-1)
    r.route(h, 0.5)
    torch.cuda.synchronize()
    assert np.array_equal(to_np(r.token[:n]), good)
    r.close()


# The kernel in front of a step may be at work for longer than any limit -- here the merge of a sharded step, which looks for a
# rank that never joins for 2.5 s -- and lets the step's kernels in early.  Their limits do not cover it.
@pytest.mark.parametrize("n,d,fp8", [(5, 64, False), (40, 64, True), (200, 64, False), (200, 1024, False), (40, 1024, True)])
def test_limits_do_not_cover_what_a_step_waits_for(pkg, n, d, fp8):
    V = 20000
    W, scale = S.make_W8(d, V, seed=2, std=0.2) if fp8 else (S.make_W(d, V, seed=2, std=0.2), None)
    r = pkg.Router(W.cuda(), max_n=n, wscale=None if scale is None else scale.cuda())
    h = S.make_h(n, d, seed=3).h.cuda()
    first = torch.zeros(n, dtype=torch.int32, device="cuda")
    out = (r.token, r.conf, r.entropy, r.route_mask, first, r.routed_idx, r.routed_count)
    r.route(h, 0.01)
    torch.cuda.synchronize()
    tau = float(r.conf.median())                     # about half of the rows are routed
    r.route(h, tau, seq_len=1, first_routed=first)
    torch.cuda.synchronize()
    want = [to_np(t).copy() for t in out]
    count = int(want[-1][0])
    assert 0 < count < n

    slow_d, slow_V = 64, 3000
    block = torch.zeros(pkg.tlr_shard_block_bytes(8, 2), dtype=torch.uint8, device="cuda")
    slow = pkg.FusedVocabShardedRouter(S.make_W(slow_d, slow_V, seed=5).cuda(), 0, 8, 0, 2, [block] * 2, keep=block)
    pkg.tlr_debug_inject(slow.ctx, 0, 2500)
    slow.push(S.make_h(8, slow_d, seed=6).h.cuda())
    torch.cuda.synchronize()
    slow.finish(8, 0.5)
    r.route(h, tau, seq_len=1, first_routed=first)
    torch.cuda.synchronize()
    assert pkg.tlr_last_device_status(slow.ctx) & pkg.TLR_DEV_WAIT_TIMEOUT
    assert pkg.tlr_last_device_status(r.ctx) == 0
    got = [to_np(t) for t in out]
    for a, b in zip(got[:5] + [got[5][:count], got[6]], want[:5] + [want[5][:count], want[6]]):
        assert np.array_equal(a, b)
    slow.close()
    r.close()


# Where the kernel behind the projection looks for the partials itself, it is the one that knows of one that never came.
@pytest.mark.parametrize("kind", ["bf16", "8bit", "odd", "summary", "push"])
def test_partials_that_never_come_raise_the_flag(pkg, kind):
    n, d, V = 16, 100 if kind == "odd" else 64, 20000
    W, scale = S.make_W8(d, V, seed=2, std=0.2) if kind == "8bit" else (S.make_W(d, V, seed=2, std=0.2), None)
    W, scale = W.cuda(), None if scale is None else scale.cuda()
    hid = S.make_h(n, d, seed=3)
    h = hid.h.cuda()
    if kind == "push":
        block = torch.zeros(pkg.tlr_shard_block_bytes(n, 1), dtype=torch.uint8, device="cuda")
        r = pkg.FusedVocabShardedRouter(W, 0, n, 0, 1, [block], keep=block)
    elif kind == "summary":
        r = pkg.VocabShardedRouter(W, 0, max_n=n, world=1)
    else:
        r = pkg.Router(W, max_n=n, wscale=scale)

    def run():
        if kind == "push":
            r.push(h)
            r.finish(n, 0.01)
        elif kind == "summary":
            r.finish(r.summarize(h)[None].contiguous(), n, 0.01)
        else:
            r.route(h, 0.01)
        torch.cuda.synchronize()
        return [to_np(t[:n]).copy() for t in (r.token, r.conf, r.entropy, r.route_mask)]

    good = run()
    assert pkg.tlr_last_device_status(r.ctx) == 0
    pkg.tlr_debug_inject(r.ctx, 3)
    run()
    assert pkg.tlr_last_device_status(r.ctx) & pkg.TLR_DEV_WAIT_TIMEOUT
    if kind in ("bf16", "8bit", "odd"):
        cnt = torch.zeros(1, dtype=torch.int32).pin_memory()
        with pytest.raises(pkg.TlrError) as e:
            pkg.tlr_route_host(r.ctx, hid.h.pin_memory(), n, 0.01, None, None, None, None, None, cnt)
        assert e.value.code == 7
        pkg.tlr_last_device_status(r.ctx)
    pkg.tlr_debug_inject(r.ctx, 0)
    again = run()
    assert pkg.tlr_last_device_status(r.ctx) == 0
    for a, b in zip(good, again):
        assert np.array_equal(a, b)
    r.close()
