"""The merge kernels behind the projection: batch sizes at the edges of their blocks, and steps that follow each other."""
import numpy as np
import pytest
import torch

import tlr_synth as S
from oracle import route_oracle as O
from tests.parity import check_against_oracle, to_np

pytestmark = pytest.mark.gpu

D, V = 64, 20000


def _head(kind):
    """(Router arguments, the matrix in 64 bits, d) of a bf16, an 8-bit and an odd-sized head."""
    if kind == "8bit":
        codes, scale = S.make_W8(D, V, seed=5, std=0.2)
        return (codes.cuda(), scale.cuda()), O.dequantize_e4m3(to_np(codes), to_np(scale)), D
    d = D - 3 if kind == "odd" else D
    W = S.make_W(d, V, seed=5, std=0.2)
    return (W.cuda(), None), O.bf16_bits_to_f64(S.bf16_bits(W)), d


def _outputs(r, n):
    return {"token": to_np(r.token[:n]), "conf": to_np(r.conf[:n]), "entropy": to_np(r.entropy[:n]),
            "route_mask": to_np(r.route_mask[:n]), "routed_idx": to_np(r.routed_idx),
            "routed_count": int(r.routed_count.item())}


# 8 and 16 row warps a block, 1 to 8 blocks, 32, 16 and fewer lanes a row, and the other merge kernels beyond
@pytest.mark.parametrize("kind,n", [(k, n) for k in ("bf16", "8bit", "odd") for n in (1, 7, 8, 9, 16, 17, 64, 65, 127, 128)] +
                         [(k, n) for k in ("bf16", "odd") for n in (129, 255, 256, 257, 511, 513, 1024, 1025)])
def test_edges_of_the_merge_blocks(pkg, kind, n):
    (W, scale), W64, d = _head(kind)
    h = S.make_h(n, d, seed=n).h
    ref = O.route_oracle(S.bf16_bits(h), None, 0.0, W64=W64)
    tau = np.float32(np.median(ref.conf) * 1.01)
    ref = O.with_threshold(ref, tau)
    r = pkg.Router(W, max_n=n, wscale=scale)
    first = torch.full((n,), -9, dtype=torch.int32, device="cuda")
    r.route(h.cuda(), float(tau), seq_len=1, first_routed=first)
    torch.cuda.synchronize()
    assert pkg.tlr_last_device_status(r.ctx) == 0
    got = _outputs(r, n)
    check_against_oracle(ref, got)
    mask = got["route_mask"]
    assert got["routed_count"] == mask.sum() and np.array_equal(got["routed_idx"][:mask.sum()], np.flatnonzero(mask))
    assert np.array_equal(to_np(first), 1 - mask)         # sequences of one row: position 0 if routed, else 1
    r.close()


# A lane owns up to six partials, the last ones of its row or fewer: 21 to 24 partials for four lanes, 37 for eight; the rows end
# inside a warp.
@pytest.mark.parametrize("n,V,chunks", [(513, 1985, 21), (765, 2082, 22), (601, 2179, 23), (700, 1500, 24), (1023, 9260, 37)])
def test_lanes_with_six_partials(pkg, n, V, chunks):
    W, h = S.make_W(D, V, seed=n, std=0.2), S.make_h(n, D, seed=V).h
    ref = O.route_oracle(S.bf16_bits(h), S.bf16_bits(W), 0.0)
    tau = float(np.float32(np.median(ref.conf) * 1.01))
    r = pkg.Router(W.cuda(), max_n=n)
    assert pkg.tlr_plan_query(r.ctx, n).vocab_chunks == chunks
    r.route(h.cuda(), tau)
    torch.cuda.synchronize()
    assert pkg.tlr_last_device_status(r.ctx) == 0
    got = _outputs(r, n)
    check_against_oracle(O.with_threshold(ref, tau), got)
    mask = got["route_mask"]
    assert got["routed_count"] == mask.sum() and np.array_equal(got["routed_idx"][:mask.sum()], np.flatnonzero(mask))
    r.close()


def _expect(kind, r, h, n):
    """What the router gives for a batch when nothing else is in flight."""
    torch.cuda.synchronize()
    r.route(h, 0.5)
    torch.cuda.synchronize()
    return [t.copy() for t in (to_np(r.token[:n]), to_np(r.conf[:n]), to_np(r.entropy[:n]), to_np(r.route_mask[:n]))]


class _Steps:
    """Steps of one context on the batches `h`, every one with output buffers of its own."""

    def __init__(self, pkg, kind, seed, sizes):
        self.pkg, self.kind = pkg, kind
        (W, scale), _, d = _head(kind)
        if seed:
            W = W.flip(0).contiguous()
            scale = None if scale is None else scale.flip(0).contiguous()
        self.h = [S.make_h(n, d, seed=seed + n).h.cuda() for n in sizes]
        top = max(sizes)
        if kind == "push":
            block = torch.zeros(pkg.tlr_shard_block_bytes(top, 1), dtype=torch.uint8, device="cuda")
            self.r = pkg.FusedVocabShardedRouter(W, 0, top, 0, 1, [block], keep=block)
        elif kind == "summary":
            self.r = pkg.VocabShardedRouter(W, 0, max_n=top, world=1)
        else:
            self.r = pkg.Router(W, max_n=top, wscale=scale)
        self.tau, self.want = [0.5] * len(sizes), []
        for k in range(len(sizes)):
            conf = self.alone(k)[1]
            self.tau[k] = float(np.median(conf)) if len(conf) > 1 else 2.0        # (a row alone is routed)
            self.want.append(self.alone(k))

    def buffers(self, k):
        n = self.h[k].shape[0]
        out = [torch.empty(n, dtype=t, device="cuda") for t in (torch.int32, torch.float32, torch.float32, torch.uint8, torch.int32)]
        return out + [torch.empty(1, dtype=torch.int32, device="cuda")]

    def step(self, k, out):
        pkg, ctx, h, n = self.pkg, self.r.ctx, self.h[k], self.h[k].shape[0]
        if self.kind == "push":
            pkg.tlr_shard_push(ctx, h, n, 0)
            pkg.tlr_shard_finish_fused(ctx, n, self.tau[k], *out)
        elif self.kind == "summary":
            pkg.tlr_shard_summary(ctx, h, n, 0, self.r.summary)
            pkg.tlr_shard_finish(ctx, self.r.summary, 1, n, self.tau[k], *out)
        else:
            pkg.tlr_route(ctx, h, n, self.tau[k], *out)

    def alone(self, k):
        """What a step gives when nothing else is in flight."""
        out = self.buffers(k)
        torch.cuda.synchronize()
        self.step(k, out)
        torch.cuda.synchronize()
        return _listed(out)


def _listed(out):
    out = [to_np(t).copy() for t in out]
    return out[:4] + [out[4][:int(out[5][0])], out[5]]


# Steps that nothing waits between, of different sizes and inputs: each merge may look for its partials while the one before is
# still at work on its own, in the same memory or, with two contexts in turn, in the other's.  More steps than there are tags
# (254); and replayed, when the tags come back.  Every step's outputs are kept and looked at.
@pytest.mark.parametrize("contexts", [1, 2])
@pytest.mark.parametrize("kind,graph", [(k, g) for k in ("bf16", "8bit", "odd", "summary") for g in (False, True)] + [("push", False)])
def test_steps_back_to_back_keep_their_partials(pkg, kind, graph, contexts):
    sizes = [1, 16, 8, 64, 17, 128] + ([] if kind == "8bit" else [256, 200, 300])
    routers = [_Steps(pkg, kind, 100 * c, sizes) for c in range(contexts)]
    steps = []
    for i in range(600 * contexts):
        s, k = routers[i % contexts], (i // contexts * 7) % len(sizes)
        steps.append((s, k, s.buffers(k)))

    def loop():
        for s, k, out in steps:
            s.step(k, out)

    def check():
        torch.cuda.synchronize()
        for s in routers:
            assert pkg.tlr_last_device_status(s.r.ctx) == 0
        for i, (s, k, out) in enumerate(steps):
            for a, b in zip(_listed(out), s.want[k]):
                assert np.array_equal(a, b), (i, sizes[k])
        for _, _, out in steps:
            for t in out:
                t.zero_()

    torch.cuda.synchronize()
    if graph:
        side = torch.cuda.Stream()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=side):
            loop()
        for _ in range(3):
            g.replay()
            check()
        del g
    else:
        torch.cuda._sleep(20_000_000)              # the host runs ahead
        loop()
        check()
    for s in routers:
        s.r.close()


# A call that fails between the projection and the merge leaves partials that nobody takes.  They are nobody's either when the
# tag comes round (after 254 steps), here in a graph captured before the failure, with other hidden states.
@pytest.mark.parametrize("kind", ["bf16", "8bit", "odd"])
def test_partials_of_a_failed_call_are_not_taken_by_later_ones(pkg, kind):
    (W, scale), _, d = _head(kind)
    n = 48
    r = pkg.Router(W, max_n=n, wscale=scale)
    h, other, one = (S.make_h(k, d, seed=s).h.cuda() for k, s in ((n, 1), (n, 2), (1, 3)))
    want = _expect(kind, r, h, n)                         # tag 1
    side = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=side):
        r.route(h, 0.5)                                   # tag 2
    for _ in range(253):
        r.route(one, 0.5)                                 # tags 3 .. 254 and 1
    pkg.tlr_set_kernel_timing(r.ctx, True)
    pkg.tlr_debug_inject(r.ctx, 4)
    with pytest.raises(pkg.TlrError) as e:
        r.route(other, 0.5)                               # tag 2
    assert e.value.code == 4
    pkg.tlr_debug_inject(r.ctx, 0)
    pkg.tlr_set_kernel_timing(r.ctx, False)
    outs = (r.token, r.conf, r.entropy, r.route_mask)
    for step in (g.replay, lambda: r.route(h, 0.5)):
        for t in outs:
            t.zero_()
        step()
        torch.cuda.synchronize()
        assert pkg.tlr_last_device_status(r.ctx) == 0
        for a, b in zip(outs, want):
            assert np.array_equal(to_np(a[:n]), b)
    del g
    r.close()
