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


def _expect(kind, r, h, n):
    """What the router gives for a batch when nothing else is in flight."""
    torch.cuda.synchronize()
    r.route(h, 0.5)
    torch.cuda.synchronize()
    return [t.copy() for t in (to_np(r.token[:n]), to_np(r.conf[:n]), to_np(r.entropy[:n]), to_np(r.route_mask[:n]))]


# Steps that nothing waits between, of different sizes and inputs: each merge may look for its partials while the one before is
# still at work on its own, in the same memory.  More steps than there are tags (254); and replayed, when the tags come back.
@pytest.mark.parametrize("kind", ["bf16", "8bit", "odd"])
@pytest.mark.parametrize("graph", [False, True])
def test_steps_back_to_back_keep_their_partials(pkg, kind, graph):
    (W, scale), _, d = _head(kind)
    sizes = [1, 16, 8, 64, 17, 128] + ([] if kind == "8bit" else [256, 200, 300])
    r = pkg.Router(W, max_n=max(sizes), wscale=scale)
    batches = [S.make_h(n, d, seed=100 + n).h.cuda() for n in sizes]
    want = [_expect(kind, r, h, n) for h, n in zip(batches, sizes)]
    steps = 600
    kept = [[torch.empty_like(t[:n]) for t in (r.token, r.conf, r.entropy, r.route_mask)] for n in sizes]

    def loop():
        for i in range(steps):
            k = (i * 7) % len(sizes)
            r.route(batches[k], 0.5)
            if i >= steps - 2 * len(sizes):               # the last rounds are looked at
                for dst, src in zip(kept[k], (r.token, r.conf, r.entropy, r.route_mask)):
                    dst.copy_(src[:sizes[k]])

    if graph:
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=side):
            loop()
        for _ in range(3):
            g.replay()
    else:
        loop()
    torch.cuda.synchronize()
    assert pkg.tlr_last_device_status(r.ctx) == 0
    for got, ref in zip(kept, want):
        for a, b in zip(got, ref):
            assert np.array_equal(to_np(a), b)
    if graph:
        del g
    r.close()


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
