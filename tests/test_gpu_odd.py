"""Hidden sizes that are no multiple of 8 on the tensor-core path, against the CPU fp64 oracle."""
import numpy as np
import pytest
import torch

import tlr_synth as S
from oracle import route_oracle as O
from tests.parity import check_against_oracle, check_self_consistency, head_with_equal_rows, run_gpu

pytestmark = pytest.mark.gpu


def check(pkg, W, h, tau):
    ref = O.route_oracle(S.bf16_bits(h), S.bf16_bits(W), tau)
    gpu = run_gpu(pkg, W.cuda(), h, tau, path=2)
    assert gpu["status"] == 0 and gpu["plan"].path == 2
    check_self_consistency(gpu, tau, W.shape[0])
    check_against_oracle(ref, gpu, O.bf16_bits_to_f64(S.bf16_bits(h)), O.bf16_bits_to_f64(S.bf16_bits(W)))
    return gpu


# 2, 4 and 8 residue classes; slabs that the shift just fills or just overflows; fewer vocabulary rows than classes,
# classes of different lengths, boxes and granules that end inside a class; either side of every switch of the kernel's
# row handling
@pytest.mark.parametrize("d", [1, 2, 3, 4, 7, 12, 57, 58, 60, 61, 100, 130, 257, 300])
@pytest.mark.parametrize("n,V", [(1, 1), (3, 7), (16, 9), (17, 260), (65, 2049), (129, 1025), (300, 5003)])
def test_small_shapes(pkg, n, d, V):
    W = S.make_W(d, V, seed=n + d + V, std=0.1)
    hid = S.make_h(n, d, seed=n + d, W=W, planted_fraction=0.1 if n >= 16 else 0.0)
    check(pkg, W, hid.h, 0.5)


@pytest.mark.parametrize("n,d,V", [(1, 2047, 20001), (64, 300, 33000), (256, 999, 30000), (100, 1500, 40000)])
def test_larger_shapes(pkg, n, d, V):
    W = S.make_W(d, V, seed=d, std=0.05)
    hid = S.make_h(n, d, seed=n, W=W, planted_fraction=0.1 if n >= 16 else 0.0)
    check(pkg, W, hid.h, 0.5)


@pytest.mark.parametrize("n,d", [(2048, 12), (2049, 12), (4500, 9)])
def test_batches_in_several_blocks(pkg, n, d):
    W = S.make_W(d, 700, seed=n, std=0.3)
    hid = S.make_h(n, d, seed=d, W=W, planted_fraction=0.1)
    check(pkg, W, hid.h, 0.5)


@pytest.mark.parametrize("d", [63, 130, 300])
@pytest.mark.parametrize("n", [40, 1100])
def test_equal_rows_of_different_classes_tie_to_the_lowest_index(pkg, n, d):
    V = 3001
    W = S.make_W(d, V, seed=d, std=0.2)
    hid = S.make_h(n, d, seed=n, W=W, planted_fraction=0.5)
    first = O.route_oracle(S.bf16_bits(hid.h), S.bf16_bits(W), 0.5)
    winners = np.unique(first.token)
    W2 = W.clone()
    for k, v in enumerate(winners[:200].tolist()):         # copies of the winners, mostly in other classes, at both ends
        W2[(5 * k) % 1000] = W[v]
        W2[V - 1 - (7 * k) % 1000] = W[v]
    ref = O.route_oracle(S.bf16_bits(hid.h), S.bf16_bits(W2), 0.5)
    exact = (O.bf16_bits_to_f64(S.bf16_bits(hid.h)) @ O.bf16_bits_to_f64(S.bf16_bits(W2)).T)
    top = exact.max(axis=1, keepdims=True)
    runner = np.where(exact >= top - 1e-9, -np.inf, exact).max(axis=1)     # the best row that is not an equal one
    sure = top[:, 0] - runner > 1e-3
    assert sure.sum() >= n // 2
    gpu = run_gpu(pkg, W2.cuda(), hid.h, 0.5)
    assert np.array_equal(gpu["token"][sure], ref.token[sure])


# Batches whose rows have four lanes in eight blocks or a warp in many (d > 128): winners with copies in other classes, the
# list and the first routed positions.
@pytest.mark.parametrize("n,d,V", [(513, 129, 2500), (640, 130, 3001), (600, 127, 2500), (1024, 300, 4000), (777, 999, 6001)])
def test_middle_batches_settle_their_winners(pkg, n, d, V):
    W, h, token, sure = head_with_equal_rows(n, d, V)
    gpu = check(pkg, W, h, 0.5)
    assert np.array_equal(gpu["token"][sure], token[sure])
    L = 3 if n % 3 == 0 else 1
    r = pkg.Router(W.cuda(), max_n=n)
    first = torch.full((n // L,), -9, dtype=torch.int32, device="cuda")
    tau = torch.from_numpy(np.where(np.arange(n) % 5 == 0, 2.0, 0.5).astype(np.float32)).cuda()
    r.route(h.cuda(), 0.0, tau_per_row=tau, seq_len=L, first_routed=first)
    torch.cuda.synchronize()
    mask = gpu["conf"] < tau.cpu().numpy()
    assert np.array_equal(r.route_mask[:n].cpu().numpy() == 1, mask) and int(r.routed_count.item()) == mask.sum()
    assert np.array_equal(r.routed_idx[:mask.sum()].cpu().numpy(), np.flatnonzero(mask))
    rows = mask.reshape(-1, L)[:n // L]
    assert np.array_equal(first.cpu().numpy(), np.where(rows.any(axis=1), rows.argmax(axis=1), L))
    r.close()


# One row whose logits all lie below -1e30: what it gives is not specified, but nothing is read beyond W for it and the other
# rows are untouched (one thread per row and four, a pair of CTAs; the call, the gathered and the pushed summaries).
@pytest.mark.parametrize("n,d", [(9, 63), (40, 100), (200, 63), (1100, 130)])
def test_a_row_of_huge_negative_logits_leaves_the_others_alone(pkg, n, d):
    V = 3001
    W = S.make_W(d, V, seed=d, std=0.2)
    W[:, :8] = -1.0
    h = S.make_h(n, d, seed=n).h
    h[:, :8] = 0
    bad = h.clone()
    bad[3, :8] = 1e30
    rows = np.arange(n) != 3
    Wd = W.cuda()
    for cls in (pkg.Router, pkg.VocabShardedRouter, pkg.FusedVocabShardedRouter):
        got = []
        for x in (h, bad):
            if cls is pkg.Router:
                r = cls(Wd, max_n=n)
                r.route(x.cuda(), 0.5)
            elif cls is pkg.VocabShardedRouter:
                r = cls(Wd, 0, max_n=n, world=1)
                r.finish(r.summarize(x.cuda()).unsqueeze(0).contiguous(), n, 0.5)
            else:
                block = torch.zeros(pkg.tlr_shard_block_bytes(n, 1), dtype=torch.uint8, device="cuda")
                r = cls(Wd, 0, n, 0, 1, [block], keep=block)
                r.push(x.cuda())
                r.finish(n, 0.5)
            torch.cuda.synchronize()
            got.append([t[:n].cpu().numpy()[rows] for t in (r.token, r.conf, r.entropy, r.route_mask)])
            r.close()
        for a, b in zip(*got):
            assert np.array_equal(a, b)


# Rows of (nearly) equal logits, as padding leaves them: every partial is a candidate for the maximum.
@pytest.mark.parametrize("n,d,V", [(3, 63, 3001), (40, 130, 3001), (300, 7, 9000), (1100, 300, 3001)])
def test_rows_of_equal_logits(pkg, n, d, V):
    W = S.make_W(d, V, seed=d, std=0.2)
    h = S.make_h(n, d, seed=n).h
    h[n // 2] = 0                                          # every logit is zero
    h[n - 1] = (h[n - 1].float() * 1e-5).to(h.dtype)       # every logit within 1e-3 of the others
    gpu = check(pkg, W, h, 0.5)
    assert gpu["token"][n // 2] == 0 and abs(gpu["conf"][n // 2] * V - 1) <= 1e-5
    z = O.bf16_bits_to_f64(S.bf16_bits(h[n - 1:]))[0] @ O.bf16_bits_to_f64(S.bf16_bits(W)).T
    assert z.max() - z[gpu["token"][n - 1]] <= 1e-6 * np.abs(z).max()     # fp32 sums of exact products settle it


@pytest.mark.parametrize("scale", [0.0, 1e-5])
def test_a_row_of_equal_logits_does_not_hold_up_the_step(pkg, scale):
    n, d, V, calls = 16, 300, 33000, 20
    W, h = S.make_W(d, V, seed=1, std=0.06).cuda(), S.make_h(n, d, seed=2).h.cuda()
    padded = h.clone()
    padded[5] = padded[5].float() * scale
    r = pkg.Router(W, max_n=n)
    stream = torch.cuda.Stream()
    times = []
    with torch.cuda.stream(stream):
        for x in (h, padded):
            r.route(x, 0.5)
            stream.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=stream):
                for _ in range(calls):
                    r.route(x, 0.5)
            took = []
            for _ in range(7):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                graph.replay()
                b.record()
                stream.synchronize()
                took.append(a.elapsed_time(b))
            times.append(sorted(took)[3])
            del graph
    r.close()
    # with every partial a candidate it was 27 times as long
    assert times[1] <= 3 * times[0], times


# The error against 64 bits: what fp32 results and the 2^-22 of ex2.approx leave, whatever d; and of large logits no more, up
# to sizes whose neighbours are further apart than the logits' differences.
@pytest.mark.parametrize("n,d,V", [(9, 255, 20000), (64, 300, 20000), (100, 999, 20000), (200, 101, 33000), (1100, 501, 9000)])
def test_scores_are_as_exact_as_fp32_sums_of_exact_products(pkg, n, d, V):
    W = S.make_W(d, V, seed=d, std=0.06)
    h = S.make_h(n, d, seed=n, W=W, planted_fraction=0.5).h
    gpu = check(pkg, W, h, 0.5)
    ref = O.route_oracle(S.bf16_bits(h), S.bf16_bits(W), 0.5)
    err = np.linalg.norm(gpu["conf"].astype(np.float64) - ref.conf) / np.linalg.norm(ref.conf)
    assert err <= 4e-7, err
    for scale in (100.0, 1e30):
        big = (h[:8].float() * scale).to(h.dtype)
        ref = O.route_oracle(S.bf16_bits(big), S.bf16_bits(W), 0.5)
        clear = ref.top2_gap >= 0.05 * scale
        assert clear.sum() >= 4
        gpu = run_gpu(pkg, W.cuda(), torch.cat([big, h[8:]]), 0.5)
        assert gpu["status"] == 0
        assert np.array_equal(gpu["token"][:8][clear], ref.token[clear])
        assert np.max(np.abs(gpu["conf"][:8][clear] - ref.conf[clear])) <= 1e-5


def test_learned_router_and_host_buffers(pkg):
    n, d, V, dh = 70, 100, 3000, 48
    W = S.make_W(d, V, seed=1, std=0.1)
    hid = S.make_h(n, d, seed=2)
    g = torch.Generator().manual_seed(5)
    W1 = (torch.randn(dh, d, generator=g) / d ** 0.5).to(torch.bfloat16)
    b1, w2 = torch.randn(dh, generator=g) * 0.1, torch.randn(dh, generator=g) * 0.5
    want = O.mlp_router_score(S.bf16_bits(hid.h), S.bf16_bits(W1), b1.numpy(), w2.numpy(), 0.1)
    ref = O.route_oracle(S.bf16_bits(hid.h), S.bf16_bits(W), 0.5)
    r = pkg.Router(W.cuda(), max_n=n)
    r.set_router_mlp(W1.cuda(), b1.cuda(), w2.cuda(), 0.1)
    score = torch.full((n,), float("nan"), device="cuda")
    r.route(hid.h.cuda(), 0.5, score_source=pkg.TLR_SCORE_MLP, mlp_score=score)
    torch.cuda.synchronize()
    assert np.max(np.abs(score.cpu().numpy() - want)) <= 1e-3
    out = [torch.zeros(n, dtype=torch.int32), torch.zeros(n), torch.zeros(n), torch.zeros(n, dtype=torch.uint8),
           torch.zeros(n, dtype=torch.int32), torch.zeros(1, dtype=torch.int32)]
    pkg.tlr_route_host(r.ctx, hid.h.pin_memory(), n, 0.5, *out)
    assert np.max(np.abs(out[1].numpy() - ref.conf) / ref.conf) <= 1e-3
    assert np.array_equal(out[0].numpy()[ref.top2_gap >= 1e-3], ref.token[ref.top2_gap >= 1e-3])
    r.close()


def test_tiny_heads_keep_the_cuda_core_kernel(pkg):
    for n, d, V, path in ((32, 36, 1820, 1), (33, 36, 1820, 2), (32, 36, 1821, 2), (32, 32, 500, 2)):
        W = S.make_W(d, V, seed=n, std=0.2)
        hid = S.make_h(n, d, seed=V)
        ref = O.route_oracle(S.bf16_bits(hid.h), S.bf16_bits(W), 0.01)
        gpu = run_gpu(pkg, W.cuda(), hid.h, 0.01)
        assert gpu["plan"].path == path and gpu["status"] == 0
        check_against_oracle(ref, gpu)


@pytest.mark.parametrize("n,d,V", [(1, 37, 100), (32, 60, 1000), (16, 300, 200), (9, 2047, 32)])
def test_tiny_heads_with_long_rows_run_on_the_tensor_cores(pkg, n, d, V):
    W = S.make_W(d, V, seed=n, std=0.1)
    hid = S.make_h(n, d, seed=V)
    ref = O.route_oracle(S.bf16_bits(hid.h), S.bf16_bits(W), 0.1)
    for path in (None, 1):
        gpu = run_gpu(pkg, W.cuda(), hid.h, 0.1, path=path)
        assert gpu["plan"].path == (path or 2) and gpu["status"] == 0
        check_against_oracle(ref, gpu)
