"""The list of routed positions of batches of more than 1024 rows: words of flags, ends of words and of passes (16384 rows)."""
import numpy as np
import pytest
import torch

import paper_2504_07878_b200 as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1025, 1031, 2048, 4097, 16383, 16384, 16385, 33001])
def test_list_of_large_batches(n):
    gen = torch.Generator(device="cuda").manual_seed(n)
    W = (torch.randn((96, 64), generator=gen, device="cuda") * 0.2).to(torch.bfloat16)
    h = torch.randn((n, 64), generator=gen, device="cuda").to(torch.bfloat16)
    r = P.Router(W, max_n=n + 5)
    out = [torch.zeros(n, dtype=t, pin_memory=True) for t in (torch.int32, torch.float32, torch.float32, torch.uint8, torch.int32)]
    out.append(torch.zeros(1, dtype=torch.int32, pin_memory=True))
    conf = r.route(h, 0.0)[1].cpu().numpy().copy()
    host = h.cpu().pin_memory()
    for tau in (2.0, 0.0, float(np.median(conf)), float(np.quantile(conf, 0.01)), 2.0):
        want = np.flatnonzero(conf < np.float32(tau))
        r.routed_idx.fill_(-1)
        _, _, _, mask, idx, count = r.route(h, tau)
        assert int(count.item()) == want.size and np.array_equal(idx.cpu().numpy()[:want.size], want)
        assert np.all(idx.cpu().numpy()[want.size:] == -1)           # nothing behind the list
        assert np.array_equal(np.flatnonzero(mask.cpu().numpy()), want)
        P.tlr_route_host(r.ctx, host, n, tau, *out)
        assert int(out[5][0]) == want.size and np.array_equal(out[4][:want.size].numpy(), want)
    L = 41 if n % 41 == 0 else (n if n % 2 else 2)
    first = torch.full((n // L,), -1, dtype=torch.int32, device="cuda")
    tau = float(np.quantile(conf, 0.3))
    r.route(h, tau, seq_len=L, first_routed=first)
    below = (conf < np.float32(tau)).reshape(n // L, L)
    assert np.array_equal(first.cpu().numpy(), np.where(below.any(axis=1), below.argmax(axis=1), L))
    r.close()


# More partials per row than the lanes of eight blocks can keep: many blocks, as above 1024 rows.  (d = 96, V = 18944: 49 per row.)
@pytest.mark.parametrize("n", [600, 639, 768])
def test_middle_batches_of_many_partials(n):
    gen = torch.Generator(device="cuda").manual_seed(n)
    W = (torch.randn((18944, 96), generator=gen, device="cuda") * 0.2).to(torch.bfloat16)
    h = torch.randn((n, 96), generator=gen, device="cuda").to(torch.bfloat16)
    r = P.Router(W, max_n=n)
    assert P.tlr_plan_query(r.ctx, n).vocab_chunks > 48
    for tau in (0.02, 2.0, 0.0, 0.02):
        _, conf, _, mask, idx, count = r.route(h, tau)
        z = h.double() @ W.double().T
        want = torch.softmax(z, dim=1).amax(dim=1)
        assert torch.all((conf - want).abs() <= 2e-5 * want)      # (fp32 sums of exact products, see the parity tests)
        flags = (conf < tau).cpu().numpy()
        assert np.array_equal(mask.cpu().numpy() != 0, flags)
        assert int(count.item()) == flags.sum() and np.array_equal(idx.cpu().numpy()[:flags.sum()], np.flatnonzero(flags))
    r.close()


# The same kernel with the options of a call: thresholds per row, first routed positions, the learned router's scores -- and where
# near-ties are settled (d % 8 != 0; chunks by residue class).
@pytest.mark.parametrize("n,d,V", [(600, 96, 18944), (869, 97, 26475), (996, 101, 33000), (440, 142, 46443)])
def test_middle_batches_with_options(n, d, V):
    gen = torch.Generator(device="cuda").manual_seed(n)
    rand = lambda *size: torch.randn(size, generator=gen, device="cuda")  # noqa: E731
    W, h = (rand(V, d) * 0.2).to(torch.bfloat16), rand(n, d).to(torch.bfloat16)
    r = P.Router(W, max_n=n)
    W1, b1, w2 = (rand(40, d) / d ** 0.5).to(torch.bfloat16), rand(40) * 0.1, rand(40) * 0.2
    r.set_router_mlp(W1, b1, w2, 0.1)
    assert P.tlr_plan_query(r.ctx, n).vocab_chunks > (96 if n <= 512 else 48)
    z = h.double() @ W.double().T
    want = torch.softmax(z, dim=1).amax(dim=1)
    learned = torch.sigmoid(torch.relu(h.double() @ W1.double().T + b1) @ w2.double() + 0.1)
    L = 4 if n % 4 == 0 else 11
    tau = torch.where(torch.rand(n, generator=gen, device="cuda") < 0.5, 0.02, 0.2)
    for source in (P.TLR_SCORE_CONF, P.TLR_SCORE_MLP):
        first = torch.full((n // L,), -1, dtype=torch.int32, device="cuda")
        score = torch.full((n,), float("nan"), device="cuda")
        token, conf, _, mask, idx, count = r.route(h, 0.0, tau_per_row=tau if source == P.TLR_SCORE_CONF else tau + 0.4,
                                                   seq_len=L, first_routed=first, score_source=source, mlp_score=score)
        assert torch.all((conf - want).abs() <= 2e-5 * want) and torch.all((score - learned).abs() <= 1e-5)
        assert torch.all(z.gather(1, token.long()[:, None])[:, 0] >= z.amax(dim=1) - 1e-4)
        flags = (conf < tau if source == P.TLR_SCORE_CONF else score < tau + 0.4).cpu().numpy()
        assert 0 < flags.sum() < n and np.array_equal(mask.cpu().numpy() != 0, flags)
        assert int(count.item()) == flags.sum() and np.array_equal(idx.cpu().numpy()[:flags.sum()], np.flatnonzero(flags))
        rows = flags.reshape(-1, L)
        assert np.array_equal(first.cpu().numpy(), np.where(rows.any(axis=1), rows.argmax(axis=1), L))
    assert P.tlr_last_device_status(r.ctx) == 0
    r.close()
