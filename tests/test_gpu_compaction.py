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
