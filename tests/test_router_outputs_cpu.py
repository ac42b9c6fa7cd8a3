"""What Router.route hands out: views of the router's current output tensors, its own for every call (no GPU needed)."""
import pytest
import torch

import paper_2504_07878_b200 as P
from paper_2504_07878_b200 import binding


def make_router(max_n):
    r = object.__new__(P.Router)
    r.ctx = None
    r.token, r.routed_idx = torch.arange(max_n, dtype=torch.int32), torch.zeros(max_n, dtype=torch.int32)
    r.conf, r.entropy = torch.rand(max_n), torch.rand(max_n)
    r.route_mask, r.routed_count = torch.zeros(max_n, dtype=torch.uint8), torch.zeros(1, dtype=torch.int32)
    return r


def test_every_call_gets_views_of_its_own():
    r = make_router(8)
    first, second = r._outputs(5), r._outputs(5)
    own = (r.token, r.conf, r.entropy, r.route_mask)
    for a, b, t in zip(first, second, own):
        assert a is not b and a.shape == b.shape == (5,)
        assert a.data_ptr() == b.data_ptr() == t.data_ptr() and a.dtype == t.dtype
        a.unsqueeze_(1)                                   # a caller's own view, changed in place
        assert b.shape == (5,)
    assert [t.shape for t in r._outputs(5)[:4]] == [(5,)] * 4
    r.token[2] = 77                                       # the views follow the router's tensors
    assert second[0][2] == 77 and r._outputs(3)[0][2] == 77


def test_a_replaced_output_tensor_is_the_one_that_is_handed_out():
    r = make_router(8)
    r._outputs(5), r._outputs(6)
    for name in ("token", "conf", "entropy", "route_mask"):
        setattr(r, name, getattr(r, name).clone() + 1)
        for n in (5, 6):
            got = dict(zip(("token", "conf", "entropy", "route_mask"), r._outputs(n)))
            assert got[name].data_ptr() == getattr(r, name).data_ptr() and got[name].shape == (n,)
    r.routed_count = torch.ones(1, dtype=torch.int32)
    assert r._outputs(5)[5] is r.routed_count


def test_many_batch_sizes():
    r = make_router(64)
    for n in list(range(65)) * 2:
        assert [t.shape[0] for t in r._outputs(n)[:4]] == [n] * 4
    assert len(r._views) <= 16


@pytest.mark.parametrize("native", [True, False])
def test_views_are_of_the_memory_that_a_tensor_has_now(monkeypatch, native):
    if not native:
        monkeypatch.setattr(binding, "_extension", False)
    r = make_router(8)
    r._outputs(5)
    before = r.conf.detach()
    r.conf.data = before + 1                              # the same object, other memory
    for n in (5, 6, 0):
        got = r._outputs(n)
        assert got[1].shape == (n,) and (n == 0 or got[1].data_ptr() == r.conf.data_ptr())
        assert torch.equal(got[1], r.conf[:n]) and got[1].dtype == torch.float32 and not got[1].requires_grad
    assert r._outputs(5)[1].data_ptr() != before.data_ptr()
    r.token = torch.arange(4, dtype=torch.int32)          # shorter than asked for: what a slice gives
    assert r._outputs(5)[0].shape == (4,)
    r.token = torch.arange(32, dtype=torch.int32).view(16, 2)[:, 1]
    assert torch.equal(r._outputs(5)[0], r.token[:5])
