"""Router.route's native call against the same call through ctypes: outputs, views, errors."""
import pytest
import torch

import tlr_synth as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [0, 1, 5])
def test_native_call_hands_out_what_the_other_does(pkg, n):
    from paper_2504_07878_b200 import binding, build
    build.build()
    r = pkg.Router(S.make_W(64, 3000, seed=1, std=0.2).cuda(), max_n=5)
    assert "built-in" in repr(binding._native_route()) and "built-in" in repr(r._native)
    h = S.make_h(max(n, 1), 64, seed=2).h[:n].cuda()
    native, r._native = r._native, lambda *args: None
    want = [t.clone() for t in r.route(h, 0.01)]                 # through ctypes; makes the views of this size
    r._native = native
    first, second = r.route(h, 0.01), r.route(h, 0.01)
    torch.cuda.synchronize()
    own = (r.token, r.conf, r.entropy, r.route_mask)
    assert all(torch.equal(a, b) for a, b in zip(first[:4], want[:4])) and torch.equal(first[5], want[5])
    assert all(a is not b for a, b in zip(first[:4], second[:4]))
    assert all(a.shape == (n,) and (n == 0 or a.data_ptr() == t.data_ptr()) for a, t in zip(first, own))
    assert first[4] is r.routed_idx and first[5] is r.routed_count
    r.conf = torch.zeros_like(r.conf)                            # a replaced tensor is the one that is written
    again = r.route(h, 0.01)
    torch.cuda.synchronize()
    assert torch.equal(again[1], want[1]) and (n == 0 or again[1].data_ptr() == r.conf.data_ptr())
    r.close()


def test_native_call_refuses_what_the_other_does(pkg):
    r = pkg.Router(S.make_W(64, 3000, seed=1, std=0.2).cuda(), max_n=4)
    h = S.make_h(4, 64, seed=2).h.cuda()
    r.route(h, 0.5)
    for bad in (h.float(), h.cpu(), h[:, :32], h.t(), h[0], torch.cat([h, h], 1)):
        with pytest.raises(ValueError):
            r.route(bad, 0.5)
    shifted = torch.empty(4 * 64 + 1, dtype=torch.bfloat16, device="cuda")[1:].view(4, 64)      # 2 bytes past 16
    with pytest.raises(pkg.TlrError) as e:
        r.route(shifted, 0.5)
    assert e.value.code == 2
    with pytest.raises(pkg.TlrError) as e:
        r.route(torch.cat([h, h]), 0.5)
    assert e.value.code == 6
    torch.cuda.synchronize()
    r.close()


def test_an_output_without_memory_is_an_error(pkg):
    r = pkg.Router(S.make_W(64, 3000, seed=1, std=0.2).cuda(), max_n=5)
    h = S.make_h(5, 64, seed=2).h.cuda()
    conf = r.conf

    def step(wrapped):
        r.conf = wrapped
        r._views[5] = (r.token, wrapped, r.entropy, r.route_mask)      # (were it kept)
        r.route(h, 0.5)
        return wrapped

    with pytest.raises(RuntimeError):
        torch.vmap(step)(torch.zeros(2, 5, device="cuda"))
    r.conf = conf
    assert r.route(h, 0.5)[1].shape == (5,)
    r.close()


def test_thresholds_are_what_ctypes_takes(pkg):
    import ctypes

    import numpy as np
    r = pkg.Router(S.make_W(64, 3000, seed=1, std=0.2).cuda(), max_n=5)
    h = S.make_h(5, 64, seed=2).h.cuda()
    tau = float(r.route(h, 0.01)[1].median())
    want = r.route(h, tau)[3].clone()
    for same in (ctypes.c_float(tau), np.float32(tau), torch.tensor(tau)):
        assert torch.equal(r.route(h, same)[3], want)
    assert int(r.route(h, 2)[5]) == 5
    for bad in (None, "0.5", 10 ** 400):
        with pytest.raises(ctypes.ArgumentError):
            r.route(h, bad)
    r.close()


def _unused(*args):
    raise AssertionError("through ctypes")


def test_native_call_takes_every_batch_size_the_first_time(pkg):
    r = pkg.Router(S.make_W(64, 3000, seed=1, std=0.2).cuda(), max_n=64)
    h = S.make_h(64, 64, seed=2).h.cuda()
    through_ctypes, r._tlr_route = r._tlr_route, _unused
    for n in list(range(65)) + [3, 64, 1]:                       # more sizes than any cache of views has
        got = r.route(h[:n], 0.01)
        assert all(t.shape == (n,) for t in got[:4])
    r._tlr_route = through_ctypes
    got[0].unsqueeze_(1)                                         # a caller's own view, changed in place
    again = r.route(h[:1], 0.01)
    native, r._native = r._native, lambda *args: None
    want = r.route(h[:1], 0.01)
    r._native = native
    assert again[0].shape == (1,) and all(a.dtype == b.dtype and a.stride() == b.stride() and a.requires_grad == b.requires_grad
                                          and a.is_inference() == b.is_inference() for a, b in zip(again[:4], want))
    r.close()


def test_native_call_writes_the_current_tensors(pkg):
    r = pkg.Router(S.make_W(64, 3000, seed=1, std=0.2).cuda(), max_n=5)
    h = S.make_h(5, 64, seed=2).h.cuda()
    want = r.route(h, 0.01)[1].clone()
    before = r.conf.detach()
    r.conf.data = torch.zeros_like(before)                       # the same object, other memory
    before.zero_()
    got = r.route(h, 0.01)[1]
    torch.cuda.synchronize()
    assert got.data_ptr() == r.conf.data_ptr() != before.data_ptr()
    assert torch.equal(r.conf, want) and not before.any()
    r.close()
