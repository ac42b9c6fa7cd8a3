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
