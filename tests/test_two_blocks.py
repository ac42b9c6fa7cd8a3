"""Batches of more than 256 rows whose work units are two blocks of 256 token rows: the schedule on the CPU, results on the GPU."""
import os
import shutil
import subprocess
import sys

import numpy as np
import pytest
import torch

import paper_2504_07878_b200 as P
import tlr_synth as S
from oracle import route_oracle as O

from .parity import check_against_oracle, check_self_consistency


@pytest.mark.parametrize("n,V,hidden", [(257, 300, 0), (512, 128256, 0), (777, 151936, 256), (1000, 17, 0), (2049, 60000, 40),
                                        (4096, 151936, 1024), (16384, 128256, 0), (27000, 3001, 0), (27000, 20000, 300),
                                        (41000, 9000, 256)])
def test_tiles_of_both_blocks_cover_every_logit_once(n, V, hidden):
    tiles, plan = P.tlr_debug_plan_tiles(n, V, 148, hidden, blocks=2)
    g, vocab_units = plan.reserved, plan.vocab_chunks * plan.row_units
    assert plan.row_units == -(-n // 512) and plan.vocab_chunks <= 192 and plan.grid <= 148
    for ru in range(plan.row_units):
        for router in (False, True) if hidden else (False,):
            sel = tiles[(tiles[:, 2] == 512 * ru) & ((tiles[:, 1] >= vocab_units) == router)]
            sel = sel[np.argsort(sel[:, 3])]
            start, end = (V, V + -(-hidden // 32) * 32) if router else (0, -(-V // g) * g)
            assert sel[0, 3] == start and sel[-1, 3] + sel[-1, 4] == end and np.all(sel[:, 4] <= 256)
            assert np.array_equal(sel[1:, 3], (sel[:, 3] + sel[:, 4])[:-1])
    first_of_unit = np.unique(tiles[:, 1], return_index=True)[1]
    assert len(np.unique(tiles[:, :2], axis=0)) == len(first_of_unit)            # one worker per unit
    # group by group of row units, the groups being equal but for the last (50 MB of h at d = 2048), and in a group chunk by chunk
    groups = -(-n * 4096 // (50 << 20))
    size = -(-plan.row_units // groups)
    vocab = tiles[first_of_unit][:vocab_units]
    ru, chunk = vocab[:, 2] // 512, np.searchsorted(np.unique(vocab[:, 3]), vocab[:, 3])
    assert np.array_equal(np.lexsort((ru, chunk, ru // size)), np.arange(vocab_units))


WALK = r"""
#include "tlr_tc_kernel.cuh"
#include <cstdio>
#include <cstdlib>
int main(int, char** argv) {
  tlr::TcParams p = {};
  p.n = atoi(argv[1]);
  p.lag = atoi(argv[2]);
  for (int slabs = 1; slabs <= 40; ++slabs) {
    const tlr::TwoWalk w(p, 0, slabs);
    for (int i = 0; i < w.items; ++i) {
      int block, slab;
      w.at(i, block, slab);
      printf("%d %d %d\n", slabs, block, slab);
    }
  }
}
"""


# The walk of one tile, as the kernel makes it: every slab of either block once and in order, the second block behind the first, and
# never more slabs of W in use than lag + 1, which is what a ring must hold.
def test_walk_of_both_blocks(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    (tmp_path / "walk.cu").write_text(WALK)
    subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-I", root + "/include",
                    "-I", root + "/paper_2504_07878_b200/csrc", str(tmp_path / "walk.cu"), "-o", str(tmp_path / "walk")], check=True)
    for n, blocks in ((256, 1), (257, 2), (512, 2)):
        for lag in (1, 2, 5):
            out = subprocess.run([str(tmp_path / "walk"), str(n), str(lag)], check=True, capture_output=True, text=True).stdout
            walk = np.array([line.split() for line in out.splitlines()], dtype=int)
            for slabs in range(1, 41):
                items = walk[walk[:, 0] == slabs, 1:]
                seen = [0, 0]
                for block, slab in items:
                    assert slab == seen[block]
                    seen[block] += 1
                    assert blocks == 1 or 0 <= seen[0] - seen[1] <= lag + 1
                assert seen == [slabs, slabs if blocks == 2 else 0]


# With a lag of one the second block reads a slab of W behind the first block's next one: two stages, or such batches stay on
# single blocks, which work with one.
@pytest.mark.parametrize("rings,status", [("5,1", 3), ("5,2", 0), ("1,8", 0), ("4,9", 0)])
def test_a_ring_that_cannot_hold_both_blocks_slabs(rings, status):
    code = ("import ctypes, paper_2504_07878_b200 as P; c = ctypes.c_int32(0)\n"
            "print(P.load_library().tlr_debug_plan_two_blocks(512, 128256, 148, 0, None, 0, ctypes.byref(c), None),"
            " P.load_library().tlr_debug_plan_tiles(512, 128256, 148, 0, None, 0, ctypes.byref(c), None))")
    run = subprocess.run([sys.executable, "-c", code], cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                         env=dict(os.environ, TLR_TC_RINGS=rings), capture_output=True, text=True)
    assert run.returncode == 0 and run.stdout.split() == [str(status), "0"], run.stdout + run.stderr


# The fewest slabs of K and more, in part; second blocks of one row, of all rows and (25 blocks) of none; several units per worker;
# with a learned router, whose tiles are the same walk; two groups of row units, of seven and six, without a router and with one.  Where W's rows begin on sectors
# (d % 16 == 0) short walks and single row units stay on single blocks.
@pytest.mark.gpu
@pytest.mark.parametrize("n,d,V,hidden,two", [(257, 1032, 67000, 0, True), (300, 712, 105000, 0, True), (769, 584, 61000, 40, True),
                                              (1000, 904, 43000, 0, True), (1500, 712, 35000, 300, True), (6200, 584, 11500, 0, True),
                                              (6656, 4104, 2800, 40, True),
                                              (6656, 4104, 2800, 0, True), (2000, 1008, 47000, 30, True),
                                              (257, 1024, 67000, 0, False), (1000, 896, 43000, 0, False), (512, 1024, 151936, 0, False)])
def test_two_blocks_match_the_oracle(n, d, V, hidden, two):
    W = S.make_W(d, V, seed=n, std=0.08)
    hid = S.make_h(n, d, seed=d, W=W, planted_fraction=0.1)
    rows = np.unique(np.concatenate([np.arange(0, n, 11 if n < 2000 else 37), np.arange(250, 262) % n, np.arange(max(0, n - 140), n)]))
    ref = O.route_oracle(S.bf16_bits(hid.h)[rows], S.bf16_bits(W), 0.5)
    r = P.Router(W.cuda(), max_n=n)
    options = {}
    if hidden:
        gen = torch.Generator().manual_seed(hidden)
        W1 = (torch.randn(hidden, d, generator=gen) / d ** 0.5).to(torch.bfloat16)
        b1, w2 = torch.randn(hidden, generator=gen) * 0.1, torch.randn(hidden, generator=gen) * 0.2
        r.set_router_mlp(W1.cuda(), b1.cuda(), w2.cuda(), 0.2)
        options["mlp_score"] = torch.full((n,), float("nan"), device="cuda")
    assert P.tlr_plan_query(r.ctx, n).reserved == (2 if two else 0)
    for _ in range(3):
        r.route(hid.h.cuda(), 0.5, **options)
    torch.cuda.synchronize()
    assert P.tlr_last_device_status(r.ctx) == 0
    names = ("token", "conf", "entropy", "route_mask", "routed_idx", "routed_count")
    full = {k: getattr(r, k).cpu().numpy()[:n] for k in names}
    full["routed_count"] = int(full["routed_count"][0])
    check_self_consistency(full, 0.5, V)
    check_against_oracle(ref, {k: full[k][rows] for k in names[:4]})
    if hidden:
        want = O.mlp_router_score(S.bf16_bits(hid.h), S.bf16_bits(W1), b1.numpy(), w2.numpy(), 0.2)
        assert np.max(np.abs(options["mlp_score"].cpu().numpy() - want)) <= 1e-5     # fp32 sums of exact products
    r.close()
