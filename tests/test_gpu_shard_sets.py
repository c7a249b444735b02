"""Shards on the other side of a size rule than their whole set: the lanes of a
team, the reverse sweep and the one-CTA Stein step are picked by a particle
count, and the shards together must still give the whole set's bits.

The shards run one after the other on one GPU, as in tests/test_gpu_sharded.py."""
import numpy as np
import pytest
import torch

from oracle import stamp_oracle as O
from paper_2310_01775_gb300 import workloads as W

from test_gpu_block_team import packed_scene

pytestmark = pytest.mark.gpu


def run_shards(P, init, goal, N, sizes, seed, th0, svgd, sgd, lr):
    from paper_2310_01775_gb300 import sharded as SH
    stream = torch.cuda.current_stream().cuda_stream
    starts = np.cumsum([0] + sizes[:-1])
    shards = [SH.LibraryShard(P, init, goal, N, int(r0), n, seed, stream) for r0, n in zip(starts, sizes)]
    th = [th0[s.row0:s.row0 + s.rows].clone() for s in shards]
    m, v = [torch.zeros_like(t) for t in th], [torch.zeros_like(t) for t in th]
    for it in range(svgd + sgd):
        g = [s.grad(t, it) for s, t in zip(shards, th)]
        th_all, g_all = torch.cat(th).contiguous(), torch.cat(g).contiguous()
        for s, t, mm, vv in zip(shards, th, m, v):
            s.step_rows(th_all, g_all, t, mm, vv, it + 1, lr, it >= svgd)
    for s in shards:
        s.prob.sync()
        s.close()
    return torch.cat(th)


# the whole set | its shards: three touching blocks, 2 lanes per block | 4; four
# blocks, 2 | 4; two blocks, 1 | 2 and 4; one block, sequential sweep |
# time-parallel; one-CTA Stein step | the general kernels
CASES = [("pusher3_h6", {"H": 1, "T": 50}, 2048, [1024, 1024]),
         ("pusher3_h6", {"H": 1, "T": 50, "n_blocks": 4}, 2600, [2100, 500]),
         ("pusher3_h6", {"H": 1, "T": 50, "n_blocks": 2}, 9800, [9000, 800]),
         ("pusher1_h4", {"H": 2, "T": 50}, 2500, [1250, 1250]),
         ("pusher1_h2", {}, 40, [20, 20]),
         ("pusher1_h2", {}, 64, [33, 31]),
         ("pusher3_h6", {"H": 2, "T": 50}, 63, [10, 53])]


@pytest.mark.parametrize("name,over,N,sizes", CASES)
def test_shards_give_the_whole_sets_bits(name, over, N, sizes):
    from paper_2310_01775_gb300 import stamp as S
    P = W.params(name, **over)
    init, goal = packed_scene(P["n_blocks"])
    seed, lr, svgd, sgd = 11, P["lr"], 3, 1
    D = O.dims(P)[2]
    th0 = torch.tensor(O.init_theta(seed, N, D), dtype=torch.float32, device="cuda")
    whole = S.Problem(P, init, goal, N, torch.cuda.current_stream().cuda_stream)
    ref = torch.empty(N, D, device="cuda")
    whole.solve(N, svgd, sgd, seed, lr, th0, ref)
    whole.close()
    assert torch.equal(run_shards(P, init, goal, N, sizes, seed, th0, svgd, sgd, lr), ref)
