"""Segment means shared by the blocks of a cluster (few segments): one, two, four and eight blocks per segment, token counts
that split unevenly, widths that end inside a block's columns or are no whole vectors."""
import pytest
import torch

import paper_2405_03133_b200 as lory
from oracle import lory_oracle as O
from paper_2405_03133_b200.workloads import Workload, make_inputs

from gpu_util import max_rel, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,d", [("bf16", 8), ("bf16", 264), ("bf16", 1000), ("fp32", 3), ("fp32", 130), ("fp32", 516)])
@pytest.mark.parametrize("N,T", [(1, 63), (1, 64), (2, 65), (1, 127), (3, 128), (1, 255), (2, 256), (1, 257), (2, 1001), (37, 256)])
def test_means_of_few_segments(N, T, dtype, d):
    wl = Workload("pool", B=1, L=N * T, T=T, d=d, f=8, E=5, dtype=dtype, w_r_std=1.0, seed=T)
    inp = make_inputs(wl)
    dims = lory.make_dims(wl.B, wl.L, wl.T, wl.d, wl.f, wl.E, dtype)
    rw = torch.full((wl.S, wl.E), float("nan"), device="cuda")
    rp = torch.full_like(rw, float("nan"))
    lory.lory_route_noalloc(dims, to_dev(inp["x"], wl), to_dev(inp["w_r"], wl), rw, rp)
    _, p, w = O.route(inp["x"], inp["w_r"], wl.T)
    assert max_rel(rw.cpu().numpy(), w) <= 1e-5 and max_rel(rp.cpu().numpy(), p) <= 1e-5
