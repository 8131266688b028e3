"""The merge on both sides of the lines between its streaming and its tcgen05 kernel (49..64 experts with more than 64 segments,
33..48 with 193..256 or more than 384), one and two tiles of 128 segments and a second launch, sizes that end inside a block; forward, and the backward that reads its
result."""
import pytest

from oracle import lory_oracle as O
from paper_2405_03133_b200.workloads import Workload, make_inputs

from gpu_util import max_rel, run_layer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S,E,d,f", [
    (64, 49, 72, 136), (65, 49, 72, 136), (127, 64, 64, 72), (128, 56, 136, 64), (129, 64, 72, 200), (256, 64, 64, 64),
    (300, 49, 64, 72), (192, 48, 72, 64), (193, 48, 72, 136), (256, 33, 136, 72), (257, 33, 64, 64), (384, 40, 64, 64), (385, 40, 64, 72),
])
def test_merge_routes(S, E, d, f):
    wl = Workload("merge", B=S, L=4, T=4, d=d, f=f, E=E, dtype="bf16", w_r_std=2.0)
    inp = make_inputs(wl)
    a = (inp["x"], inp["w_r"], inp["W1"], inp["W2"], inp["W3"], wl.T)
    y, w, p = O.forward(*a)
    ref = dict(y=y, route_w=w, route_p=p, **O.backward(*a, inp["dy"]))
    got = run_layer(wl, inp)
    errs = {k: max_rel(got[k], ref[k]) for k in ref}
    assert all(v <= 2e-2 for v in errs.values()), errs
