"""The grouped GEMMs' tile shapes: segment lengths and widths that pick CTA pairs with a ragged second half, 128- and
64-column tiles, one and several rounds."""
import pytest

from oracle import lory_oracle as O
from paper_2405_03133_b200.workloads import Workload, make_inputs

from gpu_util import max_rel, run_layer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,N,T,d,f", [
    (1, 1, 200, 72, 136),      # one pair, its second CTA partly past the segment
    (1, 2, 600, 264, 520),     # pairs whose last tile has an empty second CTA
    (1, 1, 1000, 640, 264), (2, 4, 130, 520, 72), (1, 3, 257, 1032, 328), (4, 10, 160, 392, 648), (1, 1, 16, 2048, 64),
    (3, 12, 100, 1000, 264),
])
def test_every_tile_shape(B, N, T, d, f):
    wl = Workload("tiles", B=B, L=N * T, T=T, d=d, f=f, E=3, dtype="bf16", w_r_std=1.0)
    inp = make_inputs(wl)
    a = (inp["x"], inp["w_r"], inp["W1"], inp["W2"], inp["W3"], wl.T)
    y, w, p = O.forward(*a)
    ref = dict(y=y, route_w=w, route_p=p, **O.backward(*a, inp["dy"]))
    got = run_layer(wl, inp)
    errs = {k: max_rel(got[k], ref[k]) for k in ref}
    assert all(v <= 2e-2 for v in errs.values()), errs
