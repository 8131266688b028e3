"""The plain-FMA GEMMs on rows of more than 2^24 elements, where an offset inside a tile takes 64 bits."""
import pytest

from oracle import lory_oracle as O
from paper_2405_03133_b200.workloads import Workload, make_inputs

from gpu_util import max_rel, run_layer

pytestmark = pytest.mark.gpu


def test_rows_past_2_to_the_24():
    wl = Workload("wide", B=1, L=5, T=5, d=1, f=(1 << 24) + 5, E=1, dtype="fp32")
    inp = make_inputs(wl)
    a = (inp["x"], inp["w_r"], inp["W1"], inp["W2"], inp["W3"], wl.T)
    y, w, p = O.forward(*a)
    ref = dict(y=y, route_w=w, route_p=p, **O.backward(*a, inp["dy"]))
    got = run_layer(wl, inp)
    # fp32 sums over K = 2^24 random terms, one after the other: about 2^-24 sqrt(K / 2) = 1.7e-4, times five for the largest
    errs = {k: max_rel(got[k], ref[k]) for k in ref}
    assert all(v <= 1e-3 for v in errs.values()), errs
