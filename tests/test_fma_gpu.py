"""The plain-FMA pipeline at the edges of its tiles: segments shorter and longer than 32-, 64- and 128-row tiles, sizes off
the 4-element vectors, more segments and experts than one chunk of the merge adjoint, and the experts past its range."""
import pytest

from oracle import lory_oracle as O
from paper_2405_03133_b200 import LORY_FLAG_SIMT
from paper_2405_03133_b200.workloads import Workload, make_inputs

from gpu_util import max_rel, run_layer

pytestmark = pytest.mark.gpu

CASES = [  # B, T, segments per sequence, d, f, E, dtype
    (1, 1, 1, 5, 3, 1, "fp32"), (2, 33, 2, 31, 65, 5, "fp32"), (1, 65, 3, 64, 68, 8, "fp32"), (2, 129, 1, 66, 132, 9, "fp32"),
    (1, 16, 33, 20, 28, 16, "fp32"), (3, 8, 40, 17, 24, 17, "fp32"), (2, 12, 4, 40, 36, 32, "fp32"), (2, 12, 4, 40, 36, 33, "fp32"),
    (5, 256, 12, 96, 260, 3, "fp32"),    # enough tiles for 128 rows each
    (2, 24, 3, 40, 72, 70, "bf16"), (2, 48, 3, 72, 136, 6, "bf16"),
]


@pytest.mark.parametrize("B,T,N,d,f,E,dtype", CASES)
def test_plain_fma_edges(B, T, N, d, f, E, dtype):
    wl = Workload("fma", B=B, L=N * T, T=T, d=d, f=f, E=E, dtype=dtype, w_r_std=1.0)
    inp = make_inputs(wl)
    a = (inp["x"], inp["w_r"], inp["W1"], inp["W2"], inp["W3"], wl.T)
    y, w, p = O.forward(*a)
    ref = dict(y=y, route_w=w, route_p=p, **O.backward(*a, inp["dy"]))
    got = run_layer(wl, inp, flags=LORY_FLAG_SIMT if dtype == "bf16" else 0)
    errs = {k: max_rel(got[k], ref[k]) for k in ref}
    assert all(v <= (1e-4 if dtype == "fp32" else 2e-2) for v in errs.values()), errs
