"""Passes of 1-2 tokens over INT4 rows (k_gate_up_q4w) against the fp64 oracle at the edges of
its tiling: the shortest and longest rows taken, groups and chunks cut short, more chunks on an
SM than one round takes, a list, and calls in a row, where a call may start while the reduction
before it runs.

Tolerance: a scale group's fp32 sum holds terms of (136 + |w|) |x| for |w| |x| with |w|
about 4, so its roundings (2^-24 each, two for the K-steps, one each for the correction
and the scale) weigh about 35 times those of a plain sum: 4 * 35 * 2^-24 = 8.3e-6 of one
group's magnitude, and the roundings of a row's 8 to 160 groups are independent, so they
shrink against the row's sum. 1e-5 bounds them.
"""
import pytest
import torch

import oracle
from paper_2406_05955_gb300 import workload as wl

from _parity import check_sets, rel_l2

pytestmark = pytest.mark.gpu
REL = 1e-5


@pytest.fixture(scope="module")
def ts():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_2406_05955_gb300 as ts

    ts.lib()
    return ts


@pytest.mark.parametrize("d,m,B,act,n_list", [
    (256, 9, 1, 0.5, 0),          # one row group a quarter, a second chunk of one row
    (256, 40000, 2, 0.25, 0),     # more chunks on an SM than a round takes
    (768, 1217, 2, 0.25, 0),      # 153 chunks on 152 SMs
    (2304, 5000, 1, 1.0, 0),      # every row gate-active
    (4352, 3001, 2, 0.10, 0),     # d / 128 odd groups a quarter
    (5120, 2048, 1, 0.25, 0),     # the longest rows taken
    (5120, 2048, 2, 0.25, 700),   # and a list
])
def test_int4_edges(ts, d, m, B, act, n_list):
    L = wl.ffn_layer_int4(d, m, activation=act, seed=8900 + m + B)
    x = wl.tokens(B, d, seed=8901)
    rows = wl.predictor_list(L.offsets, n_list, seed=8902) if n_list else None
    idx = rows.cuda() if n_list else None
    f = ts.Ffn(L.w_gate.cuda(), L.w_up.cuda(), L.w_down.cuda(), max_batch=B)
    y = f.forward(x.cuda(), active_idx=idx).double().cpu().numpy()
    ref = oracle.ffn(x, L.w_gate, L.w_up, L.w_down, rows=None if rows is None else rows.numpy())
    assert rel_l2(y, ref["y"]) <= REL
    for t in range(B):
        check_sets(*f.get_active(t), ref, t, rows=None if rows is None else rows.numpy())


@pytest.mark.parametrize("B", [1, 2])
def test_int4_calls_in_a_row(ts, B):
    d, m = 1024, 4000
    layers = [wl.ffn_layer_int4(d, m, activation=0.10, seed=wl.layer_seed(8910, l)) for l in range(2)]
    ffns = [ts.Ffn(L.w_gate.cuda(), L.w_up.cuda(), L.w_down.cuda(), max_batch=B) for L in layers]
    xs = [wl.tokens(B, d, seed=8911 + i).cuda() for i in range(4)]
    one = []
    for f in ffns:
        for x in xs:
            one.append(f.forward(x).clone())
            torch.cuda.synchronize()
    for _ in range(5):
        ys = [torch.empty_like(one[0]) for _ in one]
        for i, y in enumerate(ys):
            ffns[i // 4].forward(xs[i % 4], y=y)
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(one, ys))
