"""Passes of 2-16 tokens over bf16 and INT4 rows (ts_mid.cu), and wider ones (ts_wide.cu), against the fp64 oracle, at
the sizes where their tiling ends: a K block that d only partly fills, fewer K
blocks than warps, groups of 16 rows and rounds of chunks cut short, list
slices longer than one piece, and batches around the widths of 8 and 16.

Tolerance: the kernels add at most 16 (K-slice) + 16 (slices) fp32 terms per
dot product and the down projection keeps c to 24 bits, so a result is off by
about 40 * 2^-24 = 2.4e-6 of the sums' magnitude; 1e-5 leaves room for cancellation.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2406_05955_gb300 import workload as wl

from _parity import check_sets, rel_l2

pytestmark = pytest.mark.gpu
REL = 1e-5
# The wide kernels: c enters the down projection as two bf16 numbers (2^-17 of it lost) and the tensor core truncates
# when it accumulates; this is about twice what that gives.
WIDE_REL = 2e-5


@pytest.fixture(scope="module")
def ts():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_2406_05955_gb300 as ts

    ts.lib()
    return ts


def _ffn(ts, L, max_batch):
    return ts.Ffn(L.w_gate.cuda(), L.w_up.cuda(), L.w_down.cuda(), max_batch=max_batch)


@pytest.mark.parametrize("d,m,B,act,n_list", [
    (8, 5, 3, 0.5, 0),          # one K block a quarter full, one chunk cut short
    (40, 1217, 16, 0.25, 0),    # a second K block one lane wide; 153 chunks on 152 SMs
    (1032, 2049, 9, 0.25, 0),   # d % 32 != 0 across slices; the narrowest 16-wide pass
    (2304, 3000, 8, 0.10, 0),   # 72 K blocks over 16 slices: uneven slices
    (4088, 16000, 12, 1.0, 0),  # every row active, d % 256 != 0: 842 rows a slice, over one piece of 768
    (4096, 20000, 5, 1.0, 0),   # 1052 rows a slice, over one piece of 1024
    (5120, 1000, 6, 0.25, 0),   # rows so long that the activations stay in shared memory: 3 stages in flight a warp,
    (6144, 700, 5, 0.25, 0),    # 2,
    (8192, 600, 2, 0.25, 0),    # 1 (the longest rows taken, by two tokens)
    (512, 40000, 5, 0.25, 0),   # several rounds of chunks per CTA
    (1024, 3000, 33, 0.25, 0),  # the wide kernels' side of the dispatch
    (1000, 3000, 33, 0.25, 0),  # d % 256 != 0: passes of 16, 16 and 1
    (1024, 3584, 7, 0.25, 1),   # a list of one row
    (1024, 3584, 16, 0.25, 100),  # a list shorter than the grid
    (2048, 3584, 4, 0.25, 3584),  # every row listed
    (2048, 2048, 2, 0.25, 0),   # two tokens: the smallest weights that leave the row kernel
    (2048, 2047, 2, 0.25, 0),   # and the largest that stay
    (688, 3072, 2, 0.25, 0),    # the fewest short rows that leave it
    (688, 3071, 2, 0.25, 0),    # and the most that stay
    (4096, 3000, 2, 0.25, 600),  # the same over a list
])
def test_mid_pass(ts, d, m, B, act, n_list):
    L = wl.ffn_layer(d, m, activation=act, dtype=torch.bfloat16, seed=7100 + m + B)
    x = wl.tokens(B, d, seed=7101)
    f = _ffn(ts, L, B)
    rows = wl.predictor_list(L.offsets, n_list, seed=7102) if n_list else None
    idx = rows.cuda() if n_list else None
    y = f.forward(x.cuda(), active_idx=idx).double().cpu().numpy()
    ref = oracle.ffn(x, L.w_gate, L.w_up, L.w_down, rows=None if rows is None else rows.numpy())
    assert rel_l2(y, ref["y"]) <= (REL if B <= 16 or d % 256 else WIDE_REL)
    for t in {0, B - 1}:
        check_sets(*f.get_active(t), ref, t, rows=None if rows is None else rows.numpy())
    assert f.get_error() == 0 and f.check_scratch() == 0
    assert np.array_equal(f.forward(x.cuda(), active_idx=idx).double().cpu().numpy(), y)


def test_mid_unaligned_buffers(ts):
    """x and y that start between 16-byte boundaries take element loads and stores, with the same bits."""
    d, m, B = 264, 500, 6
    L = wl.ffn_layer(d, m, activation=0.25, dtype=torch.bfloat16, seed=7200)
    f = _ffn(ts, L, B)
    x = wl.tokens(B, d, seed=7201).cuda()
    y = f.forward(x)
    xu = torch.empty(B * d + 1, dtype=torch.bfloat16, device="cuda")[1:].view(B, d)
    yu = torch.empty(B * d + 1, device="cuda")[1:].view(B, d)
    xu.copy_(x)
    f.forward(xu, y=yu)
    assert torch.equal(y, yu)


@pytest.mark.parametrize("B", [2, 3, 8])
def test_mid_moe_many_rounds(ts, B):
    """Several rounds of chunks per CTA, ranges that cross from one expert to the next."""
    d, m, E = (256 if B == 2 else 64), 6001, 8
    experts = [wl.ffn_layer(d, m, activation=0.20, dtype=torch.bfloat16, seed=wl.layer_seed(7300, 0, e)) for e in range(E)]
    wr = wl.router(E, d, seed=7301)
    x = wl.tokens(B, d, seed=7302)
    moe = ts.Moe(wr.cuda(), [_ffn(ts, L, B) for L in experts], top_k=2, max_batch=B)
    y = moe.forward(x.cuda()).double().cpu().numpy()
    sel, w = moe.get_routing(B)
    ref = oracle.moe(x, wr, [(L.w_gate, L.w_up, L.w_down) for L in experts], top_k=2, sel=sel, w=w)
    assert rel_l2(y, ref["y"]) <= REL
    assert moe.get_error() == 0 and moe.check_scratch() == 0


@pytest.mark.parametrize("B", [5, 16, 20])
def test_mid_stack_graph_equals_layers(ts, B):
    d, m, n = 1000, 2000, 3
    layers = [wl.ffn_layer(d, m, activation=0.10, dtype=torch.bfloat16, seed=wl.layer_seed(7400, l)) for l in range(n)]
    ffns = [_ffn(ts, L, B) for L in layers]
    h0 = wl.residual(B, d, seed=7401).cuda()
    h_one, h_graph = h0.clone(), h0.clone()
    for f in ffns:
        ts.stack_forward([f], h_one)
    g = ts.Graph.stack(ffns, h_graph)
    g.launch()
    torch.cuda.synchronize()
    assert torch.equal(h_graph, h_one)


@pytest.mark.parametrize("B", [3, 4])
def test_short_pass_before_dense_layer(ts, B):
    """A short list's pass ends in k_down, which prefetches the next layer's rows: 251 chunks for 152 CTAs."""
    d, m, n = 1000, 2001, 3
    layers = [wl.ffn_layer(d, m, activation=0.10, dtype=torch.bfloat16, seed=wl.layer_seed(7450, l)) for l in range(n)]
    ffns = [_ffn(ts, L, B) for L in layers]
    lists = [wl.predictor_list(L.offsets, 90, seed=7451).cuda() if l != 1 else None for l, L in enumerate(layers)]
    h0 = wl.residual(B, d, seed=7452).cuda()
    h_one, h_all = h0.clone(), h0.clone()
    for f, r in zip(ffns, lists):
        ts.stack_forward([f], h_one, active_idx=[r])
    ts.stack_forward(ffns, h_all, active_idx=lists)
    assert torch.equal(h_all, h_one) and all(f.get_error() == 0 and f.check_scratch() == 0 for f in ffns)


@pytest.mark.parametrize("d,m,B,act,n_list", [
    (256, 9, 3, 0.5, 0),          # one stage, one K slice
    (768, 1217, 16, 0.25, 0),     # three stages over four slices, one of them empty
    (4096, 16000, 9, 1.0, 0),     # every row active: 842 rows a slice, over one piece of 768
    (4352, 1000, 5, 0.25, 0),     # rows so long that the activations stay in shared memory
    (1024, 3000, 19, 0.25, 0),    # a pass of 16, then one of 3
    (2048, 3584, 6, 0.25, 900),   # a predictor list
])
def test_mid_int4(ts, d, m, B, act, n_list):
    L = wl.ffn_layer_int4(d, m, activation=act, seed=7500 + m + B)
    x = wl.tokens(B, d, seed=7501)
    rows = wl.predictor_list(L.offsets, n_list, seed=7502) if n_list else None
    idx = rows.cuda() if n_list else None
    f = ts.Ffn(L.w_gate.cuda(), L.w_up.cuda(), L.w_down.cuda(), max_batch=B)
    y = f.forward(x.cuda(), active_idx=idx).double().cpu().numpy()
    ref = oracle.ffn(x, L.w_gate, L.w_up, L.w_down, rows=None if rows is None else rows.numpy())
    assert rel_l2(y, ref["y"]) <= REL
    for t in {0, B - 1}:
        check_sets(*f.get_active(t), ref, t, rows=None if rows is None else rows.numpy())
    assert f.get_error() == 0 and f.check_scratch() == 0
    xu = torch.empty(B * d + 1, dtype=torch.bfloat16, device="cuda")[1:].view(B, d)
    xu.copy_(x)
    if B <= 16:  # (a longer batch is split into other passes when x is not aligned)
        assert rel_l2(f.forward(xu, active_idx=idx).double().cpu().numpy(), y) <= REL


@pytest.mark.parametrize("d,m,B,act,n_list", [
    (256, 20, 17, 0.5, 0),       # two tiles of 16 rows, the second cut short; two K stages
    (1024, 3584, 9, 0.25, 0),    # the narrowest wide batch; 9-16 tokens over enough rows
    (512, 20000, 40, 0.25, 0),   # more than 128 rows per SM: two waves of tiles
    (768, 2435, 33, 1.0, 0),     # every row active; tiles that end inside a bitmap word; three token tiles
    (512, 3584, 64, 0.10, 777),  # a predictor list
])
def test_wide_tiles(ts, d, m, B, act, n_list):
    """ts_wide.cu at the ends of its tiling."""
    L = wl.ffn_layer(d, m, activation=act, dtype=torch.bfloat16, seed=7600 + m + B)
    x = wl.tokens(B, d, seed=7601)
    rows = wl.predictor_list(L.offsets, n_list, seed=7602) if n_list else None
    idx = rows.cuda() if n_list else None
    f = _ffn(ts, L, B)
    y = f.forward(x.cuda(), active_idx=idx)
    ref = oracle.ffn(x, L.w_gate, L.w_up, L.w_down, rows=None if rows is None else rows.numpy())
    assert rel_l2(y.double().cpu().numpy(), ref["y"]) <= WIDE_REL
    for t in {0, B // 2, B - 1}:
        check_sets(*f.get_active(t), ref, t, rows=None if rows is None else rows.numpy())
    assert f.get_error() == 0 and f.check_scratch() == 0
    assert torch.equal(f.forward(x.cuda(), active_idx=idx), y)


@pytest.mark.parametrize("d,m,B,n_list", [
    (1280, 3124, 3, 48),      # a short list: k_down instead of the slices
    (4096, 14336, 4, 256),    # the most rows of that width that count as few
    (4096, 14336, 4, 257),    # and one more
    (512, 1408, 3, 0),        # few rows without a list
    (1000, 300, 19, 0),       # passes of 16, then of 3 over few rows
])
def test_short_passes(ts, d, m, B, n_list):
    L = wl.ffn_layer(d, m, activation=0.10, dtype=torch.bfloat16, seed=7600 + m + B)
    x = wl.tokens(B, d, dtype=torch.bfloat16, seed=7601)
    rows = wl.predictor_list(L.offsets, n_list, seed=7602) if n_list else None
    idx = rows.cuda() if n_list else None
    f = _ffn(ts, L, B)
    y = f.forward(x.cuda(), active_idx=idx)
    ref = oracle.ffn(x, L.w_gate, L.w_up, L.w_down, rows=None if rows is None else rows.numpy())
    assert rel_l2(y.double().cpu().numpy(), ref["y"]) <= REL
    for t in {0, B - 1}:
        check_sets(*f.get_active(t), ref, t, rows=None if rows is None else rows.numpy())
    if B <= 8:
        f.gate_up(x.cuda(), active_idx=idx)
        assert torch.equal(f.down(B), y)


@pytest.mark.parametrize("d,m,B", [(264, 700, 3), (512, 3000, 5), (520, 3000, 16), (2048, 2100, 2)])
def test_mid_infinite_weights(ts, d, m, B):
    """An infinite W_down weight gives an infinite sum where every token is active, as in fp32: c = 6 has one
    significant bf16 part, and a part of zero times the weight would be NaN."""
    w = torch.zeros(m, d, dtype=torch.bfloat16)
    wg, wu, wd = w.clone(), w.clone(), torch.ones_like(w)
    wg[:, d - 1], wu[:, d - 1] = 2.0, 3.0
    wd[m // 2, 7], wd[m - 1, d - 1] = float("inf"), float("-inf")
    f = ts.Ffn(wg.cuda(), wu.cuda(), wd.cuda(), max_batch=B)
    y = f.forward(wl.tokens(B, d, seed=7800).cuda()).cpu()
    ref = torch.full((B, d), 6.0 * m)
    ref[:, 7], ref[:, d - 1] = float("inf"), float("-inf")
    assert torch.equal(y, ref)


@pytest.mark.parametrize("d,m,B", [(1024, 3000, 9), (1000, 3000, 16), (1024, 4000, 16), (1024, 4000, 40)])
def test_weights_written_by_the_kernel_before(ts, d, m, B):
    """More than 8 tokens: weights that the kernel before the call writes are read as written."""
    a, b = (wl.ffn_layer(d, m, activation=0.10, dtype=torch.bfloat16, seed=s) for s in (7900, 7901))
    sets = [[w.cuda() for w in (L.w_gate, L.w_up, L.w_down)] for L in (a, b)]
    w = [t.clone() for t in sets[0]]
    f = ts.Ffn(*w, max_batch=B)
    x = wl.tokens(B, d, seed=7902).cuda()
    want = [ts.Ffn(*s, max_batch=B).forward(x) for s in sets]
    got = []
    for i in range(20):
        for k in (1, 2, 0):  # w_gate last: its rows are the first that the call reads
            torch.mul(sets[i % 2][k], 1.0, out=w[k])  # (a kernel: copy_ is a memcpy)
        got.append(f.forward(x))
    assert all(torch.equal(y, want[i % 2]) for i, y in enumerate(got))


def test_router_written_by_the_kernel_before(ts):
    d, m, B, E = 1024, 600, 3, 8
    experts = [_ffn(ts, wl.ffn_layer(d, m, activation=0.20, dtype=torch.bfloat16, seed=7910 + e), B) for e in range(E)]
    sets = [wl.router(E, d, seed=s).cuda() for s in (7920, 7921)]
    wr = sets[0].clone()
    x = wl.tokens(B, d, seed=7922).cuda()
    want = [ts.Moe(s, experts, top_k=2, max_batch=B).forward(x) for s in sets]
    moe = ts.Moe(wr, experts, top_k=2, max_batch=B)
    got = []
    for i in range(20):
        torch.mul(sets[i % 2], 1.0, out=wr)
        got.append(moe.forward(x))
    assert all(torch.equal(y, want[i % 2]) for i, y in enumerate(got))
