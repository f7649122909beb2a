"""ts_ffn_down after calls other than ts_ffn_gate_up: it sums what the last call on the handle left (partial sums,
bitmaps and c, or the lists of ts_mid.cu, masked or not), and stays within the scratch where a replayed graph has
left the lists of another row space."""
import pytest
import torch

from paper_2406_05955_gb300 import workload as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ts():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_2406_05955_gb300 as ts

    ts.lib()
    return ts


def _ffn(ts, d, m, B, dtype=torch.bfloat16, seed=8100):
    L = wl.ffn_layer(d, m, activation=0.25, dtype=dtype, seed=seed)
    return L, ts.Ffn(L.w_gate.cuda(), L.w_up.cuda(), L.w_down.cuda(), max_batch=B)


@pytest.mark.parametrize("dtype,d,m,B", [
    (torch.bfloat16, 512, 1408, 1),
    (torch.bfloat16, 512, 1408, 2),     # the row kernel, the bitmaps
    (torch.bfloat16, 2048, 3000, 2),    # ts_mid.cu
    (torch.bfloat16, 512, 1408, 3),
    (torch.bfloat16, 1024, 3000, 8),
    (torch.float32, 512, 1408, 2),
    (torch.float32, 512, 1408, 5),
])
def test_down_after_topk(ts, dtype, d, m, B):
    _, f = _ffn(ts, d, m, B, dtype)
    x, x2 = (wl.tokens(B, d, dtype=dtype, seed=s).cuda() for s in (8101, 8102))
    f.forward(x2)  # leaves sums and lists of other activations
    y = f.forward_topk(x, m // 20)
    assert torch.any(y) and torch.equal(f.down(B), y)


@pytest.mark.parametrize("d,m,B", [(512, 1408, 1), (2048, 3000, 2), (512, 1408, 3), (1024, 3000, 8)])
def test_down_after_stack(ts, d, m, B):
    _, f = _ffn(ts, d, m, B)
    f.forward(wl.tokens(B, d, seed=8103).cuda())
    h0 = wl.residual(B, d, seed=8104).cuda()
    h = h0.clone()
    ts.stack_forward([f], h)
    assert torch.equal(h0 + f.down(B), h)


@pytest.mark.parametrize("B", [1, 2, 5])
def test_down_after_empty_predicted_list(ts, B):
    L, f = _ffn(ts, 2048, 3000, B)
    w = wl.predictor_weights(2048, 256, 3000, L.offsets, seed=8105)
    p = ts.Predictor(w.w1.cuda(), w.w2.cuda(), max_batch=B)
    f.forward(wl.tokens(B, 2048, seed=8106).cuda())
    h0 = wl.residual(B, 2048, seed=8107).cuda()
    h = h0.clone()
    ts.stack_forward_predicted([f], [p], h, [0], [torch.zeros(1, dtype=torch.int32, device="cuda")])
    assert torch.equal(h, h0) and not torch.any(f.down(B))


def test_down_over_lists_of_a_replayed_graph(ts):
    """The graph's dense pass lists more rows per CTA than the list of the gate_up before it has."""
    d, m, B = 1024, 14336, 6
    L, f = _ffn(ts, d, m, B)
    x = wl.tokens(B, d, seed=8108).cuda()
    idx = wl.predictor_list(L.offsets, 1200, seed=8109).cuda()
    h = wl.residual(B, d, seed=8110).cuda()
    y = f.forward(x, active_idx=idx)
    g = ts.Graph.stack([f], h)
    f.gate_up(x, active_idx=idx)
    assert torch.equal(f.down(B), y)
    g.launch()
    f.down(B)
    assert f.check_scratch() == 0 and f.get_error() == 0
    assert torch.equal(f.forward(x, active_idx=idx), y)
