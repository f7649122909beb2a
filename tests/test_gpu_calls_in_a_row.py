"""Calls in a row without a wait between them, each on other activations, against the same calls one at a time: the
next call's first kernel may start while the reduction of a dense bf16 call of 1-2 tokens over at least 2^24 weights, or
of a wide one, still runs, and must not write scratch or read activations before it has ended."""
import pytest
import torch

from paper_2406_05955_gb300 import workload as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,m,batches", [
    (4096, 4096, [1] * 8),                      # the smallest weights that trigger early
    (4096, 4096, [2] * 8),
    (1024, 4000, [16] * 8),                     # wide
    (1024, 4000, [40] * 8),
    (4096, 4096, [40, 1, 5, 16, 2, 1, 64, 3]),  # every kind of pass on one handle
    (256, 65536, [1, 1, 40, 40, 16, 2, 2, 9]),  # short rows, many of them: CTAs that leave an SM room for the next call's
])
def test_calls_in_a_row(d, m, batches):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_2406_05955_gb300 as ts

    L = wl.ffn_layer(d, m, activation=0.10, dtype=torch.bfloat16, seed=8200, device=torch.device("cuda"))
    f = ts.Ffn(L.w_gate, L.w_up, L.w_down, max_batch=max(batches))
    xs = [wl.tokens(b, d, seed=8201 + i).cuda() for i, b in enumerate(batches)]
    one = []
    for x in xs:
        one.append(f.forward(x))
        torch.cuda.synchronize()
    for _ in range(5):
        ys = [torch.empty_like(y) for y in one]
        torch.cuda.synchronize()
        for x, y in zip(xs, ys):
            f.forward(x, y=y)
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(one, ys))
    assert f.get_error() == 0 and f.check_scratch() == 0
