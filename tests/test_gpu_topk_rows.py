"""The two selection kernels of the top-k mask on either side of the row count
that divides them, at row counts that end inside a bitmap word, with one token
(whose select also writes the union) and several, and with ties at the cut."""
import numpy as np
import pytest
import torch

import oracle
from paper_2406_05955_gb300 import workload as wl

from _parity import check_y
from test_gpu_topk import _check_kept

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,B,keep,act", [(7, 1, 2, 0.25), (33, 3, 5, 0.25), (16384, 1, 900, 0.25),
                                          (16384, 3, 16000, 0.25), (16385, 1, 900, 0.25), (16385, 2, 40, 0.25),
                                          # the most rows kept that k_down gathers, and one a token more
                                          (3000, 4, 512, 0.5), (3000, 4, 513, 0.5),
                                          # every row a candidate: 16 a thread, words cleared by two threads
                                          (16384, 1, 5461, 1.0), (16383, 2, 8000, 1.0), (1057, 1, 1056, 1.0)])
def test_topk_row_counts(m, B, keep, act):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_2406_05955_gb300 as ts

    d = 256
    L = wl.ffn_layer(d, m, activation=act, dtype=torch.bfloat16, seed=7700 + m + B)
    # equal neurons tie at the cut wherever it falls between them: the lower index is kept
    for w in (L.w_gate, L.w_up):
        w[1::2] = w[0:m - m % 2:2].clone()[: w[1::2].shape[0]]
    x = wl.tokens(B, d, seed=7701)
    f = ts.Ffn(L.w_gate.cuda(), L.w_up.cuda(), L.w_down.cuda(), max_batch=B)
    y = f.forward_topk(x.cuda(), keep).double().cpu().numpy()
    ref = oracle.ffn_topk(x, L.w_gate, L.w_up, L.w_down, keep)
    check_y(y, ref["y"], "bf16")
    for t in range(B):
        kept = f.get_active(t)[1]
        _check_kept(kept, ref, t, keep)
        if np.array_equal(np.sort(kept), np.nonzero(ref["sel"][t] & (ref["c"][t] > 0))[0]):
            continue
        assert len(kept) == min(keep, int((ref["c"][t] > 0).sum()))
    assert f.get_error() == 0 and f.check_scratch() == 0
