"""The batched down projection: splits of the list that are a cluster and add their sums up themselves, and splits that are not."""
import pytest
import torch

import synthetic_inputs as syn
from parity import assert_y_close, run_oracle

DEV = "cuda:0"


@pytest.mark.gpu
@pytest.mark.parametrize("D,H,B,s", [
    (512, 700, 2, 0.9),       # clusters of eight, most splits of the list empty
    (512, 700, 33, 0.9),
    (256, 300, 256, 0.9),     # few blocks, whose ring is smaller than the sums
    (4096, 1200, 200, 0.9),   # a CTA alone on its SM, clusters of four
    (8192, 1200, 9, 0.7),
    (8192, 900, 70, 0.9),     # pairs of CTAs
    (14336, 400, 130, 0.7),   # one CTA for a tile
    (3072, 9000, 5, 0.5),     # partials: more splits than clusters
    (640, 1200, 17, 0.8),     # exact sums in clusters
    (2688, 6000, 20, 0.5),    # and in partials
])
def test_splits_of_the_list_add_up(D, H, B, s):
    """bf16 rows against the oracle, and the same bits again."""
    import paper_2609_31975_b200 as m

    w = syn.standard_ffn(D, H, torch.bfloat16, 85, DEV, sparsity=s)
    ffn = m.SparseFFN(D, H, torch.bfloat16, B_max=B)
    x = syn.tokens(B, D, torch.bfloat16, 85, DEV)
    args = (x, {"W_g": w["W_g"]}, w["b_g"], w["W_up"], w["W_down"], "relu")
    y = ffn.sparse_ffn_forward(*args).clone()
    again = ffn.sparse_ffn_forward(*args)
    torch.cuda.synchronize()
    assert ffn.device_status() == 0
    assert torch.equal(y, again)
    ref = run_oracle(x, args[1], w["b_g"], w["W_up"], w["W_down"], "relu", threads=16)
    assert_y_close(y, ref["y"], what=f"{D}x{H} B={B}")


@pytest.mark.gpu
@pytest.mark.parametrize("qbits", [8, 4])
@pytest.mark.parametrize("D,H,B", [(512, 700, 33), (4096, 600, 200), (640, 600, 200), (640, 600, 24), (8192, 1200, 64), (3072, 9000, 40)])
def test_splits_of_codes_add_up(D, H, B, qbits):
    """Against the single-token calls (a bf16 h in the batch where D is a multiple of 256: 1e-2)."""
    import paper_2609_31975_b200 as m

    w = (syn.standard_ffn_q8 if qbits == 8 else syn.standard_ffn_q4)(D, H, 86, DEV, sparsity=0.7)
    ffn = m.SparseFFN(D, H, torch.bfloat16, B_max=B)
    x = syn.tokens(B, D, torch.bfloat16, 86, DEV)
    call = ffn.sparse_ffn_forward_q8 if qbits == 8 else ffn.sparse_ffn_forward_q4
    args = ({"W_g": w["W_g"]}, w["b_g"], w["W_up"], w["W_down"], "relu")
    y = call(x, *args)
    one = torch.stack([call(x[b], *args) for b in range(B)])
    torch.cuda.synchronize()
    assert ffn.device_status() == 0
    assert ((y - one).norm(dim=1) / one.norm(dim=1)).max().item() < 1e-2


@pytest.mark.gpu
@pytest.mark.parametrize("D,B", [(512, 5), (4096, 200), (640, 20)])
def test_nothing_fires(D, B):
    import paper_2609_31975_b200 as m

    w = syn.standard_ffn(D, 700, torch.bfloat16, 87, DEV, sparsity=0.9)
    ffn = m.SparseFFN(D, 700, torch.bfloat16, B_max=B)
    y = ffn.sparse_ffn_forward(syn.tokens(B, D, torch.bfloat16, 87, DEV), {"W_g": w["W_g"]}, w["b_g"] - 100.0, w["W_up"], w["W_down"], "relu")
    torch.cuda.synchronize()
    assert ffn.device_status() == 0 and not y.any() and len(ffn.last_active()) == 0
