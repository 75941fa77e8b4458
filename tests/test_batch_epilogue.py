"""Epilogues of the batched gate and up GEMMs: steps of eight (codes: four) tokens over one or three warps."""
import pytest
import torch

import synthetic_inputs as syn
from parity import assert_active_set, assert_y_close, run_oracle

DEV = "cuda:0"


@pytest.mark.gpu
@pytest.mark.parametrize("lopa", [False, True])
@pytest.mark.parametrize("act,act_up", [("relu", None), ("sqrelu", "relu"), ("rsplus", "silu")])
@pytest.mark.parametrize("B", [2, 7, 9, 17, 33, 57, 133])  # one token past a step, a warp's last step short, no third warp's step
def test_tokens_of_short_and_full_steps(B, act, act_up, lopa):
    """bf16 rows against the oracle; 603 rows leave a ragged last tile."""
    import paper_2609_31975_b200 as m

    D, H, r = 512, 603, 64
    w = syn.lopa_ffn(D, H, r, torch.bfloat16, 81, DEV, sparsity=0.7) if lopa else syn.standard_ffn(D, H, torch.bfloat16, 81, DEV, sparsity=0.7)
    sign = torch.where(torch.arange(H, device=DEV) % 3 == 0, -1, 1).to(torch.int8)
    gate = {"V": w["V"], "U": w["U"], "g_idx": m.g_diagonal(H, D, DEV), "g_sign": sign} if lopa else {"W_g": w["W_g"]}
    x = syn.tokens(B, D, torch.bfloat16, 81, DEV)
    ffn = m.SparseFFN(D, H, torch.bfloat16, r_max=r if lopa else 0, B_max=B)
    ffn.set_up_activation(act_up)
    y = ffn.sparse_ffn_forward(x, gate, w["b_g"], w["W_up"], w["W_down"], act)
    torch.cuda.synchronize()
    assert ffn.device_status() == 0
    ref = run_oracle(x, gate, w["b_g"], w["W_up"], w["W_down"], act, act_up=act_up)
    assert_y_close(y, ref["y"], what=f"B={B} {act} {act_up}")
    assert_active_set(ffn.last_active(), ref, what=f"B={B} {act} {act_up}")


@pytest.mark.gpu
@pytest.mark.parametrize("qbits", [8, 4])
@pytest.mark.parametrize("D", [512, 640])  # against limbs; codes expanded to bf16, h in two terms
@pytest.mark.parametrize("B", [5, 13, 23, 37, 64])
def test_tokens_of_short_and_full_steps_of_codes(B, D, qbits):
    """Against the single-token calls (a bf16 h in the batch where D is a multiple of 256: 1e-2)."""
    import paper_2609_31975_b200 as m

    H = 603
    w = (syn.standard_ffn_q8 if qbits == 8 else syn.standard_ffn_q4)(D, H, 82, DEV, sparsity=0.6)
    ffn = m.SparseFFN(D, H, torch.bfloat16, B_max=B)
    ffn.set_up_activation("silu")
    x = syn.tokens(B, D, torch.bfloat16, 82, DEV)
    call = ffn.sparse_ffn_forward_q8 if qbits == 8 else ffn.sparse_ffn_forward_q4
    args = ({"W_g": w["W_g"]}, w["b_g"], w["W_up"], w["W_down"], "rsplus")
    y = call(x, *args)
    one = torch.stack([call(x[b], *args) for b in range(B)])
    torch.cuda.synchronize()
    assert ffn.device_status() == 0
    assert ((y - one).norm(dim=1) / one.norm(dim=1)).max().item() < 1e-2
