"""Epilogues of the batched gate and up GEMMs: steps of eight (codes: four) tokens over one or three warps."""
import pytest
import torch

import synthetic_inputs as syn
from parity import assert_active_set, assert_y_close, run_oracle

DEV = "cuda:0"


def in_pairs(R, K, qbits, B, cols):
    """Whether a gate over R rows of K columns, or an up projection of 32 tokens and more, runs in pairs of CTAs (qbits 1: int8 codes
    against limbs)."""
    import paper_2609_31975_b200 as m

    return m.load_library().sffn_test_umma_pairs(R, K, qbits, B, cols, torch.cuda.get_device_properties(0).multi_processor_count)


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
    """Against the single-token calls: a bf16 h in the batch where D is a multiple of 256, 1e-2; else h has 16 bits, and the single
    tokens' two limbs are what is left, some 1e-4 (the second term of h lost: 1.1e-3)."""
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
    assert ((y - one).norm(dim=1) / one.norm(dim=1)).max().item() < (1e-2 if D % 256 == 0 else 4e-4)


@pytest.mark.gpu
@pytest.mark.parametrize("qbits,D,H,B,s", [
    (0, 256, 6001, 250, 0.5),    # pairs of CTAs; every row walked, a ragged last tile
    (0, 256, 6001, 250, 0.999),  # the union listed, in tiles of eight rows or so
    (0, 256, 28003, 200, 0.9),   # 219 tiles: the last pair has one
    (0, 256, 28003, 180, 0.999),
    (0, 1280, 24001, 256, 0.9),  # two tiles for each CTA of a pair
    (8, 256, 6001, 64, 0.5),
    (8, 256, 6001, 61, 0.97),    # 244 limbs in 256 columns
    (8, 256, 28003, 45, 0.9),    # 180 limbs in 192
    (8, 1280, 24001, 57, 0.97),
])
def test_pairs_of_ctas_share_the_token_rows(qbits, D, H, B, s):
    """Two calls of one handle, the second on other tokens.  bf16 rows against the oracle, codes against the single-token calls (a
    bf16 h in the batch: 1e-2)."""
    import paper_2609_31975_b200 as m

    assert in_pairs(H, D, 1 if qbits else 0, B, 4 * B if qbits else B)
    w = syn.standard_ffn_q8(D, H, 83, DEV, sparsity=s) if qbits else syn.standard_ffn(D, H, torch.bfloat16, 83, DEV, sparsity=s)
    ffn = m.SparseFFN(D, H, torch.bfloat16, B_max=B)
    call = ffn.sparse_ffn_forward_q8 if qbits else ffn.sparse_ffn_forward
    args = ({"W_g": w["W_g"]}, w["b_g"], w["W_up"], w["W_down"], "relu")
    xs = syn.tokens(2 * B, D, torch.bfloat16, 83, DEV)
    for x in (xs[:B], xs[B:]):
        y = call(x, *args)
        torch.cuda.synchronize()
        assert ffn.device_status() == 0
        if qbits:
            one = torch.stack([call(x[b], *args) for b in range(B)])
            torch.cuda.synchronize()
            assert ((y - one).norm(dim=1) / one.norm(dim=1).clamp(min=1e-3)).max().item() < 1e-2
        else:
            ref = run_oracle(x, args[0], w["b_g"], w["W_up"], w["W_down"], "relu", threads=16)
            active = ffn.last_active()
            assert_y_close(y, ref["y"], what=f"{D}x{H} B={B}")
            assert_active_set(active, ref, what=f"{D}x{H} B={B}")


@pytest.mark.gpu
def test_a_copy_that_never_comes_ends_both_ctas_of_a_pair():
    """A wait that runs out in the even CTA, whose barrier the copies of both complete on: a status, and the next call is right."""
    import paper_2609_31975_b200 as m
    from paper_2609_31975_b200 import binding

    D, H, B = 256, 6001, 250
    assert in_pairs(H, D, 0, B, B)
    w = syn.standard_ffn(D, H, torch.bfloat16, 84, DEV, sparsity=0.9)
    ffn = m.SparseFFN(D, H, torch.bfloat16, B_max=B)
    args = (syn.tokens(B, D, torch.bfloat16, 84, DEV), {"W_g": w["W_g"]}, w["b_g"], w["W_up"], w["W_down"], "relu")
    want = ffn.sparse_ffn_forward(*args).clone()
    torch.cuda.synchronize()
    try:
        binding.test_set_knob("wait_cycles", 20_000_000)
        binding.test_set_knob("drop_stage", 1)
        ffn.sparse_ffn_forward(*args)
        torch.cuda.synchronize()
        assert ffn.device_status() == 5
    finally:
        binding.test_set_knob("drop_stage", -1)
        binding.test_set_knob("wait_cycles", 0)
    ffn.reset()
    got = ffn.sparse_ffn_forward(*args)
    torch.cuda.synchronize()
    assert ffn.device_status() == 0
    assert torch.equal(got, want)
