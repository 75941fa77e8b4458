"""Single-token LoPA calls over 4-bit rows of less than 1024 codes: the fused kernel, whose act slots are longer than their two rows."""
import pytest
import torch

import synthetic_inputs as syn

DEV = "cuda:0"
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,H,r,s", [(256, 149, 32, 0.2), (256, 1027, 64, 0.9), (480, 3000, 96, 0.7), (512, 1500, 64, 0.9), (992, 777, 256, 0.5)])
def test_narrow_rows_take_one_launch(D, H, r, s):
    """Against the CUDA-core path, whose arithmetic is fp32 too (sums of up to 3000 terms in another order: 1e-5), and its fired set."""
    import paper_2609_31975_b200 as m

    w = syn.lopa_ffn_q4(D, H, r, 91, DEV, sparsity=s)
    gate = {"V": w["V"], "U": w["U"], "g_idx": m.g_diagonal(H, D, DEV)}
    x = syn.tokens(3, D, torch.bfloat16, 91, DEV)
    ffn = m.SparseFFN(D, H, torch.bfloat16, r_max=r, B_max=1)
    got = {}
    for path in ("general", "auto"):
        ffn.set_path(path)
        for t in (0, 1, 2, 0):
            n = ffn.launch_count()
            y = ffn.sparse_ffn_forward_q4(x[t], gate, w["b_g"], w["W_up"], w["W_down"], "sqrelu").clone()
            assert path == "general" or ffn.launch_count() - n == 1
            active = ffn.last_active()
            torch.cuda.synchronize()
            assert ffn.device_status() == 0, ffn.status_words()
            if path == "auto":
                if (path, t) in got:
                    assert torch.equal(y, got[path, t][0])
                want, fired = got["general", t]
                assert (y - want).norm() <= 1e-5 * want.norm()
                assert len(set(active.tolist()) ^ set(fired.tolist())) <= 1  # a neuron within rounding of zero
            got[path, t] = (y, active)


def test_the_fused_path_by_name_keeps_its_widths():
    import paper_2609_31975_b200 as m

    w = syn.lopa_ffn_q4(512, 300, 64, 91, DEV, sparsity=0.9)
    gate = {"V": w["V"], "U": w["U"], "g_idx": m.g_diagonal(300, 512, DEV)}
    ffn = m.SparseFFN(512, 300, torch.bfloat16, r_max=64, B_max=1)
    ffn.set_path("fused")
    with pytest.raises(m.SFFNError):
        ffn.sparse_ffn_forward_q4(syn.tokens(1, 512, torch.bfloat16, 91, DEV)[0], gate, w["b_g"], w["W_up"], w["W_down"], "relu")


@pytest.mark.parametrize("D,refused", [(256, True), (896, True), (928, False), (1024, False)])
def test_the_fused_path_by_name_ends_where_slots_are_longer_than_rows(D, refused):
    """One token and three, sparse and dense: the automatic choice takes all of them."""
    import paper_2609_31975_b200 as m

    w = syn.lopa_ffn_q4(D, 300, 64, 91, DEV, sparsity=0.9)
    gate = {"V": w["V"], "U": w["U"], "g_idx": m.g_diagonal(300, D, DEV)}
    ffn = m.SparseFFN(D, 300, torch.bfloat16, r_max=64, B_max=3)
    x = syn.tokens(3, D, torch.bfloat16, 91, DEV)
    for path in ("fused", "auto"):
        ffn.set_path(path)
        for call in (ffn.sparse_ffn_forward_q4, ffn.dense_ffn_forward_q4):
            for tokens in (x[0], x):
                args = (tokens, gate, w["b_g"], w["W_up"], w["W_down"], "relu")
                if refused and path == "fused":
                    with pytest.raises(m.SFFNError):
                        call(*args)
                else:
                    call(*args)
    torch.cuda.synchronize()
    assert ffn.device_status() == 0
