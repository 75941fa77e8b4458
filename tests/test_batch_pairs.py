"""Batched gate and up GEMMs in pairs of CTAs: the gates, options and lists that they meet, against the formulas in 64 bits."""
import pytest
import torch

import synthetic_inputs as syn

DEV = "cuda:0"
pytestmark = pytest.mark.gpu


def pairs(R, K, qbits, B, cols):
    import paper_2609_31975_b200 as m

    return m.load_library().sffn_test_umma_pairs(R, K, qbits, B, cols, torch.cuda.get_device_properties(0).multi_processor_count)


def wide(w):
    return w["q"].double() * w["s"].double()[:, None] if isinstance(w, dict) else w.double()


def act64(name, z):
    p = z.clamp(min=0)
    return {None: z, "relu": p, "sqrelu": p * p, "rsplus": p * torch.sigmoid(p), "silu": z * torch.sigmoid(z)}[name]


def reference(x, gate, b_g, W_up, W_down, act, act_up=None):
    """y, and z for the list of fired neurons."""
    x = x.double()
    if "V" in gate:
        v = x @ wide(gate["V"]).T
        z = v / torch.sqrt((v * v).mean(dim=1, keepdim=True) + 1e-5) @ wide(gate["U"]).T
        sign = gate["g_sign"].double() if "g_sign" in gate else 1.0
        z = z + sign * x[:, gate["g_idx"].long()]
    else:
        z = x @ wide(gate["W_g"]).T
    z = z + b_g.double()
    return (act64(act, z) * act64(act_up, x @ wide(W_up).T)) @ wide(W_down), z


def check(ffn, y, want, z, fired=True):
    """h is bf16 for the down projection: 1.7e-3 over a token, some of the largest sums 4e-2."""
    torch.cuda.synchronize()
    assert ffn.device_status() == 0
    y = y.double()
    assert ((y - want).norm(dim=1) / want.norm(dim=1)).max().item() < 7e-3
    assert ((y - want).abs().amax(dim=1) / want.pow(2).mean(dim=1).sqrt()).max().item() < 4e-2
    if fired:
        got = torch.zeros(z.shape[1], dtype=torch.bool, device=DEV)
        got[ffn.last_active().long()] = True
        unsure = (z.abs() < 1e-3).any(dim=0)
        assert torch.equal(got | unsure, (z > 0).any(dim=0) | unsure)


@pytest.mark.parametrize("act,act_up", [("relu", None), ("sqrelu", "relu"), ("rsplus", "silu")])
@pytest.mark.parametrize("qbits,H,B", [(0, 6001, 128), (0, 18001, 112), (0, 18001, 101), (8, 6001, 64), (8, 18001, 45)])
def test_low_parameter_gates_with_signs(qbits, H, B, act, act_up):
    """Two bf16 terms a token, or four limbs, in the columns that the two CTAs share out; 112 and 101 tokens leave the up GEMM alone."""
    import paper_2609_31975_b200 as m

    D, r = 256, 128
    w = (syn.lopa_ffn_q8(D, H, r, 93, DEV, sparsity=0.9) if qbits else syn.lopa_ffn(D, H, r, torch.bfloat16, 93, DEV, sparsity=0.9))
    assert pairs(H, r, 1 if qbits else 0, B, 4 * B if qbits else 2 * ((B + 7) // 8 * 8))
    sign = torch.where(torch.arange(H, device=DEV) % 3 == 0, -1, 1).to(torch.int8)
    gate = {"V": w["V"], "U": w["U"], "g_idx": m.g_diagonal(H, D, DEV), "g_sign": sign}
    x = syn.tokens(B, D, torch.bfloat16, 93, DEV)
    ffn = m.SparseFFN(D, H, torch.bfloat16, r_max=r, B_max=B)
    ffn.set_up_activation(act_up)
    args = (x, gate, w["b_g"], w["W_up"], w["W_down"], act)
    y = (ffn.sparse_ffn_forward_q8 if qbits else ffn.sparse_ffn_forward)(*args)
    check(ffn, y, *reference(*args, act_up))


@pytest.mark.parametrize("act,act_up", [("sqrelu", "relu"), ("rsplus", "silu")])
@pytest.mark.parametrize("qbits,H,B,s", [(0, 6001, 250, 0.9), (0, 18001, 200, 0.97), (8, 6001, 63, 0.9), (8, 18001, 48, 0.97)])
def test_a_second_activation(qbits, H, B, s, act, act_up):
    """Every row walked, and a list of some."""
    import paper_2609_31975_b200 as m

    D = 256
    w = syn.standard_ffn_q8(D, H, 94, DEV, sparsity=s) if qbits else syn.standard_ffn(D, H, torch.bfloat16, 94, DEV, sparsity=s)
    if s > 0.95:
        w["b_g"][: H // 2] -= 10.0  # half of the neurons never fire
    assert pairs(H, D, 1 if qbits else 0, B, 4 * B if qbits else B)
    x = syn.tokens(B, D, torch.bfloat16, 94, DEV)
    ffn = m.SparseFFN(D, H, torch.bfloat16, B_max=B)
    ffn.set_up_activation(act_up)
    args = (x, {"W_g": w["W_g"]}, w["b_g"], w["W_up"], w["W_down"], act)
    y = (ffn.sparse_ffn_forward_q8 if qbits else ffn.sparse_ffn_forward)(*args)
    check(ffn, y, *reference(*args, act_up))


@pytest.mark.parametrize("qbits,H,B", [(0, 6001, 250), (8, 18001, 61)])
def test_the_dense_comparator(qbits, H, B):
    """Its gate in pairs, its up GEMM, which has no list to look at, alone."""
    import paper_2609_31975_b200 as m

    D = 256
    w = syn.standard_ffn_q8(D, H, 95, DEV) if qbits else syn.standard_ffn(D, H, torch.bfloat16, 95, DEV)
    assert pairs(H, D, 1 if qbits else 0, B, 4 * B if qbits else B)
    x = syn.tokens(B, D, torch.bfloat16, 95, DEV)
    ffn = m.SparseFFN(D, H, torch.bfloat16, B_max=B)
    args = (x, {"W_g": w["W_g"]}, w["b_g"], w["W_up"], w["W_down"], "sqrelu")
    y = (ffn.dense_ffn_forward_q8 if qbits else ffn.dense_ffn_forward)(*args)
    check(ffn, y, *reference(*args), fired=False)


@pytest.mark.parametrize("s", [0.9, 0.99])
def test_more_tiles_than_the_list_in_the_kernel_takes(s):
    """Byte flags from a gate in pairs, and a launch that compacts them."""
    import ctypes

    import paper_2609_31975_b200 as m

    D, H, B = 256, 50001, 200
    tr, nt, own = ctypes.c_int(), ctypes.c_int(), ctypes.c_int()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    m.load_library().sffn_test_umma_pass_tiling(H, D, 0, B, sms, ctypes.byref(tr), ctypes.byref(nt), ctypes.byref(own))
    assert not own.value and pairs(H, D, 0, B, B)
    w = syn.standard_ffn(D, H, torch.bfloat16, 96, DEV, sparsity=s)
    if s > 0.95:
        w["b_g"][: H // 2] -= 10.0  # a list of fewer than 70 % of the rows
    x = syn.tokens(B, D, torch.bfloat16, 96, DEV)
    ffn = m.SparseFFN(D, H, torch.bfloat16, B_max=B)
    args = (x, {"W_g": w["W_g"]}, w["b_g"], w["W_up"], w["W_down"], "relu")
    check(ffn, ffn.sparse_ffn_forward(*args), *reference(*args))
