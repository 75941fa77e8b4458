"""Single-token LoPA calls whose CTAs share out the rows of fired neurons in pairs, at sizes that are quick to check."""
import pytest
import torch

import synthetic_inputs as syn
from parity import assert_active_set, assert_y_close, run_oracle

DEV = "cuda:0"
pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def in_pairs():
    import paper_2609_31975_b200 as m

    m.test_set_knob("pairs", 1)  # (by their sizes these calls would go alone: too few neurons a CTA)
    yield lambda D, H, r, dtype: m.load_library().sffn_test_fused_pairs(
        0 if dtype == torch.float32 else 1, D, H, r, torch.cuda.get_device_properties(0).multi_processor_count, -1)
    m.test_set_knob("pairs", -1)


def make(m, D, H, r, dtype, s):
    w = syn.lopa_ffn(D, H, r, dtype, 88, DEV, sparsity=s)
    return {"V": w["V"], "U": w["U"], "g_idx": m.g_diagonal(H, D, DEV)}, w


@pytest.mark.parametrize("D,H,r,dtype,s", [
    (3840, 1531, 480, torch.float32, 0.9),    # slabs of unequal length
    (3840, 300, 480, torch.float32, 0.5),     # two rows a CTA, CTAs without rows
    (3840, 149, 64, torch.float32, 0.05),
    (4096, 5003, 512, torch.float32, 0.97),
    (4096, 5003, 512, torch.float32, 0.2),    # many rows a CTA: the rings wrap
    (8192, 3001, 1024, torch.bfloat16, 0.8),
])
def test_pairs_share_the_fired_rows(D, H, r, dtype, s, in_pairs):
    import paper_2609_31975_b200 as m

    assert in_pairs(D, H, r, dtype)

    gate, w = make(m, D, H, r, dtype, s)
    ffn = m.SparseFFN(D, H, dtype, r_max=r, B_max=1)
    x = syn.tokens(3, D, dtype, 88, DEV)
    ys = []
    for t in (0, 1, 2, 0):
        ys.append(ffn.sparse_ffn_forward(x[t], gate, w["b_g"], w["W_up"], w["W_down"], "relu").clone())
        active = ffn.last_active()
        torch.cuda.synchronize()
        assert ffn.device_status() == 0, ffn.status_words()
        ref = run_oracle(x[t:t + 1], gate, w["b_g"], w["W_up"], w["W_down"], "relu")
        tol = 1e-5 if dtype == torch.float32 else 1e-2  # fp32: sums of up to 5000 terms, in another order
        assert_y_close(ys[-1], ref["y"][0], rel_l2=tol, max_abs=2 * tol, what=f"{D}x{H} r={r} token {t}")
        assert_active_set(active, ref, what=f"{D}x{H} r={r} token {t}")
    assert torch.equal(ys[0], ys[3])


def test_pairs_do_every_row_of_a_dense_call_once(in_pairs):
    import paper_2609_31975_b200 as m

    assert in_pairs(3840, 700, 480, torch.float32)

    gate, w = make(m, 3840, 700, 480, torch.float32, None)
    ffn = m.SparseFFN(3840, 700, torch.float32, r_max=480, B_max=1)
    x = syn.tokens(1, 3840, torch.float32, 88, DEV)[0]
    hi = torch.full((700,), 1e3, device=DEV)
    y = ffn.sparse_ffn_forward(x, gate, hi, w["W_up"], w["W_down"], "relu").clone()
    assert torch.equal(y, ffn.dense_ffn_forward(x, gate, hi, w["W_up"], w["W_down"], "relu"))  # same rows, same order
    torch.cuda.synchronize()
    assert ffn.device_status() == 0


@pytest.mark.parametrize("knob,value", [("skip_arrival_cta", 3), ("wait_cycles", 2000), ("wait_cycles", 20000)])
def test_pairs_end_together_when_a_wait_runs_out(knob, value, in_pairs):
    """A CTA that never hands in its sums, and budgets that run out in the middle of the call: a status, and a good call after a
    reset."""
    import paper_2609_31975_b200 as m

    assert in_pairs(3840, 1531, 480, torch.float32)

    gate, w = make(m, 3840, 1531, 480, torch.float32, 0.9)
    ffn = m.SparseFFN(3840, 1531, torch.float32, r_max=480, B_max=1)
    x = syn.tokens(1, 3840, torch.float32, 88, DEV)[0]
    args = (x, gate, w["b_g"], w["W_up"], w["W_down"], "relu")
    want = ffn.sparse_ffn_forward(*args).clone()
    torch.cuda.synchronize()
    try:
        m.test_set_knob("wait_cycles", 20_000_000)
        m.test_set_knob(knob, value)
        ffn.sparse_ffn_forward(*args)
        torch.cuda.synchronize()
        assert ffn.device_status() in ((5,) if knob == "skip_arrival_cta" else (0, 5))
    finally:
        m.test_set_knob("skip_arrival_cta", -1)
        m.test_set_knob("wait_cycles", 0)
    ffn.reset()
    got = ffn.sparse_ffn_forward(*args)
    torch.cuda.synchronize()
    assert ffn.device_status() == 0
    assert torch.equal(got, want)


@pytest.mark.parametrize("dtype,D,H,r", [(torch.float32, 3840, 1531, 480), (torch.bfloat16, 8192, 1001, 512)])
@pytest.mark.parametrize("options", ["sign", "gain", "no norm", "no fixed matrix"])
def test_pairs_take_every_option_of_the_gate(dtype, D, H, r, options, in_pairs):
    import paper_2609_31975_b200 as m

    assert in_pairs(D, H, r, dtype)
    gate, w = make(m, D, H, r, dtype, 0.8)
    if options == "sign":
        gate["g_sign"] = torch.where(torch.arange(H, device=DEV) % 3 == 0, -1, 1).to(torch.int8)
    elif options == "gain":
        gate["rms_gain"] = 0.5 + torch.rand(r, generator=torch.Generator(device=DEV).manual_seed(5), device=DEV)
    elif options == "no norm":
        gate["use_rmsnorm"] = False
    else:
        del gate["g_idx"]
    x = syn.tokens(1, D, dtype, 97, DEV)
    ffn = m.SparseFFN(D, H, dtype, r_max=r, B_max=1)
    y = ffn.sparse_ffn_forward(x[0], gate, w["b_g"], w["W_up"], w["W_down"], "sqrelu")
    active = ffn.last_active()
    torch.cuda.synchronize()
    assert ffn.device_status() == 0, ffn.status_words()
    ref = run_oracle(x, gate, w["b_g"], w["W_up"], w["W_down"], "sqrelu")
    assert_y_close(y, ref["y"][0], rel_l2=1e-5, max_abs=2e-5, what=f"{D}x{H} {options}")  # fp32 sums of up to 1500 terms
    assert_active_set(active, ref, what=f"{D}x{H} {options}")


def test_pairs_token_by_token_leave_the_union_of_the_batch(in_pairs):
    """A batch of fp32 tokens is as many calls: each the bits of a call of its own, the flags those of any."""
    import paper_2609_31975_b200 as m

    D, H, r, B = 3840, 1531, 480, 3
    assert in_pairs(D, H, r, torch.float32)
    gate, w = make(m, D, H, r, torch.float32, 0.9)
    x = syn.tokens(B, D, torch.float32, 98, DEV)
    ffn = m.SparseFFN(D, H, torch.float32, r_max=r, B_max=B)
    args = (gate, w["b_g"], w["W_up"], w["W_down"], "relu")
    y = ffn.sparse_ffn_forward(x, *args).clone()
    union = set(ffn.last_active().tolist())
    fired = set()
    for b in range(B):
        assert torch.equal(ffn.sparse_ffn_forward(x[b], *args), y[b])
        fired |= set(ffn.last_active().tolist())
    torch.cuda.synchronize()
    assert ffn.device_status() == 0
    assert union == fired
