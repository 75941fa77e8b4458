"""Which single-token LoPA calls run in pairs of CTAs: the rule is host code."""
import pytest


def in_pairs(wkind, D, H, r, sms=148, at_once=-1):
    import paper_2609_31975_b200 as m

    return m.load_library().sffn_test_fused_pairs(wkind, D, H, r, sms, at_once)


@pytest.mark.parametrize("wkind,D,H,r", [(0, 3840, 14230, 480), (1, 8192, 24000, 1024)])
def test_all_pairs_of_a_call_have_to_fit_at_once(wkind, D, H, r):
    """The CTAs of a call wait for one another: one pair that gets no second SM would end the call in a timeout."""
    assert in_pairs(wkind, D, H, r, at_once=74) == 1
    assert in_pairs(wkind, D, H, r, at_once=73) == 0
    assert in_pairs(wkind, D, H, r, at_once=0) == 0
    assert in_pairs(wkind, D, H, r, sms=132, at_once=66) == 1
    assert in_pairs(wkind, D, H, r, sms=132, at_once=65) == 0
    assert in_pairs(wkind, D, H, r, sms=147, at_once=100) == 0  # an odd one out


@pytest.mark.parametrize("wkind,D,H,r,want", [
    (0, 4096, 14336, 512, 1), (0, 3840, 12000, 224, 1), (1, 8192, 28672, 1024, 1), (1, 7680, 15769, 448, 1),
    (0, 3836, 14336, 256, 0), (1, 7672, 24000, 448, 0),       # rows below 15 KB
    (0, 4096, 80 * 148, 512, 1), (0, 4096, 80 * 148 - 1, 512, 0), (1, 8192, 9000, 512, 0),  # CTAs of few neurons
    (0, 4096, 14336, 516, 0), (1, 8192, 28672, 1032, 0),      # a gate row longer than an eighth of a row
    (2, 8192, 28672, 512, 0), (3, 8192, 28672, 512, 0),       # codes
])
def test_calls_that_gain(wkind, D, H, r, want):
    """Calls whose CTAs have few fired neurons lose the microsecond that two SMs take longer to start together."""
    assert in_pairs(wkind, D, H, r, at_once=74) == want


@pytest.mark.gpu
def test_without_an_answer_a_call_goes_alone():
    import paper_2609_31975_b200 as m
    import synthetic_inputs as syn
    import torch

    D, H, r = 3840, 14230, 480
    w = syn.lopa_ffn(D, H, r, torch.float32, 90, "cuda:0", sparsity=0.95)
    gate = {"V": w["V"], "U": w["U"], "g_idx": m.g_diagonal(H, D, "cuda:0")}
    x = syn.tokens(1, D, torch.float32, 90, "cuda:0")[0]
    ffn = m.SparseFFN(D, H, torch.float32, r_max=r, B_max=1)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    y = []
    try:
        for fails in (1, 0, 1):
            m.test_set_knob("cluster_query_fails", fails)
            assert in_pairs(0, D, H, r, sms) == 1 - fails
            y.append(ffn.sparse_ffn_forward(x, gate, w["b_g"], w["W_up"], w["W_down"], "relu").clone())
            torch.cuda.synchronize()
            assert ffn.device_status() == 0
    finally:
        m.test_set_knob("cluster_query_fails", 0)
    assert torch.equal(y[0], y[2])
    assert (y[0] - y[1]).norm() <= 1e-5 * y[0].norm()  # sums of some 700 terms in another order


@pytest.mark.gpu
def test_dense_calls_go_alone():
    """Every row is done: nothing to even out between two CTAs."""
    import paper_2609_31975_b200 as m
    import synthetic_inputs as syn
    import torch

    D, H, r = 3840, 12000, 256
    w = syn.lopa_ffn(D, H, r, torch.float32, 99, "cuda:0")
    gate = {"V": w["V"], "U": w["U"], "g_idx": m.g_diagonal(H, D, "cuda:0")}
    x = syn.tokens(1, D, torch.float32, 99, "cuda:0")[0]
    ffn = m.SparseFFN(D, H, torch.float32, r_max=r, B_max=1)
    assert in_pairs(0, D, H, r, torch.cuda.get_device_properties(0).multi_processor_count)
    y = {}
    try:
        for knob in (-1, 0, 1):
            m.test_set_knob("pairs", knob)
            y[knob] = ffn.dense_ffn_forward(x, gate, w["b_g"], w["W_up"], w["W_down"], "relu").clone()
    finally:
        m.test_set_knob("pairs", -1)
    torch.cuda.synchronize()
    assert ffn.device_status() == 0
    assert torch.equal(y[-1], y[0]) and not torch.equal(y[1], y[0])  # sums of 12000 rows in another order
    assert (y[1] - y[0]).norm() <= 1e-5 * y[0].norm()
