"""The batched down projection: splits of the list that are a cluster and add their sums up themselves, and splits that are not."""
import ctypes

import pytest
import torch

import synthetic_inputs as syn
from parity import assert_y_close, run_oracle

DEV = "cuda:0"


def splits(D, H, qbits, cols, exact):
    """CTAs of a cluster, or 0: partials, which a launch of their own adds up."""
    import paper_2609_31975_b200 as m

    n = ctypes.c_int()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return n.value if m.load_library().sffn_test_umma_down_splits(D, H, qbits, cols, exact, sms, 16, None, ctypes.byref(n)) else 0


@pytest.mark.gpu
@pytest.mark.parametrize("D,H,B,s,cluster", [  # cluster: CTAs of one, 0 = partials, None = what the device's GPCs have room for
    (512, 700, 2, 0.9, 8),         # most splits of the list empty
    (512, 700, 33, 0.9, 8),
    (256, 300, 256, 0.9, 8),       # few blocks, whose ring is smaller than the sums
    (4096, 1200, 200, 0.9, None),  # a CTA alone on its SM, clusters of four
    (8192, 1200, 9, 0.7, None),
    (8192, 900, 70, 0.9, 2),
    (14336, 400, 130, 0.7, 1),     # one CTA for a tile
    (3072, 9000, 5, 0.5, 0),       # more splits than a cluster has CTAs
    (640, 1200, 17, 0.8, 8),       # exact sums
    (2688, 6000, 20, 0.5, None),   # exact sums, partials
])
def test_splits_of_the_list_add_up(D, H, B, s, cluster):
    """bf16 rows against the oracle, and the same bits again."""
    import paper_2609_31975_b200 as m

    w = syn.standard_ffn(D, H, torch.bfloat16, 85, DEV, sparsity=s)
    ffn = m.SparseFFN(D, H, torch.bfloat16, B_max=B)
    x = syn.tokens(B, D, torch.bfloat16, 85, DEV)
    args = (x, {"W_g": w["W_g"]}, w["b_g"], w["W_up"], w["W_down"], "relu")
    cols = (B + 7) // 8 * 8
    route = splits(D, H, 0, cols * (1 if D % 256 == 0 else 3), D % 256 != 0)
    assert cluster is None or route == cluster
    n = ffn.launch_count()
    y = ffn.sparse_ffn_forward(*args).clone()
    assert ffn.launch_count() - n == (3 if route else 4)  # gate, up, down, and the partials' sum
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
    """Against the single-token calls: a bf16 h in the batch where D is a multiple of 256, 1e-2; else h has 16 bits, and the single
    tokens' two limbs are what is left, some 1e-4 (the second term of h lost: 1.1e-3)."""
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
    assert ((y - one).norm(dim=1) / one.norm(dim=1)).max().item() < (1e-2 if D % 256 == 0 else 4e-4)


@pytest.mark.gpu
@pytest.mark.parametrize("D,B", [(512, 5), (4096, 200), (640, 20)])
def test_nothing_fires(D, B):
    import paper_2609_31975_b200 as m

    w = syn.standard_ffn(D, 700, torch.bfloat16, 87, DEV, sparsity=0.9)
    ffn = m.SparseFFN(D, 700, torch.bfloat16, B_max=B)
    y = ffn.sparse_ffn_forward(syn.tokens(B, D, torch.bfloat16, 87, DEV), {"W_g": w["W_g"]}, w["b_g"] - 100.0, w["W_up"], w["W_down"], "relu")
    torch.cuda.synchronize()
    assert ffn.device_status() == 0 and not y.any() and len(ffn.last_active()) == 0


@pytest.mark.gpu
def test_batches_of_two_streams_share_sms():
    """Clusters of two calls whose CTAs fit an SM together but for the tensor memory of one that has it all: each as if alone."""
    import paper_2609_31975_b200 as m

    calls, want = [], []
    for D, H, B in ((256, 300, 200), (512, 700, 33), (256, 500, 256), (512, 300, 16)):
        w = syn.standard_ffn(D, H, torch.bfloat16, 88, DEV, sparsity=0.8)
        ffn = m.SparseFFN(D, H, torch.bfloat16, B_max=B)
        x = syn.tokens(B, D, torch.bfloat16, 88, DEV)
        y = torch.empty(B, D, dtype=torch.float32, device=DEV)
        calls.append((ffn, (x, {"W_g": w["W_g"]}, w["b_g"], w["W_up"], w["W_down"], "relu", y)))
        want.append(ffn.sparse_ffn_forward(*calls[-1][1]).clone())
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in calls]
    for _ in range(200):
        for (ffn, args), stream in zip(calls, streams):
            ffn.sparse_ffn_forward(*args, stream=stream)
    torch.cuda.synchronize()
    for (ffn, args), y in zip(calls, want):
        assert ffn.device_status() == 0
        assert torch.equal(args[-1], y)
