"""How the batched down projection splits the list of fired neurons: the rule is host code."""
import ctypes

import pytest


def splits(D, R, qbits, cols, at_once, exact=0, sms=148, most=16):
    """(clustered, splits) on a device that runs at_once(n) clusters of n CTAs at once (None: the current one)."""
    import paper_2609_31975_b200 as m

    fit = (ctypes.c_int * 9)(*([0] + [at_once(n) for n in range(1, 9)])) if at_once else None
    n = ctypes.c_int()
    return m.load_library().sffn_test_umma_down_splits(D, R, qbits, cols, exact, sms, most, fit, ctypes.byref(n)), n.value


def plenty(n):
    return 296 // n


@pytest.mark.parametrize("qbits", [0, 8, 4])
def test_a_cluster_for_every_tile_or_partials(qbits):
    for D, R in ((512, 1500), (4096, 14336), (8192, 24000), (640, 600)):
        for cols in (8, 64, 72, 200):
            clustered, n = splits(D, R, qbits, cols, plenty)
            assert 1 <= n <= (8 if clustered else 16)
            if clustered:
                assert n == 1 or plenty(n) >= D // 128
            else:
                assert n * (D // 128) <= (296 if cols <= 64 else 148) or n == 1


def test_without_an_answer_the_list_is_cut_into_partials():
    """No cluster fits, or the runtime could not tell: as many splits as without clusters, short lists too."""
    for D, R in ((512, 700), (1024, 3000), (4096, 14336), (8192, 24000)):
        for cols in (8, 64, 200):
            clustered, n = splits(D, R, 0, cols, lambda size: 0)
            want = min(16, (2 if cols <= 64 else 1) * 148 // (D // 128))
            assert n == want and clustered == (want == 1)


@pytest.mark.parametrize("D,R,qbits,cols,exact,clustered", [
    (1024, 64 * 64, 0, 24, 0, 1), (1024, 64 * 64 + 1, 0, 24, 0, 0),   # eight blocks a CTA
    (1024, 64 * 64 + 1, 0, 8, 0, 1), (1024, 96 * 64, 0, 8, 0, 1), (1024, 96 * 64 + 1, 0, 8, 0, 0),
    (1024, 96 * 64, 8, 64, 0, 1), (1024, 96 * 64, 4, 64, 0, 1), (1024, 96 * 64 + 1, 4, 64, 0, 0),
    (640, 48 * 64, 0, 72, 1, 1), (640, 48 * 64 + 1, 0, 72, 1, 0),     # exact sums
    (640, 24 * 64, 0, 96, 1, 1), (640, 24 * 64 + 1, 0, 96, 1, 0),
    (5504, 16512, 0, 24, 1, 0), (5504, 16512, 8, 120, 1, 0), (16512, 200, 0, 120, 1, 1),
])
def test_clusters_for_lists_of_few_blocks(D, R, qbits, cols, exact, clustered):
    """Narrow rows, whose tiles leave room for more splits than a cluster has."""
    assert splits(D, R, qbits, cols, plenty, exact)[0] == clustered


@pytest.mark.parametrize("tiles,cols,size,most,clustered", [
    (42, 100, 3, 45, 1), (43, 100, 3, 45, 0), (45, 100, 3, 45, 0), (45, 100, 3, 48, 1),
    (52, 24, 5, 56, 1), (54, 24, 5, 56, 0), (56, 24, 5, 56, 0),
    (32, 100, 4, 33, 1), (32, 24, 8, 33, 1), (33, 100, 4, 33, 1),
])
def test_odd_clusters_need_room_to_spare(tiles, cols, size, most, clustered):
    """As many clusters of an even size as the device takes, of an odd one 15 for every 16."""
    got = splits(128 * tiles, 30000, 0, cols, lambda n: most if n == size else 0 if n > size else 296 // n)
    assert got[0] == clustered
    if clustered:
        assert got[1] == size


@pytest.mark.gpu
def test_a_question_that_failed_is_asked_again():
    """Partials and the kernel that adds them up while the runtime has no answer, one launch less once it has."""
    import paper_2609_31975_b200 as m
    import synthetic_inputs as syn
    import torch

    D, H, B = 512, 1500, 16
    w = syn.standard_ffn(D, H, torch.bfloat16, 92, "cuda:0", sparsity=0.8)
    ffn = m.SparseFFN(D, H, torch.bfloat16, B_max=B)
    x = syn.tokens(B, D, torch.bfloat16, 92, "cuda:0")
    launches, y = [], []
    try:
        for fails in (1, 0, 1, 0):
            m.test_set_knob("cluster_query_fails", fails)
            assert splits(D, H, 0, B, None) == ((0, 16) if fails else (1, 8))
            n = ffn.launch_count()
            y.append(ffn.sparse_ffn_forward(x, {"W_g": w["W_g"]}, w["b_g"], w["W_up"], w["W_down"], "relu").clone())
            launches.append(ffn.launch_count() - n)
    finally:
        m.test_set_knob("cluster_query_fails", 0)
    torch.cuda.synchronize()
    assert ffn.device_status() == 0
    assert launches[0] == launches[2] == launches[1] + 1 == launches[3] + 1
    assert torch.equal(y[0], y[2]) and torch.equal(y[1], y[3])
    assert (y[0] - y[1]).norm() <= 1e-5 * y[0].norm()  # fp32 sums of the same products in another order
