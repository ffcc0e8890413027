"""What a cache allocated longer than its prefixes changes: the capacity may choose the
kernel, the accuracy is the same, and with bf16 keys and values of 128-wide heads so are
the bits."""
import pytest
import torch

from tests.device_util import Call, assert_rows
from tests.test_gpu_columns import E4M3, EDGES, ROWS
from tests.test_gpu_f8 import run_f8, small as small_f8

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("G,T", ROWS)
@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("kap,nu", E4M3)
def test_step_edges_e4m3_in_a_small_cache(G, T, D, kap, nu):
    """The inputs of test_step_edges_e4m3 under the smallest capacity, to the same
    tolerance (with e4m3 values rounded weights need more than bf16's 8 bits there)."""
    P = EDGES
    block = [(T, 1, T - 1)[i % 3] for i in range(len(P))]
    run_f8(small_f8(batch=len(P), layers=1, q_heads=2 * G, head_dim=D, prefix=(0, 1000),
                    block=(T,)), kap, nu, layer=0, prefix=P, block=block, poison_tail=True)


@pytest.mark.parametrize("G,T", [(1, 8), (4, 5), (4, 15)])
@pytest.mark.parametrize("P", [[600, 64, 0, 1300], [12000, 11999, 70, 9000]], ids=["short", "long"])
def test_the_same_bits_under_any_capacity(G, T, P):
    c = Call(P, [T, T - 1, 1, T], G, 8, 128, seed=11)
    o1, l1 = c.run()
    o2, l2 = c.with_capacity(40000).run()
    torch.cuda.synchronize()
    assert torch.equal(o1, o2) and torch.equal(l1, l2)
    assert_rows(o1, l1, c.reference())


@pytest.mark.parametrize("kf8,vf8", [(False, False), (True, False), (True, True), (False, True)])
@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("G,T", ROWS)
def test_step_edges_in_a_long_cache(kf8, vf8, D, G, T):
    """Every prefix length around a tile and a step of two tiles, full and shorter
    blocks, empty prefixes, under a capacity that takes the kernel for longer ranges."""
    block = [(T, 1, T - 1)[i % 3] for i in range(len(EDGES))]
    c = Call(EDGES, block, G, 2, D, kf8, vf8, capacity=30000, seed=13)
    out, lse = c.run()
    assert_rows(out, lse, c.reference())
    assert c.status() == 0


@pytest.mark.parametrize("kf8,vf8,D", [(False, False, 64), (True, False, 128), (True, True, 128)])
def test_calls_over_a_long_cache(kf8, vf8, D):
    """The kernel for longer ranges in a graph, back to back on one workspace with
    lengths that change between the calls, with lengths out of range, and again: the
    bits of a call alone."""
    cap = 30000
    c = Call([cap, cap, 0], [8, 3, 8], 2, 8, D, kf8, vf8, capacity=cap, seed=17)
    lens = [([9000, 8000, 0], [8, 3, 8]), ([64, 8001, 129], [1, 8, 0]), ([0, 0, 0], [8, 8, 8]),
            ([cap, 0, 1], [8, 0, 8])]
    c.q.nan_to_num_(0.25)
    c.kb.nan_to_num_(0.25)
    c.vb.nan_to_num_(0.25)
    for t in (c.k, c.v):  # (sequence 2 has no prefix of its own: NaN codes there)
        t[2] = t[0]
    want = []
    for pl, bl in lens:
        c.P, c.T = pl, bl
        c.pl.copy_(torch.tensor(pl))
        c.bl.copy_(torch.tensor(bl))
        out, lse = c.run()
        torch.cuda.synchronize()
        assert_rows(out, lse, c.reference())
        want.append((out.clone(), lse.clone()))
    assert c.status() == 0
    on_device = [(torch.tensor(pl, dtype=torch.int32, device="cuda"),
                  torch.tensor(bl, dtype=torch.int32, device="cuda")) for pl, bl in lens]
    outs = [(torch.zeros_like(o), torch.zeros_like(l)) for o, l in want]

    def all_calls():
        for (pl, bl), (o, l) in zip(on_device, outs):
            c.pl.copy_(pl)
            c.bl.copy_(bl)
            c.run(out=o, lse=l)

    all_calls()
    torch.cuda.synchronize()
    for (o, l), (wo, wl) in zip(outs, want):
        assert torch.equal(o, wo) and torch.equal(l, wl)
        o.zero_()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        all_calls()
    graph.replay()
    torch.cuda.synchronize()
    for (o, l), (wo, wl) in zip(outs, want):
        assert torch.equal(o, wo) and torch.equal(l, wl)
    assert c.status() == 0
    c.pl.copy_(torch.tensor([cap + 100, -5, 1]))  # clamped to the last lengths, and flagged
    c.bl.copy_(torch.tensor([9, 0, 8]))
    out, lse = c.run()
    torch.cuda.synchronize()
    assert c.status() == 2
    assert torch.equal(out, want[3][0]) and torch.equal(lse, want[3][1])


@pytest.mark.parametrize("vf8", [False, True])
@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("cap", [1, 8, 63, 64, 65, 127, 128, 129])
def test_smallest_caches_of_e4m3_keys(vf8, D, cap):
    """Up to 16 rows over e4m3 keys with D = 128 always take the kernel that loads two
    tiles of keys at once: caches of less than that."""
    c = Call([cap, cap - 1, 0], [3, 1, 2], 2, 4, D, True, vf8, capacity=cap, seed=19)
    out, lse = c.run()
    assert_rows(out, lse, c.reference())
    assert c.status() == 0
