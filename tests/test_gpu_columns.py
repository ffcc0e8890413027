"""The attention kernel's forms: query columns 16, 32 and 64 (one or two softmax
groups), keys and values bf16 or e4m3, head dimensions 64 and 128, at the edges
of its 64-key tiles and two-tile steps, and with references that move.
Tolerances are those of tests/gpu_util.py (bf16 weights and outputs)."""
import pytest

from tests.gpu_util import run_small
from tests.test_gpu_attention import small
from tests.test_gpu_f8 import run_f8, small as small_f8

pytestmark = pytest.mark.gpu

ROWS = [(1, 15), (4, 5), (4, 13)]  # (G, T): 15, 20 and 52 rows of 16, 32 and 64 columns
EDGES = [0, 1, 16, 63, 64, 65, 127, 128, 129, 191, 192, 193, 1000]
E4M3 = [(2, 6), (3, 3), (6, 2)]    # e4m3 keys, keys and values, values


@pytest.mark.parametrize("G,T", ROWS)
@pytest.mark.parametrize("D", [64, 128])
def test_step_edges(G, T, D):
    """Every prefix length around a tile and a step (two tiles, the block tile
    the second of a step or alone), full and shorter blocks, in one batch: NaN
    past each length."""
    P = EDGES
    block = [(T, 1, T - 1)[i % 3] for i in range(len(P))]
    run_small(small(batch=len(P), layers=1, q_heads=2 * G, head_dim=D, prefix=(0, 1000),
                    block=(T,), depths=2, key_depth=1, value_depth=2, extra_capacity=6000),
              prefix=P, block=block, poison_tail=True)


@pytest.mark.parametrize("G,T", ROWS)
@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("kap,nu", E4M3)
def test_step_edges_e4m3(G, T, D, kap, nu):
    P = EDGES
    block = [(T, 1, T - 1)[i % 3] for i in range(len(P))]
    run_f8(small_f8(batch=len(P), layers=1, q_heads=2 * G, head_dim=D, prefix=(0, 1000),
                    block=(T,), extra_capacity=8000), kap, nu, layer=0, prefix=P, block=block,
           poison_tail=True)


@pytest.mark.parametrize("G,T", ROWS)
@pytest.mark.parametrize("D", [64, 128])
def test_long_ranges(G, T, D):
    """Many steps a range (every ring turns over), pairs split over many CTAs."""
    run_small(small(batch=1, layers=1, depths=2, key_depth=1, value_depth=2, q_heads=2 * G,
                    head_dim=D, prefix=(50000, 50000), block=(T,)))


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("kap,nu", E4M3)
def test_long_ranges_e4m3(D, kap, nu):
    run_f8(small_f8(batch=1, layers=1, q_heads=16, kv_heads=4, head_dim=D, prefix=(42000, 42000),
                    block=(13,)), kap, nu, layer=0)


@pytest.mark.parametrize("G,T", ROWS)
@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("extra", [0, 15000])
def test_either_side_of_the_short_range_rule(G, T, D, extra):
    """The kernel is chosen by the cache's capacity: the same prefixes under a
    small and a large one take the one for short ranges and the other."""
    run_small(small(batch=3, layers=1, q_heads=2 * G, head_dim=D, prefix=(0, 1000), block=(T,),
                    depths=2, key_depth=1, value_depth=2, extra_capacity=extra),
              prefix=[1000, 65, 0], block=[T, 1, T - 1])


@pytest.mark.parametrize("G,T", ROWS)
def test_references_move(G, T):
    """Scores of deviation 20 (29 in base 2): rows exceed their first keys'
    maximum by more than 2^30 and 2^15 many times over a prefix, and O, the sums
    and the row sums are rescaled."""
    run_small(small(batch=2, q_heads=2 * G, prefix=(3000, 3000), block=(T,), layers=1, depths=2,
                    key_depth=1, value_depth=2, extra_capacity=22000), scale=20.0)


def test_references_move_e4m3_values():
    run_f8(small_f8(q_heads=8, prefix=(3000, 3000), block=(13,), layers=1, extra_capacity=28000),
           6, 2, layer=0, scale=20.0)


@pytest.mark.parametrize("kap,nu", [(2, 6), (3, 3)])
def test_references_move_e4m3_keys(kap, nu):
    """e4m3 keys: the query split leaves an element below about 2^-9 of its row's
    largest an error of up to 2^-18 of that, which moves a score by about 1e-6 of
    the scores' size.  At scale 6 these caches' scores reach about 70, so that
    the lse may be off by about 7e-5 of the 1e-4 allowed; their deviation, about
    26 in base 2, still moves references by more than 2^15 and 2^30."""
    run_f8(small_f8(q_heads=8, prefix=(3000, 3000), block=(13,), layers=1, extra_capacity=28000),
           kap, nu, layer=0, scale=6.0)
