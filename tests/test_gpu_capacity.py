"""The result does not depend on how much cache is allocated past the prefixes."""
import pytest

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
