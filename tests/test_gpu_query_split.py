"""e4m3 keys scored against queries split into 8-bit parts: rows whose elements span
many powers of two, in caches long enough for the kernel that splits into three
parts (it has to lose nothing against keys widened to bf16)."""
import pytest
import torch

from tests.device_util import Call, assert_rows

pytestmark = pytest.mark.gpu

FORMS = [(64, False), (64, True), (128, True)]  # (D, e4m3 values): three parts


@pytest.mark.parametrize("D,vf8", FORMS)
@pytest.mark.parametrize("down", [8, 12, 16, 20])
@pytest.mark.parametrize("G,T", [(1, 8), (4, 5), (4, 15)])
def test_small_elements_decide(D, vf8, down, G, T):
    """The large elements meet zeros of the keys, so that the scores are those of
    elements 2^-down of the row's largest, times a scale that makes them about 1."""
    c = Call([9000, 9001, 8963], [T, T, T - 1], G, 8, D, True, vf8, 30000, seed=down)
    even = torch.zeros((), device="cuda").to(c.k.dtype)
    c.k[..., ::2] = even
    c.kb[..., ::2] = 0.0
    c.q[..., ::2] = 1.0
    c.q[..., 1::2] *= 2.0 ** -down
    scale = 2.0 ** down / (D / 2) ** 0.5
    out, lse = c.run(scale=scale)
    assert_rows(out, lse, c.reference(scale))


@pytest.mark.parametrize("D,vf8", FORMS + [(128, False)])
def test_magnitudes(D, vf8):
    """Rows of magnitudes 2^-8 to 2^3, some with elements 2^-12 of the largest, a row
    of zeros and one of each extreme bf16 exponent (2^-126 and 2^100, with keys that
    meet zeros)."""
    T = 12
    c = Call([9000, 9001, 8963], [T] * 3, 4, 8, D, True, vf8, 30000, seed=7)
    for i in range(T):
        c.q[:, i] *= 2.0 ** (i - 8)
        if i % 3 == 0:
            c.q[:, i, :, 1::2] *= 2.0 ** -12
    c.q[:, 3, 1], c.q[:, 4, 2], c.q[:, 5, 3] = 0.0, 2.0 ** -126, 0.0
    c.q[:, 5, 3, 0] = 2.0 ** 100
    c.k[..., 0] = torch.zeros((), device="cuda").to(c.k.dtype)
    c.kb[..., 0] = 0.0
    out, lse = c.run()
    assert_rows(out, lse, c.reference())
