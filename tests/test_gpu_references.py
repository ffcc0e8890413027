"""The rows' references (what is subtracted from the scores before the exponential):
they move over a segment's steps, large values do not overflow the sums, and small
weights under a strong early key are not lost."""
import pytest
import torch

from tests.device_util import Call, assert_rows

pytestmark = pytest.mark.gpu

STORES = [(False, False), (True, False), (True, True), (False, True)]
ROWS = [(1, 15), (4, 5), (4, 15)]  # (G, T): 16, 32 and 64 query columns
CAPACITY = 30000  # with 24 pairs and more: every form that the longer kernel has takes it


def ramp(c, rise):
    """Scores that rise by `rise` (natural units) over every 512 keys and fall back, each
    time to a peak 6.5 (9.4 in base 2) above the last: whatever the split, the maxima of
    a segment of 18 tiles or more pass its first step's by far more than 2^12."""
    at = torch.arange(c.k.shape[1], device="cuda")
    c.k[..., 0] = (at.remainder(512).float() / 32)[None, :, None].to(c.k.dtype)  # 0 .. 16
    c.k[..., 1] = (at // 512).clamp(max=24).float()[None, :, None].to(c.k.dtype)
    c.q[..., 0] = rise / 16 * c.D ** 0.5
    c.q[..., 1] = 6.5 * c.D ** 0.5
    return c


@pytest.mark.parametrize("kf8,vf8", STORES)
@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("G,T", ROWS)
def test_references_move_within_a_segment(kf8, vf8, D, G, T):
    """24 pairs of 12000 keys: about 29 tiles a CTA, so that most segments have 9 to 15
    steps and move their references after the first, over and over: O, the sums and the
    rounded sums are rescaled.  (The split replayed for 152 CTAs: 156 to 163 of about
    170 segments move after their first step, 413 to 667 times in all.)"""
    c = ramp(Call([12000, 11937, 12001], [T, T, T - 1], G, 8, D, kf8, vf8, CAPACITY,
                  seed=1), 60.0)
    out, lse = c.run()
    assert_rows(out, lse, c.reference())
    assert c.status() == 0


@pytest.mark.parametrize("kf8,vf8", STORES)
@pytest.mark.parametrize("D", [64, 128])
def test_sharp_scores(kf8, vf8, D):
    """Random scores of deviation 20 over segments of many steps."""
    c = Call([12000, 11937, 12001], [13] * 3, 4, 8, D, kf8, vf8, CAPACITY, seed=2, sharp=20.0)
    out, lse = c.run()
    assert_rows(out, lse, c.reference())


@pytest.mark.parametrize("kf8", [False, True])
@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("G,T", ROWS)
@pytest.mark.parametrize("P", [700, 12000])
def test_large_values(kf8, D, G, T, P):
    """bf16 values of about 2^100, under scores that exceed a segment's first by far:
    the sums of P V stay finite (weights of up to 2^8, at most 2^15 keys near them)."""
    c = ramp(Call([P] * 3, [T] * 3, G, 8, D, kf8, False, CAPACITY if P > 1000 else None, seed=4), 60.0)
    c.v.mul_(2.0 ** 100)
    c.vb.mul_(2.0 ** 100)
    out, lse = c.run()
    assert bool(out.isfinite().all())
    assert_rows(out, lse, c.reference())


@pytest.mark.parametrize("kf8,vf8", STORES)
@pytest.mark.parametrize("D", [64, 128])
def test_flat_tail_under_a_strong_key(kf8, vf8, D):
    """One key of weight 1 and value 0, 16383 of weight 2^-25.5 and value 1 each: they are
    the output.  160 pairs, so that a CTA has a whole pair's keys in one segment."""
    c = Call([16384] * 40, [2] * 40, 4, 4, D, kf8, vf8, seed=5)
    c.k.zero_()
    c.kb.zero_()
    c.q.zero_()
    c.k[:, 0, :, 0] = 8.0
    c.q[..., 0] = 25.5 * 0.6931 * D ** 0.5 / 8
    c.v[:] = torch.ones((), device="cuda").to(c.v.dtype)
    c.v[:, 0] = torch.zeros((), device="cuda").to(c.v.dtype)
    c.vb.zero_()
    out, lse = c.run()
    assert_rows(out, lse, c.reference())
