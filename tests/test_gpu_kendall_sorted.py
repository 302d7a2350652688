"""rwc_kendall by sorting (more than 16384 elements) against all pairs compared
one by one: run and tile edges, ties in one, in the other and in both vectors,
signed zeros and infinities; the counts are whole numbers, so equal exactly."""
import numpy as np
import pytest
import torch

import paper_2510_20604_gb300 as rwc

pytestmark = pytest.mark.gpu


def _all_pairs(a, b):
    n, diff = a.numel(), 0
    step = max(1, (1 << 27) // n)
    for i in range(0, n, step):
        sa = (a[i:i + step, None] > a[None]).to(torch.int8) - (a[i:i + step, None] < a[None]).to(torch.int8)
        sb = (b[i:i + step, None] > b[None]).to(torch.int8) - (b[i:i + step, None] < b[None]).to(torch.int8)
        diff += int((sa * sb).sum(dtype=torch.int64))
    return diff // 2


def _vectors(n, kind):
    g = torch.Generator(device="cuda").manual_seed(n)
    a = torch.randn(n, generator=g, device="cuda", dtype=torch.float64)
    b = a + 0.3 * torch.randn(n, generator=g, device="cuda", dtype=torch.float64)
    if kind == "ties":
        a, b = (a * 4).round() / 4, (b * 3).round() / 3          # -0.0 among them
    elif kind == "ties_a":
        a = (a * 2).round()
    elif kind == "equal":
        b = torch.full_like(b, 2.5)
    elif kind == "reversed":
        b = -a
    elif kind == "same":
        b = a.clone()
    elif kind == "special":
        a[::7], a[1::7], b[::5], b[1::5] = float("inf"), -0.0, float("-inf"), 0.0
        a[2::7] = 0.0
    return a.contiguous(), b.contiguous()


@pytest.mark.parametrize("kind", ["plain", "ties", "ties_a", "equal", "reversed", "same", "special"])
@pytest.mark.parametrize("n", [8192, 8193, 10240, 16385, 40961])
def test_sorted_equals_all_pairs(n, kind):
    a, b = _vectors(n, kind)
    tau, diff = rwc.rwc_kendall(a, b)
    ref = _all_pairs(a, b)
    assert diff == ref
    assert tau == 2.0 * ref / (n * (n - 1.0))


# the first size that is sorted, a part tile behind an odd number of tiles, two levels
# of runs with a part run
@pytest.mark.parametrize("kind", ["plain", "ties", "ties_a", "equal", "reversed", "same", "special"])
@pytest.mark.parametrize("n", [16384, 16385, 18433, 22528, 24577])
def test_sorted_equals_all_pairs_above_the_bound(n, kind):
    a, b = _vectors(n, kind)
    assert rwc.rwc_kendall(a, b)[1] == _all_pairs(a, b)


def test_one_launch_up_to_the_bound():
    for n in (8193, 12000, 16384):
        a, b = _vectors(n, "plain")
        before = rwc.rwc_launch_count()
        rwc.rwc_kendall(a, b)
        assert rwc.rwc_launch_count() == before + 1


def test_sorted_on_a_side_stream_and_repeated():
    a, b = _vectors(300_001, "ties")
    _, ref = rwc.rwc_kendall(a, b)
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        for _ in range(3):
            assert rwc.rwc_kendall(a, b)[1] == ref
