"""The packed prefill on both sides of the line between a CTA per (q-tile, head) and units of several
heads (two units an SM: 304 on 152 SMs), for groups that go to CTA pairs, to two heads a CTA and to one,
with ragged last tiles. Reference and tolerances of the unit tests."""
import pytest

from paper_2608_06146_gb300.inputs import PageSpec
from tests.test_gpu_prefill_units import _build, check  # noqa: F401  (the module's build fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hq,hkv", [(16, 2), (32, 16), (24, 24), (48, 4)])
@pytest.mark.parametrize("over", [0, 1])
def test_prefill_around_the_small_call_line(hq, hkv, over):
    tokens = 128 * (304 // hq) + (37 if over else -5)   # the last q-tile of the small side, the first above it
    pages, left = [], tokens
    while left > 0:
        n = min(left, 301)
        pages.append(PageSpec(n - 60, 20, [3, 20], [15, 25]) if n > 100 else PageSpec(n, 0, [], []))
        left -= n
    check(pages, hq, hkv, 31 * hq + over)
