"""The dK/dV pass of the prefill backward on both sides of each line of its cluster size: clusters of 8, 4, 2
and 1 CTAs for one, four and eight query heads a KV head, units of fewer steps than CTAs, short pages and
long ones. Against the oracle, and two calls agree bit for bit. Tolerances of the backward tests."""
import numpy as np
import pytest
import torch

from paper_2608_06146_gb300.inputs import PageSpec, Workload
from tests.test_gpu_prefill_bwd import _build, check  # noqa: F401  (the module's build fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hq,hkv,tokens,page", [
    (2, 2, 60, 60), (1, 1, 1500, 300), (4, 4, 1130, 140), (4, 4, 1190, 1190), (8, 8, 1200, 140), (8, 8, 1290, 400),
    (3, 1, 1500, 60), (4, 1, 1700, 140), (12, 4, 2300, 700), (16, 4, 2330, 60), (16, 4, 2600, 2600),
    (8, 1, 5700, 900), (8, 1, 5900, 140), (16, 2, 10300, 140)])
def test_prefill_bwd_cluster_lines(hq, hkv, tokens, page):
    pages, left = [], tokens
    while left > 0:
        n = min(left, page)
        pages.append(PageSpec(n - 13, 5, [2, 5], [3, 5]) if n > 20 else PageSpec(n, 0, [], []))
        left -= n
    got = check(Workload("lines", pages, hq, hkv, 128, torch.bfloat16, "prefill"), 13, repeat=2)
    for a, b in zip(got[0], got[1]):
        np.testing.assert_array_equal(a, b)
