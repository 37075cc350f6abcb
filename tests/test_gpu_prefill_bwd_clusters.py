"""The dK/dV pass of the prefill backward at each cluster size (8, 4, 2 and 1 CTAs for up to 45, 160, 560
and more (128-key tile, KV head) units), with groups of one query head, whose units have fewer steps than
a cluster has CTAs, and ragged last tiles; two calls agree bit for bit. Tolerances of the backward tests."""
import numpy as np
import pytest
import torch

from paper_2608_06146_gb300.inputs import PageSpec, Workload
from tests.test_gpu_prefill_bwd import _build, check  # noqa: F401  (the module's build fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hq,hkv,tokens", [(1, 1, 40), (2, 2, 130), (8, 1, 700), (9, 9, 640), (16, 8, 900), (16, 16, 1400),
                                           (34, 34, 2200)])
def test_prefill_bwd_cluster_sizes(hq, hkv, tokens):
    rng = np.random.default_rng(hq * 1000 + tokens)
    pages, left = [], tokens
    while left > 0:
        n = min(left, int(rng.integers(30, 260)))
        pages.append(PageSpec(n - 5, 3, [2], [2]) if n > 6 else PageSpec(n, 0, [], []))
        left -= n
    got = check(Workload("clusters", pages, hq, hkv, 128, torch.bfloat16, "prefill"), 11, repeat=2)
    for a, b in zip(got[0], got[1]):
        np.testing.assert_array_equal(a, b)
