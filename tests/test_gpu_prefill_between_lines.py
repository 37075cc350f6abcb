"""The packed prefill between one and two (q-tile, head) units an SM, where the map decides whether a CTA runs
one head or two: sizes just above one unit an SM, between, and just below two, as one causal page (many tiles
a q-tile: one head) and as short pages (two heads). Each KV head's queries in a call of their own have half
of the units or fewer and take a CTA a head: the arithmetic of a row is the same, so the bits are. Repeated
calls agree too. (The oracle checks of either kind of unit are those of the unit and small-call tests.)"""
import math

import pytest
import torch

from paper_2608_06146_gb300 import inputs
from paper_2608_06146_gb300 import padoc_attn as pa
from paper_2608_06146_gb300.engine import PrefillPlan
from paper_2608_06146_gb300.inputs import PageSpec, Workload
from tests.test_gpu_prefill_units import DEV, _build  # noqa: F401  (the module's build fixture)

pytestmark = pytest.mark.gpu


def pages_of(tokens, page):
    pages, left = [], tokens
    while left > 0:
        n = min(left, page)
        pages.append(PageSpec(n - 40, 10, [4, 10], [17, 13]) if n > 60 else PageSpec(n, 0, [], []))
        left -= n
    return pages


def run(plan, q, k, v):
    out, lse = torch.full_like(q, float("nan")), torch.full(q.shape[:2], float("nan"), dtype=torch.float32, device=DEV)
    plan.run(q, k, v, 1 / math.sqrt(128), out, lse)
    return out, lse


@pytest.mark.parametrize("hq,hkv", [(16, 2), (12, 2), (8, 4), (32, 4)])
@pytest.mark.parametrize("page", [90, 400, 10 ** 6])
@pytest.mark.parametrize("where", ["one", "middle", "two"])
def test_prefill_between_one_and_two_units_an_sm(hq, hkv, page, where):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    tiles = {"one": sms // hq + 1, "middle": 3 * sms // (2 * hq), "two": 2 * sms // hq}[where]
    pages = pages_of(128 * tiles - (0 if where == "two" else 29), page)
    q, k, v = (x.to(DEV) for x in inputs.packed_qkv(Workload("lines", pages, hq, hkv, 128, torch.bfloat16, "prefill"), 5))
    plan = PrefillPlan(pages, torch.bfloat16, 128, DEV)
    out, lse = run(plan, q, k, v)
    group = hq // hkv
    for g in range(hkv):
        h = slice(g * group, (g + 1) * group)
        o, x = run(plan, q[:, h].contiguous(), k[:, g:g + 1].contiguous(), v[:, g:g + 1].contiguous())
        assert torch.equal(out[:, h], o) and torch.equal(lse[:, h], x)
    for _ in range(8):
        o, x = run(plan, q, k, v)
        assert torch.equal(out, o) and torch.equal(lse, x)
    pa.padoc_check_device_errors()
