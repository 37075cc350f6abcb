"""The packed prefill on CTA pairs with several times more units than pairs, most of them one tile long:
the first CTA announces a unit to the second in one of two slots and writes that slot again two units on,
which may not overtake the second CTA's reads of it. Against the oracle once, then bit for bit over
repeated calls."""
import math

import pytest
import torch

from paper_2608_06146_gb300 import inputs
from paper_2608_06146_gb300 import padoc_attn as pa
from paper_2608_06146_gb300.engine import PrefillPlan
from paper_2608_06146_gb300.inputs import PageSpec, Workload
from tests.test_gpu_prefill_units import DEV, _build, check  # noqa: F401  (the module's build fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hq,hkv,long_every", [(16, 2, 1000), (16, 2, 7), (4, 1, 5), (64, 4, 3)])
def test_prefill_announced_units(hq, hkv, long_every):
    n = max(24, 1400 // hq)
    pages = [PageSpec(700, 16, [4, 16], [40, 30]) if i % long_every == long_every - 1 else PageSpec(100, 8, [8], [20])
             for i in range(n)]
    check(pages, hq, hkv, 17)
    wl = Workload("handover", pages, hq, hkv, 128, torch.bfloat16, "prefill")
    q, k, v = (x.to(DEV) for x in inputs.packed_qkv(wl, 18))
    plan = PrefillPlan(pages, wl.dtype, 128, DEV)
    runs = []
    for _ in range(20):
        out = torch.full((plan.T, hq, 128), float("nan"), dtype=wl.dtype, device=DEV)
        lse = torch.full((plan.T, hq), float("nan"), dtype=torch.float32, device=DEV)
        plan.run(q, k, v, 1 / math.sqrt(128), out, lse)
        runs.append((out, lse))
    pa.padoc_check_device_errors()
    assert all(torch.equal(o, runs[0][0]) and torch.equal(x, runs[0][1]) for o, x in runs[1:])
