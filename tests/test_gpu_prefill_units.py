"""GPU parity of the packed prefill at the edges of its work units: CTA pairs (four query heads of a
KV head), single CTAs with two heads or one, one row and one row more or less than a q-tile, many
more units than SMs (the CTAs that run take over the pending ones), and scores that grow along the
keys, so that rows rescale what they have accumulated. Reference: softmax in fp64 over the dense
mask of the packed pages, from the oracle; tolerances of the bf16 path (outputs 1.5e-2, LSE 1e-3)."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2608_06146_gb300 import build as pbuild
from paper_2608_06146_gb300 import inputs
from paper_2608_06146_gb300 import padoc_attn as pa
from paper_2608_06146_gb300.engine import PrefillPlan
from paper_2608_06146_gb300.inputs import PageSpec, Workload

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.fixture(scope="module", autouse=True)
def _build():
    pbuild.build()
    pa.load_library()


def check(pages, hq, hkv, seed, ramp=0.0):
    wl = Workload("units", pages, hq, hkv, 128, torch.bfloat16, "prefill")
    q, k, v = inputs.packed_qkv(wl, seed)
    if ramp:   # later keys score higher for every query: 0 .. ramp on top of N(0, 1)
        k = k.float()
        q = q.float()
        q[..., 0] = 8.0
        k[..., 0] = torch.linspace(0.0, ramp * math.sqrt(128.0) / 8.0, k.shape[0])[:, None]
        q, k = q.to(torch.bfloat16), k.to(torch.bfloat16)
    plan = PrefillPlan(pages, wl.dtype, 128, DEV)
    out = torch.full((plan.T, hq, 128), float("nan"), dtype=wl.dtype, device=DEV)
    lse = torch.full((plan.T, hq), float("nan"), dtype=torch.float32, device=DEV)
    scale = 1.0 / math.sqrt(128)
    plan.run(q.to(DEV), k.to(DEV), v.to(DEV), scale, out, lse)
    pa.padoc_check_device_errors()
    ref_o, ref_lse = oracle.prefill_gather(pages, q, k, v, scale)
    assert np.abs(out.float().cpu().numpy() - ref_o).max() <= 1.5e-2
    assert np.abs(lse.cpu().numpy() - ref_lse).max() <= 1e-3


@pytest.mark.parametrize("hq,hkv", [(4, 1), (8, 2), (12, 1), (2, 1), (6, 3), (3, 1), (5, 1)])
@pytest.mark.parametrize("pages", [[PageSpec(1, 0, [], [])], [PageSpec(127, 0, [], [])], [PageSpec(100, 8, [8, 3], [20, 1])],
                                   [PageSpec(200, 16, [16, 8], [70, 1]), PageSpec(64, 0, [], [])]],
                         ids=["1", "127", "129", "ragged"])
def test_prefill_units(pages, hq, hkv):
    check(pages, hq, hkv, 3)


@pytest.mark.parametrize("hq,hkv", [(16, 2), (6, 3), (5, 1)])
def test_prefill_more_units_than_sms(hq, hkv):
    rng = np.random.default_rng(hq)
    pages = [PageSpec(int(p), 16, [16, 8, 0], [int(x) for x in rng.integers(1, 90, 3)]) for p in rng.integers(1, 400, 24)]
    check(pages, hq, hkv, 4)


@pytest.mark.parametrize("hq,hkv", [(8, 1), (2, 1), (3, 1)])
def test_prefill_growing_scores(hq, hkv):
    check([PageSpec(500, 32, [32, 16], [150, 40])], hq, hkv, 5, ramp=60.0)
