"""Decode over an E4M3 pool whose queries and block scales span the range of their types (the kernels work
on f16 operands): query rows scaled by powers of two from 2^-60 to 2^60 with K scales that undo them, V
scales from 2^-60 to 2^40 mixed block by block, zero blocks at a history's start, one-M-tile and two-M-tile
pieces, private histories of one row, of part of a block and of many blocks. Reference: the oracle's fp64
decode of the dequantized cache. An output of row magnitude r carries the bf16 rounding of its partials and
of itself and the rounding of P: 2^-6 r covers them; LSE within 1e-3."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2608_06146_gb300 import build as pbuild
from paper_2608_06146_gb300 import inputs
from paper_2608_06146_gb300 import padoc_attn as pa
from paper_2608_06146_gb300.engine import DecodePlan
from paper_2608_06146_gb300.inputs import PageSpec, Workload

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.fixture(scope="module", autouse=True)
def _build():
    pbuild.build()
    pa.load_library()


@pytest.mark.parametrize("q_exp", [0, 60, -60])
@pytest.mark.parametrize("v_exps", [(0, 0), (-20, 20), (-60, 40), (-60, -50)])
def test_decode_e4m3_ranges(q_exp, v_exps):
    pages = [PageSpec(400, 24, [8, 16, 24] * 7, [1, 5, 16, 17, 40, 33, 200] * 3),       # 21 streams: two M-tiles
             PageSpec(300, 8, [8] * 9, [3, 300, 16, 15, 64, 1, 2, 48, 90]),              # one M-tile
             PageSpec(130, 8, [8, 4], [70, 9])]                                          # warp items only
    wl = Workload("ranges", pages, 16, 2, 128, torch.bfloat16, "decode")
    di = inputs.decode_inputs(wl, 77)
    rng = np.random.default_rng(5)
    nb = di.num_blocks
    pool = pa.E4M3Pool(nb, 2, 128, DEV)
    codes = [torch.from_numpy(rng.integers(0, 256, (nb, 2, 16, 128)).astype(np.uint8)) for _ in range(2)]
    for c in codes:                                     # no NaN codes; small exponents keep scores moderate
        c &= 0xBF
        c[(c & 0x7F) == 0x7F] = 0
    ks = np.full((nb, 2), 2.0 ** -q_exp * 0.5, np.float32) * rng.uniform(0.5, 2, (nb, 2)).astype(np.float32)
    vs = np.exp2(rng.uniform(v_exps[0], v_exps[1] + 1, (nb, 2))).astype(np.float32)
    zero = [int(b) for b in di.page_table[:, 0]] + [int(b) for b in di.stream_table[::3, 0]]
    vs[zero] = 0.0                                      # a zero scale: codes 0
    codes[1][zero] = 0
    ks[di.page_table[1, 2]] = 0.0
    codes[0][int(di.page_table[1, 2])] = 0
    for t, x in ((pool.k_codes, codes[0]), (pool.v_codes, codes[1]), (pool.k_scales, torch.from_numpy(ks)),
                 (pool.v_scales, torch.from_numpy(vs))):
        t.copy_(x)
    q = (di.q.float() * 2.0 ** q_exp).to(torch.bfloat16)
    plan = DecodePlan(pages, 16, 2, 128, DEV)
    S = plan.num_streams
    out = torch.full((S, 16, 128), float("nan"), dtype=torch.bfloat16, device=DEV)
    lse = torch.full((S, 16), float("nan"), dtype=torch.float32, device=DEV)
    pa.padoc_branch_decode_attn_e4m3(pool, plan.info, plan.plan_dev, torch.from_numpy(di.page_table).to(DEV),
                                     torch.from_numpy(di.stream_table).to(DEV), q.to(DEV), 1 / math.sqrt(128), out, lse,
                                     plan.workspace)
    pa.padoc_check_device_errors()
    ref_o, ref_l = oracle.decode_paged(pages, oracle.dequantize_kv_blocks(codes[0].numpy(), ks),
                                       oracle.dequantize_kv_blocks(codes[1].numpy(), vs), di.page_table, di.stream_table, q,
                                       1 / math.sqrt(128), False)
    got = out.float().cpu().numpy()
    assert np.isfinite(got).all()
    row = np.abs(ref_o).max(-1, keepdims=True)
    assert (np.abs(got - ref_o) <= 2.0 ** -6 * row + 1e-30).all()
    assert np.abs(lse.cpu().numpy() - ref_l).max() <= 1e-3
