"""Decode over E4M3 pools at the ends of what their types hold, where the f16 operands and the split of a
block's V scale between exponent and probability could lose a row without a word. Pages whose shared
streams go to the tensor cores (two M-tiles, one) and to warps, cutoffs inside tiles and blocks. Reference:
the oracle's fp64 decode of the dequantized cache; per row, outputs within 2^-6 of its largest magnitude
(the bf16 roundings of partials, output and P), LSE within 1e-3."""
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
PAGES = [PageSpec(400, 24, [8, 16, 24] * 7, [1, 5, 16, 17, 40, 33, 200] * 3),       # 21 streams: two M-tiles
         PageSpec(300, 8, [8] * 9, [3, 300, 16, 15, 64, 1, 2, 48, 90]),              # one M-tile
         PageSpec(130, 8, [8, 4], [70, 9])]                                          # warp items only


@pytest.fixture(scope="module", autouse=True)
def _build():
    pbuild.build()
    pa.load_library()


def cache(seed):
    """Page tables and queries of PAGES, and codes of small exponents for every block of the pool."""
    di = inputs.decode_inputs(Workload("extremes", PAGES, 16, 2, 128, torch.bfloat16, "decode"), seed)
    rng = np.random.default_rng(seed)
    codes = [rng.integers(0, 256, (di.num_blocks, 2, 16, 128)).astype(np.uint8) & 0xBF for _ in range(2)]
    return di, codes, rng


def check(di, codes, ks, vs, q, **plan_args):
    pool = pa.E4M3Pool(di.num_blocks, 2, 128, DEV)
    for t, x in ((pool.k_codes, codes[0]), (pool.v_codes, codes[1]), (pool.k_scales, ks), (pool.v_scales, vs)):
        t.copy_(torch.from_numpy(x))
    plan = DecodePlan(PAGES, 16, 2, 128, DEV, **plan_args)
    assert plan.info.num_tc_items > 0 and plan.info.num_warps > 0
    out = torch.full((plan.num_streams, 16, 128), float("nan"), dtype=torch.bfloat16, device=DEV)
    lse = torch.full((plan.num_streams, 16), float("nan"), dtype=torch.float32, device=DEV)
    pa.padoc_branch_decode_attn_e4m3(pool, plan.info, plan.plan_dev, torch.from_numpy(di.page_table).to(DEV),
                                     torch.from_numpy(di.stream_table).to(DEV), q.to(DEV), 1 / math.sqrt(128), out, lse,
                                     plan.workspace)
    pa.padoc_check_device_errors()
    ref_o, ref_l = oracle.decode_paged(PAGES, oracle.dequantize_kv_blocks(codes[0], ks),
                                       oracle.dequantize_kv_blocks(codes[1], vs), di.page_table, di.stream_table, q,
                                       1 / math.sqrt(128), False)
    got, got_l = out.double().cpu().numpy(), lse.double().cpu().numpy()
    seen = np.isfinite(ref_o).all((1, 2))            # streams that see no NaN
    assert seen.any() and np.isfinite(got[seen]).all() and np.isfinite(got_l[seen]).all()
    err = np.abs(got - ref_o)[seen] / (np.abs(ref_o[seen]).max(-1, keepdims=True) + 2.0 ** -130)
    assert err.max() <= 2.0 ** -6, f"outputs: {err.max():.3e} of the row"
    assert np.abs(got_l - ref_l)[seen].max() <= 1e-3


@pytest.mark.parametrize("k_exp", [-20, -24, -40])
@pytest.mark.parametrize("q_exp", [None, -120])
def test_multiplier_of_masked_columns(q_exp, k_exp):
    # A zero query row (or a tiny one) beside a tiny K scale: their product, which multiplies a tile's masked
    # columns (-inf) too, must stay above zero.
    di, codes, rng = cache(91)
    q = di.q.clone()
    q[:, ::3] = 0.0 if q_exp is None else q[:, ::3] * 2.0 ** q_exp
    q[2] = 0.0
    ks = (2.0 ** k_exp * rng.uniform(0.5, 1, (di.num_blocks, 2))).astype(np.float32)
    vs = rng.uniform(0.5, 2, (di.num_blocks, 2)).astype(np.float32)
    check(di, codes, ks, vs, q)


def test_nan_codes_in_rows_no_stream_sees():
    # Rows past a stream's end keep whatever a former owner left there, NaN codes too, and a row that
    # only later branches see is nothing to the earlier ones.
    di, codes, rng = cache(92)
    for p, pg in enumerate(PAGES):
        first = pg.prefix_len + (9 if p == 0 else max(pg.fork_offset))   # page 0: row 409 is seen from fork 16 on
        for t in range(first, 16 * math.ceil((pg.prefix_len + pg.layout_len) / 16)):
            for c in codes:
                c[di.page_table[p, t // 16], :, t % 16] = rng.choice([0x7F, 0xFF], (2, 128))
    for s, n in enumerate(di.priv_len):
        for c in codes:
            c[di.stream_table[s, (n - 1) // 16], :, (n - 1) % 16 + 1:] = 0x7F
    ks, vs = (rng.uniform(0.2, 0.5, (di.num_blocks, 2)).astype(np.float32) for _ in range(2))
    check(di, codes, ks, vs, di.q)
    check(di, codes, ks, vs, di.q, tc_ctas=2, warp_ctas=2)


@pytest.mark.parametrize("first,then", [(None, 40), (None, 15), (-100, 30), (-125, 15), (30, -100), (15, None)])
def test_row_sums_do_not_depend_on_v_scales(first, then):
    # A history's blocks with V scales of 2^first up to a point and 2^then from there (None: zero blocks, whose
    # codes are zeros), all at like scores: each token counts in the row sum whatever its V scale.
    di, codes, rng = cache(93)
    vs = np.zeros((di.num_blocks, 2), np.float32)
    for table in list(di.page_table) + list(di.stream_table):
        blocks = table[table >= 0]
        cut = max(len(blocks) * 2 // 3, 1)
        for part, e in ((blocks[:cut], first), (blocks[cut:], then)):
            vs[part] = 0.0 if e is None else 2.0 ** e * rng.uniform(0.5, 1, (len(part), 2))
    codes[1][vs == 0.0] = 0
    ks = rng.uniform(0.2, 0.5, (di.num_blocks, 2)).astype(np.float32)
    check(di, codes, ks, vs, di.q)
    check(di, codes, ks, vs, di.q, tc_ctas=2, warp_ctas=2)


@pytest.mark.parametrize("v_exp", [-98, -104, -112, -116])
def test_v_scales_below_2_to_the_minus_100(v_exp):
    # tensor-core and warp items alike carry the scale's own value
    di, codes, rng = cache(94)
    vs = (2.0 ** v_exp * rng.uniform(0.25, 1, (di.num_blocks, 2))).astype(np.float32)
    check(di, codes, rng.uniform(0.2, 0.5, (di.num_blocks, 2)).astype(np.float32), vs, di.q)
