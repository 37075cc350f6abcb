"""The E4M3 writers on infinite values: the block's scale is infinite, finite values become zeros of their
sign, infinity over infinity the NaN code, and the other heads and blocks stay what they are. Every byte
equal to the oracle's, for whole blocks and for rows appended to blocks that hold some."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_06146_gb300 import build as pbuild
from paper_2608_06146_gb300 import padoc_attn as pa

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
INF = float("inf")


@pytest.fixture(scope="module", autouse=True)
def _build():
    pbuild.build()
    pa.load_library()


@pytest.mark.parametrize("count,heads", [(1, 1), (1, 2), (5, 3)])
def test_quantize_infinities(count, heads):
    rng = np.random.default_rng(count + heads)
    k, v = (torch.from_numpy(rng.standard_normal((count, heads, 16, 128)).astype(np.float32)).to(torch.bfloat16) for _ in range(2))
    k[0, 0, 7, 9], k[0, 0, 3, 4], k[0, 0, 5], k[0, 0, 6, ::2] = INF, -INF, 0.0, -0.0
    v[-1, -1, 0, 127] = -INF
    pool = pa.E4M3Pool(count, heads, 128, DEV)
    pa.padoc_quantize_kv_blocks(pool, k.to(DEV), v.to(DEV), torch.arange(count, dtype=torch.int32, device=DEV))
    pa.padoc_check_device_errors()
    for src, codes, scales in ((k, pool.k_codes, pool.k_scales), (v, pool.v_codes, pool.v_scales)):
        c, s = oracle.quantize_kv_blocks(src.float())
        assert (c == 0x7F).any() and np.isinf(s).sum() == 1
        np.testing.assert_array_equal(scales.cpu().numpy(), s)
        np.testing.assert_array_equal(codes.cpu().numpy(), c)


@pytest.mark.parametrize("heads", [1, 3])
def test_append_infinities(heads):
    rng = np.random.default_rng(heads)
    nb = 4
    pool = pa.E4M3Pool(nb, heads, 128, DEV)
    want = [np.zeros((nb, heads, 16, 128), np.uint8), np.zeros((nb, heads), np.float32)]
    src = torch.from_numpy(rng.standard_normal((nb, heads, 5, 128)).astype(np.float32)).to(torch.bfloat16)
    src[0, 0, 0, 3], src[1, 0, 2, 5], src[2, -1, 4, 0] = INF, -INF, INF   # as the first row, between and last
    for r in range(5):
        row = src[:, :, r].contiguous()
        slots = np.arange(nb, dtype=np.int32) * 16 + r
        pa.padoc_append_inputs_e4m3(pool, row.to(DEV), row.to(DEV), torch.from_numpy(slots).to(DEV))
        want = oracle.append_kv_quantized(want[0], want[1], slots, row.float())
    pa.padoc_check_device_errors()
    for codes, scales in ((pool.k_codes, pool.k_scales), (pool.v_codes, pool.v_scales)):
        np.testing.assert_array_equal(scales.cpu().numpy(), want[1])
        np.testing.assert_array_equal(codes.cpu().numpy(), want[0])
