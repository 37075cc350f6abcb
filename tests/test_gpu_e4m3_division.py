"""The E4M3 writers take a reciprocal instead of a division wherever the code cannot depend on the
difference: bytes equal to the oracle's (IEEE fp32 division) on values at and beside the midpoints
between codes, on scales from subnormal to past the reciprocal's range, with infinities, for counts
and heads that do not fill a CTA, and for an append to a pool whose codes are not 4-byte aligned."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_06146_gb300 import build as pbuild
from paper_2608_06146_gb300 import padoc_attn as pa

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.fixture(scope="module", autouse=True)
def _build():
    pbuild.build()
    pa.load_library()


def midpoint_blocks(rng, count, heads):
    """bf16 blocks whose values lie on, or a bf16 step beside, (code midpoint) x (amax / 448)."""
    vals = oracle.e4m3_decode(np.arange(0, 0x7F, dtype=np.uint8)).astype(np.float64)
    mids = (vals[:-1] + vals[1:]) / 2
    amax = np.exp2(rng.uniform(-132, 127, (count, heads, 1, 1)))
    amax[:, 0] = rng.uniform(0.01, 100, (count, 1, 1))
    amax = torch.from_numpy(amax).to(torch.bfloat16).double().numpy()
    x = rng.choice(np.concatenate([mids, vals]), (count, heads, 16, 128)) * amax / 448 * rng.choice([-1, 1], (count, heads, 16, 128))
    b = torch.from_numpy(x).float().to(torch.bfloat16).view(torch.int16)
    b = b + torch.from_numpy(rng.integers(-1, 2, b.shape).astype(np.int16)) * (b != 0)
    b = b.view(torch.bfloat16)
    lim = torch.from_numpy(amax).to(torch.bfloat16).expand_as(b)
    b = torch.where((b.abs() <= lim) & torch.isfinite(b), b, torch.zeros_like(b))
    b[:, :, 3, 5] = torch.from_numpy(amax[:, :, 0, 0]).to(torch.bfloat16)
    return b.contiguous()


@pytest.mark.parametrize("count,heads", [(1, 1), (7, 3), (64, 2), (301, 2)])
def test_quantize_bytes(count, heads):
    rng = np.random.default_rng(count)
    k, v = midpoint_blocks(rng, count, heads), midpoint_blocks(rng, count, heads)
    k[0, 0, 7, 9] = float("inf")                       # scale inf: finite values become 0, inf / inf the NaN code
    v[-1, -1] = 0.0
    dst = torch.from_numpy(rng.permutation(count + 2)[:count].astype(np.int32))
    pool = pa.E4M3Pool(count + 2, heads, 128, DEV)
    pa.padoc_quantize_kv_blocks(pool, k.to(DEV), v.to(DEV), dst.to(DEV))
    pa.padoc_check_device_errors()
    for src, codes, scales in ((k, pool.k_codes, pool.k_scales), (v, pool.v_codes, pool.v_scales)):
        c, s = oracle.quantize_kv_blocks(src.float())
        rows = slice(1, None) if src is k else slice(None)
        np.testing.assert_array_equal(scales.cpu().numpy()[dst.numpy()], s)
        np.testing.assert_array_equal(codes.cpu().numpy()[dst.numpy()][rows], c[rows])


@pytest.mark.parametrize("heads,shift", [(1, 0), (3, 0), (2, 1)])
def test_append_bytes(heads, shift):
    rng = np.random.default_rng(heads)
    nb = 9
    pool = pa.E4M3Pool(nb, heads, 128, DEV)
    n = pool.k_codes.numel()
    raw = [torch.zeros(n + 16, dtype=torch.uint8, device=DEV) for _ in range(2)]
    pool.c.k_codes, pool.c.v_codes = (r.data_ptr() + shift for r in raw)
    want = [np.zeros((nb, heads, 16, 128), np.uint8), np.zeros((nb, heads), np.float32)]
    src = midpoint_blocks(rng, nb, heads)
    src = src * torch.from_numpy(np.exp2(rng.integers(-3, 4, (nb, 1, 16, 1)))).to(torch.bfloat16)   # scales grow within a block
    src = torch.where(torch.isfinite(src), src, torch.zeros_like(src))
    for r in range(16):
        row = src[:, :, r].contiguous()
        slots = np.arange(nb, dtype=np.int32) * 16 + r
        pa.padoc_append_inputs_e4m3(pool, row.to(DEV), row.to(DEV), torch.from_numpy(slots).to(DEV))
        want = oracle.append_kv_quantized(want[0], want[1], slots, row.float())
    pa.padoc_check_device_errors()
    for r, scales in zip(raw, (pool.k_scales, pool.v_scales)):
        np.testing.assert_array_equal(scales.cpu().numpy(), want[1])
        np.testing.assert_array_equal(r[shift:shift + n].cpu().numpy().reshape(want[0].shape), want[0])
