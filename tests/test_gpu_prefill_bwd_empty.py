"""The prefill backward over tile maps with q-tiles that hold no entries (rows that see nothing: a map made
by a caller; the library's own builder gives every row itself): their dQ is zero, the units before and
after them are as without them. Such units first, last, alone and in runs, taken over by CTAs that ran
others. Reference: the oracle with dO = 0 in those rows, whose gradients' parts are then all zero;
tolerances of the backward tests."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2608_06146_gb300 import inputs
from paper_2608_06146_gb300 import padoc_attn as pa
from paper_2608_06146_gb300.engine import PrefillPlan
from paper_2608_06146_gb300.inputs import PageSpec, Workload
from tests.test_gpu_prefill_bwd import DEV, _build, assert_grad_close  # noqa: F401  (the module's build fixture)

pytestmark = pytest.mark.gpu


def without_rows(ptr, idx, kind, drop):
    """A row-major map without the entries of the rows in drop."""
    keep = [np.zeros(0, int) if r in drop else np.arange(ptr[r], ptr[r + 1]) for r in range(len(ptr) - 1)]
    sel = np.concatenate(keep)
    return np.concatenate([[0], np.cumsum([len(x) for x in keep])]).astype(np.int32), idx[sel], kind[sel]


@pytest.mark.parametrize("empty", [(1, 2, 4), (0,), (19,), (0, 1, 2, 3, 4, 5, 6, 7, 9, 18, 19), tuple(range(20))])
def test_prefill_bwd_units_without_entries(empty):
    pages = [PageSpec(500, 32, [8, 32], [60, 48])] * 4       # 20 q-tiles x 16 heads: twice the SMs
    wl = Workload("empty", pages, 16, 2, 128, torch.bfloat16, "prefill")
    q, k, v = inputs.packed_qkv(wl, 21)
    g = inputs.packed_dout(wl, 21)
    T, scale = q.shape[0], 1 / math.sqrt(128)
    assert T == 20 * 128
    rows = np.concatenate([np.arange(128 * t, 128 * t + 128) for t in empty])
    g[rows] = 0.0
    qd, kd, vd, gd = (x.to(DEV) for x in (q, k, v, g))
    fwd = PrefillPlan(pages, wl.dtype, 128, DEV)
    out = torch.empty((T, 16, 128), dtype=wl.dtype, device=DEV)
    lse = torch.empty((T, 16), dtype=torch.float32, device=DEV)
    fwd.run(qd, kd, vd, scale, out, lse)
    dev_rows = torch.from_numpy(rows).to(DEV)
    out[dev_rows], lse[dev_rows] = 0.0, -math.inf

    (qq, qk), (kq, kk) = pa.padoc_prefill_bwd_tile_shapes(pa.PADOC_DTYPE_BF16, 128)
    spans = pa.padoc_build_query_spans(pages).copy()
    spans[rows] = 0
    ptr, idx, kind = without_rows(*pa.padoc_build_tile_map(pages, qq, qk), set(empty))
    cptr, cidx, ckind, order = pa.padoc_build_key_tile_map(pages, kq, kk)
    gone = {r * qq // kq + i for r in empty for i in range(qq // kq)}
    keep = np.array([x not in gone for x in cidx], bool)
    cptr = np.concatenate([[0], np.cumsum([keep[a:b].sum() for a, b in zip(cptr[:-1], cptr[1:])])]).astype(np.int32)
    up = lambda a, dt: torch.from_numpy(np.ascontiguousarray(a if len(a) else np.zeros(1, dt))).to(DEV)
    held = [up(ptr, np.int32), up(idx, np.int32), up(kind, np.int8), up(cptr, np.int32), up(cidx[keep], np.int32),
            up(ckind[keep], np.int8), up(order, np.int32)]
    qmap, kmap = pa.make_tile_map_dev(*held[:3], qq, qk), pa.make_tile_map_dev(*held[3:6], kq, kk, order=held[6])
    ws = torch.empty(pa.padoc_prefill_bwd_workspace_size(T, 16), dtype=torch.uint8, device=DEV)
    got = []
    for _ in range(3):
        d = [torch.full_like(x, float("nan")) for x in (qd, kd, vd)]
        pa.padoc_ancestor_prefill_bwd(qd, kd, vd, out, gd, lse, torch.from_numpy(spans).to(DEV), qmap, kmap, scale, *d, ws)
        pa.padoc_check_device_errors()
        got.append(d)
    assert all(torch.equal(a, b) for d in got[1:] for a, b in zip(got[0], d))
    dq, dk, dv = (x.float().cpu().numpy() for x in got[0])
    assert not dq[rows].any()
    ref = oracle.prefill_bwd(pages, q, k, v, g, scale, None, None)
    for a, r, name in zip((dq, dk, dv), ref, ("dq", "dk", "dv")):
        assert_grad_close(a, r, torch.bfloat16, name)
