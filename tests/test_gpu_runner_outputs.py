"""The step runner's outputs: fresh slices of a longer buffer on every step decode as one buffer does,
and what it refuses (type, shape, strides, device) is refused on every call, before the step begins."""
import numpy as np
import pytest
import torch

from paper_2608_06146_gb300 import build as pbuild
from paper_2608_06146_gb300 import engine

pytestmark = pytest.mark.gpu
HQ, HKV, D = 16, 2, 128


@pytest.fixture(scope="module", autouse=True)
def _build():
    pbuild.build()


def _loop(g):
    loop = engine.MaskedParallelLoop(64, HQ, HKV, D, torch.bfloat16, "cuda")
    src = [torch.randn(40, h, D, device="cuda", generator=g).to(torch.bfloat16) for h in (HQ, HKV, HKV)]
    loop.add_page(20, 3, False, src[1], src[2], np.arange(20))
    return loop, src


def _steps(loop, src, outs):
    row_of = np.zeros(16, np.int32)
    for step, (o, l) in enumerate(outs):
        row_of[:] = np.arange(16) + 20 + step
        n, ids = loop.run_step(src[1], src[2], src[0], row_of, 0.1, o, l)
        assert n == 4 and list(ids) == [1, 2, 3, 0]
        loop.end_step(num_streams=n)


def test_slices_decode_as_whole_buffers():
    got = []
    for fresh in (False, True):
        loop, src = _loop(torch.Generator("cuda").manual_seed(5))
        out = torch.zeros(3, 8, HQ, D, device="cuda", dtype=torch.bfloat16)
        lse = torch.zeros(3, 8, HQ, device="cuda")
        flat_o, flat_l = out.view(24, HQ, D), lse.view(24, HQ)
        whole, part = list(zip(out, lse)), [(flat_o[8 * i:8 * i + 5], flat_l[8 * i:8 * i + 6]) for i in range(3)]
        _steps(loop, src, part if fresh else whole)
        torch.cuda.synchronize()
        got.append((out, lse))
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
    assert got[0][1][:, :4].abs().min() > 0 and got[0][1][:, 4:].abs().max() == 0


@pytest.mark.parametrize("out, lse, err", [
    (lambda: torch.zeros(8, HQ, D, device="cuda"), None, TypeError),
    (lambda: torch.zeros(8, HQ, D, dtype=torch.bfloat16), None, ValueError),
    (lambda: torch.zeros(8, HQ, 2 * D, device="cuda", dtype=torch.bfloat16)[:, :, :D], None, ValueError),
    (lambda: torch.zeros(8, HQ * D, device="cuda", dtype=torch.bfloat16), None, ValueError),
    (lambda: torch.zeros(8, HQ // 2, D, device="cuda", dtype=torch.bfloat16), None, ValueError),
    (None, lambda: torch.zeros(8, HQ, device="cuda", dtype=torch.bfloat16), TypeError),
    (None, lambda: torch.zeros(8, HQ), ValueError),
    (None, lambda: torch.zeros(8, HQ, 1, device="cuda"), ValueError),
    (None, lambda: torch.zeros(8, HQ + 1, device="cuda"), ValueError),
    (None, lambda: torch.zeros(HQ, 8, device="cuda").t(), ValueError),
])
def test_refused_outputs(out, lse, err):
    loop, src = _loop(torch.Generator("cuda").manual_seed(6))
    good = (torch.zeros(8, HQ, D, device="cuda", dtype=torch.bfloat16), torch.zeros(8, HQ, device="cuda"))
    _steps(loop, src, [good])
    bad = (out() if out else good[0], lse() if lse else good[1])
    for _ in range(2):
        with pytest.raises(err):
            loop.run_step(src[1], src[2], src[0], np.zeros(16, np.int32), 0.1, *bad)
    _steps(loop, src, [good])   # nothing had begun
