"""Groups with enough tiles for the interleaved unit order (eight a CTA), with
problems of one tile and one k-chunk, of many, and empty ones among them:
whole-numbered operands, every problem exact."""
from __future__ import annotations

import pytest
import torch

import paper_1804_10694_gb300 as pkg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["bf16x3", "tf32x3", "bf16x6"])
@pytest.mark.parametrize("longest", [1, 64, 700])
def test_interleaved_units(mode, longest):
    g = torch.Generator().manual_seed(800)
    shapes = [(900, 1000, 1 + (i * 37) % longest) for i in range(24)] + [(5, 3, 9), (0, 8, 8), (130, 1, 600)]
    ops = [[torch.randint(-9, 10, s, generator=g).float().cuda() for s in ((m, k), (k, n), (m, n))] for m, n, k in shapes]
    want = [2.0 * (a.double() @ b.double()) - c.double() for a, b, c in ops]   # below 2^24: exact in FP32
    plan = pkg.GroupedPlan(shapes, mode=mode)
    A, B, C = ([o[j] for o in ops] for j in range(3))
    plan.prepare(A, B, C, [2.0] * len(ops), [-1.0] * len(ops))
    plan.execute()
    torch.cuda.synchronize()
    for s, c, w in zip(shapes, C, want):
        assert torch.equal(c.double(), w), s
    pkg.device_error()
