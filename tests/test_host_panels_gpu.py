"""Products on page-locked host buffers, run panel by panel with the tile
configuration of a panel: the bits of the same product on device buffers,
where panels take other tiles than the whole product (pair tiles there, 128 x
64 or 128 x 128 here), the same ones, and ragged last panels."""
from __future__ import annotations

import pytest
import torch

import paper_1804_10694_gb300 as pkg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["bf16x3", "tf32x3"])
@pytest.mark.parametrize("M,N,K", [(4096, 2048, 1024), (4099, 2050, 260), (3000, 4097, 96), (8192, 8192, 200)])
@pytest.mark.parametrize("beta", [0.0, 0.5])
def test_panels_match_device_buffers(mode, M, N, K, beta):
    g = torch.Generator().manual_seed(700)
    A, B, C = (torch.empty(s).uniform_(-1, 1, generator=g).pin_memory() for s in ((M, K), (K, N), (M, N)))
    want = pkg.gemm(A.cuda(), B.cuda(), C.cuda(), 1.5, beta, mode=mode).cpu()
    got = pkg.gemm_host(A, B, C, 1.5, beta, mode=mode)
    assert torch.equal(got.view(torch.int32), want.view(torch.int32))
    pkg.device_error()
