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


@pytest.mark.parametrize("M,N,K", [(1202, 5016, 1057), (2048, 2048, 2048), (4099, 2050, 1000)])
@pytest.mark.parametrize("beta", [0.0, 0.5])
def test_six_product_panels_are_as_accurate(M, N, K, beta):
    """BF16X6, whose pair tiles fold half as often as the single ones by
    default: panels on pairs of a product that runs on single tiles keep its
    folds (the first shape: the same bits), and none is less accurate."""
    g = torch.Generator().manual_seed(710)
    A, B, C = (torch.empty(s).uniform_(-1, 1, generator=g).pin_memory() for s in ((M, K), (K, N), (M, N)))
    a, b, c = A.cuda(), B.cuda(), C.cuda()
    exact = 1.5 * (a.double() @ b.double()) + beta * c.double()
    want = pkg.gemm(a, b, c, 1.5, beta, mode="bf16x6")
    got = pkg.gemm_host(A, B, C, 1.5, beta, mode="bf16x6").cuda()
    assert (got.double() - exact).norm() <= (want.double() - exact).norm()
    if (M, N, K) == (1202, 5016, 1057):
        assert torch.equal(got.view(torch.int32), want.view(torch.int32))
    pkg.device_error()


def test_host_calls_use_the_shape_s_own_plan():
    """Panels in other tiles than the whole product's take no plan of their
    own: a shape that went through host buffers can be captured on device
    buffers, and further host calls allocate nothing on the device."""
    n = 2048
    g = torch.Generator().manual_seed(720)
    A, B, C = (torch.empty(n, n).uniform_(-1, 1, generator=g).pin_memory() for _ in range(3))
    a, b, c = A.cuda(), B.cuda(), C.cuda()
    want = 1.5 * (a.double() @ b.double()) + 0.5 * c.double()
    s, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    for beta in (0.0, 0.5):
        pkg.gemm_host(A, B, C.clone().pin_memory(), 1.5, beta, mode="bf16x3", stream=s)
    free = torch.cuda.mem_get_info()[0]
    for beta in (0.5, 0.0, 0.5):
        pkg.gemm_host(A, B, C.clone().pin_memory(), 1.5, beta, mode="bf16x3", stream=s)
    assert torch.cuda.mem_get_info()[0] >= free
    with torch.cuda.graph(graph, stream=s):
        pkg.gemm(a, b, c, 1.5, 0.5, mode="bf16x3", stream=s)
    graph.replay()
    torch.cuda.synchronize()
    assert (c.double() - want).norm() <= 1e-5 * want.norm()
    pkg.device_error()
