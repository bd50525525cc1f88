"""The plain FP32 kernel's two tiles (64 x 64 for problems that would leave
SMs without work, 128 x 128 otherwise) at their edges: whole and partial
tiles, k-slices of 16 with remainders, 16-byte and 4-byte loads, transposes.
Bound: gamma_K of a recursive FP32 sum, per element, plus the final update."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import paper_1804_10694_gb300 as pkg
import workloads as W
from gpu_helpers import dev

pytestmark = pytest.mark.gpu

SHAPES = [(64, 64, 16), (65, 63, 17), (128, 192, 15), (1, 129, 33), (200, 60, 31), (1536, 1536, 20), (1537, 1663, 19)]


@pytest.mark.parametrize("M,N,K", SHAPES)
@pytest.mark.parametrize("pad", [0, 1, 4])
@pytest.mark.parametrize("ta,tb", [(0, 0), (1, 1)])
def test_tiles(M, N, K, pad, ta, tb):
    A, B = W.uniform(M, K, 400 + M), W.uniform(K, N, 401 + N)
    C0 = W.uniform(M, N, 402, ld=N + pad)
    As = W._with_ld(np.ascontiguousarray(A.T if ta else A), (M if ta else K) + pad, np.nan)
    Bs = W._with_ld(np.ascontiguousarray(B.T if tb else B), (K if tb else N) + pad, np.nan)
    dA, dB, dC = dev(As), dev(Bs), dev(C0)
    pkg.gemm_f32_t(ta, tb, M, N, K, 1.5, dA.data_ptr(), As.shape[1], dB.data_ptr(), Bs.shape[1], 0.5,
                   dC.data_ptr(), C0.shape[1], "simt", "default", torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    got = dC.cpu().numpy()
    A64, B64, c = A.astype(np.float64), B.astype(np.float64), C0[:, :N].astype(np.float64)
    u = 2.0 ** -24
    bound = (K + 3) * u / (1 - (K + 3) * u) * (1.5 * (np.abs(A64) @ np.abs(B64)) + 0.5 * np.abs(c))
    assert (np.abs(got[:, :N] - (1.5 * (A64 @ B64) + 0.5 * c)) <= bound).all()
    assert np.array_equal(got[:, N:].view(np.uint32), C0[:, N:].view(np.uint32))
