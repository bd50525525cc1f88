"""Default BF16X3 plans that run without a packing pass (tall thin and small
products whose rows TMA can load) at the edges of their tiles: items of 32 of
K with remainders, tiles of 128 x 32 and 128 x 64, several tiles a CTA, every
transpose.  The same plan takes the packed path for operands that start off a
16-byte boundary: unscaled operands give the same bits either way."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
import paper_1804_10694_gb300 as pkg
import workloads as W
from gpu_helpers import TOL

pytestmark = pytest.mark.gpu

SHAPES = [(128, 64, 32), (512, 512, 512), (640, 260, 300), (1, 1, 1), (129, 33, 31), (300, 100, 65), (128, 128, 260), (1024, 1024, 1024),
          (20100, 64, 144), (20000, 16, 130), (40000, 96, 70)]


def place(x, offset):
    """x as stored with a leading dimension that is a multiple of 4, `offset`
    floats past an aligned address; NaN around it."""
    r, c = x.shape
    ld = (c + 3) // 4 * 4
    buf = torch.full((r * ld + 8,), float("nan"), device="cuda")
    v = buf[offset:offset + r * ld].view(r, ld)
    v[:, :c] = torch.from_numpy(np.ascontiguousarray(x)).cuda()
    return v


def call(A, B, C0, ta, tb, alpha, beta, offset):
    M, N = C0.shape
    K = A.shape[1]
    a = place(A.T if ta else A, offset)
    b = place(B.T if tb else B, offset)
    c = torch.from_numpy(C0.copy()).cuda()
    pkg.gemm_f32_t(ta, tb, M, N, K, alpha, a.data_ptr(), a.stride(0), b.data_ptr(), b.stride(0), beta, c.data_ptr(), N,
                   "bf16x3", "default", torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return c.cpu().numpy()


@pytest.mark.parametrize("M,N,K", SHAPES)
@pytest.mark.parametrize("ta,tb", [(0, 0), (0, 1), (1, 0), (1, 1)])
def test_edges(M, N, K, ta, tb):
    A, B, C0 = W.uniform(M, K, 500), W.uniform(K, N, 501), W.uniform(M, N, 502)
    for beta in (0.0, 0.5):
        got, packed = (call(A, B, C0, ta, tb, 1.5, beta, offset) for offset in (0, 1))
        assert np.array_equal(got.view(np.uint32), packed.view(np.uint32)), beta
        assert oracle.rel_frob(got, oracle.gemm_f64(M, N, K, 1.5, A, B, beta, C0)) <= TOL
    Ai, Bi = W.integers(M, K, 503), W.integers(K, N, 504)
    got = call(Ai, Bi, C0, ta, tb, 1.0, 0.0, 0)
    assert np.array_equal(got, oracle.gemm_f64(M, N, K, 1.0, Ai, Bi, 0.0, None).astype(np.float32))
    pkg.device_error()


@pytest.mark.parametrize("ta,tb", [(0, 0), (1, 1)])
def test_scaled_blocks(ta, tb):
    """Tiles whose rows or columns lie outside the unscaled range are computed
    a second time with their exponents, tiles next to them are not; each
    128 x 32 block against the oracle."""
    M, N, K = 20000, 30, 100
    A, B, C0 = W.uniform(M, K, 510), W.uniform(K, N, 511), W.uniform(M, N, 512)
    A[128:256] = W.scaled(A[128:256], -100)
    A[640:700] = W.scaled(A[640:700], 50)
    for scale in (0, 60):
        Bs = W.scaled(B, scale)
        got = call(A, Bs, C0, ta, tb, 1.0, 0.0, 0)
        ref = oracle.gemm_f64(M, N, K, 1.0, A, Bs, 0.0, None)
        for r in (0, 128, 256, 512, 640, 19968):
            assert oracle.rel_frob(got[r:r + 128], ref[r:r + 128]) <= TOL, (scale, r)


def test_non_finite_values():
    """Inf and NaN reach exactly the rows and columns that hold them."""
    M, N, K = 1000, 64, 96
    A, B = W.uniform(M, K, 520), W.uniform(K, N, 521)
    A[3, 5], A[700, 95], B[40, 33] = np.inf, np.nan, -np.inf
    got = call(A, B, np.zeros((M, N), np.float32), 0, 0, 1.0, 0.0, 0)
    ref = oracle.gemm_f64(M, N, K, 1.0, A, B, 0.0, None)
    assert np.array_equal(np.isfinite(got), np.isfinite(ref))
    ok = np.isfinite(ref)
    assert oracle.rel_frob(got[ok][None], ref[ok][None]) <= TOL


@pytest.mark.parametrize("ta,tb", [(0, 0), (0, 1), (1, 0), (1, 1)])
@pytest.mark.parametrize("M,N,K", [(1060, 1060, 100), (1088, 1028, 1060), (1025, 1080, 36), (820, 1470, 260)])
def test_turned_tiles(M, N, K, ta, tb):
    """More 128 x 64 tiles than SMs, but not with the last rows (up to 64) in
    tiles of 64 x 128 whose operands change places: the packed path's bits."""
    A, B, C0 = W.uniform(M, K, 520), W.uniform(K, N, 521), W.uniform(M, N, 522)
    for beta in (0.0, 0.5):
        got, packed = (call(A, B, C0, ta, tb, 1.5, beta, offset) for offset in (0, 1))
        assert np.array_equal(got.view(np.uint32), packed.view(np.uint32)), beta
        assert oracle.rel_frob(got, oracle.gemm_f64(M, N, K, 1.5, A, B, beta, C0)) <= TOL
    # scaled rows in the last strip and scaled columns: the second pass of both kinds of tile
    last = M // 128 * 128
    A[last:] = W.scaled(A[last:], -100)
    B[:, 130:200] = W.scaled(B[:, 130:200], 60)
    got, want = call(A, B, C0, ta, tb, 1.5, 0.0, 0), oracle.gemm_f64(M, N, K, 1.5, A, B, 0.0, None)
    for r in (slice(0, last), slice(last, M)):
        for c in (slice(0, 130), slice(130, 200), slice(200, N)):
            assert oracle.rel_frob(got[r, c], want[r, c]) <= TOL, (r, c)
    pkg.device_error()


@pytest.mark.parametrize("M,N,K", [(50176, 64, 576), (100000, 32, 512), (1060, 1060, 1060)])
def test_stage_reuse(M, N, K):
    """Long runs of items through the staging ring, pass after pass: a copy
    that overtook a split warp's reads of the item before would change bits."""
    g = torch.Generator(device="cuda").manual_seed(530)
    a, b = (torch.empty(s, device="cuda").uniform_(-1, 1, generator=g) for s in ((M, K), (K, N)))
    ab = torch.full((M * K + 1,), float("nan"), device="cuda")
    ab[1:] = a.view(-1)
    want, got = torch.empty(M, N, device="cuda"), torch.empty(M, N, device="cuda")
    s = torch.cuda.current_stream().cuda_stream
    pkg.gemm_f32_ex(M, N, K, 1.0, ab.data_ptr() + 4, K, b.data_ptr(), N, 0.0, want.data_ptr(), N, "bf16x3", "default", s)
    for _ in range(20):
        got.fill_(float("nan"))
        pkg.gemm(a, b, got, mode="bf16x3")
        assert torch.equal(got.view(torch.int32), want.view(torch.int32))
    pkg.device_error()


@pytest.mark.parametrize("M,N,K,lda,ldb", [(512, 512, 512, 513, 512), (512, 512, 512, 512, 1001), (384, 384, 384, 385, 390)])
def test_rows_off_16_bytes_keep_their_configuration(M, N, K, lda, ldb):
    """Leading dimensions that are not multiples of 4 rule the kernel out for
    every call of the plan, which then runs what it would without it: the
    default split-K configuration, its bits and its workspace."""
    c = pkg.config_default("bf16x3", M, N, K)
    assert pkg.config_get("bf16x3", c)["split_k"] > 1
    A, B, C0 = W._with_ld(W.uniform(M, K, 540), lda, np.nan), W._with_ld(W.uniform(K, N, 541), ldb, np.nan), W.uniform(M, N, 542)
    a, b = (torch.from_numpy(x).cuda() for x in (A, B))
    out, info = [], []
    for config in (None, c):
        plan = pkg.Plan(M, N, K, lda, ldb, N, mode="bf16x3", config_id=config)
        info.append(plan.info())
        d = torch.from_numpy(C0.copy()).cuda()
        plan.execute_ptrs(1.5, a.data_ptr(), b.data_ptr(), 0.5, d.data_ptr())
        out.append(d.cpu().numpy())
        plan.destroy()
    assert info[0] == info[1] and info[0]["config_id"] == c
    assert np.array_equal(out[0].view(np.uint32), out[1].view(np.uint32))
    assert oracle.rel_frob(out[0], oracle.gemm_f64(M, N, K, 1.5, A, B, 0.5, C0)) <= TOL


@pytest.mark.parametrize("ta,tb,M,N,K", [(0, 0, 1, 64, 64), (0, 0, 64, 64, 1), (1, 0, 64, 64, 1), (0, 1, 64, 1, 64)])
def test_single_rows_with_any_leading_dimension(ta, tb, M, N, K):
    """A single stored row's leading dimension is never used: one past a
    tensor map's strides runs the packed path, with the same bits."""
    A, B = W.uniform(M, K, 550), W.uniform(K, N, 551)
    a, b = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (A.T if ta else A, B.T if tb else B))
    far = [2 ** 38 if x.shape[0] == 1 else x.shape[1] for x in (a, b)]
    out = []
    for lda, ldb in ((a.shape[1], b.shape[1]), far):
        c = torch.zeros(M, N, device="cuda")
        pkg.gemm_f32_t(ta, tb, M, N, K, 1.5, a.data_ptr(), lda, b.data_ptr(), ldb, 0.0, c.data_ptr(), N, "bf16x3", "default",
                       torch.cuda.current_stream().cuda_stream)
        out.append(c.cpu().numpy())
    assert 2 ** 38 in far
    assert np.array_equal(out[0].view(np.uint32), out[1].view(np.uint32))
    assert oracle.rel_frob(out[0], oracle.gemm_f64(M, N, K, 1.5, A, B, 0.0, None)) <= TOL


@pytest.mark.parametrize("n", [384, 448, 512, 640])
def test_unsplit_sums_are_the_split_ones(n):
    """In place of a split-K configuration whose parts are one fold each, the
    kernel folds at the parts' ends: without alpha and beta the sums of the
    parts in their order, the same bits."""
    c = pkg.config_default("bf16x3", n, n, n)
    cfg = pkg.config_get("bf16x3", c)
    chunks = (n + 63) // 64
    assert cfg["split_k"] > 1 and -(-chunks // cfg["split_k"]) <= cfg["kb"]
    a, b = (torch.from_numpy(W.uniform(n, n, s)).cuda() for s in (560, 561))
    got = pkg.gemm(a, b, torch.empty(n, n, device="cuda"), mode="bf16x3")
    plan = pkg.Plan(n, n, n, mode="bf16x3", config_id=c)
    want = plan.execute(a, b, torch.empty(n, n, device="cuda"))
    assert torch.equal(got.view(torch.int32), want.view(torch.int32))
    plan.destroy()
