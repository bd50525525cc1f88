"""The halo-tile convolution (default plans without split-K, at least nine
taps, C a multiple of 16) at the edges of its tiles: blocks of 16 rows and 16
or 32 columns, feature tiles of 16, 32 and 64, ragged features, filters that
are one row or one column, several channel groups, accumulation blocks longer
than one fold, both output paths (staged, and straight for K not a multiple
of 4 or a misaligned output), images that need their exponent."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from oracle import conv
import oracle
import paper_1804_10694_gb300 as pkg
import workloads as W
from gpu_helpers import TOL

pytestmark = pytest.mark.gpu

# batch, H, W, C, K, R, S
SHAPES = [(1, 16, 32, 16, 16, 3, 3), (2, 17, 33, 16, 20, 3, 3), (24, 15, 31, 16, 7, 5, 3), (1, 40, 9, 16, 16, 9, 1),
          (1, 9, 70, 16, 32, 1, 9), (18, 30, 35, 16, 33, 11, 11), (6, 70, 90, 48, 64, 3, 3), (6, 80, 96, 32, 100, 3, 3),
          (1, 1, 1, 16, 16, 3, 3), (12, 66, 64, 64, 30, 5, 5)]


def run(x, f, out0, alpha, beta, mode, offset=0):
    n, H, Wd, C = x.shape
    R, S, _, K = f.shape
    plan = pkg.ConvPlan(n, H, Wd, C, K, R, S, mode=mode)
    es = 2 if mode == "bf16x3" else 4
    # no planes of the image in the workspace: the halo kernel runs (TF32's
    # slots of an 11 x 11 halo do not fit beside 64 features' filter)
    fits = not (mode == "tf32x3" and R == 11 and K > 32)
    assert (plan.info()["workspace_bytes"] < 2 * es * (x.size + K * R * S * C)) == fits or x.size < 9000
    dx, df = torch.from_numpy(x).cuda(), torch.from_numpy(f).cuda()
    buf = torch.full((out0.size + 8,), float("nan"), device="cuda")
    do = buf[offset:offset + out0.size]
    do.copy_(torch.from_numpy(out0.reshape(-1)))
    plan.execute_ptrs(alpha, dx.data_ptr(), df.data_ptr(), beta, do.data_ptr())
    torch.cuda.synchronize()
    plan.destroy()
    got = buf.cpu().numpy()
    assert np.isnan(np.delete(got, np.s_[offset:offset + out0.size])).all()   # nothing outside the output
    return got[offset:offset + out0.size].reshape(out0.shape)


@pytest.mark.parametrize("mode", ["bf16x3", "tf32x3"])
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("beta", [0.0, 0.5])
def test_tile_edges(mode, shape, beta):
    n, H, Wd, C, K, R, S = shape
    x = W.conv_image(n, H, Wd, C, 300)
    f = W.conv_filter(C, K, 301, R=R, S=S)
    out0 = W.conv_image(n, H, Wd, K, 302)
    ref = conv.conv_f64(x, f, 1.5, beta, out0)
    for offset in ((0, 1) if x.size < 100000 else (0,)):
        got = run(x, f, out0, 1.5, beta, mode, offset)
        assert oracle.rel_frob(got.reshape(-1, K), ref.reshape(-1, K)) <= TOL, offset
    xi = W.conv_image(n, H, Wd, C, 303, kind="integers")
    fi = W.conv_filter(C, K, 304, kind="integers", R=R, S=S)
    oi = W.conv_image(n, H, Wd, K, 305, kind="integers")
    goti = run(xi, fi, oi, 1.0, beta * 2, mode)
    assert np.array_equal(goti, conv.conv_f64(xi, fi, 1.0, beta * 2, oi).astype(np.float32))
    pkg.device_error()


@pytest.mark.parametrize("mode", ["bf16x3", "tf32x3"])
@pytest.mark.parametrize("shift", [-100, 60])
@pytest.mark.parametrize("beta", [0.0, 0.5])
def test_scaled_image(mode, shift, beta):
    """The exponent is found while the image is split (beta = 0: a second
    launch starts over) or before (beta != 0); the plan's state is clean for
    the ordinary image that follows."""
    n, H, Wd, C, K = 2, 33, 40, 32, 24
    base = W.conv_image(n, H, Wd, C, 310)
    f = W.conv_filter(C, K, 311)
    out0 = W.scaled(W.conv_image(n, H, Wd, K, 312), shift)
    plan = pkg.ConvPlan(n, H, Wd, C, K, 3, 3, mode=mode)
    df = torch.from_numpy(f).cuda()
    for x, o in ((W.scaled(base, shift), out0), (base, out0), (W.scaled(base, shift), out0)):
        dx, do = torch.from_numpy(x).cuda(), torch.from_numpy(o.copy()).cuda()
        plan.execute(dx, df, do, 1.0, beta)
        torch.cuda.synchronize()
        ref = conv.conv_f64(x, f, 1.0, beta, o)
        assert oracle.rel_frob(do.cpu().numpy().reshape(-1, K), ref.reshape(-1, K)) <= TOL
    plan.destroy()


@pytest.mark.parametrize("mode", ["bf16x3", "tf32x3"])
def test_non_finite_pixels(mode):
    """Inf and NaN pixels reach exactly the outputs whose window holds them."""
    x = W.conv_image(1, 20, 37, 16, 320)
    x[0, 3, 8, 5], x[0, 17, 36, 0] = np.inf, np.nan
    f = W.conv_filter(16, 16, 321)
    ref = conv.conv_f64(x, f)
    got = run(x, f, np.zeros((1, 20, 37, 16), np.float32), 1.0, 0.0, mode)
    assert np.array_equal(np.isfinite(got), np.isfinite(ref))
    ok = np.isfinite(ref).all(axis=-1)
    assert oracle.rel_frob(got[ok], ref[ok]) <= TOL


# up to 16 features, several units a CTA, and a last column block whose columns
# do not fill the tiles of every epilogue warp (one tile in two or none of them)
RAGGED = [(100, 24, 8, 16, 12, 3, 3), (64, 40, 40, 16, 16, 3, 3), (64, 40, 48, 16, 16, 3, 3), (40, 60, 40, 16, 16, 7, 7),
          (16, 300, 300, 16, 16, 3, 3)]


@pytest.mark.parametrize("mode", ["bf16x3", "tf32x3"])
@pytest.mark.parametrize("shape", RAGGED)
@pytest.mark.parametrize("beta", [0.0, 2.0])
def test_ragged_columns_many_units(mode, shape, beta):
    """Output pieces that are skipped take no staging buffer: every pixel of
    the units before and after them is exact, in repeated passes."""
    n, H, Wd, C, K, R, S = shape
    x = W.conv_image(n, H, Wd, C, 330, kind="integers")
    f = W.conv_filter(C, K, 331, kind="integers", R=R, S=S)
    out0 = W.conv_image(n, H, Wd, K, 332, kind="integers")
    want = conv.conv_f64(x, f, 1.0, beta, out0).astype(np.float32)
    plan = pkg.ConvPlan(n, H, Wd, C, K, R, S, mode=mode)
    dx, df = torch.from_numpy(x).cuda(), torch.from_numpy(f).cuda()
    for _ in range(5):
        do = torch.from_numpy(out0.copy()).cuda()
        plan.execute(dx, df, do, 1.0, beta)
        assert np.array_equal(do.cpu().numpy(), want)
    plan.destroy()
    pkg.device_error()


@pytest.mark.parametrize("mode", ["bf16x3", "tf32x3"])
@pytest.mark.parametrize("shape", [(8, 112, 112, 128, 64, 3, 3), (8, 112, 112, 64, 64, 7, 7), (8, 112, 112, 16, 16, 3, 3)])
def test_as_accurate_as_the_im2col_kernel(mode, shape):
    """Folds are short enough that the error against 64 bits is no larger than
    that of the im2col kernel on the same layer (its configuration named)."""
    n, H, Wd, C, K, R, S = shape
    g = torch.Generator(device="cuda").manual_seed(340)
    x, f = (torch.empty(s, device="cuda").uniform_(-1, 1, generator=g) for s in ((n, H, Wd, C), (R, S, C, K)))
    pad = torch.nn.functional.pad(x.double(), (0, 0, S // 2, S // 2, R // 2, R // 2))
    exact = torch.zeros(n * H * Wd, K, dtype=torch.float64, device="cuda")
    for r in range(R):
        for s in range(S):
            exact.addmm_(pad[:, r:r + H, s:s + Wd].reshape(-1, C), f[r, s].double())
    err = []
    for named in (False, True):
        plan = pkg.ConvPlan(n, H, Wd, C, K, R, S, mode=mode, config_id=config if named else None)
        config = plan.info()["config_id"]
        out = plan.execute(x, f, torch.empty(n, H, Wd, K, device="cuda"))
        err.append((out.view(-1, K).double() - exact).norm().item())
        plan.destroy()
    assert err[0] <= err[1]


@pytest.mark.parametrize("mode,shape", [("bf16x3", (64, 17, 17, 64, 64, 11, 11)), ("tf32x3", (64, 17, 17, 64, 64, 3, 3)),
                                        ("tf32x3", (64, 17, 17, 128, 48, 5, 5)), ("tf32x3", (64, 28, 28, 128, 128, 3, 3))])
def test_mostly_padding_runs_the_im2col_kernel(mode, shape):
    """Images that fill little of the halo kernel's blocks, or need a wave more
    of them, keep the im2col kernel, with folds short enough for errors no
    larger than those of its own default."""
    n, H, Wd, C, K, R, S = shape
    x = W.conv_image(n, H, Wd, C, 350)
    f = W.conv_filter(C, K, 351, R=R, S=S)
    ref = conv.conv_f64(x, f)
    dx, df = torch.from_numpy(x).cuda(), torch.from_numpy(f).cuda()
    plan = pkg.ConvPlan(n, H, Wd, C, K, R, S, mode=mode)
    info = plan.info()
    assert info["workspace_bytes"] > (4 if mode == "bf16x3" else 8) * x.size   # the image's planes
    cfg = pkg.config_get(mode, info["config_id"])
    usual = next(i for i in range(pkg.config_count(mode)) if pkg.config_get(mode, i) == {**cfg, "kb": 4})
    err = []
    for p in (plan, pkg.ConvPlan(n, H, Wd, C, K, R, S, mode=mode, config_id=usual)):
        out = p.execute(dx, df, torch.empty(n, H, Wd, K, device="cuda")).cpu().numpy()
        err.append(oracle.rel_frob(out.reshape(-1, K), ref.reshape(-1, K)))
        p.destroy()
    assert err[0] <= err[1] <= TOL
    pkg.device_error()
