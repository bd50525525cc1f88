"""The work that users of this library have it do, as a list of cases: single
gemms over the range of sizes and modes, a gemm on host buffers, a grouped
gemm and direct convolutions, each through the public Python entry points.

listed() names the fixed cases, draw(rng) gives further ones of the same
ranges, prepare(case, seed) makes what a program holds before the call, run()
is one pass, work() the bytes and operations a pass cannot do without, and
exact() the result in 64 bits by plain torch.
"""
from __future__ import annotations

import math

import torch

import paper_1804_10694_gb300 as gemm_lib

# Products of the conv-as-gemm kind: (output pixels, output features, taps x
# channels) of 3x3 convolutions over 224 x 224 images.
CONV_GEMMS = ((50176, 64, 576), (12544, 128, 1152), (3136, 256, 2304))


def _gemm(name, M, N, K, mode="bf16x3", alpha=1.5, beta=0.5, trans_a=False, trans_b=False, dist="uniform"):
    return {"name": name, "kind": "gemm", "mode": mode, "M": M, "N": N, "K": K, "alpha": alpha, "beta": beta,
            "trans_a": trans_a, "trans_b": trans_b, "dist": dist}


def listed():
    return [
        # the smallest call: one small product inside a larger program, where
        # the launches and the call itself count
        _gemm("small_512", 512, 512, 512),
        # the paper's sgemm benchmark size, not a multiple of any tile
        _gemm("paper_1060", 1060, 1060, 1060),
        # an odd size (a prime): every row unaligned, ragged in all dimensions
        _gemm("ragged_4099", 4099, 4099, 4099),
        # the largest square product, the headline workload of the benchmark
        _gemm("square_8192", 8192, 8192, 8192),
        # a 3x3 convolution layer of a 224 x 224 image written as a product:
        # very many rows, few columns
        _gemm("skinny_50176x64x576", 50176, 64, 576, alpha=1.0, beta=0.0),
        # a linear layer x W^T with the weights stored N x K, in the TF32 split
        _gemm("linear_tf32x3_2048", 2048, 2048, 2048, mode="tf32x3", alpha=1.0, beta=0.0, trans_b=True),
        # full single-precision accuracy on operands of widely spread magnitude
        _gemm("accurate_bf16x6_2048", 2048, 2048, 2048, mode="bf16x6", dist="wide"),
        # the plain single-precision kernel, used where every product must be
        # an FP32 one
        _gemm("plain_simt_1024", 1024, 1024, 1024, mode="simt"),
        # matrices in (page-locked) host memory: copies in, product, copy out
        {"name": "host_4096", "kind": "host", "mode": "bf16x3", "M": 4096, "N": 4096, "K": 4096, "alpha": 1.5,
         "beta": 0.5, "dist": "uniform"},
        # 512 products of uneven sizes in one call (batched small solvers,
        # mixture-of-experts blocks)
        {"name": "grouped_512", "kind": "grouped", "mode": "bf16x3", "count": 512, "lo": 32, "hi": 1024,
         "alpha": 1.0, "beta": 1.0, "shapes_seed": 4000},
        # the paper's convolution benchmark: 32 images of 512 x 512, 16
        # features in and out
        {"name": "conv_paper_3x3", "kind": "conv", "mode": "bf16x3", "batch": 32, "H": 512, "W": 512, "C": 16,
         "K": 16, "R": 3, "S": 3, "alpha": 1.0, "beta": 0.0},
        # a convolution layer of an ordinary network, 64 features in and out
        {"name": "conv_64_3x3", "kind": "conv", "mode": "bf16x3", "batch": 8, "H": 256, "W": 256, "C": 64,
         "K": 64, "R": 3, "S": 3, "alpha": 1.0, "beta": 0.0},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    kind = rng.choice(("gemm", "gemm", "gemm", "gemm", "skinny", "host", "grouped", "conv", "conv"))
    alpha, beta = rng.choice(((1.0, 0.0), (1.5, 0.5)))
    if kind in ("gemm", "skinny"):
        mode = rng.choice(("bf16x3", "bf16x3", "tf32x3", "bf16x6", "simt"))
        if kind == "skinny":   # conv-as-gemm: many rows, few columns
            mode = rng.choice(("bf16x3", "bf16x3", "tf32x3"))
            M, N, K = _log_int(rng, 3136, 65536), rng.choice((16, 32, 64, 128, 256)), 9 * rng.choice((16, 32, 64, 128))
        else:
            # sizes spread over their logarithm; the slower modes stay within
            # the cost of the largest listed case
            most = {"bf16x3": 2.0 ** 39, "tf32x3": 2.0 ** 37, "bf16x6": 2.0 ** 37, "simt": 2.0 ** 35}[mode]
            while True:
                M, N, K = (_log_int(rng, 128, 8192) for _ in range(3))
                if M * N * K <= most:
                    break
            if rng.random() < 0.5:   # half of the sizes round, as layers have them
                M, N, K = (max(128, x // 64 * 64) for x in (M, N, K))
        trans_a, trans_b = rng.choice(((False, False), (False, False), (False, True), (True, False)))
        return {"kind": "gemm", "mode": mode, "M": M, "N": N, "K": K, "alpha": alpha, "beta": beta,
                "trans_a": trans_a, "trans_b": trans_b, "dist": rng.choice(("uniform", "uniform", "wide"))}
    if kind == "host":
        M, N, K = (_log_int(rng, 512, 4096) for _ in range(3))
        return {"kind": "host", "mode": rng.choice(("bf16x3", "bf16x3", "tf32x3")), "M": M, "N": N, "K": K,
                "alpha": alpha, "beta": beta, "dist": "uniform"}
    if kind == "grouped":
        return {"kind": "grouped", "mode": rng.choice(("bf16x3", "bf16x3", "tf32x3")), "count": _log_int(rng, 16, 512),
                "lo": 32, "hi": rng.choice((256, 512, 1024)), "alpha": 1.0, "beta": rng.choice((0.0, 1.0)),
                "shapes_seed": rng.randrange(1 << 20)}
    # convolutions: images of 16 to 512 pixels a side, filters 3x3 to 11x11,
    # at most the operations of the paper's layer
    C, K = rng.choice(((16, 16), (16, 32), (32, 32), (64, 64), (64, 128), (128, 128)))
    R = rng.choice((3, 3, 3, 5, 7, 9, 11))
    H, W = _log_int(rng, 28, 512), _log_int(rng, 28, 512)
    most = 32 * 512 * 512 * 16 * 16 * 9 / (H * W * C * K * R * R)
    batch = _log_int(rng, 1, max(1, min(64, int(most))))
    while batch * H * W * C * K * R * R > 32 * 512 * 512 * 16 * 16 * 9:
        H = max(1, H // 2)
    return {"kind": "conv", "mode": rng.choice(("bf16x3", "bf16x3", "tf32x3")), "batch": batch, "H": H, "W": W,
            "C": C, "K": K, "R": R, "S": R, "alpha": alpha, "beta": beta}


# ------------------------------------------------------------------- inputs
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _uniform(shape, gen):
    return torch.rand(shape, generator=gen, device="cuda", dtype=torch.float32).mul_(2.0).sub_(1.0)


def _values(shape, gen, dist):
    """uniform: iid in [-1, 1); wide: random signs times 2^u, u in [-10, 10)."""
    x = _uniform(shape, gen)
    if dist == "wide":
        x = torch.sign(x) * torch.exp2(_uniform(shape, gen).mul_(10.0))
    return x


def _stored(case):
    """Shapes of A, B and C as stored."""
    M, N, K = case["M"], case["N"], case["K"]
    ta, tb = case.get("trans_a", False), case.get("trans_b", False)
    return ((K, M) if ta else (M, K)), ((N, K) if tb else (K, N)), (M, N)


def _operands(case, seed):
    g = _generator(seed)
    return [_values(s, g, case["dist"]) for s in _stored(case)]


def _group_shapes(case):
    """(M, N, K) of a grouped call, each spread over its logarithm in [lo, hi]."""
    g = torch.Generator().manual_seed(case["shapes_seed"])
    u = torch.rand((case["count"], 3), generator=g, dtype=torch.float64)
    lo, hi = math.log(case["lo"]), math.log(case["hi"])
    return [tuple(int(x) for x in row) for row in torch.exp(lo + (hi - lo) * u).round().long()]


def _group_operands(case, seed):
    """All matrices of a group in three flat buffers, each matrix on a 256-byte
    boundary, and views of the single ones."""
    g = _generator(seed)
    shapes = _group_shapes(case)
    flats, views = [], []
    for dims in (lambda m, n, k: (m, k), lambda m, n, k: (k, n), lambda m, n, k: (m, n)):
        sizes = [dims(*s) for s in shapes]
        starts, total = [], 0
        for r, c in sizes:
            starts.append(total)
            total += (r * c + 63) // 64 * 64
        flat = torch.zeros(total, device="cuda")
        v = [flat[o:o + r * c].view(r, c) for o, (r, c) in zip(starts, sizes)]
        values = _uniform((total,), g)
        for x, o in zip(v, starts):
            x.copy_(values[o:o + x.numel()].view_as(x))
        flats.append(flat)
        views.append(v)
    return shapes, flats, views


def _conv_operands(case, seed):
    g = _generator(seed)
    n, H, W, C, K, R, S = (case[k] for k in ("batch", "H", "W", "C", "K", "R", "S"))
    x = _uniform((n, H, W, C), g)
    f = _uniform((R, S, C, K), g)
    out = _uniform((n, H, W, K), g)
    return x, f, out


# ------------------------------------------------------------------- passes
def prepare(case, seed):
    kind = case["kind"]
    if kind == "gemm":
        A, B, C = _operands(case, seed)
        plan = None
        if case["trans_a"] or case["trans_b"]:
            plan = gemm_lib.Plan(case["M"], case["N"], case["K"], mode=case["mode"], trans_a=case["trans_a"],
                                 trans_b=case["trans_b"])
        return {"case": case, "A": A, "B": B, "C": C, "plan": plan}
    if kind == "host":
        A, B, C = (t.cpu().pin_memory() for t in _operands(case, seed))
        return {"case": case, "A": A, "B": B, "C": C}
    if kind == "grouped":
        shapes, flats, (As, Bs, Cs) = _group_operands(case, seed)
        plan = gemm_lib.GroupedPlan(shapes, mode=case["mode"])
        n = len(shapes)
        plan.prepare(As, Bs, Cs, [case["alpha"]] * n, [case["beta"]] * n)
        return {"case": case, "plan": plan, "flats": flats}
    x, f, out = _conv_operands(case, seed)
    plan = gemm_lib.ConvPlan(case["batch"], case["H"], case["W"], case["C"], case["K"], case["R"], case["S"],
                             mode=case["mode"])
    return {"case": case, "plan": plan, "x": x, "f": f, "out": out}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "gemm":
        if state["plan"] is not None:
            return state["plan"].execute(state["A"], state["B"], state["C"], case["alpha"], case["beta"])
        return gemm_lib.gemm(state["A"], state["B"], state["C"], case["alpha"], case["beta"], mode=case["mode"])
    if kind == "host":
        return gemm_lib.gemm_host(state["A"], state["B"], state["C"], case["alpha"], case["beta"], mode=case["mode"])
    if kind == "grouped":
        state["plan"].execute()
        return state["flats"][2]
    return state["plan"].execute(state["x"], state["f"], state["out"], case["alpha"], case["beta"])


def _products(case):
    """(M, N, K) of every product of a pass."""
    if case["kind"] == "grouped":
        return _group_shapes(case)
    return [(case["M"], case["N"], case["K"])]


def work(case):
    """Operands read once, the result written once (and read once when beta is
    not 0); two operations a multiply-add of the defining product."""
    out = 4 if case["beta"] == 0.0 else 8
    if case["kind"] == "conv":
        n, H, W, C, K, R, S = (case[k] for k in ("batch", "H", "W", "C", "K", "R", "S"))
        pix = n * H * W
        return {"bytes": 4 * (pix * C + R * S * C * K) + out * pix * K, "flops": 2 * pix * R * S * C * K}
    shapes = _products(case)
    return {"bytes": sum(4 * (m * k + k * n) + out * m * n for m, n, k in shapes),
            "flops": sum(2 * m * n * k for m, n, k in shapes)}


# -------------------------------------------------------------------- exact
def exact(case, seed):
    alpha, beta = case["alpha"], case["beta"]
    if case["kind"] in ("gemm", "host"):
        A, B, C = _operands(case, seed)
        A = (A.t() if case.get("trans_a") else A).double()
        B = (B.t() if case.get("trans_b") else B).double()
        out = torch.matmul(A, B).mul_(alpha)
        if beta != 0.0:
            out.add_(C.double(), alpha=beta)
        return out.cpu() if case["kind"] == "host" else out
    if case["kind"] == "grouped":
        _, flats, (As, Bs, Cs) = _group_operands(case, seed)
        out = torch.zeros(flats[2].numel(), dtype=torch.float64, device="cuda")
        for a, b, c in zip(As, Bs, Cs):
            at = c.storage_offset()
            r = torch.matmul(a.double(), b.double()).mul_(alpha)
            if beta != 0.0:
                r.add_(c.double(), alpha=beta)
            out[at:at + c.numel()] = r.reshape(-1)
        return out
    x, f, out0 = _conv_operands(case, seed)
    n, H, W, C = x.shape
    R, S, _, K = f.shape
    pad = torch.nn.functional.pad(x.double(), (0, 0, S // 2, S // 2, R // 2, R // 2))
    acc = torch.zeros((n * H * W, K), dtype=torch.float64, device="cuda")
    for r in range(R):
        for s in range(S):
            acc.addmm_(pad[:, r:r + H, s:s + W].reshape(-1, C), f[r, s].double())
    acc.mul_(alpha)
    if beta != 0.0:
        acc.add_(out0.reshape(-1, K).double(), alpha=beta)
    return acc.view(n, H, W, K)
