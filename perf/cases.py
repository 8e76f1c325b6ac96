"""The calls whose speed is measured, and how their results are judged.

Each case is one call (or one short chain of calls) that a program using this
library makes through its Python entry points, with the buffers, descriptors
and workspaces such a program keeps between calls:

  dynamic      one activation tensor, global scale computed in the call
  group        all weights of a layer (or K, V, Q) in one call, scales computed in it
  static       one tensor at a global scale the program already has
  simulate     simulated quantisation: global scale, AbsMax, dequantisation to bf16
  four_six     the 4/6 baseline at a known global scale
  optimal      the optimal-scale study of a weight slice
  ldlq_prepare the Hessian factorisation of the LDLQ (GPTQ) pass
  ldlq         the LDLQ pass of one weight

Sizes are those of the repository's own synthetic workloads and of ordinary
model layers; `draw` spreads over the same ranges, odd sizes among them.
"""
import math

import torch

from paper_2606_07618_gb300 import binding as B
from paper_2606_07618_gb300.step import QuantizeStep

WIN = B.NVFP4_WINDOW_DEFAULT
MSE, WMSE = B.NVFP4_OBJ_MSE, B.NVFP4_OBJ_WMSE


def listed():
    return [
        # a decode batch: one activation of 16 tokens, scaled per call
        {"name": "dynamic_decode", "kind": "dynamic", "rows": 16, "cols": 4096, "obj": "mse", "block": 16, "dt": "bf16"},
        # a prefill batch: 8192 tokens of hidden size 4096, scaled per call
        {"name": "dynamic_prefill", "kind": "dynamic", "rows": 8192, "cols": 4096, "obj": "mse", "block": 16,
         "dt": "bf16"},
        # all linear weights of an 8B layer (4096 / 14336, k and v of 1024 rows), weighted by channel importance
        {"name": "group_layer", "kind": "group", "rows": 4096, "cols": 4096, "shape": "layer", "obj": "wmse",
         "block": 16, "dt": "bf16"},
        # the two MLP matrices of a 72B layer: the largest call
        {"name": "group_largest", "kind": "group", "rows": 8192, "cols": 29568, "shape": "pair", "obj": "wmse",
         "block": 16, "dt": "bf16"},
        # K, V and Q of a batch (head size 128; Q has four times the heads), unweighted
        {"name": "group_kvq", "kind": "group", "rows": 131072, "cols": 128, "shape": "kvq", "obj": "mse", "block": 16,
         "dt": "bf16"},
        # one weight with blocks of 32, one tensor to the call
        {"name": "group_block32", "kind": "group", "rows": 8192, "cols": 29568, "shape": "one", "obj": "mse",
         "block": 32, "dt": "bf16"},
        # an fp32 master weight of ragged size at a known scale, with the loss of every block
        {"name": "static_f32_ragged", "kind": "static", "rows": 3001, "cols": 2832, "obj": "wmse", "block": 16,
         "dt": "f32"},
        # simulated quantisation of one MLP weight (what an accuracy study runs over a model)
        {"name": "simulate_absmax", "kind": "simulate", "rows": 14336, "cols": 4096, "obj": "mse", "block": 16,
         "dt": "bf16"},
        # the 4/6 baseline on a square weight
        {"name": "four_six", "kind": "four_six", "rows": 8192, "cols": 8192, "obj": "wmse", "block": 16, "dt": "bf16"},
        # the scale study: distance to the best real scale on a slice of a weight
        {"name": "optimal_study", "kind": "optimal", "rows": 512, "cols": 8192, "obj": "wmse", "block": 16,
         "dt": "bf16"},
        # LDLQ of a 4096-wide layer: the factor once per Hessian, the pass once per weight
        {"name": "ldlq_prepare", "kind": "ldlq_prepare", "rows": 4096, "cols": 4096, "obj": "wmse", "block": 16,
         "dt": "bf16"},
        {"name": "ldlq_weight", "kind": "ldlq", "rows": 4096, "cols": 4096, "obj": "wmse", "block": 16, "dt": "bf16"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cols(rng, lo, hi, block):
    return max(1, round(_log(rng, lo, hi) / block)) * block


def draw(rng):
    kind = rng.choice(["dynamic", "dynamic", "group", "group", "group", "static", "static", "simulate", "four_six",
                       "optimal", "ldlq_prepare", "ldlq"])
    block = rng.choice([16, 16, 32, 64])
    dt = rng.choice(["bf16", "bf16", "bf16", "f32"])
    obj = rng.choice(["mse", "wmse"])
    if kind == "dynamic":
        return {"kind": kind, "rows": _log(rng, 1, 8192), "cols": _cols(rng, 512, 4096, block), "obj": obj,
                "block": block, "dt": dt}
    if kind == "group":
        shape = rng.choice(["layer", "pair", "kvq", "one"])
        if shape == "kvq":
            return {"kind": kind, "rows": _log(rng, 512, 131072), "cols": rng.choice([64, 128]), "shape": shape,
                    "obj": obj, "block": block, "dt": dt}
        if shape == "layer":
            return {"kind": kind, "rows": 0, "cols": 64 * _log(rng, 16, 64), "shape": shape, "obj": obj,
                    "block": block, "dt": dt}
        return {"kind": kind, "rows": _log(rng, 256, 8192), "cols": _cols(rng, 1024, 14784, block), "shape": shape,
                "obj": obj, "block": block, "dt": dt}
    if kind in ("static", "simulate", "four_six"):
        return {"kind": kind, "rows": _log(rng, 16, 8192), "cols": _cols(rng, 512, 8192, block),
                "obj": "mse" if kind == "simulate" else obj, "block": block, "dt": dt}
    if kind == "optimal":
        return {"kind": kind, "rows": _log(rng, 16, 512), "cols": _cols(rng, 512, 4096, 16), "obj": obj, "block": 16,
                "dt": dt}
    n = _cols(rng, 256, 4096, 16)
    rows = n if kind == "ldlq_prepare" else _log(rng, 512, 4096)
    return {"kind": kind, "rows": rows, "cols": n, "obj": "wmse", "block": 16, "dt": dt}


def _shapes(case):
    r, c = case["rows"], case["cols"]
    shape = case.get("shape", "one")
    if shape == "layer":      # q, k, v, o, gate, up, down of a layer with hidden size c
        kv, ff = c // 4, c * 7 // 2
        return [(c, c), (kv, c), (kv, c), (c, c), (ff, c), (ff, c), (c, ff)]
    if shape == "pair":
        return [(r, c), (c - c % case["block"], r - r % case["block"])]
    if shape == "kvq":
        return [(r, c), (r, c), (4 * r, c)]
    return [(r, c)]


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _values(case, rows, cols, g):
    """The repository's synthetic distributions: activations are Student-t(3)
    with 16 large channels, K/V/Q normal with a factor per head, weights
    Laplace with 0.1% large input channels."""
    if case["kind"] == "dynamic":
        x = torch.randn(rows, cols, device="cuda", generator=g)
        chi = torch.zeros(rows, cols, device="cuda")
        for _ in range(3):
            chi += torch.randn(rows, cols, device="cuda", generator=g).square_()
        x /= (chi / 3.0).sqrt_()
        at = torch.randperm(cols, device="cuda", generator=g)[:16]
        x[:, at] *= 50.0
    elif case.get("shape") == "kvq":
        x = torch.randn(rows, cols, device="cuda", generator=g)
        heads = torch.exp(0.5 * torch.randn(8, device="cuda", generator=g))
        x *= heads[torch.arange(rows, device="cuda") * 8 // rows].unsqueeze(1)
    else:
        x = torch.rand(rows, cols, device="cuda", generator=g).clamp_(min=2.0 ** -25).sub_(0.5)
        sign = torch.sign(x)
        x = x.abs_().mul_(-2.0).log1p_().mul_(-0.015).mul_(sign)
        at = torch.randperm(cols, device="cuda", generator=g)[: max(1, cols // 1000)]
        x[:, at] *= 20.0
    return x if case["dt"] == "f32" else x.to(torch.bfloat16)


def _importance(cols, g):
    return torch.exp(torch.randn(cols, device="cuda", generator=g))


def _hessian(n, g):
    """Gram matrix of 256 calibration directions plus a diagonal, with
    lognormal channel scales (symmetric)."""
    scale = torch.exp(0.8 * torch.randn(n, device="cuda", generator=g))
    A = torch.randn(n, 256, device="cuda", generator=g) * scale[:, None]
    H = A.double() @ A.double().T / 256 + torch.diag(scale.double().square() * 0.05)
    return H.float()


def _udu64(H, damp=0.01):
    """perm, U, D of (U + I) D (U + I)^T = H[perm][:, perm] + damp * mean(diag H) in 64 bits."""
    d = torch.diagonal(H).double()
    perm = torch.argsort(d, descending=True, stable=True)
    Hp = H.double()[perm][:, perm]
    Hp.diagonal().add_(damp * float(d.mean()))
    L = torch.linalg.cholesky(Hp.flip(0, 1))
    R = L.flip(0, 1)
    diag = torch.diagonal(R).clone()
    U = torch.triu(R / diag[None, :], 1)
    return perm.to(torch.int32), U, diag.square()


def _inputs(case, seed):
    """Everything that depends on the seed, without this repository's code."""
    g = _gen(seed)
    if case["kind"] == "ldlq_prepare":
        return {"H": _hessian(case["cols"], g)}
    xs = [_values(case, r, c, g) for r, c in _shapes(case)]
    ws = [_importance(c, g) if case["obj"] == "wmse" else None for _, c in _shapes(case)]
    return {"xs": xs, "ws": ws}


def _scale(x, D=256.0):
    amax = x.abs().max().float()
    return (amax / torch.tensor(6.0 * D, device=x.device)).reshape(1)


def prepare(case, seed):
    kind, block = case["kind"], case["block"]
    obj = WMSE if case["obj"] == "wmse" else MSE
    v = _inputs(case, seed)
    s = {"kind": kind, "block": block, "obj": obj}
    if kind in ("dynamic", "group"):
        s["step"] = QuantizeStep(v["xs"], v["ws"], block=block, objective=obj, activation=kind == "dynamic")
        return s
    if kind == "ldlq_prepare":
        n = case["cols"]
        s.update(H=v["H"], perm=torch.empty(n, dtype=torch.int32, device="cuda"), U=torch.empty(n, n, device="cuda"),
                 D=torch.empty(n, device="cuda"), status=torch.zeros(1, dtype=torch.int32, device="cuda"),
                 ws=torch.empty(B.nvfp4_ldlq_prepare_workspace(n), dtype=torch.uint8, device="cuda"))
        return s
    x, w = v["xs"][0], v["ws"][0]
    rows, cols = x.shape
    s.update(x=x, w=w, S=_scale(x))
    if kind == "ldlq":
        g = _gen(seed + 1)
        H = _hessian(cols, g)
        perm, U, _ = _udu64(H)
        sf = torch.empty(rows, cols // block, dtype=torch.uint8, device="cuda")
        codes = torch.empty(rows, cols // 2, dtype=torch.uint8, device="cuda")
        B.scalesweep_quantize(x, block, s["S"], WMSE, torch.diagonal(H).contiguous(), 0, WIN, WIN, codes, sf)
        s.update(perm=perm, U=U.float(), sf=sf, codes=codes, status=torch.zeros(1, dtype=torch.int32, device="cuda"),
                 ws=torch.empty(B.nvfp4_ldlq_workspace(rows, cols), dtype=torch.uint8, device="cuda"))
        return s
    if kind == "optimal":
        nb = rows * cols // block
        s.update(s_opt=torch.empty(nb, device="cuda"), loss=torch.empty(nb, device="cuda"),
                 code=torch.empty(nb, dtype=torch.uint8, device="cuda"), loss_fp8=torch.empty(nb, device="cuda"))
        return s
    s["out"] = B.empty_outputs(rows, cols, block, linear=True, swizzled=block == 16, loss=kind != "simulate")
    if kind == "simulate":
        s.update(deq=torch.empty(rows, cols, dtype=torch.bfloat16, device="cuda"),
                 ws=torch.empty(B.nvfp4_global_scale_workspace(x.numel()), dtype=torch.uint8, device="cuda"))
    return s


def run(s):
    kind, block = s["kind"], s["block"]
    if kind in ("dynamic", "group"):
        step = s["step"]
        step()
        return {"S": step.S, "status": step.status, "outs": step.outs}
    if kind == "ldlq_prepare":
        B.nvfp4_ldlq_prepare(s["H"], 0.01, s["perm"], s["U"], s["D"], s["status"], s["ws"])
        return {"perm": s["perm"], "U": s["U"], "D": s["D"], "status": s["status"]}
    if kind == "ldlq":
        B.ldlq_quantize(s["x"], block, s["S"], s["sf"], s["perm"], s["U"], s["codes"], s["status"], s["ws"])
        return {"codes": s["codes"], "status": s["status"]}
    if kind == "optimal":
        B.nvfp4_optimal_scale(s["x"], block, s["S"], s["obj"], s["w"], 0, s["s_opt"], s["loss"], s["code"],
                              s["loss_fp8"])
        return {"s_opt": s["s_opt"], "loss": s["loss"], "code": s["code"], "loss_fp8": s["loss_fp8"]}
    o = s["out"]
    if kind == "static":
        B.scalesweep_quantize(s["x"], block, s["S"], s["obj"], s["w"], 0, WIN, WIN, o["codes"], o["sf_linear"],
                              o["sf_swizzled"], o["block_loss"])
    elif kind == "four_six":
        B.four_over_six_quantize(s["x"], block, s["S"], s["obj"], s["w"], 0, o["codes"], o["sf_linear"],
                                 o["sf_swizzled"], o["block_loss"])
    else:
        x = s["x"]
        B.nvfp4_global_scale(x, 256.0, s["S"], None, s["ws"])
        B.absmax_quantize(x, block, s["S"], o["codes"], o["sf_linear"], o["sf_swizzled"])
        B.nvfp4_dequantize(o["codes"], o["sf_linear"], B.NVFP4_SF_LINEAR, s["S"], x.shape[0], x.shape[1], block,
                           s["deq"])
        return {"S": s["S"], "out": o, "deq": s["deq"]}
    return {"out": o}


def work(case):
    """Inputs read once and outputs written once.  The sweeps' own operations
    depend on how many scale candidates an implementation has to score, so only
    the LDLQ entry points, whose sums are fixed, and the study state any."""
    kind, block = case["kind"], case["block"]
    n = sum(r * c for r, c in _shapes(case))
    size = 4 if case["dt"] == "f32" else 2
    layouts = 2 if block == 16 else 1
    weights = sum(4 * c for _, c in _shapes(case)) if case["obj"] == "wmse" else 0
    if kind == "ldlq_prepare":
        c = case["cols"]
        return {"bytes": 8 * c * c + 8 * c, "flops": 2 * c ** 3 / 3}
    if kind == "ldlq":
        r, c = case["rows"], case["cols"]
        return {"bytes": r * c * (size + 0.5 + 1 / block) + 2 * c * c, "flops": r * c * c}
    if kind == "optimal":
        # one trial assignment for each of the 7 rounding midpoints of each element of a block
        return {"bytes": n * size + weights + n // block * 13, "flops": n * 7 * block * 8}
    out = n * (0.5 + layouts / block)
    if kind == "simulate":
        return {"bytes": n * size + out + 2 * n, "flops": 0}
    if kind in ("static", "four_six"):
        out += 4 * n // block
    return {"bytes": n * size + weights + out, "flops": 0}


def tolerance(case):
    """About four times what the same call differs by with its sums in another
    order: the elements of every block reversed (static, four_six, optimal), or
    the fp32-pipe updates in place of the tensor-core ones (ldlq_prepare, ldlq;
    there a target next to a rounding boundary flips, and the rest of its row
    follows, on up to 1% of the rows)."""
    kind = case["kind"]
    if kind in ("static", "four_six"):     # measured: rel 6.5e-8, max 3e-7 (fp32 losses)
        return {"rel": 3e-7, "max": 1.2e-6}
    if kind == "optimal":                  # measured: rel 4.5e-6, max 2.3e-3 (a scale on the other of two equal segments)
        return {"rel": 2e-5, "max": 9e-3}
    if kind == "ldlq_prepare":             # measured: rel 1.5e-5, max 5.6e-5
        return {"rel": 6e-5, "max": 2.2e-4}
    if kind == "ldlq":                     # measured: 1.1e-3 of the bytes
        return {"differ": 4.4e-3}
    return "exact"


# ------------------------------------------------------------------ the same in 64 bits
_CODES = [(1.0 + (c & 7) / 8.0) * 2.0 ** ((c >> 3) - 7) if c >= 8 else c * 2.0 ** -9 for c in range(127)]
_MIDS = [0.25, 0.75, 1.25, 1.75, 2.5, 3.5, 5.0]
_GRID = [0.0, 0.5, 1.0, 1.5, 2.0, 3.0, 4.0, 6.0]


def _nearest(t):
    """Nearest E2M1 magnitude of t >= 0 (a tie's side does not change a loss)."""
    mids = torch.tensor(_MIDS, dtype=torch.float64, device=t.device)
    grid = torch.tensor(_GRID, dtype=torch.float64, device=t.device)
    return grid[torch.bucketize(t, mids)]


def _blocks(case, v):
    """[blocks, block] magnitudes in units of the global scale, and their weights."""
    x, w, block = v["xs"][0], v["ws"][0], case["block"]
    rows, cols = x.shape
    a = (x.double().abs() / _scale(x).double()).reshape(-1, block)
    if w is None:
        return a, torch.ones_like(a)
    return a, w.double().reshape(1, -1).expand(rows, cols).reshape(-1, block)


def _loss(a, w, s):
    e = a - _nearest(a / s[:, None]) * s[:, None]
    return (w * e * e).sum(1)


def _study64(a, w):
    """Least sum w (a - s q)^2 over real s: every midpoint of every element
    starts a segment on which the rounding is fixed."""
    best = (w * a * a).sum(1)
    for i in range(a.shape[1]):
        for k, mid in enumerate(_MIDS):
            s = a[:, i] / mid
            q = _nearest(a / s.clamp_min(1e-300)[:, None] * (1 - 1e-9))
            q[:, i] = _GRID[k]
            b, c = (w * a * q).sum(1), (w * q * q).sum(1)
            s = torch.where(c > 0, b / c.clamp_min(1e-300), torch.zeros_like(b))
            e = a - s[:, None] * q
            best = torch.minimum(best, torch.where(a[:, i] > 0, (w * e * e).sum(1), best))
    return best


def exact(case, seed):
    kind = case["kind"]
    v = _inputs(case, seed)
    if kind == "ldlq_prepare":
        perm, U, D = _udu64(v["H"])
        return {"perm": perm, "U": U, "D": D, "status": None}
    if kind in ("dynamic", "group"):
        S = torch.stack([x.abs().max().double() / (6.0 * 256.0) for x in v["xs"]])
        return {"S": S, "status": None, "outs": None}
    if kind == "optimal":
        a, w = _blocks(case, v)
        return {"s_opt": None, "loss": _study64(a, w), "code": None, "loss_fp8": None}
    if kind == "simulate":
        return {"S": v["xs"][0].abs().max().double().reshape(1) / (6.0 * 256.0), "out": None, "deq": None}
    if kind == "ldlq" or v["xs"][0].numel() > 1 << 24:
        return None
    # the loss of the chosen scale code of each block
    a, w = _blocks(case, v)
    codes = torch.tensor(_CODES, dtype=torch.float64, device=a.device)
    m = a.max(1).values
    if kind == "static":
        i0 = torch.bucketize(m / 6.0, codes, right=True) - 1
        best = torch.full_like(m, math.inf)
        for off in range(-3 if case["obj"] == "mse" and case["block"] == 16 else -8, 8):
            c = (i0 + off).clamp(1, 126)
            best = torch.minimum(best, _loss(a, w, codes[c]))
    else:
        best = torch.full_like(m, math.inf)
        for top in (6.0, 4.0):
            s = (m / top).float().clamp(max=448.0).to(torch.float8_e4m3fn).double().clamp_min(2.0 ** -9)
            best = torch.minimum(best, _loss(a, w, s))
    best = torch.where(m > 0, best, torch.zeros_like(best))
    return {"out": {"codes": None, "sf_linear": None, "sf_swizzled": None, "block_loss": best}}
