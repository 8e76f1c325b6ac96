"""Paths chosen by size or range, against the general ones, bit for bit.

* One-cluster dynamic-scale launch (up to 4096 segments) against the global scale
  and the static sweep as two calls, at the edges of a CTA, of the portable and of
  the largest cluster, and one segment past it, with ragged swizzled scales.
* Default windows, whose codes are scored an octave apart where they are normal (WMSE)
  and whose low end is left out once saturated terms rule it out, against the same
  codes scored one call each, with block scales from the smallest code to the largest.
* The screened optimal scale against every segment scored.
* Zeroed padding of the swizzled layout at rows and columns off its atoms.
"""
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_07618_gb300 import binding
    binding.lib()
    return binding


def _tensor(rows, cols, dt, seed, special=False):
    g = torch.Generator().manual_seed(seed)
    x = torch.randn(rows, cols, generator=g) * torch.exp(torch.randn(rows, cols, generator=g))
    if special:
        x[0, 3], x[-1, -1] = float("nan"), float("-inf")
    return x.to(dt).to(DEV)


def _outs(B, x, block, swizzled):
    o = B.empty_outputs(x.shape[0], x.shape[1], block, device=DEV, linear=True, swizzled=swizzled, loss=True)
    for t in o.values():
        if t is not None:
            t.fill_(7)
    return o


def _same(a, b):
    for k, v in a.items():
        if v is not None:
            assert torch.equal(v, b[k]) or torch.equal(v.nan_to_num(-1.0), b[k].nan_to_num(-1.0)), k


# segments: one, a CTA and one more, 8 CTAs and one more, 16 CTAs and one more
@pytest.mark.parametrize("rows,cols", [(1, 16), (1, 64), (8, 512), (257, 16), (64, 512), (2049, 16), (16, 4096),
                                       (4097, 16), (3, 1360)])
@pytest.mark.parametrize("obj", [0, 1])
@pytest.mark.parametrize("dt", [torch.bfloat16, torch.float32])
def test_cluster_launch(B, rows, cols, obj, dt):
    for block in (16, 64):
        if cols % block:
            continue
        for special in (False, True):
            x = _tensor(rows, cols, dt, rows + cols, special)
            w = torch.rand(cols, generator=torch.Generator().manual_seed(3)).to(DEV) if obj else None
            win = (B.NVFP4_WINDOW_DEFAULT, B.NVFP4_WINDOW_DEFAULT)
            S, S2 = torch.zeros(1, device=DEV), torch.zeros(1, device=DEV)
            st, st2 = (torch.zeros(1, dtype=torch.int32, device=DEV) for _ in range(2))
            ws = torch.empty(B.nvfp4_dynamic_workspace(), dtype=torch.uint8, device=DEV)
            gws = torch.empty(B.nvfp4_global_scale_workspace(x.numel()), dtype=torch.uint8, device=DEV)
            a, b = _outs(B, x, block, block == 16), _outs(B, x, block, block == 16)
            B.scalesweep_quantize_dynamic(x, block, 256.0, obj, w, 0, *win, S, st, ws, a["codes"], a["sf_linear"],
                                          a["sf_swizzled"], a["block_loss"])
            B.nvfp4_global_scale(x, 256.0, S2, st2, gws)
            B.scalesweep_quantize(x, block, S2, obj, w, 0, *win, b["codes"], b["sf_linear"], b["sf_swizzled"],
                                  b["block_loss"])
            torch.cuda.synchronize()
            assert torch.equal(S, S2) and torch.equal(st, st2)
            _same(a, b)


def _one_code_at_a_time(B, x, block, S, obj, w, lo):
    """Losses and linear outputs of the window's codes, each scored by a call whose
    window holds that code alone, folded on the host side: lowest code on ties."""
    best = None
    for d in range(lo, 8):
        o = _outs(B, x, block, False)
        B.scalesweep_quantize(x, block, S, obj, w, 0, d, d, o["codes"], o["sf_linear"], None, o["block_loss"])
        rows, kb = o["sf_linear"].shape if o["sf_linear"].dim() == 2 else (x.shape[0], x.shape[1] // block)
        loss, sf = o["block_loss"].view(rows, kb), o["sf_linear"].view(rows, kb)
        codes = o["codes"].view(rows, kb, block // 2)
        if best is None:
            best = [loss, sf, codes]
        else:
            m = loss < best[0]
            best = [torch.where(m, loss, best[0]), torch.where(m, sf, best[1]),
                    torch.where(m[..., None], codes, best[2])]
    return best


@pytest.mark.parametrize("dt", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("block", [16, 32, 64])
@pytest.mark.parametrize("weights", [None, "positive", "mixed", "negative"])
def test_window_against_single_codes(B, dt, block, weights):
    """Octave pairs and the end of the walk down: block maxima from below the smallest
    code to above the largest, uniform over a warp and mixed within one, with heavy
    tails (many terms saturate); negative weights allow neither skips nor an end."""
    g = torch.Generator().manual_seed(11)
    rows, cols = 512, 512
    scale = torch.exp2(torch.linspace(-14.0, 14.0, rows))[:, None]
    mixed = torch.exp2(torch.randint(-12, 12, (rows, cols // 16, 1), generator=g).float()).expand(-1, -1, 16)
    tails = torch.exp(torch.randn(rows, cols, generator=g))
    w = None
    if weights:
        w = torch.exp(torch.randn(cols, generator=g))
        w = {"positive": w, "mixed": w * torch.where(torch.arange(cols) % 96 < 80, 1.0, -1.0), "negative": -w}[weights]
        w = w.to(DEV)
    obj = 1 if weights else 0
    lo = -3 if (block == 16 and not weights) else -8
    S = torch.tensor([0.25], device=DEV)
    for s in (scale, mixed.reshape(rows, cols), scale * tails):
        x = (torch.randn(rows, cols, generator=g) * s).to(dt).to(DEV)
        a = _outs(B, x, block, False)
        B.scalesweep_quantize(x, block, S, obj, w, 0, *(B.NVFP4_WINDOW_DEFAULT,) * 2, a["codes"], a["sf_linear"], None,
                              a["block_loss"])
        gr = _outs(B, x, block, False)
        desc = B.group_descriptors([x], [w], [0], [gr["codes"]], [gr["sf_linear"]], [None])
        B.scalesweep_quantize_group(desc, B.NVFP4_IN_BF16 if dt == torch.bfloat16 else B.NVFP4_IN_F32, obj, 0.0, S, None,
                                    None, block=block)
        loss, sf, codes = _one_code_at_a_time(B, x, block, S, obj, w, lo)
        torch.cuda.synchronize()
        fin = torch.isfinite(loss)
        if weights in ("mixed", "negative"):         # an offset outside the codes has no loss to compare
            o = _outs(B, x, block, False)
            B.scalesweep_quantize(x, block, S, obj, w, 0, 0, 0, o["codes"], o["sf_linear"], None, o["block_loss"])
            base = o["sf_linear"].view(loss.shape).int()
            fin &= (base + lo >= 1) & (base + 7 <= 126)
        assert fin.float().mean() > 0.4                # 14 of 28 octaves lie inside the codes
        shape = (rows, cols // block, -1)
        for o in (a, gr):
            assert torch.equal(o["sf_linear"].view(shape[:2])[fin], sf[fin])
            assert torch.equal(o["codes"].view(shape)[fin], codes[fin])
        assert torch.equal(a["block_loss"].view(shape[:2])[fin], loss[fin])


@pytest.mark.parametrize("rows,cols", [(1, 16), (127, 48), (129, 80), (130, 4112), (256, 64)])
def test_swizzle_padding(B, rows, cols):
    x = _tensor(rows, cols, torch.bfloat16, 5)
    S = torch.tensor([0.01], device=DEV)
    kb, kpad4 = cols // 16, -(-(cols // 16) // 4)
    o = _outs(B, x, 16, True)
    B.absmax_quantize(x, 16, S, o["codes"], o["sf_linear"], o["sf_swizzled"])
    torch.cuda.synchronize()
    want = torch.zeros_like(o["sf_swizzled"]).cpu()
    lin = o["sf_linear"].cpu()
    r, k = torch.meshgrid(torch.arange(rows), torch.arange(kb), indexing="ij")
    off = ((r // 128) * kpad4 + k // 4) * 512 + (r % 32) * 16 + (r // 32 % 4) * 4 + k % 4
    want[off.reshape(-1)] = lin.reshape(-1)
    assert torch.equal(o["sf_swizzled"].cpu(), want)


@pytest.mark.parametrize("block", [16, 32, 64])
@pytest.mark.parametrize("kind", ["normal", "tails", "equal", "few", "zero_weights"])
def test_optimal_screen(B, block, kind):
    """The screened optimum against every segment scored: weights times 2^100 are past
    the screen's range, and a power of two changes no rounding of the scored form."""
    g = torch.Generator().manual_seed(block)
    rows, cols = 64, 512
    x = torch.randn(rows, cols, generator=g)
    if kind == "tails":
        x = x * torch.exp(torch.randn(rows, cols, generator=g))
    elif kind == "equal":                              # every segment coincides: past the list
        x = torch.sign(x) * torch.arange(1, rows + 1)[:, None] / 16
    elif kind == "few":
        x = torch.sign(x) * torch.randint(0, 4, (rows, cols), generator=g)
    w = torch.exp(torch.randn(cols, generator=g))
    if kind == "zero_weights":
        w[torch.rand(cols, generator=g) < 0.6] = 0.0
    x, S = x.to(torch.bfloat16).to(DEV), torch.ones(1, device=DEV)
    nb = rows * cols // block
    res = []
    for f in (1.0, 2.0 ** 100):
        o = (torch.empty(nb, device=DEV), torch.empty(nb, device=DEV), torch.empty(nb, dtype=torch.uint8, device=DEV),
             torch.empty(nb, device=DEV))
        B.nvfp4_optimal_scale(x, block, S, 1, (w * f).to(DEV), 0, *o)
        res.append(o)
    torch.cuda.synchronize()
    (s1, l1, c1, f1), (s2, l2, c2, f2) = res
    assert torch.equal(s1, s2) and torch.equal(c1, c2)
    assert torch.equal(l1 * 2.0 ** 100, l2) and torch.equal(f1 * 2.0 ** 100, f2)


@pytest.mark.parametrize("block", [16, 32, 64])
@pytest.mark.parametrize("kind", ["normal", "tails", "few", "negative"])
def test_optimal_screen_unweighted(B, block, kind):
    """The MSE form's screen against equal weights of 2^100, which are past it; and
    (negative) blocks with a negative weight, which have no screen: their scale is that
    of the same weights times 2^100."""
    g = torch.Generator().manual_seed(block + 1)
    rows, cols = 64, 512
    x = torch.randn(rows, cols, generator=g)
    if kind == "tails":
        x = x * torch.exp(torch.randn(rows, cols, generator=g))
    elif kind == "few":
        x = torch.sign(x) * torch.randint(0, 4, (rows, cols), generator=g)
    x, S = x.to(torch.bfloat16).to(DEV), torch.ones(1, device=DEV)
    w = torch.ones(cols, device=DEV)
    if kind == "negative":
        w = torch.exp(torch.randn(cols, generator=g)).to(DEV)
        w[::block] *= -0.1
    nb = rows * cols // block
    res = []
    for obj, f in ((int(kind == "negative"), 1.0), (1, 2.0 ** 100)):
        o = (torch.empty(nb, device=DEV), torch.empty(nb, device=DEV), torch.empty(nb, dtype=torch.uint8, device=DEV),
             torch.empty(nb, device=DEV))
        B.nvfp4_optimal_scale(x, block, S, obj, w * f if obj else None, 0, *o)
        res.append(o)
    torch.cuda.synchronize()
    (s1, l1, c1, f1), (s2, l2, c2, f2) = res
    assert torch.equal(s1, s2) and torch.equal(c1, c2)
    assert torch.equal(l1 * 2.0 ** 100, l2) and torch.equal(f1 * 2.0 ** 100, f2)
