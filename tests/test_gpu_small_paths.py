"""Paths chosen by size or range, against the general ones, bit for bit.

* One-cluster dynamic-scale launch (up to 4096 segments) against the global scale
  and the static sweep as two calls, at the edges of a CTA, of the portable and of
  the largest cluster, and one segment past it, with ragged swizzled scales.
* Windows scored an octave apart (WMSE, every code from 8 to 126) against the same
  window given explicitly, with block scales from the smallest code to the largest.
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


@pytest.mark.parametrize("dt", [torch.bfloat16, torch.float32])
def test_octave_windows(B, dt):
    """Block maxima from below the smallest code to above the largest, several
    mixed in a warp and uniform over one."""
    g = torch.Generator().manual_seed(11)
    rows, cols = 512, 512
    scale = torch.exp2(torch.linspace(-14.0, 14.0, rows))[:, None]
    mixed = torch.exp2(torch.randint(-12, 12, (rows, cols // 16, 1), generator=g).float()).expand(-1, -1, 16)
    for s in (scale, mixed.reshape(rows, cols)):
        x = (torch.randn(rows, cols, generator=g) * s).to(dt).to(DEV)
        w = torch.exp(torch.randn(cols, generator=g)).to(DEV)
        S = torch.tensor([0.25], device=DEV)
        for block in (16, 32, 64):
            a, b = _outs(B, x, block, block == 16), _outs(B, x, block, block == 16)
            for o, win in ((a, (B.NVFP4_WINDOW_DEFAULT,) * 2), (b, (-8, 7))):
                B.scalesweep_quantize(x, block, S, 1, w, 0, *win, o["codes"], o["sf_linear"], o["sf_swizzled"],
                                      o["block_loss"])
            # the default window given explicitly takes the same path: one code wider on one side does not
            c = _outs(B, x, block, block == 16)
            B.scalesweep_quantize(x, block, S, 1, w, 0, -9, 7, c["codes"], c["sf_linear"], c["sf_swizzled"],
                                  c["block_loss"])
            torch.cuda.synchronize()
            _same(a, b)
            # a wider window changes a block only where its extra code wins
            keep = c["sf_linear"] == a["sf_linear"]
            assert float(keep.float().mean()) > 0.999
            assert torch.equal(a["block_loss"][keep.reshape(-1)], c["block_loss"][keep.reshape(-1)])


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
