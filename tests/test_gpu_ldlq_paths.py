"""LDLQ paths chosen by size and alignment.

* Row and column counts off the walk's tiles (32 rows, 64 and 256 columns) and off the
  update's (128, alone and in strips of two and four), with the walk scheduled beside
  the update and after it.
* A factor that is not 16-byte aligned: the same arithmetic, so the same codes.
* Rows too long for the gather's and the packer's shared memory: with a zero factor the
  codes are plain rounding.
* Factorizations off the panels of 64, with outputs that are not 16-byte aligned.
* The least workspaces, without the split operands: updates on the FP32 pipe.
* Sums of errors: kept where each is below the target's last place, and as close to 64
  bits as sums on the FP32 pipe.
* Dependencies of a captured pass: only a walk behind an update may start before it ends.
"""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from oracle import ldlq as L
from test_gpu_ldlq import B, DEV, conditional_parity, prepare, quantize  # noqa: F401
from test_oracle_ldlq import fixed_scales, rand_problem

pytestmark = pytest.mark.gpu


def _misaligned(t):
    out = torch.empty(t.numel() + 1, dtype=t.dtype, device=DEV)[1:].view(t.shape)
    out.copy_(t)
    assert out.data_ptr() % 16 != 0
    return out


@pytest.mark.parametrize("rows,cols", [(1, 16), (31, 272), (32, 320), (33, 528), (129, 784), (4900, 528), (24000, 1296)])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_walk_and_update_tiles(B, rows, cols, dtype):
    W64, H = rand_problem(rows, cols, rows + cols)
    Wt = torch.from_numpy(W64.astype(np.float32)).to(dtype)
    W = Wt.float().numpy().astype(np.float64)
    H = H.astype(np.float32).astype(np.float64)
    S, sf = fixed_scales(W, H)
    perm, U, _, st = prepare(B, H)
    assert st == 0
    codes, st = quantize(B, Wt.to(DEV), S, sf, perm, U)
    assert st == 0
    idx = np.unique(np.linspace(0, rows - 1, 130).astype(np.int64))        # first and last rows among them
    bad, exempt, total, first = conditional_parity(W[idx], S, sf[idx], 16, perm.cpu().numpy().astype(np.int64),
                                                   U.double().cpu().numpy(), codes[idx])
    assert bad == 0 and first == 0
    assert exempt <= max(2, total // 200)
    again, st = quantize(B, Wt.to(DEV), S, sf, perm, _misaligned(U))
    assert st == 0 and np.array_equal(codes, again)


# 4 rows of fp32 past 200 KB; of bf16; and of code bytes
@pytest.mark.parametrize("n,dtype", [(12784, torch.float32), (12816, torch.float32), (25616, torch.bfloat16),
                                     (51216, torch.float32)])
def test_long_rows(B, n, dtype):
    g = torch.Generator().manual_seed(n)
    rows = 5
    Wt = (torch.randn(rows, n, generator=g) * 0.02).to(dtype)
    sf = torch.randint(30, 80, (rows, n // 16), generator=g).to(torch.uint8).numpy()
    perm = torch.randperm(n, generator=g).to(torch.int32).to(DEV)
    U = torch.zeros(n, n, device=DEV)
    codes, st = quantize(B, Wt.to(DEV), 0.01, sf, perm, U)
    assert st == 0
    _, ref = oracle.block_losses_at(Wt.float().numpy(), 16, np.float32(0.01), sf, want_codes=True)
    assert np.array_equal(codes, ref)


@pytest.mark.parametrize("n", [1, 63, 65, 129, 193, 330, 580])
def test_least_factor_workspace(B, n):
    _, H = rand_problem(2, n, n)
    perm, U, D, _ = prepare(B, H)
    pb = _least(1, n)[0]
    w = _guarded(pb)
    perm2, U2, D2 = torch.empty_like(perm), torch.empty_like(U), torch.empty_like(D)
    st = torch.zeros(1, dtype=torch.int32, device=DEV)
    B.nvfp4_ldlq_prepare(torch.as_tensor(H, dtype=torch.float32, device=DEV), 0.01, perm2, U2, D2, st, w[:pb])
    torch.cuda.synchronize()
    assert st.item() == 0 and torch.all(w[pb:] == 0xA5)
    assert torch.equal(perm, perm2) and torch.all(torch.tril(U2) == 0)
    assert torch.allclose(D2, D, rtol=2e-4) and (U2 - U).abs().max() <= 2e-4 * max(1.0, float(U.abs().max()))


@pytest.mark.parametrize("n", [1, 63, 65, 128, 193, 330, 580])
def test_prepare_panels(B, n):
    _, H = rand_problem(2, n, n)
    H = H.astype(np.float32).astype(np.float64)
    Hd, perm_ref = L.damp_and_order(H)
    Hp = Hd[np.ix_(perm_ref, perm_ref)]
    U_ref, D_ref = L.udu(Hp)
    perm, U, D, st = prepare(B, H)
    Hm = _misaligned(torch.as_tensor(H, dtype=torch.float32))
    Um, Dm, permm = _misaligned(torch.zeros_like(U)), torch.empty_like(D), torch.empty_like(perm)
    stm = torch.zeros(1, dtype=torch.int32, device=DEV)
    ws = torch.empty(B.nvfp4_ldlq_prepare_workspace(n), dtype=torch.uint8, device=DEV)
    B.nvfp4_ldlq_prepare(Hm, 0.01, permm, Um, Dm, stm, ws)
    torch.cuda.synchronize()
    assert st == 0 and int(stm.item()) == 0
    for pg, Ug, Dg in ((perm, U, D), (permm, Um, Dm)):
        assert np.array_equal(pg.cpu().numpy(), perm_ref)
        Ug, Dg = Ug.double().cpu().numpy(), Dg.double().cpu().numpy()
        assert np.all(np.tril(Ug) == 0)
        # the bounds of the aligned factorization's test: fp32 rounding of n-term sums
        assert np.allclose(Dg, D_ref, rtol=2e-4)
        assert np.abs(Ug - U_ref).max() <= 2e-4 * max(1.0, np.abs(U_ref).max())
        R = (Ug + np.eye(n)) @ np.diag(Dg) @ (Ug + np.eye(n)).T - Hp
        assert np.abs(R).max() <= 2e-5 * np.abs(Hp).max()


def _guarded(nbytes):
    return torch.full((nbytes + 4096,), 0xA5, dtype=torch.uint8, device=DEV)


def _least(rows, n):
    up = lambda b: -(-b // 256) * 256
    return (up(4 * n) + 256 + 4 * 64 * 64,
            2 * up(4 * rows * n) + 2 * up(rows * n) + 2 * up(1024 * rows) + up(4 * n))


# one panel; a ragged second one; several, off and on multiples of 4; several super-panels
@pytest.mark.parametrize("rows,n", [(5, 64), (33, 80), (40, 304), (129, 784), (600, 1040)])
def test_least_workspaces(B, rows, n):
    W64, H = rand_problem(rows, n, rows * n)
    W = W64.astype(np.float32)
    S, sf = fixed_scales(W64, H)
    pb, qb = _least(rows, n)
    wp, wq = _guarded(pb), _guarded(qb)
    Hd = torch.as_tensor(H, dtype=torch.float32, device=DEV)
    perm, U, D, _ = prepare(B, Hd.double().cpu().numpy())     # with its full workspace
    perm2, U2, D2 = torch.empty_like(perm), torch.empty_like(U), torch.empty_like(D)
    codes = torch.empty(rows, n // 2, dtype=torch.uint8, device=DEV)
    st = torch.zeros(1, dtype=torch.int32, device=DEV)
    B.nvfp4_ldlq_prepare(Hd, 0.01, perm2, U2, D2, st, wp[:pb])
    sfd = torch.as_tensor(np.ascontiguousarray(sf), dtype=torch.uint8).to(DEV)
    B.ldlq_quantize(torch.from_numpy(W).to(DEV), 16, torch.tensor([S], dtype=torch.float32, device=DEV), sfd, perm2, U2,
                    codes, st, wq[:qb])
    torch.cuda.synchronize()
    assert st.item() == 0
    assert torch.all(wp[pb:] == 0xA5) and torch.all(wq[qb:] == 0xA5)
    assert torch.equal(perm, perm2) and torch.all(torch.tril(U2) == 0)
    # two fp32 factorizations of one matrix: the bounds of the tests against 64 bits
    assert torch.allclose(D2, D, rtol=2e-4) and (U2 - U).abs().max() <= 2e-4 * max(1.0, float(U.abs().max()))
    bad, exempt, total, first = conditional_parity(W.astype(np.float64), S, sf, 16, perm2.cpu().numpy().astype(np.int64),
                                                   U2.double().cpu().numpy(), codes.cpu().numpy())
    assert bad == 0 and first == 0 and exempt <= max(2, total // 200)


def programmatic_edges(graph):
    """How many of a captured graph's edges let a node start before the one ahead of it ends."""
    class Edge(ctypes.Structure):
        _fields_ = [("from_port", ctypes.c_ubyte), ("to_port", ctypes.c_ubyte), ("type", ctypes.c_ubyte),
                    ("reserved", ctypes.c_ubyte * 5)]

    get = ctypes.CDLL("libcuda.so.1").cuGraphGetEdges_v2
    h, n = ctypes.c_void_p(graph.raw_cuda_graph()), ctypes.c_size_t(0)
    assert get(h, None, None, None, ctypes.byref(n)) == 0 and n.value > 0
    src, dst, data = (ctypes.c_void_p * n.value)(), (ctypes.c_void_p * n.value)(), (Edge * n.value)()
    assert get(h, src, dst, data, ctypes.byref(n)) == 0
    return sum(e.type != 0 for e in data)


# super-panels of 256 columns; 64 rows: every walk but the first is scheduled beside an update
@pytest.mark.parametrize("cols,behind_update", [(256, 0), (528, 2)])
def test_first_walk_waits_for_the_gather(B, cols, behind_update):
    """The walk reads the gathered weights and scales before it waits for the grid ahead
    of it: the gather must have ended by then, so its edge is a full dependency."""
    rows = 64
    W64, H = rand_problem(rows, cols, cols)
    S, sf = fixed_scales(W64, H)
    Wt = torch.from_numpy(W64.astype(np.float32)).to(DEV)
    perm, U, _, _ = prepare(B, H)                             # also the first call on the device
    eager, _ = quantize(B, Wt, S, sf, perm, U)
    codes = torch.empty(rows, cols // 2, dtype=torch.uint8, device=DEV)
    st = torch.zeros(1, dtype=torch.int32, device=DEV)
    ws = torch.empty(B.nvfp4_ldlq_workspace(rows, cols), dtype=torch.uint8, device=DEV)
    Sd = torch.tensor([S], dtype=torch.float32, device=DEV)
    sfd = torch.as_tensor(np.ascontiguousarray(sf), dtype=torch.uint8).to(DEV)
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g, stream=s):
        B.ldlq_quantize(Wt, 16, Sd, sfd, perm, U, codes, st, ws, stream=s)
    assert programmatic_edges(g) == behind_update
    g.replay()
    torch.cuda.synchronize()
    assert st.item() == 0 and np.array_equal(codes.cpu().numpy(), eager)


# rows not a multiple of 4; a factor off 16 bytes
@pytest.mark.parametrize("rows,aligned", [(64, True), (33, True), (64, False)])
def test_small_errors_add_up(B, rows, aligned):
    """Every column's error is 2^-12 and reaches the columns k = 64, 128, 192 and 256
    with factor 2^-16: 2^-28 each, 1/32 of those targets' last place.  Column k lies
    k / 64 places below the boundary 1.25, which rounds down to 1; its errors, 2 k / 64
    places less 1/32 for each earlier k, take it above.  Every product and every sum of
    errors is exact."""
    cols, at = 272, [64, 128, 192, 256]
    W = torch.full((rows, cols), 1 + 2.0 ** -12)
    U = torch.zeros(cols, cols)
    for k in at:
        W[:, k] = 1.25 - k / 64 * 2.0 ** -23
        U[:k, k] = 2.0 ** -16
    U[at] = 0                                                 # their own errors go nowhere
    sf = np.full((rows, cols // 16), 56, dtype=np.uint8)      # E4M3 1.0
    perm = torch.arange(cols, dtype=torch.int32, device=DEV)
    Ud = U.to(DEV) if aligned else _misaligned(U)
    codes, st = quantize(B, W.to(DEV), 1.0, sf, perm, Ud)
    assert st == 0
    nib = np.stack([codes & 15, codes >> 4], axis=-1).reshape(rows, cols)
    want = np.full((rows, cols), 2)                           # E2M1 1.0
    want[:, at] = 3                                           # 1.5
    assert np.array_equal(nib, want)


def _factor64(H):
    perm = torch.argsort(torch.diagonal(H), descending=True, stable=True)
    Hp = H.double()[perm][:, perm]
    Hp.diagonal().add_(0.01 * float(torch.diagonal(H).double().mean()))
    R = torch.linalg.cholesky(Hp.flip(0, 1)).flip(0, 1)
    return perm, torch.triu(R / torch.diagonal(R)[None, :], 1).float()


@pytest.mark.parametrize("rows,cols", [(4096, 4096), (4095, 4096), (16384, 1040)])
def test_decisions_follow_64_bits(B, rows, cols):
    """How many codes differ from those of 64-bit targets formed from the same earlier
    codes.  A target with error d crosses a rounding boundary with probability rho d, rho
    the density of targets around the boundaries, so errors of 2^-22 of the rows' rms
    (2.4e-7; all sums on the FP32 pipe give 2.0e-7 at 4096 columns) flip about
    rho E|d| of them.  (Adding the 8-column sums to the targets one by one: 3 to 5
    times as many as that pipe's.)"""
    g = torch.Generator(device=DEV).manual_seed(rows + cols)
    scale = torch.exp(0.8 * torch.randn(cols, device=DEV, generator=g))
    A = torch.randn(cols, 256, device=DEV, generator=g) * scale[:, None]
    H = (A.double() @ A.double().T / 256 + torch.diag(scale.double() ** 2 * 0.05)).float()
    perm, U = _factor64(H)
    W = torch.randn(rows, cols, device=DEV, generator=g) * 0.02
    S = (W.abs().max() / 1536).reshape(1)
    win = (B.NVFP4_WINDOW_DEFAULT, B.NVFP4_WINDOW_DEFAULT)
    sf = torch.empty(rows, cols // 16, dtype=torch.uint8, device=DEV)
    codes = torch.empty(rows, cols // 2, dtype=torch.uint8, device=DEV)
    B.scalesweep_quantize(W, 16, S, B.NVFP4_OBJ_WMSE, torch.diagonal(H).contiguous(), 0, *win, codes, sf)
    st = torch.zeros(1, dtype=torch.int32, device=DEV)
    ws = torch.empty(B.nvfp4_ldlq_workspace(rows, cols), dtype=torch.uint8, device=DEV)
    B.ldlq_quantize(W, 16, S, sf, perm.to(torch.int32), U, codes, st, ws)
    assert st.item() == 0
    grid = torch.tensor([0, .5, 1, 1.5, 2, 3, 4, 6], device=DEV)
    mids = torch.tensor([.25, .75, 1.25, 1.75, 2.5, 3.5, 5.], dtype=torch.float64, device=DEV)
    e4m3 = torch.tensor([(8 + (c & 7)) * 2.0 ** ((c >> 3) - 10) if c >= 8 else c * 2.0 ** -9 for c in range(127)],
                        device=DEV)
    nib = torch.stack([codes & 15, codes >> 4], -1).reshape(rows, cols)[:, perm].long()
    v = e4m3[sf.long()][:, perm // 16]
    q = torch.where(nib > 7, -grid[nib & 7], grid[nib & 7])
    Wp = W[:, perm]
    T = Wp.double() + (Wp - (q * v) * S).double() @ U.double()
    unit = v.double() * S.double()
    t = T.abs() / unit.clamp_min(1e-300)
    flips = int((((torch.bucketize(t, mids)) != (nib & 7)) & (v > 0)).sum())
    gap = (t[..., None] - mids).abs().amin(-1) * unit / T.square().mean().sqrt()      # in units of the rms
    rho = int((gap < 1e-4).sum()) / 2e-4
    mean = rho * (2 / np.pi) ** 0.5 * 2.0 ** -22                                      # E|d| of a normal error
    print(f"[ldlq] {rows} x {cols}: {flips} codes off their 64-bit targets' (FP32 sums: about {mean:.1f})")
    assert flips <= mean + 4 * mean ** 0.5
