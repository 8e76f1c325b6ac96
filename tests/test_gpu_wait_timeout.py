"""Failure detection on the GPU without a fault: every device wait is bounded.

nvfp4_selftest_wait_timeout makes a barrier expect one arrival more than it can get:
the grouped launch's scale wait (which = 0 and 1), the LDLQ walk's wait for its copies
of U (2), and the waits of LDLQ's trailing updates for their operands (3; one tile to a
CTA, and strips of tiles).  Each wait must give up after its limit (about a second),
report it in the status word (bit 1; LDLQ: bit 16), leave the outputs as documented --
unwritten; zero codes and no errors fed on; an update not applied -- and leave the
context usable: the same call without the raised target right after gives the normal
result.
"""
import time

import pytest
import torch

from paper_2606_07618_gb300 import workloads as W

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_07618_gb300 import binding
    binding.lib()
    return binding


@pytest.mark.parametrize("which", [0, 1])
def test_wait_runs_out_and_is_reported(B, which):
    x = W.small_tensor(256, 1024, 3).to(DEV)
    ws = torch.empty(max(B.nvfp4_dynamic_workspace(), B.scalesweep_quantize_group_workspace()), dtype=torch.uint8,
                     device=DEV)
    codes = torch.full((256, 512), 0xEE, dtype=torch.uint8, device=DEV)
    sfl = torch.full((256, 64), 0xEE, dtype=torch.uint8, device=DEV)
    S = torch.full((1,), -1.0, device=DEV)
    st = torch.zeros(1, dtype=torch.int32, device=DEV)
    torch.cuda.synchronize()
    t0 = time.time()
    B.nvfp4_selftest_wait_timeout(which, x, S, st, ws, codes, sfl)
    torch.cuda.synchronize()
    dt = time.time() - t0
    assert st.item() & 2
    assert 0.5 < dt < 60
    assert torch.all(codes == 0xEE) and torch.all(sfl == 0xEE)      # the waiting warps wrote nothing
    # the context is still usable: the real call gives the normal result
    st.zero_()
    win = (B.NVFP4_WINDOW_DEFAULT, B.NVFP4_WINDOW_DEFAULT)
    S2 = torch.empty(1, device=DEV)
    if which == 0:
        B.scalesweep_quantize_dynamic(x, 16, 256.0, 0, None, 0, *win, S2, st, ws, codes, sfl)
    else:
        d = B.group_descriptors([x], [None], [0], [codes], [sfl], [None])
        B.scalesweep_quantize_group(d, B.NVFP4_IN_BF16, 0, 256.0, S2, st, ws)
    ref = B.empty_outputs(256, 1024, 16, device=DEV, linear=True)
    S3 = torch.empty(1, device=DEV)
    gws = torch.empty(B.nvfp4_global_scale_workspace(x.numel()), dtype=torch.uint8, device=DEV)
    B.nvfp4_global_scale(x, 256.0, S3, None, gws)
    B.scalesweep_quantize(x, 16, S3, 0, None, 0, *win, ref["codes"], ref["sf_linear"])
    torch.cuda.synchronize()
    assert st.item() == 0 and S2.item() == S3.item()
    assert torch.equal(codes, ref["codes"]) and torch.equal(sfl, ref["sf_linear"])


def ldlq_buffers(B, rows, cols, seed):
    g = torch.Generator().manual_seed(seed)
    x = (torch.randn(rows, cols, generator=g) * 0.02).to(torch.bfloat16).to(DEV)
    sf = torch.randint(40, 80, (rows, cols // 16), generator=g).to(torch.uint8).to(DEV)
    perm = torch.randperm(cols, generator=g).to(torch.int32).to(DEV)
    U = torch.triu(torch.randn(cols, cols, generator=g) * 0.05, 1).to(DEV)
    pad = lambda n: -(-n // 256) * 256
    head = pad(4 * cols) + pad(4 * cols * cols)
    # stale bytes everywhere the call writes: none of them may come back
    ws = torch.full((head + B.nvfp4_ldlq_workspace(rows, cols),), 0xEE, dtype=torch.uint8, device=DEV)
    ws[:4 * cols].view(torch.int32).copy_(perm)
    ws[pad(4 * cols):pad(4 * cols) + 4 * cols * cols].view(torch.float32).copy_(U.reshape(-1))
    return x, sf, perm, U, ws, torch.full((rows, cols // 2), 0xEE, dtype=torch.uint8, device=DEV)


def ldlq_pass(B, x, S, sf, perm, U):
    rows, cols = x.shape
    codes = torch.empty(rows, cols // 2, dtype=torch.uint8, device=DEV)
    st = torch.zeros(1, dtype=torch.int32, device=DEV)
    ws = torch.empty(B.nvfp4_ldlq_workspace(rows, cols), dtype=torch.uint8, device=DEV)
    B.ldlq_quantize(x, 16, S, sf, perm, U, codes, st, ws)
    torch.cuda.synchronize()
    assert st.item() == 0
    return codes


# 2: three super-panels, the last of 16 columns.  3: one update of 256 columns, as two
# tiles alone, and as 229 x 2 on 152 SMs, which go in strips.
@pytest.mark.parametrize("which,rows,cols", [(2, 45, 528), (3, 45, 512), (3, 29300, 512)])
def test_ldlq_wait_runs_out_and_is_reported(B, which, rows, cols):
    x, sf, perm, U, ws, codes = ldlq_buffers(B, rows, cols, rows + cols)
    S = torch.full((1,), 0.01, device=DEV)
    st = torch.zeros(1, dtype=torch.int32, device=DEV)
    want = torch.zeros_like(codes) if which == 2 else None
    if which == 3:                                  # the update of columns 256.. left out
        cut = U.clone()
        cut[:256, 256:] = 0.0
        want = ldlq_pass(B, x, S, sf, perm, cut)
    torch.cuda.synchronize()
    t0 = time.time()
    B.nvfp4_selftest_wait_timeout(which, x, S, st, ws, codes, sf)
    torch.cuda.synchronize()
    assert 0.5 < time.time() - t0 < 60
    assert st.item() == 16
    assert torch.equal(codes, want)
    ref = ldlq_pass(B, x, S, sf, perm, U)           # the context is still usable
    assert not torch.equal(ref, want)
    assert torch.equal(ref, ldlq_pass(B, x, S, sf, perm, U))
