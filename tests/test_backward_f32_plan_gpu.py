"""The backward's plan for fp32, of which an SM holds three CTAs (bf16: four):
even shares are at most three per SM, which the workspace tells, and the spans
at the edges of the rules (three segments, unsplit, shares of two and of three
per SM) equal the unsplit sweep of a 256-byte workspace; only sums over channels
and over segments come in another order."""
import pytest
import torch

from paper_2401_13660_gb300 import mbscan as mb
from paper_2401_13660_gb300.inputs import make_inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("dtype, most", [("f32", 3), ("bf16", 4)])
@pytest.mark.parametrize("per_sm", [2.1, 3.1, 3.5, 4.25, 5.1])
def test_shares_are_resident(dtype, most, per_sm):
    sms, L, D = torch.cuda.get_device_properties(0).multi_processor_count, 288, 64
    t = torch.empty(-(-int(per_sm * sms) // 2), L, D, device=DEV, dtype=torch.float32 if dtype == "f32" else torch.bfloat16)
    bc = t[..., :16].contiguous()
    n = mb.mb_workspace_size(mb.make_args(t, t, bc, bc, torch.empty(D, 16, device=DEV), torch.empty_like(t)))

    def scratch(shares):   # a ticket and a flag each, in whole 256 bytes; the state or adjoint of 32 channels
        return 256 + -(-4 * (shares + 1) // 256) * 256 + shares * 32 * 16 * 4
    assert n in [256] + [scratch(k * sms) for k in range(1, most + 1)]


@pytest.mark.parametrize("per_sm, L, D", [(0.5, 300, 64), (1.2, 200, 64), (1.33, 140, 40), (1.7, 160, 64), (2.1, 300, 72),
                                          (3.1, 290, 40), (5.1, 272, 64)])
def test_plan_equals_the_unsplit_sweep(per_sm, L, D):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    b = -(-int(per_sm * sms) // -(-D // 32))
    i = make_inputs(b, L, D, 16, "f32", "normal", seed=L, device=DEV)
    args = tuple(i[k] for k in ("x", "dt", "B", "C", "A"))
    kw = {k: i[k] for k in ("z", "D", "dt_bias", "h0")}
    y = torch.empty_like(i["x"])
    full = max(256, mb.mb_workspace_size(mb.make_args(*args, y, **kw)))
    small, ws = torch.zeros(256, dtype=torch.uint8, device=DEV), torch.full((full,), 255, dtype=torch.uint8, device=DEV)
    ws[:256] = 0
    _, _, ck = mb.mb_scan_prefill_ckpt(*args, y, ws=small, **kw)
    g = torch.Generator(device=DEV).manual_seed(L)
    dout = torch.randn(b, L, D, device=DEV, generator=g)
    dh = torch.randn(b, D, 16, device=DEV, generator=g)
    want = mb.mb_scan_backward(*args, ck, dout, dh_last=dh, ws=small, **kw)
    got = mb.mb_scan_backward(*args, ck, dout, dh_last=dh, ws=ws, **kw)
    assert mb.mb_check(ws) == (mb.MB_OK, -1)
    for k, w in want.items():   # bars of test_backward_edges_gpu.py, of the largest value
        bar = 1e-3 if k in ("dB", "dC", "dA", "dD", "ddt_bias") else 1e-4
        torch.testing.assert_close(got[k], w, rtol=bar, atol=bar * w.abs().max().item(), msg=lambda m, k=k: f"{k}: {m}")
