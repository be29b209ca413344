"""The backward scan at the edges of its tiles (16-step chunks in halves and
pairs of steps, 32-channel CTAs of 16-channel warps with two channels per lane)
against the oracle, with general A, and the same spans split over L (the
workspace mb_workspace_size asks for) and not (256 bytes). Bars: those of
test_backward_gpu.py (fp32 inputs 1e-4, sums over channels 1e-3; bf16 2e-2)."""
import pytest
import torch

import oracle
from paper_2401_13660_gb300 import mbscan as mb
from paper_2401_13660_gb300.inputs import make_inputs

from _parity import rel_err, to_np

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("b, L, Dn, gate, h0, dhl", [(1, 1, 8, True, "normal", True), (2, 9, 40, False, "zeros", True),
                                                     (1, 16, 16, True, "zeros", False), (3, 23, 24, True, "normal", True),
                                                     (1, 64, 72, False, "normal", False), (2, 129, 48, True, "normal", True),
                                                     (1, 250, 136, True, "zeros", True), (2, 516, 8, True, "normal", True)])
def test_backward_edges(dtype, b, L, Dn, gate, h0, dhl):
    inp = make_inputs(b, L, Dn, 16, dtype, h0, seed=100 * L + Dn, device=DEV, gate=gate)
    g = torch.Generator(device=DEV).manual_seed(L)
    inp["A"] = (inp["A"] * torch.exp(0.5 * torch.randn(Dn, 16, device=DEV, generator=g))).contiguous()
    x = inp["x"]
    dout = torch.randn(b, L, Dn, device=DEV, generator=g).to(x.dtype)
    dh = torch.randn(b, Dn, 16, device=DEV, generator=g) if dhl else None
    args = (x, inp["dt"], inp["B"], inp["C"], inp["A"])
    kw = {k: inp[k] for k in ("z", "D", "dt_bias", "h0")}
    y = torch.empty_like(x)
    _, _, ck = mb.mb_scan_prefill_ckpt(*args, y, **kw)
    want = oracle.scan_backward(*map(to_np, args), to_np(dout), **{k: to_np(v) for k, v in kw.items()},
                                dh_last=to_np(dh))
    full = mb.mb_workspace_size(mb.make_args(*args, y, **kw))
    assert (full > 256) == (L >= 128)   # 8 chunks and more of so few channels are split
    for n in {256, full}:
        ws = torch.zeros(n, dtype=torch.uint8, device=DEV)
        got = mb.mb_scan_backward(*args, ck, dout, dh_last=dh, ws=ws, **kw)
        for k, v in got.items():
            if v is None:
                continue
            sums = k in ("dB", "dC", "dA", "dD", "ddt_bias")
            assert rel_err(v, want[k]) <= ({True: 1e-3, False: 1e-4}[sums] if dtype == "f32" else 2e-2), (k, n)
        assert mb.mb_check(ws) == (mb.MB_OK, -1)
