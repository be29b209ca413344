"""Even shares of a prefill or backward whose channel tiles are little over a
multiple of the SMs or of the resident slots (prefill_shares, backward_shares):
the same arithmetic as one CTA per tile (a 256-byte workspace), so everything
but the backward's atomic sums over channels is equal bit for bit, on ragged
spans, part-filled tiles, with and without gate and h0; twice on one workspace
with nothing in between; sampled rows against the oracle. Tile counts are taken
from the device's SMs."""
import pytest
import torch

from paper_2401_13660_gb300 import mbscan as mb
from paper_2401_13660_gb300.inputs import make_inputs

from _parity import TOL, TOL_STATE, oracle_channels, rel_err

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("dtype, per_sm, L, D, gate, h0", [("bf16", 1.07, 2051, 40, True, "normal"),
                                                           ("bf16", 2.1, 1500, 72, False, "zeros"),
                                                           ("bf16", 3.05, 1040, 136, True, "normal"),
                                                           ("bf16", 3.4, 2313, 64, True, "zeros"),
                                                           ("bf16", 4.2, 1040, 40, True, "zeros"),
                                                           ("bf16", 8.15, 1041, 64, True, "normal"),
                                                           ("f32", 4.3, 1000, 72, False, "normal"),
                                                           ("f32", 1.05, 1777, 40, True, "normal"),
                                                           ("f32", 2.05, 1600, 64, False, "zeros"),
                                                           ("f32", 3.1, 1025, 104, True, "normal")])
def test_shares_equal_one_cta_per_tile(dtype, per_sm, L, D, gate, h0):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    b = -(-int(per_sm * sms) // -(-D // 32))
    i = make_inputs(b, L, D, 16, dtype, h0, seed=L, device=DEV, gate=gate)
    args = (i["x"], i["dt"], i["B"], i["C"], i["A"])
    kw = {k: i[k] for k in ("z", "D", "dt_bias", "h0")}
    full = mb.mb_workspace_size(mb.make_args(*args, torch.empty_like(i["x"]), **kw))
    assert full > 4096   # shares
    got = {}
    for n in (256, full):
        ws = torch.full((n,), 255, dtype=torch.uint8, device=DEV)   # scratch needs no clearing by the caller
        ws[:256] = 0
        for r in range(2):
            y, hl = torch.empty_like(i["x"]), torch.empty(b, D, 16, device=DEV)
            mb.mb_scan_prefill(*args, y, h_last=hl, ws=ws, **kw)
            y2, hl2, ck = torch.empty_like(y), torch.empty_like(hl), torch.empty(b, -(-L // 16), D, 16, device=DEV)
            mb.mb_scan_prefill_ckpt(*args, y2, ck, h_last=hl2, ws=ws, **kw)
            got[n, r] = (y, hl, y2, hl2, ck)
        assert mb.mb_check(ws) == (mb.MB_OK, -1)
    for k in got:
        assert all(torch.equal(x, w) for x, w in zip(got[k], got[256, 0])), k
    rows, chans = [0, b // 2, b - 1], [0, D // 2, D - 1]
    ry, rh, _ = oracle_channels(i, rows, chans)
    pick = lambda t: t[torch.tensor(rows, device=DEV)]
    assert rel_err(pick(got[full, 1][0])[:, :, torch.tensor(chans, device=DEV)], ry) <= TOL[dtype]
    assert rel_err(pick(got[full, 1][1])[:, torch.tensor(chans, device=DEV)], rh) <= TOL_STATE[dtype]


@pytest.mark.parametrize("dtype, per_sm, L, D, gate, h0", [("bf16", 2.07, 700, 40, True, "normal"),
                                                           ("bf16", 2.3, 529, 64, False, "zeros"),
                                                           ("bf16", 4.1, 300, 72, True, "normal"),
                                                           ("bf16", 8.2, 410, 64, True, "zeros"),
                                                           ("f32", 2.2, 515, 72, True, "normal"),
                                                           ("f32", 4.25, 288, 40, False, "zeros")])
def test_backward_shares_equal_one_cta_per_tile(dtype, per_sm, L, D, gate, h0):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    b = -(-int(per_sm * sms) // -(-D // 32))
    i = make_inputs(b, L, D, 16, dtype, h0, seed=L, device=DEV, gate=gate)
    args = (i["x"], i["dt"], i["B"], i["C"], i["A"])
    kw = {k: i[k] for k in ("z", "D", "dt_bias", "h0")}
    y = torch.empty_like(i["x"])
    small = torch.zeros(256, dtype=torch.uint8, device=DEV)
    _, _, ck = mb.mb_scan_prefill_ckpt(*args, y, ws=small, **kw)
    g = torch.Generator(device=DEV).manual_seed(L)
    dout = torch.randn(b, L, D, device=DEV, generator=g).to(i["x"].dtype)
    dh = torch.randn(b, D, 16, device=DEV, generator=g)
    full = mb.mb_workspace_size(mb.make_args(*args, y, **kw))
    assert full > 4096   # shares
    big = torch.full((full,), 255, dtype=torch.uint8, device=DEV)   # scratch needs no clearing by the caller
    big[:256] = 0
    want = mb.mb_scan_backward(*args, ck, dout, dh_last=dh, ws=small, **kw)
    got = [mb.mb_scan_backward(*args, ck, dout, dh_last=dh, ws=big, **kw) for _ in range(2)]
    assert mb.mb_check(big) == (mb.MB_OK, -1) and mb.mb_check(small) == (mb.MB_OK, -1)
    for r in got:
        for k in ("dx", "ddt", "dz", "dh0"):
            assert (r[k] is None and want[k] is None) or torch.equal(r[k], want[k]), k
        for k in ("dB", "dC", "dA", "dD", "ddt_bias"):   # fp32 atomics: their order is not fixed
            torch.testing.assert_close(r[k], want[k], rtol=1e-3, atol=1e-3 * want[k].abs().max().item())
