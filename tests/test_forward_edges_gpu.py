"""The forward scan at the edges of its tiles (16-step chunks scanned in pairs
of steps, 32-channel CTAs of 8-channel warps), against the oracle: spans that
end within a pair, a chunk or the ring, widths that leave warps or the last
tile part-filled, with and without gate, h0 and checkpoints, general A. Bars:
those of every parity test (_parity.py)."""
import pytest
import torch

from paper_2401_13660_gb300 import mbscan as mb
from paper_2401_13660_gb300.inputs import make_inputs

from _parity import TOL, TOL_STATE, oracle_scan, rel_err

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("b, L, Dn, gate, h0", [(1, 1, 8, True, "normal"), (2, 2, 40, False, "zeros"),
                                                (3, 15, 32, True, "zeros"), (1, 16, 72, True, "normal"),
                                                (2, 17, 8, False, "normal"), (1, 33, 136, True, "zeros"),
                                                (2, 63, 24, True, "normal"), (1, 65, 64, False, "normal"),
                                                (1, 257, 40, True, "normal")])
def test_forward_edges(dtype, b, L, Dn, gate, h0):
    inp = make_inputs(b, L, Dn, 16, dtype, h0, seed=100 * L + Dn, device=DEV, gate=gate)
    g = torch.Generator(device=DEV).manual_seed(L)
    inp["A"] = (inp["A"] * torch.exp(0.5 * torch.randn(Dn, 16, device=DEV, generator=g))).contiguous()
    ry, rh, rall = oracle_scan(inp, want_h_all=True)
    args = (inp["x"], inp["dt"], inp["B"], inp["C"], inp["A"])
    kw = {k: inp[k] for k in ("z", "D", "dt_bias", "h0")}
    for ckpt in (False, True):
        y, hl = torch.full_like(inp["x"], float("nan")), torch.empty(b, Dn, 16, device=DEV)
        ws = torch.zeros(256, dtype=torch.uint8, device=DEV)
        if ckpt:
            _, _, ck = mb.mb_scan_prefill_ckpt(*args, y, h_last=hl, ws=ws, **kw)
            for i in range(1, ck.shape[1]):   # the state before step 16 i
                assert rel_err(ck[:, i], rall[:, 16 * i - 1]) <= TOL_STATE[dtype]
        else:
            mb.mb_scan_prefill(*args, y, h_last=hl, ws=ws, **kw)
        assert rel_err(y, ry) <= TOL[dtype] and rel_err(hl, rh) <= TOL_STATE[dtype]
        assert mb.mb_check(ws) == (mb.MB_OK, -1)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("b, L, Dn, h0", [(1, 256, 8, "normal"), (2, 257, 40, "zeros"), (1, 289, 64, "normal"),
                                          (3, 511, 1024, "normal"), (1, 777, 2048, "zeros"), (4, 545, 1216, "normal")])
def test_segments_of_a_split_span(dtype, b, L, Dn, h0):
    """Split spans (the first segment shorter than the others and scanned in the first pass, a ragged last one, few
    and many channel tiles up to one per SM); h_last written over h0."""
    inp = make_inputs(b, L, Dn, 16, dtype, h0, seed=L + Dn, device=DEV)
    ry, rh, rall = oracle_scan(inp, want_h_all=True)
    args = (inp["x"], inp["dt"], inp["B"], inp["C"], inp["A"])
    kw = {k: inp[k] for k in ("z", "D", "dt_bias")}
    a = mb.make_args(*args, torch.empty_like(inp["x"]), z=inp["z"])
    assert mb.mb_workspace_size(a) > 256
    for ckpt in (False, True):
        y = torch.full_like(inp["x"], float("nan"))
        hl = torch.empty(b, Dn, 16, device=DEV) if inp["h0"] is None else inp["h0"].clone()
        ws = mb.new_workspace(a, DEV)
        kw["h0"] = None if inp["h0"] is None else hl
        if ckpt:
            _, _, ck = mb.mb_scan_prefill_ckpt(*args, y, h_last=hl, ws=ws, **kw)
            for i in range(1, ck.shape[1]):
                assert rel_err(ck[:, i], rall[:, 16 * i - 1]) <= TOL_STATE[dtype]
        else:
            mb.mb_scan_prefill(*args, y, h_last=hl, ws=ws, **kw)
        assert rel_err(y, ry) <= TOL[dtype] and rel_err(hl, rh) <= TOL_STATE[dtype]
        assert mb.mb_check(ws) == (mb.MB_OK, -1)
