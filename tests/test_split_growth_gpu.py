"""A time split with states that grow (A > 0), where the product of a segment's
decays overflows. Before the first input the state is zero, after the last loss
the adjoint is, and zero times that product must stay zero: the step-by-step
scan (a 256-byte workspace) gives finite values, and so must the split, the same
up to the order of sums."""
import pytest
import torch

from paper_2401_13660_gb300 import mbscan as mb
from paper_2401_13660_gb300.inputs import make_inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("b, L, D", [(1, 1024, 64), (2, 519, 40)])
def test_zero_state_over_an_overflowing_segment(dtype, b, L, D):
    i = make_inputs(b, L, D, 16, dtype, "zeros", seed=L, device=DEV)
    A = torch.full_like(i["A"], 4.0)                 # 32 steps with Delta about 1: e^128
    x, dout = i["x"].clone(), torch.zeros_like(i["x"])
    x[:, :L - 8] = 0                                 # inputs in the last steps, losses on the first
    dout[:, :8] = 1
    args = (x, i["dt"], i["B"], i["C"], A)
    kw = dict(z=i["z"], D=i["D"], dt_bias=torch.full_like(i["dt_bias"], 0.5))
    full = mb.mb_workspace_size(mb.make_args(*args, torch.empty_like(x), **kw))
    assert full > 256   # split
    got = []
    for n in (256, full):
        ws = torch.zeros(n, dtype=torch.uint8, device=DEV)
        y, h, ck = torch.empty_like(x), torch.empty(b, D, 16, device=DEV), torch.empty(b, -(-L // 16), D, 16, device=DEV)
        mb.mb_scan_prefill_ckpt(*args, y, ck, h_last=h, ws=ws, **kw)
        got.append(dict(mb.mb_scan_backward(*args, ck, dout, ws=ws, **kw), y=y, h=h, ck=ck))
        assert mb.mb_check(ws) == (mb.MB_OK, -1)
    for k, want in got[0].items():
        assert want.isfinite().all()
        torch.testing.assert_close(got[1][k].float(), want.float(), rtol=1e-3, atol=1e-4 * want.abs().max().item(),
                                   msg=lambda m, k=k: f"{k}: {m}")
