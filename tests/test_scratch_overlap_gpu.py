"""A workspace whose scratch overlaps an argument (one large buffer for both):
the span runs without scratch, bit for bit as with a 256-byte workspace, and
nothing else is touched. Checkpoints in the workspace are refused, as ever."""
import pytest
import torch

from paper_2401_13660_gb300 import mbscan as mb
from paper_2401_13660_gb300.inputs import make_inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("where", ["y", "h_last", "h0"])
@pytest.mark.parametrize("dtype, per_sm, L, D", [("bf16", None, 900, 64), ("f32", None, 300, 40), ("bf16", 2.1, 1040, 64)])
def test_scratch_that_overlaps_an_argument_is_left_alone(where, dtype, per_sm, L, D):
    b = 1 if per_sm is None else -(-int(per_sm * torch.cuda.get_device_properties(0).multi_processor_count) // -(-D // 32))
    i = make_inputs(b, L, D, 16, dtype, "normal", seed=L, device=DEV)
    args = tuple(i[k] for k in ("x", "dt", "B", "C", "A"))
    kw = {k: i[k] for k in ("z", "D", "dt_bias")}
    full = mb.mb_workspace_size(mb.make_args(*args, torch.empty_like(i["x"]), **kw))
    assert full > 256   # a split (few tiles) or even shares

    def call(f, ws, y, h_last, h0, *ck):
        return f(*args, y, *ck, h0=h0, h_last=h_last, ws=ws, **kw)
    want = torch.empty_like(i["x"]), torch.empty_like(i["h0"])
    call(mb.mb_scan_prefill, torch.zeros(256, dtype=torch.uint8, device=DEV), *want, i["h0"])
    big = torch.zeros(full + 2 * i["x"].nbytes + 2 * i["h0"].nbytes, dtype=torch.uint8, device=DEV)
    inside = {"y": i["x"], "h_last": i["h0"], "h0": i["h0"]}[where]
    t = big[512:512 + inside.nbytes].view(inside.dtype).view(inside.shape)   # begins inside the scratch
    got = {"y": torch.empty_like(i["x"]), "h_last": torch.empty_like(i["h0"]), "h0": i["h0"].clone(), where: t}
    for f in (mb.mb_scan_prefill, mb.mb_scan_prefill_ckpt):
        got["h0"].copy_(i["h0"])
        ck = () if f is mb.mb_scan_prefill else (torch.empty(b, -(-L // 16), D, 16, device=DEV),)
        call(f, big[:full], got["y"], got["h_last"], got["h0"], *ck)
        torch.cuda.synchronize()
        assert torch.equal(got["y"], want[0]) and torch.equal(got["h_last"], want[1])
        assert torch.equal(got["h0"], i["h0"])
    assert mb.mb_check(big[:256]) == (mb.MB_OK, -1)


def test_checkpoints_in_the_workspace_are_refused():
    L, D = 600, 64
    i = make_inputs(1, L, D, 16, "f32", "zeros", seed=1, device=DEV)
    args = tuple(i[k] for k in ("x", "dt", "B", "C", "A"))
    n = 38 * D * 16 * 4
    big = torch.zeros(1024 + n, dtype=torch.uint8, device=DEV)
    ck = big[512:512 + n].view(torch.float32).view(1, 38, D, 16)
    with pytest.raises(mb.MbError) as e:
        mb.mb_scan_prefill_ckpt(*args, torch.empty_like(i["x"]), ck, ws=big)
    assert e.value.status == mb.MB_ERR_INVALID_ARG
