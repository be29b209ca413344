"""The native argument marshalling (csrc/binding.cpp) against the plain Python
path, which a `stream` argument selects: the same results bit for bit on every
entry point it serves (contiguous B, C and column blocks of wider rows; with
and without the optional tensors), the same errors where arguments are wrong."""
import pytest
import torch

from paper_2401_13660_gb300 import mbscan as mb
from paper_2401_13660_gb300.inputs import make_inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _spy(monkeypatch):
    """Count the native calls that were served."""
    served, fast = [], mb._native()

    class Spy:
        def __getattr__(self, name):
            def f(*a):
                rc = getattr(fast, name)(*a)
                if rc >= 0:
                    served.append(name)
                return rc
            return f
    monkeypatch.setattr(mb, "_fast", Spy())
    return served


@pytest.mark.parametrize("full", [True, False])
@pytest.mark.parametrize("b, L, D, block", [(1, 3, 8, False), (2, 16, 40, True), (1, 1, 64, True), (3, 1, 24, True)])
def test_native_equals_plain(monkeypatch, full, b, L, D, block):
    served = _spy(monkeypatch)
    dt = torch.bfloat16 if full else torch.float32
    i = make_inputs(b, L, D, 16, "bf16" if full else "f32", "normal", seed=L + D, device=DEV, accept=True)
    if block:   # columns of [dt_low | B | C] rows
        rows = torch.cat([i["x"][..., :8], i["B"], i["C"]], -1).contiguous()
        i["B"], i["C"] = rows[..., 8:24], rows[..., 24:]
    a = (i["x"], i["dt"], i["B"], i["C"], i["A"])
    kw = dict(z=i["z"], D=i["D"], dt_bias=i["dt_bias"]) if full else {}
    h0 = i["h0"] if full else None
    one = tuple(t[:, :1].contiguous() for t in a[:4]) + (i["A"],)
    kw1 = dict(kw, z=i["z"][:, :1].contiguous()) if full else {}
    g = torch.Generator(device=DEV).manual_seed(b)
    logits = torch.randn(b, L, 256, device=DEV, generator=g).to(dt)
    drafted = torch.randint(0, 256, (b, L), device=DEV, generator=g).to(torch.uint8)
    conv_w = torch.randn(D, 4, device=DEV, generator=g)
    cx = dict(w=128, n=40)
    xc_x = torch.randn(b, cx["w"], device=DEV, generator=g).bfloat16()
    xc_s = torch.randn(b, 3, cx["w"], device=DEV, generator=g).bfloat16()
    xc_W = torch.randn(cx["n"], cx["w"], device=DEV, generator=g).bfloat16()
    xc_w = torch.randn(cx["w"], 4, device=DEV, generator=g)

    def every(stream):
        n = dict(stream=stream)
        e = lambda *s, dtype=torch.float32: torch.zeros(*s, device=DEV, dtype=dtype)
        ws = lambda k=256: e(max(k, 256), dtype=torch.uint8)
        out = []
        y, hl = torch.zeros_like(i["x"]), e(b, D, 16)
        out += [*mb.mb_scan_prefill(*a, y, h0=h0, h_last=hl if full else None, ws=ws(), **kw, **n)]
        y, ck = torch.zeros_like(i["x"]), e(b, -(-L // 16), D, 16)
        out += [*mb.mb_scan_prefill_ckpt(*a, y, ck, h0=h0, h_last=hl.clone(), ws=ws(), **kw, **n)]
        y, ha = torch.zeros_like(i["x"]), e(b, L, D, 16)
        out += [*mb.mb_scan_verify(*a, y, ha, h0=h0, ws=ws(), **kw, **n)]
        out.append(mb.mb_accept_topk(logits, drafted, 100, e(b, dtype=torch.int32), **n))
        out.append(mb.mb_rollback(h0, ha, i["accept"], e(b, D, 16), ws=ws() if full else None, **n))
        y2, ha2 = torch.zeros_like(i["x"]), e(b, L, D, 16)
        out += [*mb.mb_scan_verify_resume(*a, y2, ha2, ha, i["accept"], h0=h0, ws=ws(), **kw, **n)]
        y1, st = torch.zeros_like(one[0]), i["h0"].clone()
        out += [*mb.mb_step(*one, y1, st, ws=ws() if full else None, **kw1, **n)]
        y1, st = torch.zeros_like(one[0]), e(b, D, 16)
        out += [*mb.mb_step_resume(*one, y1, ha, i["accept"], st, h0=h0, ws=ws() if full else None, **kw1, **n)]
        res = i["h0"][..., 0].contiguous().clone()
        out.append(mb.mb_rmsnorm(res, i["D"], torch.zeros(b, D, device=DEV, dtype=dt),
                                 add=i["x"][:, 0].contiguous() if full else None, **n))
        win = torch.zeros(b, 3, D, device=DEV, dtype=dt)
        out.append(mb.mb_conv1d_step(i["x"][:, 0].contiguous(), win, conv_w, torch.zeros(b, D, device=DEV, dtype=dt),
                                     bias=i["D"] if full else None, **n))
        s2, xc = xc_s.clone(), torch.zeros_like(xc_x)
        out += [mb.mb_conv_xproj(xc_x, s2, xc_w, xc_W, xc, e(b, cx["n"], dtype=torch.bfloat16),
                                 ws(mb.mb_conv_xproj_workspace_size(b, cx["w"], cx["n"]))), s2, xc, res, win]
        return out
    native = every(None)
    names = {"prefill", "prefill_ckpt", "verify", "accept_topk", "rollback", "verify_resume", "step", "step_resume",
             "rmsnorm", "conv1d_step", "conv_xproj"}
    assert set(served) == names
    for x, y in zip(native, every(torch.cuda.current_stream())):
        assert (x is None and y is None) or torch.equal(x, y)


def test_native_leaves_wrong_arguments_to_the_plain_path(monkeypatch):
    served = _spy(monkeypatch)
    i = make_inputs(2, 1, 16, 16, "bf16", "normal", seed=1, device=DEV)
    ok = dict(x=i["x"], dt=i["dt"], B=i["B"], C=i["C"], A=i["A"], y=torch.empty_like(i["x"]), state=i["h0"])

    class Sub(torch.Tensor):
        pass
    wrong = [("x", i["x"].float(), ValueError), ("dt", i["dt"][:1], ValueError), ("B", i["B"].cpu(), ValueError),
             ("A", i["A"].double(), TypeError), ("y", torch.empty(2, 1, 32, device=DEV, dtype=torch.bfloat16)[..., ::2],
                                                 ValueError), ("state", i["h0"][:, :8], ValueError),
             ("x", [1.0], Exception)]
    for k, v, err in wrong:
        for stream in (None, torch.cuda.current_stream()):
            with pytest.raises((err, TypeError, ValueError, AttributeError)):
                mb.mb_step(**dict(ok, **{k: v}), stream=stream)
    assert not served
    y0, s0 = (t.clone() for t in mb.mb_step(**dict(ok, state=i["h0"].clone(), y=torch.empty_like(i["x"]))))
    assert served == ["step"]
    y1, s1 = mb.mb_step(**dict(ok, x=i["x"].as_subclass(Sub), state=i["h0"].clone()))   # a subclass: plain path
    assert served == ["step"] and torch.equal(y0, y1) and torch.equal(s0, s1)
