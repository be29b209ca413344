"""Launch overlap: rounds of verify, accept and resume, and split prefill and
backward calls on one workspace, issued with nothing in between (eagerly and
from a CUDA graph), equal the same calls with a synchronisation after each, bit
for bit (the backward's sums over channels are atomic: close, not equal)."""
import pytest
import torch

from paper_2401_13660_gb300 import mbscan as mb
from paper_2401_13660_gb300.inputs import make_inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _graphed(f):
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        f(lambda: None)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        r = f(lambda: None)
    g.replay()
    torch.cuda.synchronize()
    return r


@pytest.mark.parametrize("b, k, D", [(32, 16, 2048), (3, 5, 72)])
def test_speculative_rounds(b, k, D):
    i = make_inputs(b, k, D, 16, "bf16", "normal", seed=k, device=DEV)
    one = [t[:, :1].contiguous() for t in (i["x"], i["dt"], i["B"], i["C"], i["z"])]
    g = torch.Generator(device=DEV).manual_seed(k)
    rounds = 4
    logits = torch.randn(rounds, b, k, 256, device=DEV, generator=g).bfloat16()
    drafted = torch.randint(0, 256, (rounds, b, k), device=DEV, generator=g).to(torch.uint8)
    kw = dict(D=i["D"], dt_bias=i["dt_bias"])
    bufs = [[torch.empty(b, k, D, device=DEV, dtype=torch.bfloat16), torch.empty(b, k, D, 16, device=DEV),
             torch.empty(b, device=DEV, dtype=torch.int32), torch.empty(b, 1, D, device=DEV, dtype=torch.bfloat16),
             torch.empty(b, D, 16, device=DEV)] for _ in range(rounds)]
    ws = torch.zeros(256, dtype=torch.uint8, device=DEV)

    def run(sync):
        h = i["h0"]
        for r, (y, ha, acc, y1, st) in enumerate(bufs):
            mb.mb_scan_verify(i["x"], i["dt"], i["B"], i["C"], i["A"], y, ha, z=i["z"], h0=h, ws=ws, **kw)
            sync()
            mb.mb_accept_topk(logits[r], drafted[r], 200, acc)
            sync()
            mb.mb_step_resume(*one[:4], i["A"], y1, ha, acc, st, z=one[4], h0=h, ws=ws, **kw)
            sync()
            h = st
        return bufs
    want = [[t.clone() for t in r] for r in run(torch.cuda.synchronize)]
    for f in (lambda: run(lambda: None), lambda: _graphed(run)):
        for t in (t for r in bufs for t in r):
            t.zero_()
        got = f()
        torch.cuda.synchronize()
        assert all(torch.equal(x, y) for a, b_ in zip(got, want) for x, y in zip(a, b_))
    assert mb.mb_check(ws) == (mb.MB_OK, -1)


@pytest.mark.parametrize("b, L, D", [(1, 600, 64), (2, 300, 520)])
def test_split_spans_on_one_workspace(b, L, D):
    n = 3
    ins = [make_inputs(b, L, D, 16, "f32", "normal", seed=s, device=DEV) for s in range(n)]
    args = [tuple(i[k] for k in ("x", "dt", "B", "C", "A")) for i in ins]
    kw = [{k: i[k] for k in ("z", "D", "dt_bias", "h0")} for i in ins]
    ws = mb.new_workspace(mb.make_args(*args[0], torch.empty_like(ins[0]["x"]), h0=ins[0]["h0"]), DEV)
    assert ws.numel() > 256
    y = [torch.empty_like(i["x"]) for i in ins]
    hl = [torch.empty(b, D, 16, device=DEV) for _ in ins]
    ck = [torch.empty(b, -(-L // 16), D, 16, device=DEV) for _ in ins]
    gr = [{} for _ in ins]

    def run(sync):
        for j in range(n):
            mb.mb_scan_prefill_ckpt(*args[j], y[j], ck[j], h_last=hl[j], ws=ws, **kw[j])
            sync()
        for j in range(n):
            gr[j].update(mb.mb_scan_backward(*args[j], ck[j], y[j], dh_last=hl[j], grads=gr[j], ws=ws, **kw[j]))
            sync()
        return y + hl + ck + [g[k] for g in gr for k in ("dx", "ddt", "dz", "dh0")], \
            [g[k] for g in gr for k in ("dB", "dC", "dA", "dD", "ddt_bias")]
    want = [[t.clone() for t in r] for r in run(torch.cuda.synchronize)]
    for f in (lambda: run(lambda: None), lambda: _graphed(run)):
        for t in y + hl + ck:
            t.zero_()
        got = f()
        torch.cuda.synchronize()
        assert all(torch.equal(x, w) for x, w in zip(got[0], want[0]))
        for x, w in zip(got[1], want[1]):   # fp32 atomics: their order is not fixed
            torch.testing.assert_close(x, w, rtol=1e-3, atol=1e-3 * w.abs().max().item())
    assert mb.mb_check(ws) == (mb.MB_OK, -1)
