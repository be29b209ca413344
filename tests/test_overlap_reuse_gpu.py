"""Launch overlap on buffers that a program keeps: every round writes the same
accept counts, per-position states, outputs and workspace as the round before,
with nothing in between, so a read that is served from before the preceding
kernel's write shows in what follows. Eagerly and from a CUDA graph, against the
same calls with a synchronisation after each, bit for bit (the backward's sums
over channels are atomic: close, not equal); outputs are NaN before each run."""
import pytest
import torch

from paper_2401_13660_gb300 import mbscan as mb
from paper_2401_13660_gb300.inputs import make_inputs

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
SUMS = ("dB", "dC", "dA", "dD", "ddt_bias")


def _graphed(f):
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        f(lambda: None)
    return g.replay


def _same_as_synchronised(run, reset, equal, close=()):
    """run(sync) from the buffers as reset() leaves them: synchronised, back to back, and twice from a graph."""
    reset()
    run(torch.cuda.synchronize)
    torch.cuda.synchronize()
    want = [t.clone() for t in equal], [t.clone() for t in close]
    replay = _graphed(run)
    for f in (lambda: run(lambda: None), replay, replay):
        reset()
        torch.cuda.synchronize()
        f()
        torch.cuda.synchronize()
        for x, w in zip(equal, want[0]):
            assert torch.equal(x, w)
        for x, w in zip(close, want[1]):
            torch.testing.assert_close(x, w, rtol=1e-3, atol=1e-3 * w.abs().max().item())


@pytest.mark.parametrize("b, k, D, verify", [(32, 16, 2048, True), (3, 5, 72, True), (32, 16, 2048, False),
                                             (5, 7, 40, False)])
def test_speculative_rounds_on_one_set_of_buffers(b, k, D, verify):
    """verify, accept, resume in place over and over; without the verify, accept and resume alone from one h_all."""
    i = make_inputs(b, k, D, 16, "bf16", "normal", seed=k, device=DEV)
    one = [t[:, :1].contiguous() for t in (i["x"], i["dt"], i["B"], i["C"], i["z"])]
    g = torch.Generator(device=DEV).manual_seed(k)
    rounds = 8
    logits = torch.randn(rounds, b, k, 256, device=DEV, generator=g).bfloat16()
    drafted = torch.randint(0, 256, (rounds, b, k), device=DEV, generator=g).to(torch.uint8)
    kw = dict(D=i["D"], dt_bias=i["dt_bias"])
    y, y1 = torch.empty_like(i["x"]), torch.empty_like(one[0])
    ha, st = torch.empty(b, k, D, 16, device=DEV), torch.empty_like(i["h0"])
    acc = torch.empty(b, device=DEV, dtype=torch.int32)
    given = torch.randn(b, k, D, 16, device=DEV, generator=g)
    ws = torch.zeros(256, dtype=torch.uint8, device=DEV)

    def reset():
        for t in (y, y1):
            t.fill_(float("nan"))
        ha.copy_(given)
        st.copy_(i["h0"])
        acc.fill_(-1)

    def run(sync):
        for r in range(rounds):
            if verify:
                mb.mb_scan_verify(i["x"], i["dt"], i["B"], i["C"], i["A"], y, ha, z=i["z"], h0=st, ws=ws, **kw)
                sync()
            mb.mb_accept_topk(logits[r], drafted[r], 200, acc)
            sync()
            mb.mb_step_resume(*one[:4], i["A"], y1, ha, acc, st, z=one[4], h0=st, ws=ws, **kw)
            sync()
    _same_as_synchronised(run, reset, [y1, ha, acc, st] + ([y] if verify else []))
    assert mb.mb_check(ws) == (mb.MB_OK, -1)


@pytest.mark.parametrize("dtype, per_sm, b, L, D", [("f32", None, 1, 600, 64), ("bf16", None, 2, 300, 520),
                                                    ("bf16", 2.1, None, 1040, 64), ("f32", 3.1, None, 1025, 72),
                                                    ("bf16", 4.25, None, 1040, 40)])
def test_training_passes_on_one_workspace(dtype, per_sm, b, L, D):
    """Time splits (few tiles) and even shares (per_sm tiles per SM) of forward and backward, the forward's h_last
    written over its h0, so that each pass starts from the state that the one before left."""
    if b is None:
        b = -(-int(per_sm * torch.cuda.get_device_properties(0).multi_processor_count) // -(-D // 32))
    i = make_inputs(b, L, D, 16, dtype, "normal", seed=L, device=DEV)
    args = tuple(i[k] for k in ("x", "dt", "B", "C", "A"))
    kw = {k: i[k] for k in ("z", "D", "dt_bias")}
    ws = mb.new_workspace(mb.make_args(*args, torch.empty_like(i["x"]), **kw), DEV)
    assert ws.numel() > 256
    y, h = torch.empty_like(i["x"]), torch.empty_like(i["h0"])
    ck = torch.empty(b, -(-L // 16), D, 16, device=DEV)
    small = torch.zeros(256, dtype=torch.uint8, device=DEV)
    gr = mb.mb_scan_backward(*args, ck.zero_(), y.zero_(), ws=small, **kw)   # allocates the gradients
    y2 = torch.empty_like(y)

    def reset():
        for t in (y, y2, ck, *gr.values()):
            t.fill_(float("nan"))
        h.copy_(i["h0"])

    def run(sync):
        for _ in range(3):
            mb.mb_scan_prefill_ckpt(*args, y, ck, h0=h, h_last=h, ws=ws, **kw)
            sync()
            mb.mb_scan_prefill(*args, y2, h0=h, h_last=h, ws=ws, **kw)
            sync()
            mb.mb_scan_backward(*args, ck, y, h0=h, dh_last=h, grads=gr, ws=ws, **kw)
            sync()
    _same_as_synchronised(run, reset, [y, y2, h, ck] + [t for k, t in gr.items() if k not in SUMS],
                          [gr[k] for k in SUMS])
    assert mb.mb_check(ws) == (mb.MB_OK, -1)


def test_even_shares_on_two_streams():
    """Two workspaces, two streams: each result is that of the call alone."""
    L, D = 1040, 64
    b = -(-int(2.1 * torch.cuda.get_device_properties(0).multi_processor_count) // 2)
    ins = [make_inputs(b, L, D, 16, "bf16", "normal", seed=s, device=DEV) for s in (1, 2)]
    streams = [torch.cuda.Stream() for _ in ins]
    outs, works = [], []
    for i in ins:
        outs.append((torch.empty_like(i["x"]), torch.empty_like(i["h0"])))
        works.append(mb.new_workspace(mb.make_args(i["x"], i["dt"], i["B"], i["C"], i["A"], outs[-1][0], z=i["z"]), DEV))
        assert works[-1].numel() > 4096

    def call(j):
        i, (y, h) = ins[j], outs[j]
        mb.mb_scan_prefill(i["x"], i["dt"], i["B"], i["C"], i["A"], y, z=i["z"], D=i["D"], dt_bias=i["dt_bias"],
                           h0=i["h0"], h_last=h, ws=works[j])
    want = []
    for j in (0, 1):
        call(j)
        torch.cuda.synchronize()
        want.append([t.clone() for t in outs[j]])
    for t in (t for o in outs for t in o):
        t.fill_(float("nan"))
    torch.cuda.synchronize()
    for _ in range(4):
        for j, s in enumerate(streams):
            with torch.cuda.stream(s):
                call(j)
    torch.cuda.synchronize()
    assert all(torch.equal(x, w) for o, ww in zip(outs, want) for x, w in zip(o, ww))
    assert all(mb.mb_check(w) == (mb.MB_OK, -1) for w in works)
