"""Performance cases: the work that programs using this library give it, over the sizes they give it.

Every case is one pass through the public entry points of paper_2401_13660_gb300.mbscan (or one
Decoder.step), on buffers, workspaces and weights that such a program keeps between calls. Kinds:

* step    mb_step: one byte for every stream through one layer, the state updated in place.
* block   mb_rmsnorm and mb_conv_xproj: what a layer runs before its step when a whole model decodes.
* spec    one speculative round on one layer: mb_scan_verify, mb_accept_topk, mb_step_resume.
* prefill mb_scan_prefill over a whole span (prompts; evaluation).
* train   mb_scan_prefill_ckpt and mb_scan_backward (the scan's part of a training step).
* decode  Decoder.step, a whole model with its cuBLAS projections, captured in one CUDA graph.

Sizes are those of the MambaByte models this repository names (d_inner 2048, 3584, 4608; dt_rank
64, 112, 144; 8192-byte spans), with small, ragged and odd ones around them. Spans take B and C as
column blocks of the x-projection's rows (`rank` + 32 wide) where a model's would be. The fused
Delta projection (dt_low) is left out: the library documents it as slower than the projection GEMM
followed by the calls measured here.

Inputs follow the distributions of trained Mamba layers: unit-variance activations, dt_bias =
softplus^-1 of steps log-uniform on [0.01, 0.1], A = -(n + 1) times a log-normal factor of its own
for every channel and state (S4D-real initialisation after training has moved it).
"""
import math

import torch

from paper_2401_13660_gb300 import mbscan as mb
from paper_2401_13660_gb300.decoder import Decoder, DecoderConfig

N = 16          # d_state
DEV = "cuda"
MOST = 8 * 8192 * 2048   # (row, step, channel) triples of the largest spans


def listed():
    return [
        # One stream generating on one 353M-sized layer: the smallest call, nothing but latency.
        dict(name="step_b1_D2048", kind="step", batch=1, D=2048, dtype="bf16", rank=64),
        # Batched serving of the 1.6B-sized model, one layer: streams its 75 MB of states.
        dict(name="step_b256_D4608", kind="step", batch=256, D=4608, dtype="bf16", rank=144),
        # The same model's steps before the scan: residual + norm, convolution, x-projection.
        dict(name="block_b256_d2304", kind="block", batch=256, d_model=2304, rank=144),
        # Speculative serving: 32 streams, 16 drafted bytes each, then the first corrector byte.
        dict(name="spec_s32_k16_D2048", kind="spec", batch=32, k=16, D=2048, dtype="bf16", rank=64, beta=3),
        # A short fp32 span (experiments, checks of a training set-up).
        dict(name="prefill_f32_b1_L256_D64", kind="prefill", batch=1, L=256, D=64, dtype="f32", rank=0,
             gate=True, h0=False),
        # One prompt of the full context on one 353M-sized layer.
        dict(name="prefill_b1_L8192_D2048", kind="prefill", batch=1, L=8192, D=2048, dtype="bf16", rank=64,
             gate=True, h0=False),
        # Evaluation or batched prompts at the full context: 353M- and 972M-sized layers, the
        # second resuming from cached states.
        dict(name="prefill_b8_L8192_D2048", kind="prefill", batch=8, L=8192, D=2048, dtype="bf16", rank=64,
             gate=True, h0=False),
        dict(name="prefill_b4_L8192_D3584", kind="prefill", batch=4, L=8192, D=3584, dtype="bf16", rank=112,
             gate=True, h0=True),
        # Prompts of no round length on an odd width, fp32.
        dict(name="prefill_f32_b3_L1003_D1544", kind="prefill", batch=3, L=1003, D=1544, dtype="f32", rank=0,
             gate=True, h0=True),
        # Training: the 353M-sized layer at the paper's span, bf16, forward and backward.
        dict(name="train_b8_L8192_D2048", kind="train", batch=8, L=8192, D=2048, dtype="bf16", rank=64,
             gate=True, h0=False),
        # A small ragged training batch (fine-tuning), carried state.
        dict(name="train_b2_L777_D1544", kind="train", batch=2, L=777, D=1544, dtype="bf16", rank=48,
             gate=True, h0=True),
        # Generating with a whole model: half the depth of the 48-layer one at its batch size.
        dict(name="decode_24x2304_b256", kind="decode", batch=256, layers=24, d_model=2304),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "block", "spec", "prefill", "prefill", "prefill", "train", "train",
                       "decode"])
    if kind == "block":
        d_model = rng.choice([1024, 1792, 2304])
        return dict(kind=kind, batch=_log(rng, 1, 300), d_model=d_model, rank=d_model // 16)
    if kind == "decode":
        return dict(kind=kind, batch=_log(rng, 1, 256), layers=rng.randint(1, 24),
                    d_model=rng.choice([1024, 1792, 2304]))
    D = rng.choice([2048, 3584, 4608, 8 * _log(rng, 8, 576), 8 * _log(rng, 8, 576)])
    rank = D // 32 // 8 * 8 if rng.random() < 0.75 else 0
    dtype = "f32" if rng.random() < 0.25 else "bf16"
    if kind == "step":
        return dict(kind=kind, batch=_log(rng, 1, 320), D=D, dtype=dtype, rank=rank)
    if kind == "spec":
        return dict(kind=kind, batch=_log(rng, 1, 64), k=rng.randint(2, 40), D=D, dtype=dtype, rank=rank,
                    beta=rng.randint(1, 5))
    most = MOST // (4 if dtype == "f32" else 1) // (2 if kind == "train" else 1)
    L = _log(rng, 17, 8192)
    batch = _log(rng, 1, max(1, min(64, most // (L * D))))
    return dict(kind=kind, batch=batch, L=L, D=D, dtype=dtype, rank=rank, gate=rng.random() < 0.85,
                h0=rng.random() < 0.5)


# ---------------------------------------------------------------------------
# inputs

def _type(case):
    return torch.float32 if case["dtype"] == "f32" else torch.bfloat16


def _layer(g, D):
    """A, D, dt_bias of one layer."""
    A = -torch.arange(1, N + 1, device=DEV, dtype=torch.float32) * \
        torch.exp(0.25 * torch.randn(D, N, device=DEV, generator=g))
    Dw = torch.randn(D, device=DEV, generator=g)
    u = torch.rand(D, device=DEV, generator=g, dtype=torch.float64)
    step = torch.exp(math.log(0.01) + u * math.log(10.0))
    return A.contiguous(), Dw, (step + torch.log(-torch.expm1(-step))).float()


def _tokens(g, batch, L, D, dtype, rank, gate=True):
    """x, z, dt [batch, L, D]; B, C [batch, L, N], columns of the x-projection's rows if rank > 0."""
    def rnd(*shape):
        return torch.randn(*shape, device=DEV, generator=g, dtype=torch.float32).to(dtype)
    x, z, dt = rnd(batch, L, D), rnd(batch, L, D) if gate else None, rnd(batch, L, D)
    rows = rnd(batch, L, rank + 2 * N)
    if rank:
        return x, z, dt, rows[..., rank:rank + N], rows[..., rank + N:]
    return x, z, dt, rows[..., :N].contiguous(), rows[..., N:].contiguous()


def _inputs(case, seed):
    """Everything random in a case."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    kind, b = case["kind"], case["batch"]
    i = {}
    if kind == "block":
        d, E, n_out = case["d_model"], 2 * case["d_model"], case["rank"] + 2 * N
        i["residual"] = torch.randn(b, d, device=DEV, generator=g)
        i["add"] = torch.randn(b, d, device=DEV, generator=g).bfloat16()
        i["norm_w"] = 1 + 0.1 * torch.randn(d, device=DEV, generator=g)
        i["x"] = torch.randn(b, E, device=DEV, generator=g).bfloat16()
        i["window"] = torch.randn(b, 3, E, device=DEV, generator=g).bfloat16()
        i["conv_w"] = torch.rand(E, 4, device=DEV, generator=g) - 0.5
        i["conv_b"] = 0.1 * torch.randn(E, device=DEV, generator=g)
        i["W"] = (torch.randn(n_out, E, device=DEV, generator=g) / math.sqrt(E)).bfloat16()
        return i
    if kind == "decode":
        i["weights"] = _model(g, case)
        E = 2 * case["d_model"]
        i["ssm"] = [0.1 * torch.randn(b, E, N, device=DEV, generator=g) for _ in range(case["layers"])]
        i["conv"] = [torch.randn(b, 3, E, device=DEV, generator=g).bfloat16() for _ in range(case["layers"])]
        i["tokens"] = torch.randint(0, 256, (b,), device=DEV, generator=g)
        return i
    D, td = case["D"], _type(case)
    i["A"], i["Dw"], i["dt_bias"] = _layer(g, D)
    L = {"step": 1, "spec": case.get("k", 0)}.get(kind, case.get("L", 0))
    i["x"], i["z"], i["dt"], i["B"], i["C"] = _tokens(g, b, L, D, td, case["rank"], case.get("gate", True))
    if case.get("h0", True):
        i["h0"] = 0.1 * torch.randn(b, D, N, device=DEV, generator=g)
    else:
        i["h0"] = None
    if kind == "spec":
        # a verifier that mostly agrees with the draft: drafted bytes are usually near the top
        k = case["k"]
        logits = torch.randn(b, k, 256, device=DEV, generator=g)
        drafted = torch.randint(0, 256, (b, k), device=DEV, generator=g)
        agree = 4.5 * (torch.rand(b, k, 1, device=DEV, generator=g) < 0.9)
        logits.scatter_add_(2, drafted[..., None], agree.float())
        i["logits"], i["drafted"] = logits.to(td), drafted.to(torch.uint8)
        i["next"] = _tokens(g, b, 1, D, td, case["rank"])
    if kind == "train":
        i["dout"] = torch.randn(b, L, D, device=DEV, generator=g).to(td)
        i["dh_last"] = 0.1 * torch.randn(b, D, N, device=DEV, generator=g) if case["h0"] else None
    return i


def _model(g, case):
    """Weights of a model as Decoder takes them: (layers, embedding, final norm)."""
    d = case["d_model"]
    E, R = 2 * d, d // 16

    def lin(n, m):
        return (torch.randn(n, m, device=DEV, generator=g) / math.sqrt(m)).bfloat16()
    layers = []
    for _ in range(case["layers"]):
        A, Dw, bias = _layer(g, E)
        L = dict(norm_w=1 + 0.1 * torch.randn(d, device=DEV, generator=g), W_in=torch.stack([lin(E, d), lin(E, d)]),
                 conv_w=torch.rand(E, 4, device=DEV, generator=g) - 0.5,
                 conv_b=0.1 * torch.randn(E, device=DEV, generator=g), W_xproj=lin(R + 2 * N, E), W_dt=lin(E, R),
                 dt_bias=bias, A=A, D=Dw, W_out=lin(d, E))
        W = L["W_xproj"]
        L.update(W_in_x=L["W_in"][0], W_in_z=L["W_in"][1], W_dtlow=W[:R], W_B=W[R:R + N], W_C=W[R + N:])
        layers.append(L)
    return layers, torch.randn(256, d, device=DEV, generator=g).bfloat16(), torch.ones(d, device=DEV)


# ---------------------------------------------------------------------------
# what a program has before the call, and the call

def prepare(case, seed):
    i = _inputs(case, seed)
    s = dict(i, case=case)
    kind, b = case["kind"], case["batch"]
    if kind == "decode":
        cfg = DecoderConfig(n_layers=case["layers"], d_model=case["d_model"], d_inner=2 * case["d_model"],
                            dt_rank=case["d_model"] // 16)
        dec = Decoder(cfg, b, DEV, weights=i["weights"])
        for mine, given in zip(dec.ssm + dec.conv, i["ssm"] + i["conv"]):
            mine.copy_(given)
        dec.capture()
        return dict(case=case, dec=dec, tokens=i["tokens"])
    if kind == "block":
        n_out = case["rank"] + 2 * N
        s["h"] = torch.empty(b, case["d_model"], device=DEV, dtype=torch.bfloat16)
        s["xc"], s["out"] = torch.empty_like(i["x"]), torch.empty(b, n_out, device=DEV, dtype=torch.bfloat16)
        s["ws"] = torch.zeros(mb.mb_conv_xproj_workspace_size(b, 2 * case["d_model"], n_out), dtype=torch.uint8,
                              device=DEV)
        return s
    s["y"] = torch.empty_like(i["x"])
    if kind == "step":
        s["state"] = i["h0"]
        s["ws"] = torch.zeros(256, dtype=torch.uint8, device=DEV)
        return s
    s["ws"] = mb.new_workspace(mb.make_args(i["x"], i["dt"], i["B"], i["C"], i["A"], s["y"], z=i["z"], h0=i["h0"]), DEV)
    L, D = i["x"].shape[1:]
    if kind == "spec":
        s["h_all"] = torch.empty(b, L, D, N, device=DEV)
        s["accept"] = torch.empty(b, device=DEV, dtype=torch.int32)
        s["state"], s["y1"] = torch.empty(b, D, N, device=DEV), torch.empty_like(i["next"][0])
        return s
    s["h_last"] = torch.empty(b, D, N, device=DEV)
    if kind == "train":
        s["h_ckpt"] = torch.empty(b, -(-L // mb.MB_CKPT_STEPS), D, N, device=DEV)
        like = {"dx": i["x"], "ddt": i["x"], "dz": i["z"], "dA": i["A"], "dD": i["Dw"], "ddt_bias": i["dt_bias"],
                "dh0": s["h_last"]}
        s["grads"] = {k: torch.empty_like(t) for k, t in like.items() if t is not None}
        s["grads"].update({k: torch.empty(b, L, N, device=DEV) for k in ("dB", "dC")})
    return s


def run(s):
    kind = s["case"]["kind"]
    if kind == "decode":
        logits = s["dec"].step(s["tokens"])
        return {"logits": logits, "ssm": s["dec"].ssm, "conv": s["dec"].conv}
    if kind == "block":
        mb.mb_rmsnorm(s["residual"], s["norm_w"], s["h"], add=s["add"])
        mb.mb_conv_xproj(s["x"], s["window"], s["conv_w"], s["W"], s["xc"], s["out"], s["ws"], bias=s["conv_b"])
        return {"residual": s["residual"], "h": s["h"], "window": s["window"], "xc": s["xc"], "out": s["out"]}
    a = (s["x"], s["dt"], s["B"], s["C"], s["A"])
    w = dict(z=s["z"], D=s["Dw"], dt_bias=s["dt_bias"], ws=s["ws"])
    if kind == "step":
        mb.mb_step(*a, s["y"], s["state"], **w)
        return {"y": s["y"], "state": s["state"]}
    w["h0"] = s["h0"]
    if kind == "prefill":
        mb.mb_scan_prefill(*a, s["y"], h_last=s["h_last"], **w)
        return {"y": s["y"], "h_last": s["h_last"]}
    if kind == "spec":
        mb.mb_scan_verify(*a, s["y"], s["h_all"], **w)
        mb.mb_accept_topk(s["logits"], s["drafted"], s["case"]["beta"], s["accept"])
        x, z, dt, B, C = s["next"]
        mb.mb_step_resume(x, dt, B, C, s["A"], s["y1"], s["h_all"], s["accept"], s["state"], **dict(w, z=z))
        return {k: s[k] for k in ("y", "h_all", "accept", "y1", "state")}
    mb.mb_scan_prefill_ckpt(*a, s["y"], s["h_ckpt"], h_last=s["h_last"], **w)
    g = mb.mb_scan_backward(*a, s["h_ckpt"], s["dout"], dh_last=s["dh_last"], grads=s["grads"], **w)
    return {"y": s["y"], "h_last": s["h_last"], "h_ckpt": s["h_ckpt"], **{k: v for k, v in g.items() if v is not None}}


# ---------------------------------------------------------------------------
# what a pass cannot do without

def work(case):
    """Each input read once, each output written once; operations of the recurrence (8 per state and step
    forward, 24 backward) and of the matrix products."""
    kind, b = case["kind"], case["batch"]
    if kind == "block":
        d, E, n_out = case["d_model"], 2 * case["d_model"], case["rank"] + 2 * N
        rows = b * d * (4 + 4 + 2 + 2) + b * E * 2 * (1 + 6 + 1) + b * n_out * 2
        return {"bytes": rows + d * 4 + E * 20 + n_out * E * 2, "flops": 2 * b * E * n_out + b * (8 * E + 4 * d)}
    if kind == "decode":
        d, n = case["d_model"], case["layers"]
        E, R = 2 * d, d // 16
        w = 2 * E * d + (R + 2 * N) * E + E * R + d * E
        per = 2 * w + 4 * (d + 4 * E + E + E + E * N + E) + 2 * b * E * (N * 4 + 6)
        head = 256 * d * 2 + d * 4 + b * (8 + 512)
        return {"bytes": n * per + head, "flops": n * (2 * b * w + 8 * b * E * N) + 2 * b * 256 * d}
    es, D = (4 if case["dtype"] == "f32" else 2), case["D"]
    const = D * N * 4 + D * 8
    state = b * D * N * 4
    if kind == "step":
        return {"bytes": 2 * state + 4 * b * D * es + 2 * b * N * es + const, "flops": 8 * b * D * N}
    if kind == "spec":
        t = b * case["k"]
        verify = state + 4 * t * D * es + 2 * t * N * es + const + t * D * N * 4
        accept = t * (256 * es + 1) + 4 * b
        resume = 2 * state + 4 * b * D * es + 2 * b * N * es
        return {"bytes": verify + accept + resume, "flops": 8 * (t + b) * D * N + 256 * t}
    t = b * case["L"]
    toks = 3 if case["gate"] else 2
    fwd = (toks + 1) * t * D * es + 2 * t * N * es + const + state * (2 if case["h0"] else 1)
    if kind == "prefill":
        return {"bytes": fwd, "flops": 8 * t * D * N}
    ckpt = b * -(-case["L"] // 16) * D * N * 4
    bwd = (toks + 1 + toks) * t * D * es + 2 * t * N * (es + 4) + 2 * const + state * (2 if case["h0"] else 1)
    return {"bytes": fwd + bwd + 2 * ckpt, "flops": (8 + 24) * t * D * N}


# ---------------------------------------------------------------------------
# the same in 64 bits

def _wide(t):
    return None if t is None else t.double()


def _scan64(x, z, dt, B, C, A, Dw, bias, h0, every=None, keep=None):
    """Eq. 2-3 step by step: y, h_last; states after each step into `every` [batch, L, D, N] (64 bits or
    fp32), states before every 16th step into `keep`."""
    b, L, D = x.shape
    h = torch.zeros(b, D, N, device=DEV, dtype=torch.float64) if h0 is None else h0.double()
    y = torch.empty(b, L, D, device=DEV, dtype=torch.float64)
    A = A.double()
    for t in range(L):
        if keep is not None and t % 16 == 0:
            keep[:, t // 16] = h
        xt, Bt, Ct = x[:, t].double(), B[:, t].double(), C[:, t].double()
        delta = torch.nn.functional.softplus(dt[:, t].double() + bias, threshold=40.0)
        h = torch.exp(delta[..., None] * A) * h + (delta * xt)[..., None] * Bt[:, None]
        y[:, t] = torch.bmm(h, Ct[..., None])[..., 0] + Dw * xt
        if every is not None:
            every[:, t] = h
    if z is not None:
        for r in range(b):   # row by row: less memory
            y[r] *= torch.nn.functional.silu(z[r].double())
    return y, h


def _train64(i):
    x, z, dt, B, C, A, dout = (i[k] for k in ("x", "z", "dt", "B", "C", "A", "dout"))
    b, L, D = x.shape
    f64 = dict(device=DEV, dtype=torch.float64)
    Dw, bias, A64 = i["Dw"].double(), i["dt_bias"].double(), A.double()
    hs = torch.empty(b, L, D, N, **f64)
    ck = torch.empty(b, -(-L // 16), D, N, device=DEV)
    y, h_last = _scan64(x, z, dt, B, C, A, Dw, bias, i["h0"], every=hs, keep=ck)
    g = torch.zeros(b, D, N, **f64) if i["dh_last"] is None else i["dh_last"].double()
    h_first = torch.zeros(b, D, N, **f64) if i["h0"] is None else i["h0"].double()
    dx, ddt = torch.empty(b, L, D, **f64), torch.empty(b, L, D, **f64)
    dz = None if z is None else torch.empty(b, L, D, **f64)
    dB, dC = torch.empty(b, L, N, **f64), torch.empty(b, L, N, **f64)
    dA, dD, dbias = torch.zeros(D, N, **f64), torch.zeros(D, **f64), torch.zeros(D, **f64)
    for t in range(L - 1, -1, -1):
        xt, Bt, Ct, h = x[:, t].double(), B[:, t].double(), C[:, t].double(), hs[:, t]
        v = dt[:, t].double() + bias
        delta = torch.nn.functional.softplus(v, threshold=40.0)
        dy = dout[:, t].double()
        if z is not None:
            zt = z[:, t].double()
            sg = torch.sigmoid(zt)
            out = torch.bmm(h, Ct[..., None])[..., 0] + Dw * xt
            dz[:, t] = dy * out * sg * (1 + zt * (1 - sg))
            dy = dy * zt * sg
        g = g + dy[..., None] * Ct[:, None]
        dC[:, t] = torch.bmm(dy[:, None], h)[:, 0]
        dB[:, t] = torch.bmm((delta * xt)[:, None], g)[:, 0]
        gB = torch.bmm(g, Bt[..., None])[..., 0]
        g = g * torch.exp(delta[..., None] * A64)
        w = g * (hs[:, t - 1] if t else h_first)
        dx[:, t] = dy * Dw + delta * gB
        dv = (xt * gB + (w * A64).sum(-1)) * torch.sigmoid(v)
        ddt[:, t] = dv
        dA += (w * delta[..., None]).sum(0)
        dD += (dy * xt).sum(0)
        dbias += dv.sum(0)
    r = dict(y=y, h_last=h_last, h_ckpt=ck.double(), dx=dx, ddt=ddt, dB=dB, dC=dC, dA=dA, dD=dD, ddt_bias=dbias,
             dh0=g)
    return r if dz is None else dict(r, dz=dz)


def _norm64(res, w):
    return res * w.double() * torch.rsqrt(res.square().mean(-1, keepdim=True) + 1e-5)


def _conv64(x, window, w, bias):
    taps = torch.cat([window.double(), x[:, None].double()], 1)
    return torch.nn.functional.silu(torch.einsum("bjd,dj->bd", taps, w.double()) + bias.double()), taps[:, 1:]


def exact(case, seed):
    i = _inputs(case, seed)
    kind = case["kind"]
    if kind == "block":
        res = i["residual"].double() + i["add"].double()
        xc, window = _conv64(i["x"], i["window"], i["conv_w"], i["conv_b"])
        return {"residual": res, "h": _norm64(res, i["norm_w"]), "window": window, "xc": xc,
                "out": xc @ i["W"].double().T}
    if kind == "decode":
        layers, emb, norm_f = i["weights"]
        E, R = 2 * case["d_model"], case["d_model"] // 16
        res, ssm, conv = emb[i["tokens"]].double(), [], []
        for n, L in enumerate(layers):
            h = _norm64(res, L["norm_w"])
            xc, window = _conv64(h @ L["W_in"][0].double().T, i["conv"][n], L["conv_w"], L["conv_b"])
            rows = xc @ L["W_xproj"].double().T
            y, state = _scan64(xc[:, None], (h @ L["W_in"][1].double().T)[:, None],
                               (rows[:, :R] @ L["W_dt"].double().T)[:, None], rows[:, None, R:R + N],
                               rows[:, None, R + N:], L["A"], L["D"].double(), L["dt_bias"].double(), i["ssm"][n])
            res = res + y[:, 0] @ L["W_out"].double().T
            ssm.append(state)
            conv.append(window)
        return {"logits": _norm64(res, norm_f) @ emb.double().T, "ssm": ssm, "conv": conv}
    if kind == "train":
        return _train64(i)
    w = (i["A"], i["Dw"].double(), i["dt_bias"].double())
    every = None
    if kind == "spec":
        every = torch.empty(*i["x"].shape, N, device=DEV, dtype=torch.float64)
    y, h = _scan64(*(i[k] for k in ("x", "z", "dt", "B", "C")), *w, i["h0"], every=every)
    if kind == "step":
        return {"y": y, "state": h}
    if kind == "prefill":
        return {"y": y, "h_last": h}
    logits = i["logits"].float()
    mine = logits.gather(2, i["drafted"].long()[..., None])
    ok = 1 + (logits > mine).sum(-1) <= case["beta"]
    accept = ok.long().cumprod(1).sum(1)
    rows = torch.arange(case["batch"], device=DEV)
    kept = torch.where((accept > 0)[:, None, None], every[rows, (accept - 1).clamp(min=0)], i["h0"].double())
    y1, state = _scan64(*i["next"], *w, kept)
    return {"y": y, "h_all": every, "accept": accept.to(torch.int32), "y1": y1, "state": state}
