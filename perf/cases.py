"""The workloads whose speed this library is judged by.

Every case is one pass that a user's program makes through the public entry
points (``paper_2607_02805_gb300.binding`` and the ``Layer`` holder): a
training step of a scan layer (forward, then the gradient of every input), a
cache build over a clean prefix, one cached active block, or a denoising loop
of active blocks that the program captured as a CUDA graph. Inputs are drawn
on the GPU from the seed alone, with the value ranges of
``paper_2607_02805_gb300/inputs.py``. ``exact`` evaluates the same functions
in 64 bits with plain torch.

A case is a dict: ``kind`` (below), sizes, and options.

* ``train``       diagonal form: forward + backward of one layer
* ``prefill``     diagonal form: cache build over a prefix
* ``active``      diagonal form: one active block, called on its own
* ``denoise``     a captured loop of active blocks from one cached state:
                  ``form`` "ssd", "diag" or "adaln"
* ``ssd_train``   SSD (Mamba-2) form: forward + backward of one layer
* ``ssd_prefill`` SSD form: cache build over a prefix
* ``mixer``       convolution, step size and gate around the diagonal scan:
                  forward + backward
"""

import math

import torch

from paper_2607_02805_gb300 import binding

EPS = 1e-5  # of the active block's layer norm
HEAD = 64   # channels per head of the SSD form

# what each tensor is drawn from, and its stream id
IDS = {k: i for i, k in enumerate(
    ("x_c", "dt_c", "B_c", "C_c", "x_n", "dt_f", "B_f", "C_f", "dt_r", "B_r", "C_r", "A_f", "D_f", "A_r", "D_r",
     "dy_c", "dy_n", "dstates", "seed", "shift", "scale", "gate", "xr_c", "xr_n", "dtr_c", "dtr_f", "dtr_r", "z_c",
     "z_n", "conv_w", "conv_b", "dt_bias_f", "dt_bias_r"))}
F32_ALWAYS = {"A_f", "D_f", "A_r", "D_r", "dstates", "seed", "shift", "scale", "gate", "conv_w", "conv_b",
              "dt_bias_f", "dt_bias_r"}
CLEAN = ("x_c", "dt_c", "B_c", "C_c")
NOISY = ("x_n", "dt_f", "B_f", "C_f", "dt_r", "B_r", "C_r")
PARAMS = ("A_f", "D_f", "A_r", "D_r")
MIX_IN = ("xr_c", "dtr_c", "B_c", "C_c", "z_c", "xr_n", "dtr_f", "B_f", "C_f", "dtr_r", "B_r", "C_r", "z_n")
MIX_PARAMS = PARAMS + ("conv_w", "conv_b", "dt_bias_f", "dt_bias_r")


def listed():
    return [
        # one denoising step of one layer of a 262,144-token context, called from Python: the smallest call there
        # is, all latency
        dict(name="active_block", kind="active", batch=1, block=16, d=2048, n=16, dtype="bf16"),
        # the inner loop of block-cached decoding with the 350M-class Mamba-2 layer: 16 denoising steps replayed
        # as one CUDA graph
        dict(name="denoise_ssd_350m", kind="denoise", form="ssd", batch=1, block=256, heads=26, n=128, steps=16),
        # the smallest training step of the test suite, fp32: launches and short kernels
        dict(name="train_tiny_f32", kind="train", batch=1, len=256, block=16, d=32, n=8, dtype="f32", dstates=False),
        # one layer of the 87M-scale training step, the benchmark's workload
        dict(name="train_87m", kind="train", batch=8, len=2048, block=16, d=1536, n=16, dtype="bf16", dstates=False),
        # the longest block of the 350M-scale block-size sweep
        dict(name="train_350m_block64", kind="train", batch=8, len=2048, block=64, d=2048, n=16, dtype="bf16",
             dstates=False),
        # ragged sizes in fp32 (three channel groups, the last one partial; a ragged last chunk), with gradients
        # arriving at the boundary states as well
        dict(name="train_odd_f32", kind="train", batch=3, len=48 * 13, block=48, d=300, n=16, dtype="f32",
             dstates=True),
        # cache build over a 65,536-token prefix for a layer above: every block-end state and the clean outputs
        dict(name="prefill_65k_all", kind="prefill", batch=1, len=65536, block=32, d=2048, n=16, dtype="bf16",
             all=True),
        # cache build over a 262,144-token prefix of which only the final state is kept
        dict(name="prefill_262k_final", kind="prefill", batch=1, len=262144, block=16, d=2048, n=16, dtype="bf16",
             all=False),
        # one 350M-class Mamba-2 layer of the training step at the paper's training length
        dict(name="ssd_train_350m", kind="ssd_train", batch=8, len=8192, block=256, heads=26, n=128, dstates=False),
        # a small odd batch of the 87M-class Mamba-2 layer with the shorter block
        dict(name="ssd_train_87m_odd", kind="ssd_train", batch=3, len=128 * 21, block=128, heads=14, n=64,
             dstates=False),
        # cache build over a 65,536-token prefix with the 350M-class Mamba-2 layer, with its outputs
        dict(name="ssd_prefill_65k", kind="ssd_prefill", batch=1, len=65536, block=256, heads=26, n=128, all=True),
        # the 87M-scale layer with the convolution, the step size and the gate around the scan
        dict(name="mixer_87m", kind="mixer", batch=8, len=2048, block=16, d=1536, n=16, dtype="bf16"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("train", "train", "prefill", "active", "denoise", "ssd_train", "ssd_prefill", "mixer"))
    dtype = rng.choice(("bf16", "bf16", "bf16", "f32"))
    align = 8 if dtype == "bf16" else 4
    d = max(align, _log(rng, 32, 2048) // align * align)
    n = rng.choice((8, 16, 16, 16, 16, 32))
    if kind in ("train", "mixer"):
        block = rng.choice((4, 8, 16, 16, 16, 32, 64, rng.randint(1, 16), 16 * rng.randint(1, 8)))
        tokens = _log(rng, 256, 16384)
        batch = min(rng.randint(1, 8), max(1, tokens // block))
        nb = max(1, tokens // batch // block)
        if kind == "mixer":
            n = min(n, 16)
            nb = max(1, min(nb, 16384 * 1536 // (d * batch * block)))
            return dict(kind=kind, batch=batch, len=nb * block, block=block, d=d, n=n, dtype=dtype)
        nb = max(1, nb if n <= 16 else nb // 3)
        return dict(kind=kind, batch=batch, len=nb * block, block=block, d=d, n=n, dtype=dtype,
                    dstates=rng.random() < 0.25)
    if kind == "prefill":
        block = rng.choice((8, 16, 16, 32, 32, 64, 128, rng.randint(5, 60)))
        nb = max(1, _log(rng, 512, 262144) // block)
        n = min(n, 16)
        emit = rng.random() < 0.5
        if emit:
            nb = max(1, min(nb, 65536 // block))
        return dict(kind=kind, batch=1, len=nb * block, block=block, d=d, n=n, dtype=dtype, all=emit)
    if kind == "active":
        return dict(kind=kind, batch=rng.choice((1, 1, 1, rng.randint(2, 16))), block=rng.choice((4, 8, 16, 16, 32, 64, rng.randint(3, 90))),
                    d=d, n=min(n, 16), dtype=dtype)
    if kind == "denoise":
        steps = rng.randint(4, 32)
        if rng.random() < 0.5:
            return dict(kind=kind, form="ssd", batch=rng.randint(1, 4), block=rng.choice((128, 256)),
                        heads=rng.randint(1, 32), n=rng.choice((64, 128)), steps=steps)
        return dict(kind=kind, form=rng.choice(("diag", "adaln")), batch=rng.randint(1, 4),
                    block=rng.choice((8, 16, 16, 32, rng.randint(3, 64))), d=d, n=min(n, 16), dtype=dtype, steps=steps)
    block = rng.choice((128, 256))
    heads = _log(rng, 2, 26)
    sn = rng.choice((64, 128))
    if kind == "ssd_train":
        batch = rng.randint(1, 8)
        nb = max(1, _log(rng, 512, 65536) // batch // block)
        return dict(kind=kind, batch=batch, len=nb * block, block=block, heads=heads, n=sn,
                    dstates=rng.random() < 0.25)
    nb = max(1, _log(rng, 1024, 65536) // block)
    return dict(kind=kind, batch=1, len=nb * block, block=block, heads=heads, n=sn, all=rng.random() < 0.6)


# ------------------------------------------------------------------ inputs
def _shapes(c):
    """Shape of every tensor that prepare() makes."""
    k, Bt, n = c["kind"], c["batch"], c["n"]
    ssd = k.startswith("ssd") or c.get("form") == "ssd"
    L = c["block"] if k in ("active", "denoise") else c["len"]
    X = (Bt, L, c["heads"], HEAD) if ssd else (Bt, L, c["d"])
    T = (Bt, L, c["heads"]) if ssd else (Bt, L, c["d"])
    S = (c["heads"], HEAD, n) if ssd else (c["d"], n)
    A, P = ((c["heads"],), (c["heads"],)) if ssd else ((c["d"], n), (c["d"],))
    if k == "mixer":
        names = MIX_IN + MIX_PARAMS + ("dy_c", "dy_n")
    elif k in ("train", "ssd_train"):
        names = CLEAN + NOISY + PARAMS + ("dy_c", "dy_n") + (("dstates",) if c["dstates"] else ())
    elif k in ("prefill", "ssd_prefill"):
        names = CLEAN + ("A_f", "D_f")
    else:
        names = NOISY + PARAMS + ("seed",) + (("shift", "scale", "gate") if c.get("form") == "adaln" else ())
    out = {}
    for s in names:
        if s.startswith(("x", "dy", "z")):
            out[s] = X
        elif s.startswith("dt_bias") or s == "conv_b":
            out[s] = (c["d"],)
        elif s.startswith("dt"):
            out[s] = T
        elif s[0] in "BC":
            out[s] = (Bt, L, n)
        elif s == "conv_w":
            out[s] = (c["d"], 4)
        elif s == "seed":
            out[s] = (Bt,) + S
        elif s in ("shift", "scale", "gate"):
            out[s] = (Bt, c["d"])
        elif s[0] == "A":
            out[s] = A
        elif s[0] == "D":
            out[s] = P
    if c.get("dstates"):
        out["dstates"] = (Bt, L // c["block"]) + S
    return out


def _in_dtype(c):
    return torch.float32 if c.get("dtype") == "f32" else torch.bfloat16


def _draw(name, shape, seed, part, dtype, device):
    g = torch.Generator(device=device)
    g.manual_seed((int(seed) * 1009 + part) * 64 + IDS[name])
    if name in ("A_f", "A_r"):
        u = torch.rand(shape, generator=g, device=device) * math.log(16.0)
        return -torch.exp(u)
    v = torch.randn(shape, generator=g, device=device)
    if name in ("dt_c", "dt_f", "dt_r"):
        v = torch.nn.functional.softplus(v.mul_(0.5).sub_(2.0))
    elif name in ("dtr_c", "dtr_f", "dtr_r"):
        v = v.mul_(0.5).sub_(2.0)
    elif name[0] in "BC":
        v = v.mul_(1.0 / math.sqrt(shape[-1]))
    elif name in ("D_f", "D_r", "conv_b", "dt_bias_f", "dt_bias_r"):
        v = v.mul_(0.1)
    elif name == "conv_w":
        v = v.mul_(0.5)
    elif name in ("shift", "scale"):
        v = v.mul_(0.3)
    elif name == "gate":
        v = v.mul_(0.3).add_(1.0)
    return v if name in F32_ALWAYS else v.to(dtype)


def _inputs(c, seed, part=0, keep=()):
    """The tensors of one draw; those in `keep` come from part 0."""
    return {k: _draw(k, s, seed, 0 if k in keep else part, _in_dtype(c), "cuda") for k, s in _shapes(c).items()}


def _dims(c):
    L = c["block"] if c["kind"] in ("active", "denoise") else c["len"]
    if "heads" in c:
        return binding.make_ssd_dims(c["batch"], L, c["block"], c["heads"], c["n"])
    return binding.make_dims(c["batch"], L, c["block"], c["d"], c["n"],
                             binding.BDSCAN_F32 if c["dtype"] == "f32" else binding.BDSCAN_BF16)


def _space(nbytes):
    return torch.empty(max(16, nbytes), dtype=torch.uint8, device="cuda")


def _state_shape(c):
    nb = 1 if c.get("all") is False else c["len"] // c["block"]
    return (c["batch"], nb) + ((c["heads"], HEAD, c["n"]) if "heads" in c else (c["d"], c["n"]))


# the steps of a denoising loop share the layer's parameters and the cached state; tokens and modulation change
STEP_KEEP = PARAMS + ("seed",)


def prepare(case, seed):
    c, k = case, case["kind"]
    dims = _dims(c)
    dt = _in_dtype(c)
    if k == "denoise":
        steps = [_inputs(c, seed, p, STEP_KEEP) for p in range(c["steps"])]
        for t in steps[1:]:
            t.update({s: steps[0][s] for s in STEP_KEEP})
        outs = [torch.empty_like(t["x_n"]) for t in steps]
        ws = None
        if c["form"] == "adaln":
            ws = _space(binding.bdscan_active_block_adaln_workspace_size(dims))

        def loop():
            for t, y in zip(steps, outs):
                if c["form"] == "ssd":
                    binding.ssd_active_block(dims, t["seed"], t, y)
                elif c["form"] == "diag":
                    binding.active_block(dims, t["seed"], t, y)
                else:
                    binding.active_block_adaln(dims, t["seed"], t, t["shift"], t["scale"], t["gate"], EPS, y, ws)

        loop()  # the first call sets kernel attributes, which a capture may not
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            loop()
        return dict(case=c, graph=graph, steps=steps, outs=outs, ws=ws, dims=dims)
    t = _inputs(c, seed)
    s = dict(case=c, dims=dims, t=t)
    if k == "active":
        s["y"] = torch.empty_like(t["x_n"])
        return s
    x = t["xr_c" if k == "mixer" else "x_c"]
    s["y_c"] = torch.empty_like(x)
    s["states"] = torch.empty(_state_shape(c), dtype=torch.float32, device="cuda")
    if k in ("prefill", "ssd_prefill"):
        if not c["all"]:
            s["y_c"] = None
        size = binding.bdscan_ssd_boundary_states_workspace_size if k == "ssd_prefill" else \
            binding.bdscan_boundary_states_workspace_size
        s["ws"] = _space(size(dims, int(c["all"])))
        return s
    s["y_n"] = torch.empty_like(x)
    fwd, bwd = {
        "train": (binding.bdscan_forward_workspace_size, binding.bdscan_backward_workspace_size),
        "ssd_train": (binding.bdscan_ssd_forward_workspace_size, binding.bdscan_ssd_backward_workspace_size),
        "mixer": (binding.bdscan_mixer_forward_workspace_size, binding.bdscan_mixer_backward_workspace_size)}[k]
    s["ws_f"], s["ws_b"] = _space(fwd(dims)), _space(bwd(dims))
    s["g"] = {n: torch.empty(v.shape, dtype=torch.float32 if n in F32_ALWAYS else dt, device="cuda")
              for n, v in t.items() if n not in ("dy_c", "dy_n", "dstates")}
    return s


def run(state):
    s = state
    c, dims = s["case"], s["dims"]
    k = c["kind"]
    if k == "denoise":
        s["graph"].replay()
        return {"y%d" % i: y for i, y in enumerate(s["outs"])}
    t = s["t"]
    if k == "active":
        binding.active_block(dims, t["seed"], t, s["y"])
        return {"y_n": s["y"]}
    if k in ("prefill", "ssd_prefill"):
        call = binding.ssd_boundary_states if k == "ssd_prefill" else binding.boundary_states
        call(dims, t, None, s["y_c"], s["states"], int(c["all"]), s["ws"])
        return {"states": s["states"]} if s["y_c"] is None else {"states": s["states"], "y_c": s["y_c"]}
    if k == "mixer":
        binding.mixer_forward(dims, t, s["y_c"], s["y_n"], s["states"], s["ws_f"])
        binding.mixer_backward(dims, t, t["dy_c"], t["dy_n"], None, s["g"], s["ws_b"])
    elif k == "train":
        binding.forward(dims, t, s["y_c"], s["y_n"], s["states"], s["ws_f"])
        binding.backward(dims, t, s["states"], t["dy_c"], t["dy_n"], t.get("dstates"), s["g"], s["ws_b"])
    else:
        binding.ssd_forward(dims, t, s["y_c"], s["y_n"], s["states"], s["ws_f"])
        binding.ssd_backward(dims, t, s["states"], t["dy_c"], t["dy_n"], t.get("dstates"), s["g"], s["ws_b"])
    out = {"y_c": s["y_c"], "y_n": s["y_n"], "states": s["states"]}
    out.update(("d" + n, v) for n, v in s["g"].items())
    return out


def work(case):
    """Bytes: each input read once, each output written once. Flops: the
    recurrences as printed (decay, update, read-out: 6 per token, channel and
    state of a scan; 20 for its adjoint with the recomputed states), or the
    SSD form's causal products."""
    c, k = case, case["kind"]
    e = 4 if c.get("dtype") == "f32" else 2
    size = {n: math.prod(s) * (4 if n in F32_ALWAYS else e) for n, s in _shapes(c).items()}
    loop = c.get("steps", 1)
    once = sum(v for n, v in size.items() if n in STEP_KEEP or loop == 1)
    each = sum(v for n, v in size.items() if n not in STEP_KEEP) if loop > 1 else 0
    nbytes = once + loop * each
    L = c["block"] if k in ("active", "denoise") else c["len"]
    tokens = c["batch"] * L * loop
    out = tokens * (c["heads"] * HEAD if "heads" in c else c["d"]) * e
    if k in ("active", "denoise"):
        nbytes += out
    else:
        st = math.prod(_state_shape(c)) * 4
        nbytes += st
        if k in ("prefill", "ssd_prefill"):
            nbytes += out if c["all"] else 0
        else:
            nbytes += 2 * out + sum(v for n, v in size.items() if n not in ("dy_c", "dy_n", "dstates"))
    if "heads" in c:
        H, n, b = c["heads"], c["n"], c["block"]
        clean = b * n + H * (b * HEAD + 4 * HEAD * n)
        if k == "ssd_prefill" and not c["all"]:
            clean = H * 2 * HEAD * n
        noisy = 2 * b * n + H * (2 * b * HEAD + 2 * HEAD * n)
        flops = {"ssd_prefill": clean, "denoise": noisy, "ssd_train": 3 * (clean + noisy)}[k]
        return {"bytes": nbytes, "flops": tokens * flops}
    per = {"train": 78, "mixer": 78, "prefill": 6, "active": 12, "denoise": 12}[k]
    return {"bytes": nbytes, "flops": tokens * c["d"] * c["n"] * per}


# ------------------------------------------------------------- 64 bits
def _scan(x, dt, B, C, A, h):
    """Selective scan over axis 1 of [M, T, d] tokens from state h [M, d, N]
    (or zero); outputs (None without C) and the last state."""
    ys = []
    for t in range(x.shape[1]):
        a = torch.exp(dt[:, t, :, None] * A)
        u = (dt[:, t] * x[:, t])[:, :, None] * B[:, t, None, :]
        h = u if h is None else a * h + u
        if C is not None:
            ys.append((h * C[:, t, None, :]).sum(-1))
    return (torch.stack(ys, 1) if ys else None), h


def _diag_clean(c, x, dt, B, C, A, D, want_y=True):
    """Clean outputs and every block-end state [Bt, nb, d, N]."""
    Bt, L, d = x.shape
    b, n = c["block"], B.shape[-1]
    nb = L // b
    cut = lambda v: v.reshape(Bt * nb, b, v.shape[-1])
    _, loc = _scan(cut(x), cut(dt), cut(B), None, A, None)
    loc = loc.reshape(Bt, nb, d, n)
    dec = torch.exp(dt.reshape(Bt, nb, b, d).sum(2)[..., None] * A)
    S = [loc[:, 0]]
    for k in range(1, nb):
        S.append(dec[:, k] * S[-1] + loc[:, k])
    S = torch.stack(S, 1)
    y = None
    if want_y:
        seeds = torch.cat([torch.zeros_like(S[:, :1]), S[:, :-1]], 1)
        y, _ = _scan(cut(x), cut(dt), cut(B), cut(C), A, seeds.reshape(Bt * nb, d, n))
        y = y.reshape(Bt, L, d) + D * x
    return y, S


def _diag_noisy(c, t, x, seeds):
    """Noisy outputs of every block; seeds [Bt, nb, d, N]."""
    Bt, L, d = x.shape
    b = c["block"]
    M = Bt * (L // b)
    cut = lambda v: v.reshape(M, b, v.shape[-1])
    rev = lambda v: cut(v).flip(1)
    yf, _ = _scan(cut(x), cut(t["dt_f"]), cut(t["B_f"]), cut(t["C_f"]), t["A_f"], seeds.reshape(M, d, -1))
    yr, _ = _scan(rev(x), rev(t["dt_r"]), rev(t["B_r"]), rev(t["C_r"]), t["A_r"], None)
    return (yf + yr.flip(1)).reshape(Bt, L, d) + (t["D_f"] + t["D_r"]) * x


def _conv(xs, w, b):
    """Width-4 causal taps over axis -2 of [..., T + 3, d]."""
    T = xs.shape[-2] - 3
    return b + sum(w[:, j] * xs[..., j:j + T, :] for j in range(4))


def _diag_layer(c, t):
    """Outputs of the whole layer (with the mixer's steps if it has them)."""
    b = c["block"]
    s = dict(t)
    if c["kind"] == "mixer":
        F = torch.nn.functional
        Bt, L, d = t["xr_c"].shape
        nb = L // b
        ext = F.pad(t["xr_c"], (0, 0, 3, 0))
        s["x_c"] = F.silu(_conv(ext, t["conv_w"], t["conv_b"]))
        before = torch.stack([ext[:, j:j + L:b] for j in range(3)], 2)  # the three clean inputs before each block
        win = torch.cat([before, t["xr_n"].reshape(Bt, nb, b, d)], 2)
        s["x_n"] = F.silu(_conv(win, t["conv_w"], t["conv_b"])).reshape(Bt, L, d)
        for q, bias in (("c", "f"), ("f", "f"), ("r", "r")):
            s["dt_" + q] = F.softplus(t["dtr_" + q] + t["dt_bias_" + bias])
    y_c, S = _diag_clean(c, s["x_c"], s["dt_c"], s["B_c"], s["C_c"], s["A_f"], s["D_f"])
    seeds = torch.cat([torch.zeros_like(S[:, :1]), S[:, :-1]], 1)
    y_n = _diag_noisy(c, s, s["x_n"], seeds)
    if c["kind"] == "mixer":
        y_c, y_n = y_c * torch.nn.functional.silu(t["z_c"]), y_n * torch.nn.functional.silu(t["z_n"])
    return y_c, y_n, S


def _ssd_mask(dt, A, upper):
    """exp(A sum of dt between s and t) on the triangle; dt [..., b, H] ->
    [..., H, b, b], zero where s does not reach t."""
    v = dt.movedim(-1, -2)
    if upper:
        v = v.flip(-1)
    cum = torch.cumsum(v, -1)
    diff = (cum[..., :, None] - cum[..., None, :]) * A[:, None, None]
    keep = torch.ones(diff.shape[-2:], dtype=torch.bool, device=diff.device).tril()
    m = torch.exp(diff.masked_fill(~keep, -math.inf))
    return m.flip(-1, -2) if upper else m


def _ssd_mix(x, dt, B, C, A, upper):
    """(mask o C B^T) diag(dt) x of every block: x [M, b, H, P], dt [M, b, H]."""
    G = C @ B.transpose(-1, -2)
    W = _ssd_mask(dt, A, upper) * G[:, None]
    return (W @ (dt[..., None] * x).transpose(1, 2)).transpose(1, 2)


def _ssd_seed(dt, C, A, seed):
    """The seed's part: exp(A cum dt) C seed^T; seed [M, H, P, N]."""
    e = torch.exp(torch.cumsum(dt, 1) * A)
    return e[..., None] * torch.einsum("mtn,mhpn->mthp", C, seed)


def _ssd_clean(c, x, dt, B, C, A, D, want_y=True):
    """One batch row: x [L, H, P], dt [L, H], B, C [L, N]."""
    b = c["block"]
    nb = x.shape[0] // b
    cut = lambda v: v.reshape((nb, b) + v.shape[1:])
    x, dt, B, C = cut(x), cut(dt), cut(B), cut(C)
    cum = torch.cumsum(dt, 1)
    w = torch.exp((cum[:, -1:] - cum) * A) * dt
    loc = torch.einsum("mth,mthp,mtn->mhpn", w, x, B)
    dec = torch.exp(cum[:, -1] * A)[..., None, None]
    S = [loc[0]]
    for k in range(1, nb):
        S.append(dec[k] * S[-1] + loc[k])
    S = torch.stack(S)
    y = None
    if want_y:
        seeds = torch.cat([torch.zeros_like(S[:1]), S[:-1]])
        y = _ssd_mix(x, dt, B, C, A, False) + _ssd_seed(dt, C, A, seeds) + D[:, None] * x
        y = y.reshape((nb * b,) + x.shape[2:])
    return y, S


def _ssd_noisy(c, t, x, seeds):
    """One batch row's noisy outputs; seeds [nb, H, P, N]."""
    nb = seeds.shape[0]
    cut = lambda v: v.reshape((nb, c["block"]) + v.shape[1:])
    x = cut(x)
    f = [cut(t[q]) for q in ("dt_f", "B_f", "C_f")]
    r = [cut(t[q]) for q in ("dt_r", "B_r", "C_r")]
    y = _ssd_mix(x, *f, t["A_f"], False) + _ssd_seed(f[0], f[2], t["A_f"], seeds)
    y = y + _ssd_mix(x, *r, t["A_r"], True) + (t["D_f"] + t["D_r"])[:, None] * x
    return y.reshape((-1,) + x.shape[2:])


def _train_exact(c, t, layer, pieces):
    """Outputs and gradients of <dy_c, y_c> + <dy_n, y_n> + <dstates, S> by
    autograd, one independent piece (a slice of every tensor) at a time."""
    out = {}
    names = [n for n in t if n not in ("dy_c", "dy_n", "dstates")]
    grads = {n: torch.zeros(t[n].shape, dtype=torch.float64, device="cuda") for n in names}
    y_c = torch.zeros(t["dy_c"].shape, dtype=torch.float64, device="cuda")
    y_n = torch.zeros_like(y_c)
    S = torch.zeros(_state_shape(c), dtype=torch.float64, device="cuda")
    for at, at_y, at_s in pieces:
        p = {n: t[n][at(n)].double().requires_grad_() for n in names}
        a, b, s = layer(c, p)
        loss = (a * t["dy_c"][at_y].double()).sum() + (b * t["dy_n"][at_y].double()).sum()
        if "dstates" in t:
            loss = loss + (s * t["dstates"][at_s].double()).sum()
        for n, g in zip(names, torch.autograd.grad(loss, [p[n] for n in names], allow_unused=True)):
            if g is not None:
                grads[n][at(n)] += g
        y_c[at_y], y_n[at_y], S[at_s] = a.detach(), b.detach(), s.detach()
        del p, a, b, s, loss
    out.update(y_c=y_c, y_n=y_n, states=S)
    out.update(("d" + n, grads[n]) for n in names)
    return out


def exact(case, seed):
    c, k = case, case["kind"]
    if k in ("active", "denoise"):
        out = {}
        for p in range(c.get("steps", 1)):
            t = {n: v.double() for n, v in _inputs(c, seed, p, STEP_KEEP).items()}
            if "heads" in c:
                y = torch.stack([_ssd_noisy(c, {n: v if n in PARAMS else v[i] for n, v in t.items()}, t["x_n"][i],
                                            t["seed"][i:i + 1]) for i in range(c["batch"])])
            else:
                x = t["x_n"]
                if c.get("form") == "adaln":
                    x = torch.nn.functional.layer_norm(x, (c["d"],), eps=EPS)
                    x = (1 + t["scale"][:, None]) * x + t["shift"][:, None]
                y = _diag_noisy(c, t, x, t["seed"][:, None])
                if c.get("form") == "adaln":
                    y = t["x_n"] + t["gate"][:, None] * y
            out["y_n" if k == "active" else "y%d" % p] = y
        return out
    t = _inputs(c, seed)
    if k == "prefill":
        ys, Ss = [], []
        step = 512
        for i in range(0, c["d"], step):
            q = slice(i, i + step)
            v = {n: (w if n in ("B_c", "C_c") else w[q] if n in PARAMS else w[..., q]).double() for n, w in t.items()}
            y, S = _diag_clean(c, v["x_c"], v["dt_c"], v["B_c"], v["C_c"], v["A_f"], v["D_f"], c["all"])
            ys.append(y)
            Ss.append(S if c["all"] else S[:, -1:].clone())
            del y, S
        out = {"states": torch.cat(Ss, 2)}
        if c["all"]:
            out["y_c"] = torch.cat(ys, 2)
        return out
    if k == "ssd_prefill":
        v = {n: w.double() if n in PARAMS else w[0].double() for n, w in t.items()}
        y, S = _ssd_clean(c, v["x_c"], v["dt_c"], v["B_c"], v["C_c"], v["A_f"], v["D_f"], c["all"])
        return {"states": S[None], "y_c": y[None]} if c["all"] else {"states": S[-1:][None]}
    if k == "ssd_train":
        def layer(c, p):
            q = {n: v if n in PARAMS else v[0] for n, v in p.items()}
            y_c, S = _ssd_clean(c, q["x_c"], q["dt_c"], q["B_c"], q["C_c"], q["A_f"], q["D_f"])
            y_n = _ssd_noisy(c, q, q["x_n"], torch.cat([torch.zeros_like(S[:1]), S[:-1]]))
            return y_c[None], y_n[None], S[None]

        def row(i):
            r = slice(i, i + 1)
            return (lambda n: slice(None) if n in PARAMS else r), r, r
        return _train_exact(c, t, layer, [row(i) for i in range(c["batch"])])

    def channels(i, step):
        q = slice(i, i + step)
        full = slice(None)

        def at(n):
            if n[0] in "BC":
                return (full,)
            return (q,) if n in MIX_PARAMS else (full, full, q)
        return at, (full, full, q), (full, full, q)
    step = max(8, min(512, (1 << 29) // (c["batch"] * c["len"] * c["n"])))
    return _train_exact(c, t, _diag_layer, [channels(i, step) for i in range(0, c["d"], step)])
