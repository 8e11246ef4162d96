"""The workloads the library is timed on, as a program of its users runs them.

A case is a dict of plain values.  `listed()` are the named ones, `draw(rng)` gives more of the same ranges, `prepare` makes
what a program holds before the call (activations, tables, gradients, workspaces), `run` is one pass through the public
binding, `work` is what the pass cannot do without and `tolerance` how far two correct implementations may lie apart.

Kinds of case:
  infer     one attention layer on one map or frame, forward only.  Frames are not multiples of the window and often not of
            8 either (a 1280 x 720 output at x2, x3, x4 has 360 x 640, 240 x 427, 180 x 320 tokens).
  train     one attention layer on a batch of training patches, forward and backward; tables shared by the heads or one per
            head, windows shifted or not, with or without the mask between the wrapped parts.
  block     the layers of a block, whose window sizes cycle, forward and backward through the cycle drivers.
  gated     one layer with the convolutional local attention gate, forward and backward.
  features  the positional features of one layer from their generator's weights, and the weights' gradients.
"""
import math

import torch
import torch.nn.functional as F

from paper_2603_06738_b200 import binding


def listed():
    return [
        # the smallest call: one 64 x 64 map, 2 heads, 16 x 16 windows; launch and host latency are what counts
        dict(name="infer_64x64_h2_w16", kind="infer", B=1, H=64, W=64, heads=2, d=32, r=16, window=16, shift=0),
        # inference on one square map, large windows
        dict(name="infer_256x256_w64_s32", kind="infer", B=1, H=256, W=256, heads=6, d=32, r=16, window=64, shift=32),
        # a 1280 x 720 output at x2: the frame is a multiple of 8 but not of the window
        dict(name="infer_360x640_w64", kind="infer", B=1, H=360, W=640, heads=6, d=32, r=16, window=64, shift=0),
        # the same output at x4: 180 rows, not a multiple of 8
        dict(name="infer_180x320_w32", kind="infer", B=1, H=180, W=320, heads=6, d=32, r=16, window=32, shift=0),
        # the training configuration of the benchmark: 16 patches of 96 x 96
        dict(name="train_w32_s16", kind="train", B=16, H=96, W=96, heads=6, d=32, r=16, window=32, shift=16, headwise=False, masked=False),
        # large windows in training
        dict(name="train_w48_s24", kind="train", B=16, H=96, W=96, heads=6, d=32, r=16, window=48, shift=24, headwise=False, masked=False),
        # the smallest window, where memory traffic and per-window costs dominate
        dict(name="train_w8", kind="train", B=16, H=96, W=96, heads=6, d=32, r=16, window=8, shift=0, headwise=False, masked=False),
        # 30-channel heads with rank 18: rows that are no multiple of 16 bytes
        dict(name="train_d30_r18_w32", kind="train", B=8, H=96, W=96, heads=6, d=30, r=18, window=32, shift=0, headwise=False, masked=False),
        # narrow heads, a table per head, shifted windows with a mask: small windows of a small batch
        dict(name="train_d16_r24_w16_masked", kind="train", B=4, H=96, W=96, heads=12, d=16, r=24, window=16, shift=8, headwise=True, masked=True),
        # a block of six layers on 64 x 64 patches, window sizes cycling
        dict(name="block_64x64_w16_32_64", kind="block", B=10, H=64, W=64, heads=6, d=32, r=16, windows="16,32,64,16,32,64"),
        # a layer with the gate, trained: gate, attention, product and the three backward passes
        dict(name="gated_96x96_w32", kind="gated", B=8, H=96, W=96, heads=6, d=32, r=16, window=32, shift=16),
        # the generator of one layer's tables, once per layer and step
        dict(name="features_w32", kind="features", window=32, L=10, dh=32, r=16),
    ]


# (channels per head, rank, heads): the widths of the network tables, the rank-32 option, and an odd one
_WIDTHS = [(32, 16, 6), (32, 16, 6), (32, 32, 6), (30, 18, 6), (16, 24, 12), (24, 8, 4)]
_MOST_FLOPS = 9e11          # below the largest listed case


def draw(rng):
    while True:
        kind = rng.choices(["infer", "train", "block", "gated", "features"], weights=[5, 5, 1, 1, 1])[0]
        d, r, heads = rng.choice(_WIDTHS)
        if kind == "features":
            case = dict(kind=kind, window=rng.choice([8, 16, 24, 32, 48, 64]), L=rng.randint(6, 12), dh=rng.choice([16, 32, 48]), r=rng.choice([16, 18, 24, 32]))
        elif kind == "infer":
            window = rng.choice([16, 32, 48, 64])
            if rng.random() < 0.3:                      # a map of whole windows, shifted or not
                H, W = window * rng.randint(1, 320 // window), window * rng.randint(1, 448 // window)
                shift = rng.choice([0, window // 2])
            else:                                       # a frame of any size; half of them multiples of 8
                H, W, shift = int(48 * (400 / 48) ** rng.random()), int(64 * (640 / 64) ** rng.random()), 0
                if rng.random() < 0.5:
                    H, W = H // 8 * 8, W // 8 * 8
            case = dict(kind=kind, B=1, H=H, W=W, heads=heads, d=d, r=r, window=window, shift=shift)
        elif kind == "train":
            window = rng.choice([8, 16, 16, 32, 32, 48, 64, 96])
            side = 96 if window in (48, 96) else rng.choice([64, 128]) if window == 64 else rng.choice([64, 96, 128])
            masked = window in (16, 32, 48) and rng.random() < 0.25
            shift = window // 2 if masked else rng.choice([0, window // 2]) if window >= 16 else 0
            case = dict(kind=kind, B=rng.randint(1, 20), H=side, W=side, heads=heads, d=d, r=r, window=window, shift=shift,
                        headwise=rng.random() < 0.3, masked=masked)
        elif kind == "block":
            side = rng.choice([64, 96])
            windows = ",".join(str(rng.choice([16, 32, 48, 64] if side == 96 else [16, 32, 64])) for _ in range(rng.randint(2, 6)))
            case = dict(kind=kind, B=rng.randint(1, 10), H=side, W=side, heads=6, d=32, r=16, windows=windows)
        else:
            d, r, heads = rng.choice([(32, 16, 6), (30, 18, 6), (16, 24, 6)])
            window = rng.choice([16, 32, 48])
            case = dict(kind=kind, B=rng.randint(1, 12), H=96, W=96, heads=heads, d=d, r=r, window=window, shift=rng.choice([0, window // 2]))
        if work(case)["flops"] <= _MOST_FLOPS:
            return case


class _Source:
    """Seeded values on the device: activations and gradients N(0, 1), tables N(0, 0.5^2), in bf16."""

    def __init__(self, seed):
        self.gen = torch.Generator(device="cuda")
        self.gen.manual_seed(int(seed))

    def bf16(self, *shape, sigma=1.0):
        return (torch.randn(shape, generator=self.gen, device="cuda") * sigma).to(torch.bfloat16)

    def f32(self, *shape, sigma=1.0):
        return torch.randn(shape, generator=self.gen, device="cuda") * sigma


def _windows(case):
    return [int(w) for w in case["windows"].split(",")]


def _generator(case, source):
    rows, dh, r = 2 + 4 * case["L"], case["dh"], case["r"]
    return [source.f32(rows, dh, sigma=rows ** -0.5), source.f32(dh, sigma=0.1), source.f32(dh, r, sigma=dh ** -0.5), source.f32(dh, r, sigma=dh ** -0.5)]


def _inputs(case, seed):
    source = _Source(seed)
    if case["kind"] == "features":
        n = case["window"] ** 2
        return dict(case=case, weights=_generator(case, source), dpq=source.f32(n, case["r"]), dpk=source.f32(n, case["r"]))
    B, H, W, heads, d, r = (case[k] for k in ("B", "H", "W", "heads", "d", "r"))
    image = (B, H, W, heads, d)
    if case["kind"] == "block":
        windows = _windows(case)
        lists = {k: [source.bf16(*image) for _ in windows] for k in ("q", "k", "v", "dout")}
        for k in ("pq", "pk"):
            lists[k] = [source.bf16(w * w, r, sigma=0.5) for w in windows]
        return dict(case=case, windows=windows, **lists)
    n = case["window"] ** 2
    table = (heads, n, r) if case.get("headwise") else (n, r)
    state = dict(case=case, q=source.bf16(*image), k=source.bf16(*image), v=source.bf16(*image),
                 pq=source.bf16(*table, sigma=0.5), pk=source.bf16(*table, sigma=0.5))
    if case["kind"] == "infer":
        return state
    state["dout"] = source.bf16(*image)
    if case["kind"] == "gated":
        D = heads * d
        state["x"] = source.bf16(B, H, W, D)
        state["conv"] = [source.f32(D, 3, 3, sigma=1 / 3), source.f32(D, sigma=0.1), source.f32(D, D, sigma=D ** -0.5), source.f32(D, sigma=0.1)]
    return state


def prepare(case, seed):
    state = _inputs(case, seed)
    if case["kind"] in ("train", "gated"):
        shape = tuple(case[k] for k in ("B", "H", "W", "heads", "d", "r", "window"))
        if case.get("headwise"):
            need = binding.rib_window_attn_bwd_headwise_workspace(case["window"] ** 2 * case["r"], *shape)
        else:
            need = binding.rib_window_attn_bwd_workspace(*shape)
        state["workspace"] = torch.empty(need, dtype=torch.uint8, device="cuda")
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "features":
        pq, pk = binding.rib_generate_features(*state["weights"], case["window"])
        return pq, pk, binding.rib_generate_features_bwd(*state["weights"], state["dpq"], state["dpk"], case["window"])
    if kind == "block":
        args = [state[k] for k in ("q", "k", "v", "pq", "pk")]
        outs, lses = binding.rib_window_cycle_fwd(*args, state["windows"])
        return outs, binding.rib_window_cycle_bwd(*args, outs, lses, state["dout"], state["windows"])
    args = [state[k] for k in ("q", "k", "v", "pq", "pk")]
    window, shift = case["window"], case["shift"]
    if kind == "infer":
        out, _ = binding.rib_window_attn_fwd_padded(*args, window, shift, want_lse=False)
        return out
    workspace, dout = state["workspace"], state["dout"]
    if kind == "gated":
        gate = binding.rib_cla_gate(state["x"], *state["conv"])
        out, lse = binding.rib_window_attn_fwd(*args, window, shift)
        gated = binding.rib_cla_product(out, gate)
        dattn, dgate = binding.rib_cla_product_bwd(out, gate, dout)
        grads = binding.rib_window_attn_bwd(*args, out, lse, dattn, window, shift, workspace=workspace)
        return gated, grads, binding.rib_cla_gate_bwd(state["x"], *state["conv"], dgate)
    if case["masked"]:
        out, lse = binding.rib_window_attn_fwd_masked(*args, window, shift)
        return out, lse, binding.rib_window_attn_bwd_masked(*args, out, lse, dout, window, shift, workspace=workspace)
    if case["headwise"]:
        out, lse = binding.rib_window_attn_fwd_headwise(*args, window, shift)
        return out, lse, binding.rib_window_attn_bwd_headwise(*args, out, lse, dout, window, shift, workspace=workspace)
    out, lse = binding.rib_window_attn_fwd(*args, window, shift)
    return out, lse, binding.rib_window_attn_bwd(*args, out, lse, dout, window, shift, workspace=workspace)


def _to_windows(t, window, shift):
    """[B, H, W, ...] laid over the extended map, rolled by the shift and cut: [B * windows, window^2, ...]."""
    B, H, W = t.shape[:3]
    Hp, Wp = -(-H // window) * window, -(-W // window) * window
    t = F.pad(t, [0, 0] * (t.dim() - 3) + [0, Wp - W, 0, Hp - H]).roll((-shift, -shift), (1, 2))
    t = t.reshape(B, Hp // window, window, Wp // window, window, -1).transpose(2, 3)
    return t.reshape(B * (Hp // window) * (Wp // window), window * window, -1)


def _from_windows(t, shape, window, shift):
    """The inverse of _to_windows for a map of shape (B, H, W)."""
    B, H, W = shape
    ny, nx = -(-H // window), -(-W // window)
    t = t.reshape(B, ny, nx, window, window, -1).transpose(2, 3).reshape(B, ny * window, nx * window, -1)
    return t.roll((shift, shift), (1, 2))[:, :H, :W]


def _attention(q, k, v, pq, pk, dout, window, shift, masked):
    """out, lse (and, given dout, dq, dk, dv, dpq, dpk) in float64, one group of windows of one head at a time."""
    B, H, W, heads, d = q.shape
    r = pq.shape[-1]
    images = [_to_windows(t, window, shift).unflatten(-1, (heads, d)) for t in (q, k, v) + ((dout,) if dout is not None else ())]
    # a label per position: different labels do not attend to each other, label 0 is no token
    label = torch.zeros((1, -(-H // window) * window, -(-W // window) * window), device=q.device)
    label[:, :H, :W] = 1
    if masked and shift:
        rows, cols = (torch.arange(side, device=q.device) < shift for side in (H, W))
        label = label + rows[None, :, None] + 2 * cols[None, None, :]
    label = _to_windows(label[..., None], window, shift)[..., 0].repeat(B, 1)
    pq, pk = (t.double().expand(heads, -1, -1) if t.dim() == 2 else t.double() for t in (pq, pk))
    results = [torch.zeros(images[0].shape, dtype=torch.float64, device=q.device) for _ in range(1 if dout is None else 4)]
    lse = torch.zeros(images[0].shape[:-1], dtype=torch.float64, device=q.device)
    dpq, dpk = torch.zeros_like(pq, memory_format=torch.contiguous_format), torch.zeros_like(pk, memory_format=torch.contiguous_format)
    group = max(1, (1 << 27) // window ** 4)
    for h in range(heads):
        for start in range(0, label.shape[0], group):
            part = slice(start, start + group)
            qw, kw, vw = (t[part, :, h].double() for t in images[:3])
            logits = qw @ kw.mT / math.sqrt(d) + pq[h] @ pk[h].T / math.sqrt(r)
            logits = logits.masked_fill_(label[part, :, None] != label[part, None, :], -math.inf)
            lse[part, :, h] = logits.logsumexp(-1)
            p = torch.exp(logits.sub_(lse[part, :, h, None]))
            results[0][part, :, h] = p @ vw
            if dout is None:
                continue
            gw = images[3][part, :, h].double()
            results[3][part, :, h] = p.mT @ gw
            ds = p * (gw @ vw.mT - (gw * results[0][part, :, h]).sum(-1, keepdim=True))
            results[1][part, :, h] = ds @ kw / math.sqrt(d)
            results[2][part, :, h] = ds.mT @ qw / math.sqrt(d)
            total = (ds * (label[part] > 0)[:, :, None]).sum(0)
            dpq[h] += total @ pk[h] / math.sqrt(r)
            dpk[h] += total.T @ pq[h] / math.sqrt(r)
    results = [_from_windows(t.flatten(-2), (B, H, W), window, shift).unflatten(-1, (heads, d)) for t in results]
    lse = _from_windows(lse, (B, H, W), window, shift).permute(0, 3, 1, 2)
    return results[0], lse, results[1:], dpq, dpk


def _gate(x, w_dw, b_dw, w_pw, b_pw):
    D = x.shape[-1]
    y = F.conv2d(x.permute(0, 3, 1, 2), w_dw[:, None], b_dw, padding=1, groups=D).permute(0, 2, 3, 1)
    return torch.sigmoid(y @ w_pw.T + b_pw)


def exact(case, seed):
    """What `run` returns, from the definitions in float64."""
    state = _inputs(case, seed)
    kind = case["kind"]
    if kind == "features":
        w_h, b_h, w_pq, w_pk = weights = [t.double().requires_grad_() for t in state["weights"]]
        axis = torch.linspace(-1, 1, case["window"], dtype=torch.float64, device="cuda")
        x = torch.stack(torch.meshgrid(axis, axis, indexing="ij"), -1).reshape(-1, 2)
        rows = torch.cat([x] + [f(2.0 ** l * x) for l in range(case["L"]) for f in (torch.sin, torch.cos)], 1)
        hidden = torch.relu(rows @ w_h + b_h)
        pq, pk = hidden @ w_pq, hidden @ w_pk
        grads = torch.autograd.grad([pq, pk], weights, [state["dpq"].double(), state["dpk"].double()])
        return pq.detach(), pk.detach(), grads
    if kind == "block":
        layers = [_attention(*(state[k][l] for k in ("q", "k", "v", "pq", "pk", "dout")), w, 0, False) for l, w in enumerate(state["windows"])]
        tables = [(dpq.sum(0), dpk.sum(0)) for _, _, _, dpq, dpk in layers]
        return [l[0] for l in layers], tuple([l[2][i] for l in layers] for i in range(3)) + tuple([t[i] for t in tables] for i in range(2))
    dout = state.get("dout")
    if kind == "gated":
        x, *conv = leaves = [t.double().requires_grad_() for t in [state["x"], *state["conv"]]]
        gate = _gate(x, *conv)
        dout = dout.double() * gate.detach().reshape(dout.shape)
    out, lse, grads, dpq, dpk = _attention(*(state[k] for k in ("q", "k", "v", "pq", "pk")), dout, case["window"], case["shift"],
                                           case.get("masked", False))
    if kind == "infer":
        return out
    if not case.get("headwise"):
        dpq, dpk = dpq.sum(0), dpk.sum(0)
    grads = (*grads, dpq, dpk)
    if kind == "gated":
        dgate = (state["dout"].double() * out).reshape(gate.shape)
        return out * gate.detach().reshape(out.shape), grads, torch.autograd.grad(gate, leaves, dgate)
    return out, lse, grads


def _attending(side, window, shift, masked):
    """Pairs of positions of one axis that attend to each other: the sum over its windows of the squared number of real
    positions in it (with a mask, of the squared sizes of the last window's two parts)."""
    extended = -(-side // window) * window
    pairs = 0
    for start in range(0, extended, window):
        places = [(start + i + shift) % extended for i in range(window)]
        wrapped = start + window == extended and masked and shift > 0
        for part in ([places[:window - shift], places[window - shift:]] if wrapped else [places]):
            pairs += sum(p < side for p in part) ** 2
    return pairs


def _layer(case, window, shift, masked, backward):
    B, H, W, heads, d, r = (case[k] for k in ("B", "H", "W", "heads", "d", "r"))
    pairs = B * heads * _attending(H, window, shift, masked) * _attending(W, window, shift, masked)
    tables = heads if case.get("headwise") else 1
    row, table = B * H * W * heads * d * 2, tables * window * window * r * 2
    work = {"flops": 2 * pairs * (2 * d + r), "bytes": 4 * row + 2 * table}            # q, k, v in, out
    if backward:
        lse = B * H * W * heads * 4
        work["flops"] += 2 * pairs * (5 * d + 3 * r)
        work["bytes"] += lse + 8 * row + lse + 2 * table + 2 * 2 * table               # lse out; q, k, v, out, dout, lse in, dq, dk, dv, dPq, dPk
    return work


def work(case):
    kind = case["kind"]
    if kind == "features":
        n, rows, dh, r = case["window"] ** 2, 2 + 4 * case["L"], case["dh"], case["r"]
        weights = 4 * (rows * dh + dh + 2 * dh * r)
        mults = n * (rows * dh + 2 * dh * r)
        return {"flops": 2 * mults * 4, "bytes": 3 * weights + 2 * 2 * n * r + 2 * 4 * n * r}
    if kind == "block":
        layers = [_layer(case, w, 0, False, True) for w in _windows(case)]
        return {k: sum(l[k] for l in layers) for k in ("flops", "bytes")}
    total = _layer(case, case["window"], case["shift"], case.get("masked", False), kind != "infer")
    if kind == "gated":
        pixels, D = case["B"] * case["H"] * case["W"], case["heads"] * case["d"]
        total["flops"] += pixels * (2 * D * D + 18 * D + 6 * D * D + 36 * D)
        total["bytes"] += pixels * D * 2 * (2 + 3 + 5 + 3)                             # gate, product, its chain rule, the gate's
    return total


def tolerance(case):
    # About four times what the tensor-core kernels and the fp32 kernels of the library differ by on these cases.
    # Attention: bf16 results (half a unit in the last place is 2^-9) of probabilities rounded to bf16, 2.9e-3 at most over
    # all results; gate weights' gradients add a bf16 product per term, 4.3e-3.  Features: bf16 results of short fp32 sums,
    # of which another order of summation turns a few roundings.
    if case["kind"] == "features":
        return {"rel": 1e-3, "max": 0.02}
    return {"rel": 1.5e-2 if case["kind"] == "gated" else 1e-2, "max": 0.2}
