"""The work that users of the gated subspace layer have it do, as cases to time.

Five kinds of case, all through the public entry points of the package:

  stack   one decode step of a whole model (``Stack.step`` as one captured CUDA graph, or
          ``Stack.step_host`` with host buffers): 1 to 64 tokens per step
  layer   one call of one group of maps (``Layer.forward``): 1 to 64 tokens
  static  the same for callers that cannot allocate (``gsi_forward_static``): 1 to 4 tokens
  image   the cached image W P of one map (``gsi_build_image``), once per map at model load
  track   a token tested against the basis in use (``Layer.extend_basis``); nearly every token
          lies inside the tracked subspace, so nothing is appended

Shapes are those of the repository's configurations (GPT-2, GPT-J, OPT: widths, ranks, eps,
gate rates) and of its tests (ragged widths).  Activations are low rank plus noise: with one
token per call the noise puts the share ``gate`` of the tokens above eps; with several tokens
per call the share ``gate`` of them are full-rank outliers and the others lie far below eps.
"""
import ctypes
import math

import torch

import paper_2605_03109_b200 as gsi

# model -> (groups of a layer: input width, output widths), layers, independent neighbours
MODELS = {
    "gpt2": (((768, (2304,)), (768, (768,)), (768, (3072,)), (3072, (768,))), 12, ()),
    "gptj": (((4096, (4096, 4096, 4096, 16384)), (4096, (4096,)), (16384, (4096,))), 28, (1,)),
    "opt": (((4096, (4096, 4096, 4096)), (4096, (4096,)), (4096, (16384,)), (16384, (4096,))), 32, ()),
}


def listed():
    def stack(name, model, k, n, eps, gate, host=False, fp8=False):
        return dict(name=name, kind="stack", model=model, layers=MODELS[model][1], k=k, n=n, eps=eps,
                    gate=gate, host=host, fp8=fp8)

    def layer(name, d, outs, k, n, gate, f32=False):
        return dict(name=name, kind="layer", d=d, outs=outs, k=k, n=n, cap=n, eps=0.05, gate=gate, f32=f32)

    qkv_fc = "4096,4096,4096,16384"
    return [
        # the smallest call: one token through one map of GPT-2, where launches are what counts
        layer("cfc_1", 768, "3072", 64, 1, 0.05),
        # one token through the widest group of GPT-J, for programs with their own layer loop
        layer("qkv_fc_1", 4096, qkv_fc, 256, 1, 0.10),
        # the same group for a full batch
        layer("qkv_fc_64", 4096, qkv_fc, 256, 64, 0.10),
        # widths that divide into nothing, an odd number of tokens
        layer("ragged_21", 3000, "1000,504,72", 200, 21, 0.25),
        # a basis kept in fp32, small batch
        layer("f32_basis_16", 768, "2304", 128, 16, 0.10, f32=True),
        # decode of a small model, most tokens gated
        stack("gpt2_step", "gpt2", 128, 1, 0.05, 0.70),
        # the headline: GPT-J decode, one token in ten gated
        stack("gptj_step", "gptj", 256, 1, 0.05, 0.10),
        # the same with host buffers, the call of a server that keeps activations on the host
        stack("gptj_step_host", "gptj", 256, 1, 0.05, 0.10, host=True),
        # OPT decode at the largest rank and threshold of the sweep
        stack("opt_step_k512", "opt", 512, 1, 0.10, 0.25),
        # batched decode, the largest case
        stack("gptj_step_64", "gptj", 256, 64, 0.05, 0.10),
        # model load: the image of the widest map
        dict(name="image_fc", kind="image", o=16384, d=4096, k=256, f32=False),
        # online basis tracking at the widest group
        dict(name="track_qkv_fc", kind="track", d=4096, outs=qkv_fc, k=256, tau=0.05, f32=False),
    ]


def _log_int(rng, lo, hi, step=1):
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(lo, min(hi, int(round(v / step)) * step))


def draw(rng):
    kind = rng.choices(("stack", "layer", "static", "image", "track"), (6, 8, 2, 2, 2))[0]
    if kind == "stack":
        model = rng.choice(sorted(MODELS))
        n = 1 if rng.random() < 0.5 else _log_int(rng, 2, 64)
        most = 26 if model == "opt" else MODELS[model][1]   # no more weights than the largest listed case
        return dict(kind=kind, model=model, layers=_log_int(rng, 2, most), k=rng.choice((128, 256, 512)), n=n,
                    eps=rng.choice((0.01, 0.05, 0.1)), gate=rng.choice((0.01, 0.1, 0.25, 0.5, 1.0)),
                    host=rng.random() < 0.2, fp8=n == 1 and rng.random() < 0.2)
    f32 = rng.random() < 0.2
    if kind == "image":
        d, o = _log_int(rng, 768, 16384, 8), _log_int(rng, 768, 16384, 8)
        most = min(512, 16384 * 6144 * 256 // (o * d) // 8 * 8)   # a matrix and rank no dearer than GPT-J's
        return dict(kind=kind, o=o, d=d, k=_log_int(rng, 64, most, 8), f32=f32)
    # half of the groups have the tidy widths of models, the others any multiple of 8
    step = 128 if rng.random() < 0.5 else 8
    d = _log_int(rng, 256, 16384, step)
    k = min(d, rng.choice((64, 128, 256, 512)) if step == 128 else _log_int(rng, 16, 512, 8))
    outs = ",".join(str(_log_int(rng, step, 8192, step)) for _ in range(rng.randint(1, 4)))
    if kind == "track":
        return dict(kind=kind, d=d, outs=outs, k=k, tau=0.05, f32=f32)
    n = _log_int(rng, 1, 4 if kind == "static" else 64)
    cap = n if kind == "static" or rng.random() < 0.7 else 64
    return dict(kind=kind, d=d, outs=outs, k=k, n=n, cap=cap, eps=0.05,
                gate=rng.choice((0.01, 0.1, 0.25, 0.5, 1.0)), f32=f32)


# ---- inputs ------------------------------------------------------------------------------
def _bases(n, d, k, gen):
    """n orthonormal d x k bases in fp32 (Cholesky QR of Gaussians)."""
    a = torch.randn((n, d, k), device="cuda", generator=gen)
    low = torch.linalg.cholesky_ex(a.transpose(1, 2) @ a)[0]
    return torch.linalg.solve_triangular(low, a.transpose(1, 2), upper=False).transpose(1, 2).contiguous()


def _weights(shapes, gen):
    """bf16 matrices iid N(0, 0.02^2), one buffer."""
    flat = torch.empty(sum(o * d for o, d in shapes), dtype=torch.bfloat16, device="cuda")
    flat.normal_(0.0, 0.02, generator=gen)
    return [v.view(o, d) for v, (o, d) in zip(flat.split([o * d for o, d in shapes]), shapes)]


def _noise(d, k, rank, eps, share):
    """Noise scale that puts the share `share` of the tokens at ||r|| >= eps ||x||:
    ||r|| ~ sigma sqrt(d - k), ||x||^2 ~ chi-squared with `rank` degrees of freedom."""
    if share >= 1.0:
        return 4.0 * eps * math.sqrt(rank / max(8, d - k))
    # quantile of the normal distribution by bisection, then Wilson and Hilferty's cube
    lo, hi = -8.0, 8.0
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if 0.5 * math.erfc(-mid / math.sqrt(2.0)) < share else (lo, mid)
    c = 2.0 / (9.0 * rank)
    return eps * math.sqrt(rank * max(0.05, 1.0 - c + lo * math.sqrt(c)) ** 3 / max(8, d - k))


def _activations(q, tokens, n, eps, gate, gen):
    """[bases][tokens][d] fp32 around the bases q [bases][d][k]; n tokens travel together."""
    b, d, k = q.shape
    rank = max(1, int(round(0.78 * k)))
    sigma = _noise(d, k, rank, eps, gate) if n == 1 else 0.2 * eps * math.sqrt(rank / max(8, d - k))
    z = torch.randn((b, tokens, rank), device="cuda", generator=gen)
    x = z @ q[:, :, :rank].transpose(1, 2)
    x.add_(torch.randn((b, tokens, d), device="cuda", generator=gen), alpha=sigma)
    if n > 1:
        out = torch.rand((b, tokens), device="cuda", generator=gen) < gate
        far = torch.randn((b, tokens, d), device="cuda", generator=gen).mul_(math.sqrt(rank / d))
        x = torch.where(out[:, :, None], far, x)
    return x


def _stored(q, f32):
    return q if f32 else q.to(torch.bfloat16)


def _outs(case):
    return [int(v) for v in case["outs"].split(",")]


def _carve(flat, sizes):
    return list(flat.split(sizes))


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    kind = case["kind"]
    if kind == "stack":
        return _prepare_stack(case, gen)
    d, k = case["d"], case["k"]
    q = _bases(1, d, k, gen)
    P = _stored(q[0], case["f32"])
    if kind == "image":
        W, = _weights([(case["o"], d)], gen)
        return dict(kind=kind, W=W, P=P)
    Ws = _weights([(o, d) for o in _outs(case)], gen)
    if kind == "track":
        P[:, k - 1] = 0   # one column still free
        layer = gsi.Layer(Ws, P, case["tau"], max_tokens=1)
        x = _activations(q, 1, 2, case["tau"], 0.0, gen)[0, 0].contiguous()
        first = ctypes.c_void_p()   # the images of all maps, one block of the layer's workspace
        gsi.lib.gsi_get_image(layer.handle, 0, ctypes.byref(first))
        at = first.value - layer.workspace.data_ptr()
        images = layer.workspace[at:at + layer.O * k * 2].view(torch.bfloat16)
        return dict(kind=kind, layer=layer, x=x, tau=case["tau"], P=P, images=images,
                    k_active=torch.full((1,), k - 1, dtype=torch.int32, device="cuda"))
    x = _activations(q, case["n"], case["n"], case["eps"], case["gate"], gen)[0].contiguous()
    if kind == "static":
        WP = torch.cat([gsi.gsi_build_image(W, P) for W in Ws])
        return dict(kind=kind, Ws=Ws, P=P, WP=WP, eps=case["eps"], x=x)
    return dict(kind=kind, layer=gsi.Layer(Ws, P, case["eps"], max_tokens=case["cap"]), x=x)


def _prepare_stack(case, gen):
    groups, _, side = MODELS[case["model"]]
    L, k, n = case["layers"], case["k"], case["n"]
    steps = 1 if case["host"] else 16 if n == 1 else 4
    layers, xs = [None] * (L * len(groups)), [None] * (L * len(groups))
    flags = gsi.GSI_FLAG_FP8_IMAGE if case["fp8"] else 0
    for gi, (d, outs) in enumerate(groups):
        q = _bases(L, d, k, gen)
        x = _activations(q, steps * n, n, case["eps"], case["gate"], gen)
        W = _weights([(o, d) for _ in range(L) for o in outs], gen)
        for layer in range(L):
            at = layer * len(groups) + gi
            layers[at] = gsi.Layer(W[layer * len(outs):(layer + 1) * len(outs)], q[layer].to(torch.bfloat16),
                                   case["eps"], max_tokens=n, flags=flags)
            xs[at] = x[layer].contiguous()
    stack = gsi.Stack(layers, concurrent=[layer * len(groups) + i for layer in range(L) for i in side])
    # the outputs of all groups in one buffer (and, with host buffers, the inputs too): one copy each way
    y = torch.empty(sum(n * layer.O for layer in layers), dtype=torch.float32, device="cuda")
    y_sizes = [n * layer.O for layer in layers]
    ys = [v.view(n, -1) for v in _carve(y, y_sizes)]
    state = dict(kind="stack", stack=stack, y=y, graph=None)
    if case["host"]:
        x_host = torch.cat([x.reshape(-1) for x in xs]).cpu().pin_memory()
        x_dev = torch.empty_like(x_host, device="cuda")
        x_sizes = [x.numel() for x in xs]
        stack.bind(_carve(x_dev, x_sizes), ys=ys, n_steps=1)
        y_host = torch.empty(y.numel(), dtype=torch.float32).pin_memory()
        state.update(xs_host=_carve(x_host, x_sizes), ys_host=_carve(y_host, y_sizes), y_host=y_host,
                     gate_host=torch.empty((len(layers), n), dtype=torch.uint8).pin_memory())
        return state
    stack.bind(xs, ys=ys, n_steps=steps)
    stack.step()
    torch.cuda.synchronize()
    state["graph"] = torch.cuda.CUDAGraph()
    with torch.cuda.graph(state["graph"]):
        stack.step()
    return state


# ---- one pass ----------------------------------------------------------------------------
def run(state):
    kind = state["kind"]
    if kind == "stack":
        stack = state["stack"]
        if state["graph"] is None:
            stack.step_host(state["xs_host"], state["ys_host"], state["gate_host"])
            return dict(y=state["y_host"], gate=state["gate_host"])
        state["graph"].replay()
        return dict(y=state["y"], gate=stack.gate_log, rho=stack.rho_log)
    if kind == "layer":
        y, gate, rho = state["layer"].forward(state["x"])
        return dict(y=y, gate=gate, rho=rho)
    if kind == "static":
        y, gate, rho = gsi.gsi_forward_static(state["Ws"], state["P"], state["WP"], state["eps"], state["x"])
        return dict(y=y, gate=gate, rho=rho)
    if kind == "image":
        return dict(image=gsi.gsi_build_image(state["W"], state["P"]))
    appended, rho = state["layer"].extend_basis(state["x"], state["tau"], state["k_active"])
    return dict(appended=appended, rho=rho, k_active=state["k_active"], P=state["P"], images=state["images"])


def work(case):
    """Weights, bases and images once each, W only where a token of the call is expected to be
    gated, activations in and out; one multiply-add per matrix entry and token that uses it."""
    kind, k = case["kind"], case["k"]
    if kind == "image":
        o, d = case["o"], case["d"]
        return dict(bytes=2 * o * d + (4 if case["f32"] else 2) * d * k + 2 * o * k, flops=2 * o * d * k)
    if kind == "track":   # the basis and the token; the images are not read for a token inside the subspace
        d = case["d"]
        return dict(bytes=(4 if case["f32"] else 2) * d * k + 4 * d, flops=4 * d * k)
    if kind == "stack":
        groups, layers = MODELS[case["model"]][0], case["layers"]
        pb, wb = 2, 1 if case["fp8"] else 2
    else:
        groups, layers = ((case["d"], _outs(case)),), 1
        pb, wb = 4 if case["f32"] else 2, 2
    n = case["n"]
    any_gated = 1.0 - (1.0 - case["gate"]) ** n
    total = flops = 0.0
    for d, outs in groups:
        o = sum(outs)
        total += pb * d * k + wb * o * k + 2.0 * o * d * any_gated + 4.0 * n * (d + o)
        flops += n * (4.0 * d * k + 2.0 * o * k + 2.0 * o * d * case["gate"])
    return dict(bytes=layers * total, flops=layers * flops)


def tolerance(case):
    """Against a restatement in fp64 from the same stored matrices: outputs differ by 2e-5 to
    7e-5 (bf16 images whose fp32 sums fall on the other side of a rounding boundary: one last
    place, at most 2^-7 of the entry), and by 5e-4 to 1.6e-3 where the layer takes the gated
    residual as bf16 (batched calls at widths of whole tensor-core tiles).  Four times that.
    An FP8 image carries a flipped bf16 entry over to codes whose spacing is sixteen times wider."""
    if case["kind"] in ("layer", "stack"):
        widths = [(case["d"], _outs(case))] if case["kind"] == "layer" else MODELS[case["model"]][0]
        if case["n"] > 1 and all(d % 64 == 0 and all(o % 128 == 0 for o in outs) for d, outs in widths):
            return dict(rel=6e-3, max=0.032)
        if case.get("fp8"):
            return dict(rel=1.2e-3, max=0.06)
    return dict(rel=3e-4, max=0.016)
