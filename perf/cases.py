"""The work a user of the OffQ library has it do, as cases that can be timed and compared.

A case is one pass through the public entry points (``paper_2606_07116_gb300.offq``) over
buffers that a serving or conversion program keeps: quantize the activations of a
transformer block's linear layers, run its W4A4 linears, quantize its KV vectors; the same
through the per-group and the MXFP4 variants; the key / query rotation; the weight
preparation of a model load. Shapes are those of the repository's workloads (Llama-2-7B,
Llama-3-8B and Llama-2-70B layers) and generic ones around them.

Kinds:
  layers   the linears of a block (``part``: attn = q k v o, mlp = gate up down, block = both,
           one = a single layer) on T token rows, in one of three formats (``path``: token =
           per-token scale with offsets, group = per-group asymmetric, mx = MXFP4), with the
           KV4 quantizer of the block's keys and values where the part has them. ``graph``:
           the pass is one CUDA graph, as serving engines replay their small batches.
  keys     KV4 under a dense per-head rotation, and the same rotation of the queries.
  weights  offline weight preparation of one layer.
"""

from __future__ import annotations

import math

import torch

from paper_2606_07116_gb300 import offq as Q

DT = {"bf16": torch.bfloat16, "f16": torch.float16, "f32": torch.float32}
BYTES = {"bf16": 2, "f16": 2, "f32": 4}
HD = 128         # head dimension
GROUP = 128      # activation group of the per-group path
GRAPH_T = 512    # batches up to this replay a CUDA graph


def block_for(K):
    """Offset / rotation block of K channels: K itself if it is a power of two up to 8192,
    else the largest power of two up to 1024 that divides it."""
    if K & (K - 1) == 0:
        return min(K, 8192)
    return min(K & -K, 1024)


def layers_case(name, part, T, hidden, inter=0, kv=0, path="token", x="bf16", out="bf16", dist="normal", n_out=4,
                mult=100.0):
    c = {"name": name, "kind": "layers", "path": path, "part": part, "T": T, "hidden": hidden, "inter": inter,
         "kv_heads": kv, "x": x, "out": out, "dist": dist, "n_out": n_out, "mult": mult, "graph": T <= GRAPH_T}
    return c


def listed():
    return [
        # The smallest layer call: 16 fp32 tokens through one rotated 512 x 512 layer, called eagerly.
        dict(layers_case("toy_f32", "one", 16, 512, 512, x="f32", out="f32", n_out=2, mult=50.0), graph=False),
        # One decode step of a Llama-2-7B block for a single stream, and for a batch of 32.
        layers_case("decode_1", "block", 1, 4096, 11008, 32),
        layers_case("decode_32", "block", 32, 4096, 11008, 32),
        # A chunk of a prefill (or a verified draft) joining a batch: between decode and prefill, an odd size.
        layers_case("chunk_201", "block", 201, 4096, 11008, 32),
        # The prefill of a 2048-token prompt through a Llama-2-7B block.
        layers_case("prefill_7b", "block", 2048, 4096, 11008, 32),
        # Llama-3-8B MLP on heavy-tailed activations, 4096 tokens.
        layers_case("mlp_8b", "mlp", 4096, 4096, 14336, dist="student_t3", n_out=3),
        # The largest: a Llama-2-70B block (8 KV heads) at 8192 tokens.
        layers_case("prefill_70b", "block", 8192, 8192, 28672, 8, n_out=6, mult=200.0),
        # A ragged half-precision MLP: odd token count, hidden size that is no power of two.
        layers_case("mlp_ragged_f16", "mlp", 777, 2560, 6912, x="f16", out="f16"),
        # The paper's evaluated setting (per-group asymmetric activations), Llama-2-7B MLP.
        layers_case("group_mlp_7b", "mlp", 2048, 4096, 11008, path="group"),
        # MXFP4 with offsets, Llama-3-8B MLP.
        layers_case("mx_mlp_8b", "mlp", 4096, 4096, 14336, path="mx", dist="student_t3", n_out=3),
        # Keys into the 4-bit cache and queries, under a dense per-head rotation.
        {"name": "keys_4096", "kind": "keys", "form": "prepared", "T": 4096, "heads": 32, "x": "bf16"},
        # Model load: a down projection's weights rotated, quantized and packed.
        {"name": "weights_down_8b", "kind": "weights", "N": 4096, "K": 14336, "x": "f32", "rotate": True},
    ]


def log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["token", "group", "mx", "keys", "weights"], [8, 3, 3, 1, 1])[0]
    if kind == "keys":
        form = rng.choice(["prepared", "reflected", "dense"])
        return {"kind": "keys", "form": form, "T": log_int(rng, 1, 8192), "heads": rng.choice([8, 16, 32, 40]),
                "x": "bf16" if form != "dense" else rng.choice(["bf16", "f16", "f32"])}
    if kind == "weights":
        K = 128 * log_int(rng, 4, 224)
        return {"kind": "weights", "N": log_int(rng, 64, 8192), "K": K, "x": rng.choice(["f32", "bf16"]),
                "rotate": rng.random() < 0.5}
    hidden = rng.choice([512, 1024, 2048, 4096, 8192, 128 * log_int(rng, 5, 64)])
    inter = 128 * max(4, int(round(hidden * rng.uniform(2.0, 4.0) / 128)))
    inter = min(inter, 28672)
    part = rng.choice(["attn", "mlp", "block", "one"])
    kv = max(1, hidden // HD // rng.choice([1, 4, 8])) if part in ("attn", "block") else 0
    # Per-pass work stays below the largest listed case's; the two slower formats below a tenth of it.
    most = {"token": 4e12, "group": 6e11, "mx": 1.2e12}[kind]
    T = log_int(rng, 1, 8192)
    while T > 1 and 2.0 * T * hidden * (3 * inter + 4 * hidden) > most:
        T //= 2
    x = rng.choices(["bf16", "f16", "f32"], [6, 2, 1])[0]
    c = layers_case("", part, T, hidden, inter, kv, path=kind, x=x, out=rng.choice([x, "bf16"]),
                    dist=rng.choice(["normal", "student_t3"]), n_out=rng.choice([2, 3, 4, 6]),
                    mult=rng.choice([50.0, 100.0, 200.0]))
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# What a case is made of
# ---------------------------------------------------------------------------

def inputs_of(case):
    """[(input, channels, rotated online, [(layer, output channels)])] of a layers case."""
    h, i, kv = case["hidden"], case["inter"], case["kv_heads"] * HD
    if case["part"] == "one":
        return [("x", h, True, [("y", i)])]
    attn = [("x_qkv", h, False, [("q", h), ("k", kv), ("v", kv)]), ("x_o", h, False, [("o", h)])]
    mlp = [("x_mlp", h, False, [("gate", i), ("up", i)]), ("x_down", i, True, [("down", h)])]
    return {"attn": attn, "mlp": mlp, "block": attn + mlp}[case["part"]]


def generator(seed, salt):
    return torch.Generator(device="cuda").manual_seed((int(seed) * 1000003 + salt * 7919) % (1 << 62))


def activations(case, K, gen):
    """Token rows in the basis the online path sees: bulk entries, and outlier channels k * (K / n_out) of
    mult * (1 + 0.1 z) on every token."""
    T = case["T"]
    x = torch.randn(T, K, generator=gen, device="cuda")
    if case["dist"] == "student_t3":
        chi = sum(torch.randn(T, K, generator=gen, device="cuda") ** 2 for _ in range(3))
        x = x / (chi / 3).sqrt()
    amp = case["mult"] * (1 + 0.1 * torch.randn(T, generator=gen, device="cuda"))
    step = K // case["n_out"]
    for c in range(case["n_out"]):
        x[:, c * step] = amp
    return x.to(DT[case["x"]])


def hadamard(g, dtype):
    h = torch.ones(1, 1, dtype=dtype, device="cuda")
    while h.shape[0] < g:
        h = torch.cat([torch.cat([h, h], 1), torch.cat([h, -h], 1)], 0)
    return h


def rotated(x, g):
    """x blockdiag(H_g), not normalised."""
    h = hadamard(g, x.dtype)
    return (x.reshape(-1, g) @ h).reshape(x.shape)


E2M1 = (0.0, 0.5, 1.0, 1.5, 2.0, 3.0, 4.0, 6.0)


def layer_weights(N, K, g, rotate, path, gen, dtype=torch.float32):
    """Weights as a weight quantizer leaves them, on the 4-bit grid of the basis they are used in (uniform per
    output channel, or MXFP4 blocks); a rotated layer's are taken back to the basis the preparation rotates from.
    So the codes the preparation finds are those of the grid, in any precision."""
    if path == "mx":
        grid = torch.tensor(E2M1, device="cuda")
        w = torch.randn(N, K // 32, 32, generator=gen, device="cuda")
        q = grid[torch.bucketize(w.abs() * 2.0, grid[1:] * 0.75).clamp(max=7)] * w.sign()
        q[:, :, 0] = 6.0 * w[:, :, 0].sign()
        sh = torch.randint(0, 3, (N, K // 32, 1), generator=gen, device="cuda")
        w = (q * torch.exp2(sh - 9.0)).reshape(N, K)
    else:
        q = (torch.randn(N, K, generator=gen, device="cuda") * 2.4).round_().clamp_(-7, 7)
        q[:, 0] = 7.0
        s = 0.02 / 2.4 * (0.8 + 0.4 * torch.rand(N, 1, generator=gen, device="cuda"))
        w = q.mul_(s)
    if rotate:
        w = rotated(w, g).mul_(1.0 / math.sqrt(g))
    return w.to(dtype)


def key_transforms(case, gen):
    """Per head the top-1 direction v, a permutation that keeps channel 0 first, and M = U3 P3 H3."""
    H = case["heads"]
    v = torch.randn(H, HD, generator=gen, device="cuda")
    perm = torch.stack([torch.cat([torch.zeros(1, dtype=torch.int64, device="cuda"),
                                   1 + torch.randperm(HD - 1, generator=gen, device="cuda")]) for _ in range(H)])
    v64 = v.double() / v.double().norm(dim=1, keepdim=True)
    w = v64.clone()
    w[:, 0] -= 1.0
    U = torch.eye(HD, dtype=torch.float64, device="cuda") - 2 * w[:, :, None] * w[:, None, :] / (w * w).sum(1)[:, None, None]
    M = torch.stack([U[h][:, perm[h]] for h in range(H)]) @ hadamard(HD, torch.float64) / math.sqrt(HD)
    return v, perm.to(torch.int32), v64, M


def key_inputs(case, gen, v64):
    """Keys with a bias along each head's direction, and queries."""
    T, H = case["T"], case["heads"]
    k = torch.randn(T, H, HD, generator=gen, device="cuda")
    k += 20.0 * (1 + 0.1 * torch.randn(T, H, 1, generator=gen, device="cuda")) * v64.float()
    return k.to(DT[case["x"]]), torch.randn(T, H, HD, generator=gen, device="cuda").to(DT[case["x"]])


# ---------------------------------------------------------------------------
# The measured pass
# ---------------------------------------------------------------------------

def bytes_(n):
    # Zeroed: rows that pad a buffer to a multiple of 32 are not written.
    return torch.zeros(n, dtype=torch.uint8, device="cuda")


def floats(*shape):
    return torch.zeros(shape, dtype=torch.float32, device="cuda")


def prepare(case, seed):
    s = {"case": case}
    if case["kind"] == "weights":
        N, K = case["N"], case["K"]
        g = block_for(K)
        s["w"] = layer_weights(N, K, g, case["rotate"], "token", generator(seed, 1), DT[case["x"]])
        s["out"] = {"codes": bytes_(Q.offq_weight_codes_bytes(N, K)), "scale": floats(N), "offsum": floats(K // g, N)}
        return s
    if case["kind"] == "keys":
        T, H, gen = case["T"], case["heads"], generator(seed, 2)
        v, perm, v64, M = key_transforms(case, gen)
        s["k"], s["q"] = key_inputs(case, gen, v64)
        if case["form"] == "prepared":
            s["rot"] = Q.prepare_key_rotation(M.float())
        elif case["form"] == "reflected":
            s["rot"] = Q.prepare_key_reflection(v, perm, device="cuda")
        else:
            s["rot"] = M.float().contiguous()
        s["out"] = {"codes": bytes_(T * H * HD // 2), "scale": floats(T, H), "offset": floats(T, H),
                    "q": torch.empty(T, H, HD, dtype=DT[case["x"]], device="cuda")}
        return s
    T, path, out = case["T"], case["path"], {}
    s.update(layers=[], x={}, w={}, out=out)
    for i, (name, K, rotate, layers) in enumerate(inputs_of(case)):
        g = block_for(K)
        s["x"][name] = activations(case, K, generator(seed, 10 + i))
        out[name] = {"codes": bytes_(Q.offq_act_codes_bytes(T, K))}
        if path == "group":
            out[name].update(scale=floats(T, K // GROUP), zero=floats(T, K // GROUP))
        else:
            out[name].update(scale=floats(T), offset=floats(T, K // g))
        if path == "mx":
            out[name]["shifts"] = bytes_(Q.mx_shift_bytes(T, K))
        for j, (layer, N) in enumerate(layers):
            w = layer_weights(N, K, g, rotate, path, generator(seed, 100 + 10 * i + j))
            if path == "mx":
                s["w"][layer] = Q.prepare_weight_mx(w, g, rotate=rotate)
            else:
                s["w"][layer] = Q.prepare_weight(w, g, rotate=rotate)
                if path == "group":
                    s["w"][layer] += (Q.weight_group_sums(s["w"][layer][0], N, K, GROUP),)
            out[layer] = torch.empty(T, N, dtype=DT[case["out"]], device="cuda")
            del w
    if case["kv_heads"]:
        gen = generator(seed, 3)
        for name in ("cache_k", "cache_v"):
            kv = torch.randn(T, case["kv_heads"], HD, generator=gen, device="cuda")
            kv[:, :, 0] = 20.0 * (1 + 0.1 * torch.randn(T, case["kv_heads"], generator=gen, device="cuda"))
            s["x"][name] = kv.to(DT[case["x"]])
            out[name] = {"codes": bytes_(T * case["kv_heads"] * HD // 2), "scale": floats(T, case["kv_heads"]),
                         "offset": floats(T, case["kv_heads"])}
    if case["graph"]:
        # As an engine does at start-up: one eager pass, then the capture that every later pass replays.
        layers_pass(s)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            layers_pass(s)
        s["graph"] = graph
    return s


def layers_pass(s):
    case, x, w, out = s["case"], s["x"], s["w"], s["out"]
    T, path = case["T"], case["path"]
    for name, K, rotate, layers in inputs_of(case):
        g, xi, o = block_for(K), x[name], out[name]
        rot = Q.OFFQ_ROTATE if rotate else 0
        if path == "token":
            Q.offq_quantize_act(xi, T, K, K, g, rot | Q.OFFQ_OFFSET, o["codes"], o["scale"], o["offset"])
        elif path == "group":
            Q.offq_quantize_act_group(xi, T, K, K, g, GROUP, rot, o["codes"], o["scale"], o["zero"])
        else:
            Q.offq_quantize_act_mx(xi, T, K, K, g, rot | Q.OFFQ_OFFSET, o["codes"], o["shifts"], o["scale"], o["offset"])
        for layer, N in layers:
            y, wl = out[layer], w[layer]
            if path == "token":
                Q.offq_w4a4_linear(o["codes"], o["scale"], o["offset"], T, N, K, g, *wl, y, N)
            elif path == "group":
                Q.offq_w4a4_linear_group(o["codes"], o["scale"], o["zero"], T, N, K, GROUP, wl[0], wl[1], wl[3], y, N)
            else:
                Q.offq_mx_linear(o["codes"], o["shifts"], o["scale"], o["offset"], T, N, K, g, *wl, y, N)
    for name, rot in (("cache_k", Q.OFFQ_ROTATE), ("cache_v", 0)):
        if name in out:
            o, H = out[name], case["kv_heads"]
            Q.offq_kv4_quantize(x[name], T, H, HD, H * HD, rot | Q.OFFQ_OFFSET, o["codes"], o["scale"], o["offset"])


def run(s):
    case, o = s["case"], s["out"]
    if case["kind"] == "weights":
        Q.offq_prepare_weight(s["w"], case["N"], case["K"], block_for(case["K"]), case["rotate"], o["codes"],
                              o["scale"], o["offsum"])
    elif case["kind"] == "keys":
        T, H, ld = case["T"], case["heads"], case["heads"] * HD
        kv4, rot = {"prepared": (Q.offq_kv4_quantize_prepared, Q.offq_rotate_heads_prepared),
                    "reflected": (Q.offq_kv4_quantize_reflected, Q.offq_rotate_heads_reflected),
                    "dense": (Q.offq_kv4_quantize_rotated, Q.offq_rotate_heads)}[case["form"]]
        kv4(s["k"], T, H, HD, ld, s["rot"], Q.OFFQ_OFFSET, o["codes"], o["scale"], o["offset"])
        rot(s["q"], T, H, HD, ld, s["rot"], o["q"], ld)
    elif "graph" in s:
        s["graph"].replay()
    else:
        layers_pass(s)
    return o


# ---------------------------------------------------------------------------
# What a pass cannot do without, and what it has to give
# ---------------------------------------------------------------------------

def work(case):
    if case["kind"] == "weights":
        N, K = case["N"], case["K"]
        return {"bytes": N * K * BYTES[case["x"]] + N * K // 2 + 4 * N * (1 + K // block_for(K)),
                "flops": N * K * (math.log2(block_for(K)) if case["rotate"] else 1)}
    if case["kind"] == "keys":
        rows = case["T"] * case["heads"]
        return {"bytes": rows * (3 * HD * BYTES[case["x"]] + HD // 2 + 8) + case["heads"] * HD * HD * 4,
                "flops": 2 * rows * 2 * HD * HD}
    T, path, b, f = case["T"], case["path"], 0, 0
    for _, K, rotate, layers in inputs_of(case):
        g = block_for(K)
        side = {"token": 4 * (1 + K // g), "group": 8 * (K // GROUP), "mx": K // 32 + 4 * (1 + K // g)}[path]
        b += T * (K * BYTES[case["x"]] + K // 2 + side)
        for _, N in layers:
            tables = {"token": 4 * (1 + K // g), "group": 4 * (1 + K // GROUP), "mx": K // 32 + 4 * (1 + K // g)}[path]
            b += N * (K // 2 + tables) + T * N * BYTES[case["out"]]
            f += 2 * T * N * K
    b += 2 * T * case["kv_heads"] * (HD * BYTES[case["x"]] + HD // 2 + 8)
    return {"bytes": b, "flops": f}


def tolerance(case):
    """A code whose value lies within the rounding error of a tie may take either neighbour: a share of the packed
    bytes may differ, and each such code moves one row's outputs by a code step (about 1 / (2.5 sqrt(K)) of their
    root mean square). The rest is the rounding of the output type."""
    if case["kind"] == "weights":
        return {"rel": 1e-6, "max": 1e-5, "differ": 1e-4} if case["x"] == "f32" else {"rel": 1e-5, "max": 1e-3, "differ": 1e-3}
    out = case["x"] if case["kind"] == "keys" else case["out"]
    rel = {"bf16": 8e-3, "f16": 1e-3, "f32": 1e-5 if case["kind"] == "keys" else 1e-3}[out]
    # A zero-point at a tie moves by one step of about eight.
    return {"rel": rel, "max": 0.3 if case.get("path") == "group" else 0.1, "differ": 1e-3}


def offsets_and_residual(y, g):
    T, K = y.shape
    o = y.reshape(T, K // g, g).mean(2)
    return o, y - o.repeat_interleave(g, 1)


def symmetric(r):
    s = r.abs().amax(-1, keepdim=True) / 7
    return s, torch.where(s > 0, r / s, torch.zeros_like(r)).round_().clamp_(-7, 7)


def mx(r):
    """Block exponents kept within 6 of the row's largest, E2M1 magnitudes (ties to the even code)."""
    T, K = r.shape
    amax = r.reshape(T, K // 32, 32).abs().amax(2)
    X = torch.where(amax > 0, torch.frexp(amax)[1].double() - 3, torch.full_like(amax, -1e9))
    top = X.amax(1, keepdim=True)
    scale = torch.exp2(torch.maximum(X, top - 6))
    v = (r.reshape(T, K // 32, 32) / scale[:, :, None])
    a = v.abs()
    step = torch.where(a < 2, 0.5, torch.where(a < 4, 1.0, 2.0))
    q = ((a / step).round() * step).clamp(max=6.0) * v.sign()
    return (q * scale[:, :, None]).reshape(T, K), torch.exp2(top - 6)


def exact(case, seed):
    if case["kind"] == "weights":
        g = block_for(case["K"])
        w = layer_weights(case["N"], case["K"], g, case["rotate"], "token", generator(seed, 1), DT[case["x"]]).double()
        s, q = symmetric(rotated(w, g) / math.sqrt(g) if case["rotate"] else w)
        return {"codes": None, "scale": s[:, 0], "offsum": q.reshape(case["N"], -1, g).sum(2).T.contiguous()}
    if case["kind"] == "keys":
        gen = generator(seed, 2)
        _, _, v64, M = key_transforms(case, gen)
        M = M.float().double() if case["form"] != "reflected" else M
        k, q = key_inputs(case, gen, v64)
        y = torch.einsum("thi,hij->thj", k.double(), M)
        o = y.mean(2)
        s, _ = symmetric(y - o[:, :, None])
        return {"codes": None, "scale": s[:, :, 0], "offset": o, "q": torch.einsum("thi,hij->thj", q.double(), M)}
    if case["path"] != "token" and work(case)["flops"] > 6e12:
        return None
    T, path, out = case["T"], case["path"], {}
    for i, (name, K, rotate, layers) in enumerate(inputs_of(case)):
        g = block_for(K)
        x = activations(case, K, generator(seed, 10 + i)).double()
        y = rotated(x, g) / math.sqrt(g) if rotate else x
        del x
        if path == "group":
            yg = y.reshape(T, K // GROUP, GROUP)
            lo, hi = yg.amin(2), yg.amax(2)
            sg, span = (hi - lo) / 15, torch.where(hi > lo, hi - lo, torch.ones_like(lo))
            z = -(15 * lo / span).round()
            u = ((15 * yg / span[:, :, None]).round() + z[:, :, None]).clamp(0, 15)
            a = ((u - z[:, :, None]) * sg[:, :, None]).reshape(T, K)
            out[name] = {"codes": None, "scale": sg, "zero": z}
        else:
            o, r = offsets_and_residual(y, g)
            if path == "token":
                sa, a = symmetric(r)
                out[name] = {"codes": None, "scale": sa[:, 0], "offset": o}
            else:
                a, sa = mx(r)
                out[name] = {"codes": None, "shifts": None, "scale": sa[:, 0], "offset": o}
            del r
        del y
        for j, (layer, N) in enumerate(layers):
            w = layer_weights(N, K, g, rotate, path, generator(seed, 100 + 10 * i + j)).double()
            w = rotated(w, g) / math.sqrt(g) if rotate else w
            if path == "mx":
                wq, _ = mx(w)
                out[layer] = a @ wq.T + o @ wq.reshape(N, K // g, g).sum(2).T
            else:
                sw, wq = symmetric(w)
                if path == "group":
                    out[layer] = (a @ wq.T) * sw.T
                else:
                    # Whole numbers below 2^24: their fp32 products and sums are exact.
                    p = (a.float() @ wq.float().T).double()
                    out[layer] = (p.mul_(sa) + o @ wq.reshape(N, K // g, g).sum(2).T) * sw.T
            del w, wq
    if case["kv_heads"]:
        gen = generator(seed, 3)
        for name in ("cache_k", "cache_v"):
            kv = torch.randn(T, case["kv_heads"], HD, generator=gen, device="cuda")
            kv[:, :, 0] = 20.0 * (1 + 0.1 * torch.randn(T, case["kv_heads"], generator=gen, device="cuda"))
            y = kv.to(DT[case["x"]]).double().reshape(-1, HD)
            y = rotated(y, HD) / math.sqrt(HD) if name == "cache_k" else y
            o, r = offsets_and_residual(y, HD)
            s, _ = symmetric(r)
            out[name] = {"codes": None, "scale": s.reshape(T, -1), "offset": o.reshape(T, -1)}
    return out
