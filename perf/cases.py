"""Performance cases of the RPD commit step: what programs that decode with it have it do.

A case names an entry point and the sizes and options of one call:

    call        "step" | "batched" | "host" | "noalloc" | "shard" | "loop"
    d, V        hidden size and vocabulary entries of the LM head (for "shard": of the slice)
    K           window layers
    B, N        canvases and positions per canvas
    masked      masked positions over all canvases
    tau, budget thresholds of the call; profile and block: the rule
    projection  "all" | "lazy" | "auto"
    parts       "shard": slices of the vocabulary;  steps: "loop": most steps of one launch

The inputs are drawn on the GPU from the seed alone, by the recipe of the repository's workloads:
a head W ~ N(0, 1.28/sqrt(d)) (0.02 at d = 4096), a gain 1 + N(0, 0.1), and hidden states
h[k][p] = a_k b_p sigma W_t/|W_t| + N(0, 1) whose signal is strong at both ends of the canvas, so
that a step meets confident, band and uncertain positions; a tenth of the positions read another
token in the penultimate window layer.
"""
import ctypes
import math

import numpy as np
import torch

import paper_2609_36452_gb300 as rpd

LLADA = {"d": 4096, "V": 126464}
DREAM = {"d": 3584, "V": 152064}
EPS = 1e-6
LARGEST_FLOPS = 2.0 * 6 * 5325 * 4096 * 126464  # the largest listed case's


def _case(name, call, head, K, B, N, masked, tau=0.9, budget=1.0, profile="llada", block=0,
          projection="all", parts=1, steps=0):
    c = dict(call=call, d=head["d"], V=head["V"], K=K, B=B, N=N, masked=masked, tau=tau,
             budget=budget, profile=profile, block=block, projection=projection, parts=parts,
             steps=steps)
    return dict(c, name=name) if name else c


def listed():
    return [
        # a small model's step: nothing but latency, launches and host work
        _case("tiny_step", "step", {"d": 256, "V": 4096}, 3, 1, 64, 64),
        # the last steps of a decode: a handful of positions, bound by reading the head
        _case("llada_tail", "step", LLADA, 4, 1, 256, 5),
        # late in a decode, a ragged row count (280) where reading the head and the contraction
        # take equally long
        _case("llada_late", "step", LLADA, 4, 1, 256, 70),
        # a decode's first step: the whole canvas is masked
        _case("llada_first", "step", LLADA, 4, 1, 256, 256),
        # another model's head and profile, half of a longer canvas left
        _case("dream_mid", "step", DREAM, 4, 1, 512, 267, 0.85, 2.0, "dream"),
        # the paper's 16-layer window, projection chosen on the device
        _case("llada_window16_auto", "step", LLADA, 16, 1, 256, 256, projection="auto"),
        # serving: many long canvases in one call, the largest one
        _case("serving", "batched", LLADA, 6, 8, 1024, 5325, budget=1.5),
        # serving of a few odd-length canvases with lazy projection
        _case("serving_lazy", "batched", DREAM, 4, 3, 333, 601, 0.85, 2.0, "dream", projection="lazy"),
        # a program whose hidden states lie in pinned host memory
        _case("llada_host", "host", LLADA, 4, 1, 256, 31),
        # a caller that owns all device memory, with the RPD-block rule
        _case("dream_noalloc_block", "noalloc", DREAM, 4, 1, 256, 203, 0.85, 2.0, "dream_block", 32),
        # one of eight vocabulary slices' statistics
        _case("llada_shard", "shard", {"d": 4096, "V": 15872}, 4, 1, 256, 187, parts=8),
        # steps repeated on the device in one launch, from the middle of a decode on
        _case("llada_loop", "loop", LLADA, 4, 1, 256, 149, steps=6),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    """Any entry point over: the two models' heads or any head of d 64..4096 (multiples of 8) and
    V 256..152064; windows of 1..16 layers; canvases of 8..2048 positions, 1..16 of them; any
    masked count; every projection and rule."""
    call = rng.choice(["step"] * 5 + ["batched"] * 2 + ["host", "noalloc", "shard", "loop"])
    pick = rng.random()
    head = LLADA if pick < 0.4 else DREAM if pick < 0.6 else {
        "d": 8 * _log_int(rng, 8, 512), "V": _log_int(rng, 256, 152064)}
    parts = 1
    if call == "shard":
        parts = rng.choice([2, 3, 4, 8])
        head = dict(head, V=max(256, (head["V"] // parts) // 256 * 256))
    K = rng.choice([1, 2, 3, 4, 4, 4, 5, 6, 8, 16])
    B = _log_int(rng, 2, 16) if call == "batched" else 1
    N = _log_int(rng, 8, 1024 // K if call == "noalloc" else 2048)
    while B * N > 8192 or K * B * N * head["d"] > 6 * 8192 * 4096:
        N = N // 2 + 1
    masked = _log_int(rng, 1, B * N)
    steps = rng.randint(2, 6) if call == "loop" else 0
    while 2.0 * K * masked * head["d"] * head["V"] * max(1, steps) > LARGEST_FLOPS:
        masked = masked // 2 + 1
    profile = rng.choice(["llada"] * 4 + ["dream"] * 3 + ["llada_block", "dream_block"])
    tau, budget = rng.choice([(0.9, 1.0), (0.9, 1.5), (0.85, 2.0), (0.95, 0.3), (0.9, 1e30)])
    return _case(None, call, head, K, B, N, masked, tau, budget, profile,
                 32 if profile.endswith("_block") else 0,
                 "all" if call in ("noalloc", "shard") else rng.choice(["all", "all", "lazy", "auto"]),
                 parts, steps)


# ------------------------------------------------------------------------------- inputs

RULES = {"llada": (0.6, 3.5, 15.0, 6, 32), "dream": (0.6, 2.5, 20.0, 6, 32)}


def _rule(case):
    return RULES[case["profile"].replace("_block", "")] + (case["block"],)


def _shares(case, gen):
    """Masked positions of each canvas: between 0.3 and 1 of each other, in a drawn order."""
    B, N, left = case["B"], case["N"], case["masked"]
    weight = [0.3 + 0.7 * (b + 0.5) / B for b in torch.randperm(B, generator=gen).tolist()]
    count = [min(N, int(left * w / sum(weight))) for w in weight]
    b = 0
    while sum(count) < left:
        count[b % B] += count[b % B] < N
        b += 1
    return count


def _inputs(case, seed):
    d, V, K, B, N = (case[k] for k in ("d", "V", "K", "B", "N"))
    cpu = torch.Generator().manual_seed(seed)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    dev = dict(device="cuda", generator=gen)
    std = 1.28 / math.sqrt(d)
    W = torch.empty(V, d, dtype=torch.bfloat16, device="cuda")
    slab = max(1, (1 << 26) // d)
    for v in range(0, V, slab):
        W[v:v + slab] = torch.randn(min(slab, V - v), d, **dev) * std
    g = (1 + 0.1 * torch.randn(d, **dev)).to(torch.bfloat16)
    # the strongest target logit lies 5 nats above the log-partition of the other logits
    sigma = (math.log(V) + 0.5 * 1.28 ** 2 + 5) / (4.0 * 1.28)
    x = torch.linspace(-1, 1, N, device="cuda") if N > 1 else torch.ones(1, device="cuda")
    signal = (sigma * (0.3 + 3.7 * x * x))[None, :, None]
    token = torch.randint(0, V, (B, N), **dev)
    other = torch.where(torch.rand(B, N, **dev) < 0.1, torch.randint(0, V, (B, N), **dev), token)
    hidden = torch.empty(K, B, N, d, dtype=torch.bfloat16, device="cuda")
    for k in range(K):
        a = 1.0 if K == 1 else 0.6 + 0.4 * k / (K - 1)
        for b in range(B):
            row = W[(other if k == K - 2 else token)[b]].float()
            row *= signal[0] * (a / row.norm(dim=1, keepdim=True))
            hidden[k, b] = row + torch.randn(N, d, **dev)
    mask = torch.zeros(B, N, dtype=torch.uint8)
    for b, n in enumerate(_shares(case, cpu)):
        mask[b, torch.randperm(N, generator=cpu)[:n]] = 1
    return W, g, hidden, mask


def prepare(case, seed):
    call, K, B, N = (case[k] for k in ("call", "K", "B", "N"))
    W, g, hidden, mask = _inputs(case, seed)
    where = "cpu" if call == "host" else "cuda"
    s = {"case": case, "W": W, "g": g, "hidden": hidden,
         "start": mask.to(where), "mask": mask.to(where),
         "commit": torch.zeros(B, N, dtype=torch.uint8, device=where),
         "token": torch.full((B, N), -1, dtype=torch.int32, device=where),
         "stats": torch.zeros(B, rpd.STATS_WORDS, dtype=torch.int32, device=where)}
    if call == "host":
        for k in ("hidden", "start", "mask", "commit", "token", "stats"):
            s[k] = s[k].cpu().pin_memory()
    if call == "noalloc":
        s["rule"] = rpd.RpdRule(*_rule(case))
        return s
    ctx = s["ctx"] = rpd.Rpd(case["d"], case["V"], K, EPS)
    ctx.set_stream(torch.cuda.current_stream())
    ctx.set_head(W, g)
    ctx.set_rule(*_rule(case))
    ctx.set_projection(case["projection"])
    ctx.reserve(B, N)
    if call == "shard":
        ctx.set_vocab_shard(case["V"] * (case["parts"] // 2), case["V"] * case["parts"])
        s["partials"] = torch.zeros(K, N, 4, device="cuda")
        return s
    # the scores that the decision was made from, which a program may show or log
    s["scores"] = {"conf": torch.zeros(B, N, device="cuda"),
                   "entropy": torch.zeros(B, N, device="cuda"),
                   "layer_argmax": torch.zeros(K, B, N, dtype=torch.int32, device="cuda"),
                   "layer_pmax": torch.zeros(K, B, N, device="cuda")}
    ctx.set_debug(**s["scores"])
    s["tau"], s["budget"] = [case["tau"]] * B, [case["budget"]] * B
    if call == "loop":
        s["steps"] = torch.zeros(1, dtype=torch.int32, device="cuda")
        s["loop"] = ctx.build_decode_loop(hidden[:, 0], s["mask"][0], case["tau"], case["budget"],
                                          s["commit"][0], s["token"][0], s["stats"][0], s["steps"],
                                          max_steps=case["steps"])
    return s


def run(s):
    case = s["case"]
    call = case["call"]
    if call == "shard":
        s["ctx"].step_shard_partials(s["hidden"][:, 0], s["mask"][0], s["partials"])
        return {"stats": s["partials"][..., :3], "argmax": s["partials"].view(torch.int32)[..., 3]}
    s["mask"].copy_(s["start"])  # a step clears the bits of what it commits
    if call == "step":
        s["ctx"].step(s["hidden"], s["mask"], case["tau"], case["budget"], s["commit"], s["token"],
                      s["stats"])
    elif call == "batched":
        s["ctx"].step_batched(s["hidden"], s["mask"], s["tau"], s["budget"], s["commit"], s["token"],
                              s["stats"])
    elif call == "host":
        s["ctx"].step_host(s["hidden"], s["mask"], case["tau"], case["budget"], s["commit"],
                           s["token"], s["stats"])
    elif call == "loop":
        s["loop"].launch()
    else:
        p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
        code = rpd.rpd_step_noalloc(
            p(s["W"]), p(s["g"]), case["d"], case["V"], case["K"], ctypes.c_float(EPS),
            ctypes.byref(s["rule"]), p(s["hidden"]), p(s["mask"]), case["N"],
            ctypes.c_float(case["tau"]), ctypes.c_float(case["budget"]), p(s["commit"]),
            p(s["token"]), p(s["stats"]), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        if code:
            raise RuntimeError(rpd.rpd_last_error().decode())
    out = {k: s[k] for k in ("mask", "commit", "token", "stats")}
    return dict(out, **s.get("scores", {}))


# ------------------------------------------------------------------- what a pass has to do

def _rows(case):
    """Rows that have to be projected: with lazy projection the final layer's only (how many
    earlier rows follow depends on the data), with RPD-block the active block's masked
    positions (their expected number)."""
    sel = case["masked"]
    if case["block"]:
        sel = max(1, round(min(case["block"], case["N"]) * sel / case["N"]))
    return sel * (1 if case["projection"] != "all" else case["K"])


def work(case):
    rows, d, V, times = _rows(case), case["d"], case["V"], max(1, case["steps"])
    return {"bytes": times * (2.0 * V * d + 2.0 * rows * d + 16.0 * case["B"] * case["N"]),
            "flops": times * 2.0 * rows * d * V}


def tolerance(case):
    """Logits are 32-bit sums over d of 16-bit products; a logit's error of 1e-5 moves a
    probability by the same part of itself.  Against 64 bits the listed cases' probabilities are
    1e-5 to 3.3e-5 off.  Decisions compare such numbers with thresholds and tokens are argmaxes,
    so that one in some hundreds may fall the other way on a near tie."""
    return {"rel": 1.2e-4, "max": 1e-3, "differ": 0.005}


# ---------------------------------------------------------------------------- 64-bit results

def _readout(case, W, g, hidden, rows):
    """Statistics of the given (k, b, n) rows in 64 bits: max, sum e^(z-max),
    sum e^(z-max)(z-max) in nats, argmax."""
    h = hidden[rows]
    u = (h.float() * g.float()).to(torch.bfloat16).double()
    rho = (h.double().square().mean(1, keepdim=True) + EPS).rsqrt()
    Wd = W.double().t()
    got = []
    for r in range(0, u.shape[0], 512):
        z = (u[r:r + 512] @ Wd) * rho[r:r + 512]
        m, a = z.max(1)
        z -= m[:, None]
        e = z.exp()
        got.append((m, e.sum(1), (e * z).sum(1), a))
    return [torch.cat(x) for x in zip(*got)]


def exact(case, seed):
    call, K, B, N = (case[k] for k in ("call", "K", "B", "N"))
    if 2.0 * K * case["masked"] * case["d"] * case["V"] > 1e13:
        return None
    W, g, hidden, mask = _inputs(case, seed)
    theta_c, theta_s, w, k_max, window, block = _rule(case)
    tau, budget = np.float32(case["tau"]), case["budget"]
    start = mask.numpy().astype(bool)
    masked = start.copy()

    def active():
        on = masked.copy()
        for b in range(B):
            if block and masked[b].any():
                lo = int(np.argmax(masked[b])) // block * block
                on[b, :lo] = on[b, lo + block:] = False
        return on

    at = torch.from_numpy(np.broadcast_to(start if call == "loop" else active(), (K, B, N)).copy()).cuda()
    m, s, t, a = _readout(case, W, g, hidden, at)
    if call == "shard":
        out, arg = torch.zeros(K, N, 3, dtype=torch.float64, device="cuda"), torch.zeros(K, N, dtype=torch.int32, device="cuda")
        log2e = 1 / math.log(2)
        out[at[:, 0]] = torch.stack([m * log2e, s, t * log2e], 1)
        arg[at[:, 0]] = (a + case["V"] * (case["parts"] // 2)).int()
        return {"stats": out, "argmax": arg}
    pmax, H, arg = np.zeros((K, B, N)), np.zeros((K, B, N)), np.full((K, B, N), -1, np.int32)
    where = at.cpu().numpy()
    pmax[where], H[where], arg[where] = (1 / s).cpu(), (s.log() - t / s).cpu(), a.cpu().numpy()
    token = np.full((B, N), -1, np.int32)
    stop, passes = math.floor(0.02 * N), max(1, case["steps"])
    for n in range(passes):
        on = active()
        commit = np.zeros((B, N), np.uint8)
        conf = np.where(on, pmax[-1], 0.0)
        band = on & (conf >= np.float32(theta_c)) & (conf < tau)
        for b in range(B):
            q, accepted, seen = 0.0, [], np.flatnonzero(on[b])
            for i in seen:
                k = K - 1
                while k and arg[k - 1, b, i] == arg[-1, b, i]:
                    k -= 1
                stab = min(K - k, k_max) - w * (pmax[k:, b, i].max() - conf[b, i])
                if conf[b, i] >= tau or (band[b, i] and stab >= theta_s):
                    if q > budget and not block:
                        break
                    accepted.append(i)
                else:
                    q += H[-1, b, i]
            if not accepted and len(seen):
                first = seen if block else seen[:window]
                accepted = [first[np.argmax(conf[b, first])]]
            commit[b, accepted] = 1
            token[b, accepted] = arg[-1, b, accepted]
        masked &= commit == 0
        if masked.sum() <= stop:
            break
    out = {"mask": masked.astype(np.uint8), "commit": commit, "token": token, "stats": None}
    if call == "noalloc":
        return out
    shown = np.broadcast_to(on, (K, B, N)).copy()
    if case["projection"] == "lazy":
        shown[:-1] &= band
    elif case["projection"] == "auto":
        shown = None  # which layers are read depends on the choice made on the device
    return dict(out, conf=conf, entropy=np.where(on, H[-1], 0.0),
                layer_argmax=None if shown is None else np.where(shown, arg, -1).astype(np.int32),
                layer_pmax=None if shown is None else np.where(shown, pmax, 0.0))
