"""What the speed of this library is measured on: the calls a program with this library makes, at the sizes it makes them.

The library is the linear attention of a video diffusion transformer and the temporal convolution of its feed-forward
block.  Such a program calls it in two settings: on a whole clip (every layer of every denoising step: ``forward``,
plain or with rotary factors, and ``tconv_forward``), and block by block on a stream with constant-memory caches (the
denoising steps of a block read the cache: ``peek``; the clean block is committed: ``step``, ``tconv_step``; a given
beginning of the video is taken in at once: ``prefill``).  Sizes are the 480p and 720p latent grids (21 frames of
30 x 52 or 45 x 80 positions, width 2240, blocks of three frames), a tiny clip where only latency counts, and in
``draw`` everything between.
"""
import torch

import paper_2509_24695_b200 as la

WIDTH = 2240                      # model width: H heads of dimension d
MOST_TOKENS = 21 * 45 * 80        # a 720p clip
F32_TOKENS = 21 * 30 * 52         # a 480p clip: the most the fp32 and odd-head-dim calls are drawn with


def _attention(op, N, H, d, B=1, **more):
    """N: tokens of the clip, or of one block; blocks: blocks of a prefill."""
    case = {"op": op, "B": B, "N": N, "H": H, "d": d, "dtype": "bf16", "rope": False, "layout": "token", "blocks": 1}
    case.update(more)
    return case


def _conv(op, T, HW, D, B=1, dtype="bf16"):
    return {"op": op, "B": B, "T": T, "HW": HW, "D": D, "dtype": dtype}


def listed():
    cases = {
        # a thumbnail clip of 3 x 8 x 8 latents: what a call costs when there is next to nothing to do
        "forward_tiny": _attention("forward", 192, 4, 32),
        # one attention layer over a five-second 480p clip
        "forward_480p": _attention("forward", 21 * 30 * 52, 20, 112),
        # one attention layer over a five-second 720p clip: the largest
        "forward_720p": _attention("forward", MOST_TOKENS, 20, 112),
        # the same width cut into smaller heads (several of them share a tensor-core operand; the last one is half full)
        "forward_720p_d64": _attention("forward", MOST_TOKENS, 35, 64),
        # the attention as the model runs it on a clip, with its rotary factors
        "forward_rope_480p": _attention("forward", 21 * 30 * 52, 20, 112, rope=True),
        # committing a clean block of three 480p frames to the stream's cache and reading it
        "step_480p": _attention("step", 3 * 30 * 52, 20, 112),
        # a step of two minute-long 720p streams together
        "step_720p_stream": _attention("step", 3 * 45 * 80, 20, 112, B=2),
        # a denoising step of a block of a 480p stream, with rotary factors: the call a stream makes most often
        "peek_rope_480p": _attention("peek", 3 * 30 * 52, 20, 112, rope=True),
        # taking seven given blocks of a 480p video into a cache in one call
        "prefill_480p": _attention("prefill", 3 * 30 * 52, 20, 112, blocks=7),
        # the fp32 path over a 480p clip: fp32 in, fp32 arithmetic, fp32 out
        "forward_480p_f32": _attention("forward", F32_TOKENS, 20, 112, dtype="f32"),
        # the temporal convolution of one layer over a 720p clip
        "tconv_forward_720p": _conv("tconv_forward", 21, 45 * 80, WIDTH),
        # the same layer on a block of three 480p frames with its one-frame cache
        "tconv_step_480p": _conv("tconv_step", 3, 30 * 52, WIDTH),
    }
    return [dict(case, name=name) for name, case in cases.items()]


def _spread(rng, low, high):
    """A whole number between low and high, even over the logarithm."""
    return max(low, min(high, round(low * (high / low) ** rng.random())))


def draw(rng):
    op = rng.choice(["forward", "forward", "forward", "step", "peek", "prefill", "tconv_forward", "tconv_step"])
    dtype = "f32" if rng.random() < 0.15 else "bf16"
    if op.startswith("tconv"):
        B = rng.choice([1, 1, 1, 2])
        D = rng.choice([WIDTH, WIDTH, 1120, 8 * rng.randint(16, 280)])
        T = rng.randint(1, 4) if op == "tconv_step" else rng.randint(4, 33)
        room = MOST_TOKENS * WIDTH // (B * T * D * (2 if dtype == "f32" else 1))
        return _conv(op, T, _spread(rng, 16, min(3600, room)), D, B, dtype)
    d = rng.choice([112, 112, 112, 128, 64, 32, rng.choice([40, 72, 80, 96])])
    H = rng.choice([-(-WIDTH // d), -(-WIDTH // d), rng.randint(1, 24)])
    B = rng.choice([1, 1, 1, 2, 3])
    room = MOST_TOKENS * WIDTH // (B * H * d)
    if dtype == "f32" or d not in (32, 64, 112, 128):
        room = F32_TOKENS * 20 * 112 * 112 // (B * H * d * d)
    case = _attention(op, 1, H, d, B, dtype=dtype, rope=op != "prefill" and rng.random() < 0.4,
                      layout="head" if op == "forward" and rng.random() < 0.2 else "token")
    if op == "prefill":
        case["blocks"] = rng.randint(2, 7)
        room //= case["blocks"]
    most = MOST_TOKENS if op == "forward" else 3 * 45 * 80
    case["N"] = _spread(rng, 64, max(64, min(most, room)))
    return case


DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}


def _angles(N, d, first):
    """cos and sin of N tokens from position `first`: one frequency per feature pair, base 10000."""
    freq = 10000.0 ** (-torch.arange(d // 2, device="cuda", dtype=torch.float32) / (d // 2))
    angle = torch.arange(first, first + N, device="cuda", dtype=torch.float32)[:, None] * freq
    return angle.cos(), angle.sin()


def _inputs(case, seed):
    """The tensors of a case, from the seed alone; k0, v0 (x0): the block that has gone before on a stream."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    dtype = DTYPES[case["dtype"]]

    def normal(*shape, scale=1.0):
        return torch.randn(*shape, device="cuda", generator=gen).mul_(scale).to(dtype)

    B, made = case["B"], {}
    if case["op"].startswith("tconv"):
        T, HW, D = case["T"], case["HW"], case["D"]
        made["x"] = normal(B, T, HW, D)
        made["taps"] = torch.randn(3, D, device="cuda", generator=gen).mul_(0.25)
        if case["op"] == "tconv_step":
            made["x0"] = normal(B, 1, HW, D)
        return made
    N, H, d = case["N"] * case["blocks"], case["H"], case["d"]
    # queries and keys as the projections of a normalised activation leave them: zero mean, 1/sqrt(d)
    for name, scale in (("q", d ** -0.5), ("k", d ** -0.5), ("v", 1.0)):
        if case["layout"] == "head":
            made[name] = normal(B, H, N, d, scale=scale).permute(0, 2, 1, 3)
        else:
            made[name] = normal(B, N, H, d, scale=scale)
    if case["op"] != "forward":
        made["k0"], made["v0"] = normal(B, case["N"], H, d, scale=d ** -0.5), normal(B, case["N"], H, d)
    return made


def prepare(case, seed):
    made = _inputs(case, seed)
    state = {"case": case, **{name: made[name] for name in ("x", "taps", "q", "k", "v") if name in made}}
    B, dtype = case["B"], DTYPES[case["dtype"]]
    if case["op"].startswith("tconv"):
        if case["op"] == "tconv_step":
            state["cache"] = la.TConvCache(B, case["HW"], case["D"], dtype, "cuda")
            state["cache"].absorb(made["x0"])
        return state

    N, H, d = case["N"] * case["blocks"], case["H"], case["d"]
    if case["op"] == "forward":
        if case["rope"]:
            state["table"] = la.rope_pack(*_angles(N, d, 0))
            state["workspace"] = la.new_rope_workspace(state["q"])
        else:
            state["workspace"] = la.new_workspace(state["q"])
        return state
    cache = la.BlockLinCache(B, H, d, dtype, "cuda", max_T_b=case["N"],
                             prefill_blocks=case["blocks"] if case["op"] == "prefill" else 0)
    state["cache"] = cache
    if case["rope"]:
        cache.step_rope(None, made["k0"], made["v0"], la.rope_pack(*_angles(case["N"], d, 0)))
        state["table"] = la.rope_pack(*_angles(N, d, case["N"]))
    else:
        cache.step(None, made["k0"], made["v0"])
    return state


def run(state):
    case = state["case"]
    op = case["op"]
    if op == "tconv_forward":
        return la.tconv_forward(state["x"], state["taps"])
    if op == "tconv_step":
        return state["cache"].step(state["x"], state["taps"]), state["cache"].frame
    q, k, v = state["q"], state["k"], state["v"]
    if op == "forward":
        if case["rope"]:
            return la.linattn_forward_rope(q, k, v, state["table"], workspace=state["workspace"])
        return la.linattn_forward(q, k, v, workspace=state["workspace"])
    cache = state["cache"]
    if op == "prefill":
        return cache.prefill(q, k, v, case["blocks"]), cache.state
    if case["rope"]:
        call = cache.step_rope if op == "step" else cache.peek_rope
        return call(q, k, v, state["table"]), cache.state
    call = cache.step if op == "step" else cache.peek
    return call(q, k, v), cache.state


def work(case):
    B, size = case["B"], 2 if case["dtype"] == "bf16" else 4
    if case["op"].startswith("tconv"):
        frame = B * case["HW"] * case["D"]
        frames = 2 * case["T"] + (2 if case["op"] == "tconv_step" else 0)   # a step: the cached frame in and out
        return {"bytes": frames * frame * size + 12 * case["D"], "flops": 6 * case["T"] * frame}
    N, H, d = case["N"] * case["blocks"], case["H"], case["d"]
    bytes_ = 4 * B * N * H * d * size                                        # q, k, v in, o out
    if case["rope"]:
        bytes_ += 2 * N * d                                                  # (cos, sin) as fp16, half of d per token
    states = {"forward": 0, "peek": 1, "step": 2, "prefill": 2}[case["op"]]  # the cache: in, or in and out
    bytes_ += states * 4 * B * H * (d + 1) * d
    return {"bytes": bytes_, "flops": 4 * B * N * H * d * (d + 1)}


def tolerance(case):
    # About four times the distance of this library's results from the same sums in 64 bits (2-norm, largest element):
    # bf16 1.7e-3, 3.9e-3, which is the rounding of the output; with rotary factors 2.8e-3, 1.8e-2 (the rotated features
    # are rounded to bf16 too); fp32 attention 1.9e-7, 1.1e-6; fp32 convolution 4.1e-8, 2.1e-7.
    if case["op"].startswith("tconv"):
        return {"rel": 2e-7, "max": 1e-6} if case["dtype"] == "f32" else {"rel": 7e-3, "max": 0.016}
    if case["dtype"] == "f32":
        return {"rel": 1e-6, "max": 6e-6}
    return {"rel": 0.012, "max": 0.08} if case["rope"] else {"rel": 7e-3, "max": 0.016}


def _rotated(x, cos, sin):
    """Feature pairs (2p, 2p+1) of x[B, N, H, d] turned by the angles of their token; the table holds fp16 values."""
    c, s = cos.half().double()[None, :, None], sin.half().double()[None, :, None]
    a, b = x[..., 0::2], x[..., 1::2]
    return torch.stack((a * c - b * s, b * c + a * s), dim=-1).flatten(-2)


def exact(case, seed):
    """What `run` returns, from the definitions, in 64 bits."""
    made = {name: t.double() for name, t in _inputs(case, seed).items()}
    op = case["op"]
    if op.startswith("tconv"):
        x, w = made["x"], made["taps"]
        y = x + w[1] * x
        y[:, 1:] += w[0] * x[:, :-1]
        y[:, :-1] += w[2] * x[:, 1:]
        if op == "tconv_forward":
            return y
        y[:, :1] += w[0] * made["x0"]
        return y, x[:, -1]

    N, d, rope = case["N"], case["d"], case["rope"]

    def state_of(k, v, first):
        k = k.relu()
        turned = _rotated(k, *_angles(k.shape[1], d, first)) if rope else k
        return torch.einsum("bnhi,bnhj->bhji", turned, v), k.sum(1)

    def read(q, S, z, first):
        q = q.relu()
        turned = _rotated(q, *_angles(q.shape[1], d, first)) if rope else q
        return torch.einsum("bnhi,bhji->bnhj", turned, S) / (torch.einsum("bnhi,bhi->bnh", q, z) + 1e-6)[..., None]

    q, k, v = made["q"], made["k"], made["v"]
    if op == "forward":
        return read(q, *state_of(k, v, 0), 0)
    S, z = state_of(made["k0"], made["v0"], 0)
    before = torch.cat((S, z[:, :, None]), dim=2)
    outs = []
    for first in range(0, N * case["blocks"], N):
        dS, dz = state_of(k[:, first:first + N], v[:, first:first + N], N + first)
        S, z = S + dS, z + dz
        outs.append(read(q[:, first:first + N], S, z, N + first))
    return torch.cat(outs, dim=1), before if op == "peek" else torch.cat((S, z[:, :, None]), dim=2)
