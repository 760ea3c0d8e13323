"""The work whose time and results are held to: selection steps, the confidence pass, the rules
and the LM-head-fused steps, each called through the package as a decoding program calls it.

A case is a dict of plain values; ``op`` names the call (or the short fixed sequence of calls)
that one pass makes:

  select     fdllm_select on device logits: one decode step
  robust     fdllm_select_robust with a per-position allowance
  decode     one block decoded by ``steps`` fdllm_select calls, fewer masked positions each time
  host       fdllm_select on page-locked host tensors, the results back on the host
  split      fdllm_confidence, fdllm_profile_terms and fdllm_select_from_conf in turn
  lm_select  fdllm_lmhead_select: hidden states and the vocabulary projection in
  lm_conf    fdllm_lmhead_confidence
  lm_logits  fdllm_lmhead_logits
  lm_loop    fdllm_decode_loop_lmhead: whole generations, block after block

Sizes are the repository's workloads (LLaDA's vocabulary of 126464 and hidden size 4096, blocks
of 32 positions, whole sequences of 1024) and generic ragged ones around the vocabularies and
block lengths of its tests.
"""
import math

import torch

import paper_2606_02955_gb300 as fd

LLADA_V = 126464
TYPES = {"bf16": torch.bfloat16, "fp16": torch.float16, "fp32": torch.float32}

# Masked share of the block at each step of the decode case, first step to last: a block starts
# whole and most of its steps find a small remainder.
SHARES = (1.0, 0.6, 0.4, 0.27, 0.18, 0.12, 0.08, 0.05, 0.03, 0.016)

# The largest pass: logits bytes of one select, multiply-adds of one LM-head step.
MOST_BYTES = 16 * 1024 * LLADA_V * 4
MOST_MACS = 64 * 32 * 4096 * LLADA_V


def listed():
    return [
        # The smallest call: one sequence, one block, bf16 logits straight from the model.
        dict(name="block_b1_bf16", op="select", B=1, L=32, V=LLADA_V, dtype="bf16", masked=1.0,
             mode="profile", param=0.75),
        # A serving batch's step while its blocks are young: the throughput workload.
        dict(name="serving_b64_bf16", op="select", B=64, L=32, V=LLADA_V, dtype="bf16",
             masked=0.72, mode="profile", param=0.75),
        # The same batch decoding one block to its end: ten steps with ever fewer positions.
        dict(name="decode_b64_bf16", op="decode", B=64, L=32, V=LLADA_V, dtype="bf16", steps=10,
             mode="profile", param=0.75),
        # Logits in host memory (a CPU-side or remote model): the end-to-end call.
        dict(name="host_b8_bf16", op="host", B=8, L=32, V=LLADA_V, dtype="bf16", masked=0.5,
             mode="profile", param=0.75),
        # The largest call: whole sequences of 1024 positions, fp32 logits.
        dict(name="sequence_b16_fp32", op="select", B=16, L=1024, V=LLADA_V, dtype="fp32",
             masked=1.0, mode="factor", param=1.0),
        # A smaller vocabulary in fp16 with calibration allowances, ragged in every size.
        dict(name="robust_v20008_fp16", op="robust", B=131, L=61, V=20008, dtype="fp16",
             masked=0.8, mode="profile", param=0.75),
        # A tiny vocabulary (codes, bytes) over long blocks, with the per-rank diagnostics
        # read before the decision: confidence, terms and rule as separate calls.
        dict(name="split_v1004_fp32", op="split", B=63, L=1000, V=1004, dtype="fp32", masked=0.7,
             mode="threshold", param=0.9),
        # LM head fused with the step, one sequence: the projection's weights stream.
        dict(name="lm_select_b1", op="lm_select", B=1, L=32, H=4096, V=LLADA_V, masked=0.75,
             mode="profile", param=0.75),
        # A mid-size batch: a few row tiles, between weight streaming and tensor-bound.
        dict(name="lm_conf_b12", op="lm_conf", B=12, L=32, H=4096, V=LLADA_V, masked=0.75),
        # The serving batch through the LM head: tensor-bound.
        dict(name="lm_conf_b64", op="lm_conf", B=64, L=32, H=4096, V=LLADA_V, masked=0.72),
        # The logits themselves, for callers that sample from them; a ragged vocabulary.
        dict(name="lm_logits_b8_v50001", op="lm_logits", B=8, L=32, H=2048, V=50001, masked=0.75),
        # Four sequences generated whole on the device, the LM head inside the loop.
        dict(name="lm_loop_b4", op="lm_loop", B=4, L=32, H=4096, V=LLADA_V, blocks=3,
             mode="profile", param=0.75),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _rule(rng):
    mode = rng.choice(("profile", "profile", "factor", "threshold"))
    return dict(mode=mode, param=round(rng.uniform(0.5, 1.0), 3))


def draw(rng):
    op = rng.choice(("select", "select", "select", "robust", "decode", "host", "split",
                     "lm_select", "lm_conf", "lm_conf", "lm_logits", "lm_loop"))
    if op.startswith("lm_"):
        B, L = _log(rng, 1, 64), rng.choice((16, 24, 32, 32, 32, 33))
        if op == "lm_loop":
            B = min(B, 8)
        if op == "lm_logits":
            B = min(B, 16)
        c = dict(op=op, B=B, L=L, H=8 * _log(rng, 64, 512), V=_log(rng, 8000, 130000))
        if op == "lm_loop":
            c["blocks"] = rng.randint(1, 3)
        else:
            c["masked"] = round(rng.uniform(0.3, 1.0), 3)
        if op in ("lm_select", "lm_loop"):
            c.update(_rule(rng))
        while B * L * c["H"] * c["V"] > MOST_MACS:
            c["V"] //= 2
        return c
    dtype = rng.choice(("bf16", "bf16", "fp16", "fp32"))
    L = rng.choice((_log(rng, 8, 64), 32, _log(rng, 64, 1024)))
    B, V = _log(rng, 1, 128), 8 * _log(rng, 125, 16250)
    if op == "split":
        V = 8 * _log(rng, 125, 2500)
    if op == "decode":
        L, B = rng.choice((16, 32, 64)), min(B, 64)
    if op == "host":
        L, B = rng.choice((16, 32, 64)), min(B, 8)
    size = 4 if dtype == "fp32" else 2
    most = MOST_BYTES // 8 if op == "decode" else MOST_BYTES // 2
    while B * L * V * size > most or B * L > 65536:
        B = (B + 1) // 2
        if B == 1:
            V = V // 16 * 8
    c = dict(op=op, B=B, L=L, V=V, dtype=dtype)
    if op == "decode":
        c["steps"] = rng.randint(2, len(SHARES))
    else:
        c["masked"] = round(rng.uniform(0.1, 1.0), 3)
    c.update(_rule(rng))
    if op == "robust":
        c["mode"] = "profile"
    return c


def _count(case, share):
    """Masked positions of a call: at least one."""
    return max(1, int(round(share * case["B"] * case["L"])))


def _shares(case):
    if case["op"] == "decode":
        return SHARES[:case["steps"]]
    return (case.get("masked", 1.0),)


class State:
    pass


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _masks(case, g):
    """uint8 [calls, B, L]: the masked positions of each call, each call's within the last's."""
    order = torch.randperm(case["B"] * case["L"], generator=g, device="cuda")
    m = torch.zeros((len(_shares(case)), order.numel()), dtype=torch.uint8, device="cuda")
    for i, share in enumerate(_shares(case)):
        m[i, order[:_count(case, share)]] = 1
    return m.view(-1, case["B"], case["L"])


def _confident(case, g, shape):
    """The confidences aimed at: from unsure to sure for a decision, spread evenly where every
    rank is looked at."""
    r = torch.rand(shape, generator=g, device="cuda", dtype=torch.float32)
    return 0.02 + 0.96 * r if case["op"] == "split" else 1.0 - 10.0 ** -(0.3 + 3.2 * r)


def _logits(case, g):
    """[B, L, V]: Gaussian noise with one planted maximum per position, in the case's type."""
    B, L, V = case["B"], case["L"], case["V"]
    out = torch.empty((B * L, V), dtype=TYPES[case["dtype"]], device="cuda")
    rows = max(1, (1 << 28) // V)
    for r in range(0, B * L, rows):
        n = min(rows, B * L - r)
        x = torch.randn((n, V), generator=g, device="cuda", dtype=torch.float32)
        u = _confident(case, g, (n, 1))
        at = torch.randint(0, V, (n, 1), generator=g, device="cuda")
        x.scatter_(1, at, math.log(V - 1) + 0.5 + torch.logit(u))
        out[r:r + n] = x
    return out.view(B, L, V)


def _head(case, g):
    """The vocabulary projection [V, H]: rows of norm about one."""
    V, H = case["V"], case["H"]
    w = torch.empty((V, H), dtype=torch.bfloat16, device="cuda")
    rows = max(1, (1 << 28) // H)
    for r in range(0, V, rows):
        n = min(rows, V - r)
        w[r:r + n] = torch.randn((n, H), generator=g, device="cuda") * H ** -0.5
    return w


def _hidden(case, g, w, n):
    """n hidden states, bf16: noise plus the direction of one token, so that its logit stands
    out by about what the confidence aimed at asks for."""
    V, H = case["V"], case["H"]
    h = torch.randn((n, H), generator=g, device="cuda")
    at = torch.randint(0, V, (n,), generator=g, device="cuda")
    t = w[at].float()
    peak = math.log(V - 1) + 0.5 + torch.logit(_confident(case, g, (n, 1)))
    return (h + t * ((peak - (h * t).sum(1, keepdim=True)) / t.square().sum(1, keepdim=True))
            ).to(torch.bfloat16)


class _Ints:
    """int32 device values at an address the library gives (the loop's step and block)."""

    def __init__(self, address, n):
        self.__cuda_array_interface__ = {"shape": (n,), "typestr": "<i4", "version": 3,
                                         "data": (address, False)}


def _forward(s):
    """The loop's forward pass: the current block's hidden states, out of the bank that stands
    for the model."""
    block = torch.as_tensor(_Ints(s.at, 2), device="cuda")[1:2]
    torch.index_select(s.bank, 0, block, out=s.hidden.view(1, *s.hidden.shape))


def prepare(case, seed):
    g = _generator(seed)
    s = State()
    s.case = case
    B, L, op = case["B"], case["L"], case["op"]
    if op == "lm_loop":
        s.w = _head(case, g)
        s.bank = _hidden(case, g, s.w, case["blocks"] * B * L).view(-1, B, L, case["H"])
        s.hidden = torch.empty((B, L, case["H"]), dtype=torch.bfloat16, device="cuda")
        return s
    s.before = _masks(case, g)
    s.mask = s.before.clone()
    s.tokens = torch.full((B, L), -1, dtype=torch.int32, device="cuda")
    s.commit = torch.zeros((B, L), dtype=torch.uint8, device="cuda")
    s.n = torch.zeros((B,), dtype=torch.int32, device="cuda")
    if op.startswith("lm_"):
        s.w = _head(case, g)
        s.hidden = _hidden(case, g, s.w, B * L).view(B, L, case["H"])
        if op == "lm_logits":
            s.logits = torch.zeros((B, L, case["V"]), dtype=torch.float32, device="cuda")
    elif op == "decode":
        s.logits = [_logits(case, g) for _ in range(case["steps"])]
        s.tokens, s.commit, s.n = ([t.clone() for _ in range(case["steps"])]
                                   for t in (s.tokens, s.commit, s.n))
    else:
        s.logits = _logits(case, g)
    if op == "robust":
        s.eta = 0.05 * torch.rand((B, L), generator=g, device="cuda", dtype=torch.float32)
    if op in ("split", "lm_conf"):
        s.conf = torch.zeros((B, L), dtype=torch.float32, device="cuda")
        s.argmax = torch.full((B, L), -1, dtype=torch.int32, device="cuda")
    if op == "host":
        for name in ("logits", "before", "mask", "tokens", "commit", "n"):
            t = getattr(s, name)
            setattr(s, name, torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t))
    return s


def run(s):
    c = s.case
    op = c["op"]
    if op == "lm_loop":
        def forward(state, mask, out, stream):
            s.at = state
            with torch.cuda.stream(torch.cuda.ExternalStream(stream)):
                _forward(s)

        tokens, nfe, steps = fd.fdllm_decode_loop_lmhead(forward, s.hidden, s.w,
                                                         c["blocks"] * c["L"], c["param"],
                                                         c["mode"])
        return {"tokens": tokens, "nfe": nfe, "steps": steps, "hidden": s.hidden}
    if op == "lm_conf":
        fd.fdllm_lmhead_confidence(s.hidden, s.w, s.mask[0], s.conf, s.argmax)
        return {"conf": s.conf, "argmax": s.argmax}
    if op == "lm_logits":
        fd.fdllm_lmhead_logits(s.hidden, s.w, s.mask[0], s.logits)
        return {"logits": s.logits}
    s.mask.copy_(s.before)  # a step clears the positions it commits
    out = {"tokens": s.tokens, "commit": s.commit, "n": s.n, "mask": s.mask}
    if op == "decode":
        for i in range(c["steps"]):
            fd.fdllm_select(s.logits[i], s.mask[i], c["param"], c["mode"], s.tokens[i],
                            s.commit[i], s.n[i])
    elif op == "robust":
        fd.fdllm_select_robust(s.logits, s.mask[0], c["param"], 0.0, s.eta, s.tokens, s.commit,
                               s.n)
    elif op == "split":
        fd.fdllm_confidence(s.logits, s.mask[0], s.conf, s.argmax)
        out.update(fd.fdllm_profile_terms(s.conf, s.mask[0], 0.25))
        out.update(conf=s.conf, argmax=s.argmax)
        fd.fdllm_select_from_conf(s.conf, s.argmax, s.mask[0], c["param"], c["mode"], s.tokens,
                                  s.commit, s.n)
    elif op == "lm_select":
        fd.fdllm_lmhead_select(s.hidden, s.w, s.mask[0], c["param"], c["mode"], s.tokens,
                               s.commit, s.n)
    else:
        fd.fdllm_select(s.logits, s.mask[0], c["param"], c["mode"], s.tokens, s.commit, s.n)
    return out


def work(case):
    """Masked rows read once (or the head's weights and the masked hidden states, and their
    products), masks read and written, results written."""
    B, L, V, op = case["B"], case["L"], case["V"], case["op"]
    rows = sum(_count(case, x) for x in _shares(case))
    step = len(_shares(case)) * B * (L * 3 + 4)  # mask read and written, commit flags, counts
    if not op.startswith("lm_"):
        n = rows * V * (4 if case["dtype"] == "fp32" else 2) + step
        if op == "split":
            n += B * L * (4 * 8 + 4 + 8)  # terms and order, confidence and argmax
        if op == "robust":
            n += B * L * 4
        return {"bytes": n, "flops": 4 * rows * V}
    H = case["H"]
    if op == "lm_loop":
        # at least one step per block, on the whole block
        rows = B * L * case["blocks"]
        return {"bytes": case["blocks"] * V * H * 2 + rows * H * 4, "flops": 2 * rows * H * V}
    n = V * H * 2 + rows * H * 2 + step
    if op == "lm_logits":
        n += rows * V * 4
    return {"bytes": n, "flops": 2 * rows * H * V}


def tolerance(case):
    """fp32 sums of exp (and, for the LM head, fp32 dot products of bf16 values); tokens and
    decisions can differ only where two values agree to the last bits of fp32.  Measured
    against 64 bits: 5e-6 through the LM head, 3e-7 from logits."""
    if case["op"] in ("lm_conf", "lm_logits"):
        return {"rel": 2e-5, "max": 2e-4, "differ": 1e-3}
    if case["op"] == "split":
        return {"rel": 1.2e-6, "max": 1.2e-5, "differ": 2e-3}
    return {"rel": 0.0, "differ": 2e-3}


def _rows(case, s):
    return s.before[0].reshape(-1).nonzero().reshape(-1)


def _softmax_max(x):
    """(max probability, first index of the maximum) of rows of 64-bit logits."""
    m, at = x.max(1)
    first = (x == m[:, None]).to(torch.uint8).argmax(1)
    return 1.0 / (x - m[:, None]).exp().sum(1), first


def exact(case, seed):
    op = case["op"]
    if op not in ("split", "lm_conf", "lm_logits"):
        return None  # whole numbers only
    s = prepare(case, seed)
    B, L, V = case["B"], case["L"], case["V"]
    rows = _rows(case, s)
    if op == "split":
        return _exact_split(case, s, rows)
    h = s.hidden.view(B * L, -1)[rows].double()
    per = max(1, (1 << 27) // h.shape[0])
    if op == "lm_logits":
        out = torch.zeros((B * L, V), dtype=torch.float64, device="cuda")
        for v in range(0, V, per):
            out[rows, v:v + per] = h @ s.w[v:v + per].double().t()
        return {"logits": out.view(B, L, V)}
    # running maximum and sum over slices of the vocabulary
    m = torch.full((rows.numel(),), -math.inf, dtype=torch.float64, device="cuda")
    t = torch.zeros_like(m)
    for v in range(0, V, per):
        x = h @ s.w[v:v + per].double().t()
        top = torch.maximum(m, x.max(1).values)
        t = t * (m - top).exp() + (x - top[:, None]).exp().sum(1)
        m = top
    conf = torch.zeros(B * L, dtype=torch.float64, device="cuda")
    conf[rows] = 1.0 / t
    return {"conf": conf.view(B, L), "argmax": None}


def _exact_split(case, s, rows):
    B, L, V = case["B"], case["L"], case["V"]
    conf = torch.zeros(B * L, dtype=torch.float64, device="cuda")
    flat = s.logits.view(B * L, V)
    per = max(1, (1 << 26) // V)
    for r in range(0, rows.numel(), per):
        conf[rows[r:r + per]], _ = _softmax_max(flat[rows[r:r + per]].double())
    conf = conf.view(B, L)
    masked = s.before[0] != 0
    c, _ = torch.where(masked, conf, torch.full_like(conf, -1.0)).sort(1, descending=True)
    live = c >= 0
    n = torch.arange(1, L + 1, device="cuda", dtype=torch.float64)
    total = torch.where(live, c, torch.zeros_like(c)).cumsum(1)
    bonus = total - n * c
    terms = {"G": (total - (n - 1)).clamp(min=0) - (1 - c), "F": (n + 1) * c - n, "B": bonus,
             "f_eff": 0.75 + bonus}
    out = {k: torch.where(live, v, torch.full_like(v, math.nan)) for k, v in terms.items()}
    out.update(conf=conf, order=None, argmax=None, tokens=None, commit=None, n=None, mask=None)
    return out
