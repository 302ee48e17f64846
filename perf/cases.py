"""Workloads that the speed of the verify-and-draft library is measured on.

A case is one call pattern of a decoding program, with its sizes, data type
and sampler options; its inputs are synthetic logits made on the GPU from a
seed. Sizes are those of paper_2603_18599_gb300/workloads.py (one image to
sixteen, windows of 16 to 64 rows, 8192 to 65536 ids) and ragged ones between
them.

Logits: the rows of one image share a base draw N(0, sigma^2) per branch and
add their own N(0, q_noise^2), the same in both branches, so that a row's
stored draft distribution (the row's position in the step before) resembles
its target as consecutive Jacobi iterates do, and a step has accepted and
rejected rows. Ids outside the allowed range hold 64.0, above every logit.

Every pass returns what the program reads (committed tokens, commit counts,
first rejections) and the updated decode state: the window with its candidate
groups and the stored distributions of all its rows.
"""

import ctypes
import math

import torch

from paper_2603_18599_gb300 import sjd

DEVICE = "cuda"
OUT_OF_RANGE = 64.0
SMEM = 227 * 1024         # shared memory a row may take (sjd_init refuses more)

DEFAULTS = {
    "entry": "step",      # step | chain | verify | draft | tree | host | decode
    "batch": 1, "window": 16, "vocab": 8192, "lo": 0, "hi": 8192, "dtype": "bf16",
    "cfg": 3.0, "temperature": 1.0, "top_k": 2000, "top_p": 1.0, "pd_k": 4, "pd_depth": 3, "ac": 1,
    "sigma": 3.0, "sigma_step": 0.0,   # sigma of image b: sigma + sigma_step * (b mod 5)
    "q_noise": 1.0, "dominant": 0.0,   # share of rows with one id raised by 12
    "bufs": 2,            # logit tensors the steps alternate between
    "steps": 1,           # steps of one pass (chain)
    "n_tokens": 0,        # tokens of one decode
}


def _case(name=None, **kw):
    c = dict(DEFAULTS, **kw)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # one image, fp32 logits: the smallest call, whose latency a
        # single-user decode pays at every step
        _case("step_b1w16v8192_f32", dtype="f32"),
        # the same with the larger vocabulary of a 90 x 90 decode, bf16
        _case("step_b1w16v32768_bf16", vocab=32768, hi=32768),
        # four images, 10 % of the rows nearly certain (one id far above)
        _case("step_b4w32v32768_bf16", batch=4, window=32, vocab=32768, hi=32768, dominant=0.1),
        # eight images from sharp to flat rows, long top-k: the longest kept rows
        _case("step_b8w32v16384_bf16_k4096", batch=8, window=32, vocab=16384, hi=16384, cfg=4.0, top_k=4096,
              sigma=1.0, sigma_step=1.0, q_noise=0.5),
        # sixteen images, image ids inside a text + image vocabulary, top-p:
        # the serving step right after a forward
        _case("step_b16w64v65536_bf16_topp", batch=16, window=64, vocab=65536, lo=4, hi=8196, top_p=0.9),
        # the same on resident logits, eight steps back to back (scoring of
        # precomputed logits; the early-logits guarantee)
        _case("chain8_b16w64v65536_bf16_topp", entry="chain", batch=16, window=64, vocab=65536, lo=4, hi=8196,
              top_p=0.9, bufs=4, steps=8),
        # verification and drafting as separate calls, the distributions read
        # between them (acceptance statistics)
        _case("verify_b8w32v16384_bf16", entry="verify", batch=8, window=32, vocab=16384, hi=16384, sigma=2.0,
              top_p=0.95, q_noise=0.5),
        # a window drafted from a draft model's logits
        _case("draft_b8w32v16384_bf16", entry="draft", batch=8, window=32, vocab=16384, hi=16384, sigma=2.0),
        # the full drafting tree, 34 logit rows per image
        _case("tree_b4w16v8192_bf16", entry="tree", batch=4, window=16, sigma=1.0, q_noise=0.5),
        # a vocabulary whose rows do not start on 16-byte boundaries, an
        # unaligned allowed range, temperature and top-p
        _case("step_b8w32v10007_bf16_ragged", batch=8, window=32, vocab=10007, lo=5, hi=9001, temperature=0.7,
              top_p=0.8, top_k=1000),
        # logits produced in pinned host memory
        _case("host_b4w32v65536_bf16_topp", entry="host", batch=4, window=32, vocab=65536, lo=4, hi=8196, top_p=0.9),
        # a whole image of 256 tokens through the decode loop
        _case("decode_b1w16v8192_bf16", entry="decode", n_tokens=256),
    ]


def _padded(c):
    epv = 8 if c["dtype"] == "bf16" else 4
    al0 = c["lo"] // epv * epv
    return -(-c["hi"] // epv) * epv - al0


def _support(c):
    veff = c["hi"] - c["lo"]
    return min(c["top_k"], veff) if c["top_k"] else veff


def _fits(c):
    """A row of the configuration fits an SM's shared memory (the library
    refuses it otherwise)."""
    nl, s = _padded(c), _support(c)
    need = 4 * nl + 16384 + 24 * s + (0 if 16 * s <= 4 * nl else 16 * s) + 4096
    return need <= SMEM


def draw(rng):
    """One more case of the ranges above: 1 to 16 images, windows of 1 to 64
    rows, 1000 to 65536 ids, both data types, every option."""
    biggest = work(listed()[5])["bytes"]

    def log_uniform(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    while True:
        entry = rng.choice(["step", "step", "step", "step", "chain", "verify", "draft", "tree", "host", "decode"])
        vocab = log_uniform(1000, 65536)
        if rng.random() < 0.5:
            vocab = -(-vocab // 64) * 64     # most models pad their vocabulary; some do not
        width = vocab if rng.random() < 0.5 else max(500, int(vocab * rng.uniform(0.1, 0.9)))
        lo = 0 if width >= vocab else rng.randrange(0, vocab - width + 1)
        hi = lo + min(width, vocab)
        c = _case(entry=entry, batch=log_uniform(1, 16), window=log_uniform(4, 64), vocab=vocab, lo=lo, hi=hi,
                  dtype=rng.choice(["bf16", "bf16", "f32"]), cfg=rng.choice([1.0, 3.0, 3.0, 4.0, 7.5]),
                  temperature=rng.choice([1.0, 1.0, 0.7, 1.3]), top_k=log_uniform(50, 4096),
                  top_p=rng.choice([1.0, 1.0, 0.95, 0.9, 0.8]), pd_k=rng.choice([1, 2, 4, 4, 8]),
                  pd_depth=rng.choice([1, 3, 3, 6]), ac=rng.choice([1, 1, 1, 0]),
                  sigma=round(rng.uniform(0.7, 4.0), 2), sigma_step=rng.choice([0.0, 0.0, 0.5]),
                  q_noise=rng.choice([0.3, 0.5, 1.0]), dominant=rng.choice([0.0, 0.0, 0.1]))
        if rng.random() < 0.1:
            c["top_k"] = 0                   # no top-k: every id with weight is kept
        if entry == "chain":
            c.update(bufs=4, steps=rng.choice([2, 4, 8]))
        elif entry == "tree":
            c.update(ac=1, pd_k=rng.choice([2, 3, 4]), pd_depth=rng.choice([2, 3]), window=max(8, c["window"] // 2))
        elif entry == "decode":
            c.update(batch=1, window=rng.choice([8, 16, 24]), n_tokens=rng.choice([64, 128, 256]))
            if vocab > 16384:
                continue                     # the stand-in forward's tables grow as vocab^2
        if entry == "host" and c["batch"] * c["window"] * vocab > 4 * 32 * 65536:
            continue                         # bounded pinned memory
        if _fits(c) and work(c)["bytes"] <= biggest:
            return c


# ---------------------------------------------------------------------------
# Inputs


def _dtype(c):
    return torch.bfloat16 if c["dtype"] == "bf16" else torch.float32


def _generator(seed, what):
    g = torch.Generator(device=DEVICE)
    g.manual_seed((int(seed) * 1000003 + what) & 0x7FFFFFFF)
    return g


def _tree_rows(c):
    return sum(c["pd_k"] ** d - 1 for d in range(1, c["pd_depth"])) if c["entry"] == "tree" else 0


def _logits(c, seed, index, rows):
    """(cond, uncond) [batch, rows, vocab] of logit tensor `index`; uncond is
    None at guidance scale 1."""
    b, veff = c["batch"], c["hi"] - c["lo"]
    g = _generator(seed, 1)
    sig = torch.tensor([c["sigma"] + c["sigma_step"] * (i % 5) for i in range(b)], device=DEVICE).view(b, 1, 1)
    base = [torch.randn((b, 1, veff), generator=g, device=DEVICE) * sig for _ in range(2)]
    g = _generator(seed, 16 + index)
    z = torch.randn((b, rows, veff), generator=g, device=DEVICE) * c["q_noise"]
    n = int(round(c["dominant"] * b * rows))
    if n:
        at = torch.randperm(b * rows, generator=g, device=DEVICE)[:n]
        z.view(b * rows, veff)[at, torch.randint(0, veff, (n,), generator=g, device=DEVICE)] += 12.0
    out = []
    for x in base if c["cfg"] != 1.0 else base[:1]:
        full = torch.full((b, rows, c["vocab"]), OUT_OF_RANGE, dtype=_dtype(c), device=DEVICE)
        full[:, :, c["lo"]:c["hi"]] = (x + z).to(_dtype(c))
        out.append(full)
    return out[0], out[1] if len(out) > 1 else None


def _config(c, seed):
    return sjd.make_config(c["batch"], c["window"], c["vocab"], c["lo"], c["hi"], c["cfg"], c["temperature"],
                           c["top_k"], c["top_p"], c["pd_k"], c["pd_depth"], c["ac"], int(seed) & 0x7FFFFFFF,
                           sjd.SJD_BF16 if c["dtype"] == "bf16" else sjd.SJD_F32,
                           max_steps=max(1, c["n_tokens"]), pd_tree=1 if c["entry"] == "tree" else 0)


class _State:
    pass


def _read_buffers(s, c):
    """Output buffers that the program keeps, and the argument lists of the C
    calls that fill them."""
    b, w, k = c["batch"], c["window"], c["pd_k"]
    i32 = dict(dtype=torch.int32, device=DEVICE)
    s.outs = [(torch.empty((b, w), **i32), torch.empty((b,), **i32), torch.empty((b,), **i32))
              for _ in range(c["steps"])]
    s.out = s.outs[0]
    s.window = [torch.empty(n, **i32) for n in ((b, w), (b, w, k), (b, w), (b,), (b,))]
    cap = s.ctx.cfg.support_cap
    s.rows = [torch.empty((b, w, cap), **i32), torch.empty((b, w, cap), dtype=torch.float32, device=DEVICE),
              torch.empty((b, w), **i32)]
    s.window_args = [ctypes.c_void_p(t.data_ptr()) for t in s.window]
    s.rows_args = [ctypes.c_void_p(t.data_ptr()) for t in s.rows]


def prepare(case, seed):
    c = dict(DEFAULTS, **case)
    s = _State()
    s.case, s.at = c, 0
    cfg = _config(c, seed)
    if c["entry"] == "decode":
        # the stand-in forward's tables: the logits after each previous token
        s.cfg = cfg
        v = c["vocab"]
        g = _generator(seed, 2)
        s.tables = []
        for _ in range(2 if c["cfg"] != 1.0 else 1):
            t = torch.randn((1, v), generator=g, device=DEVICE) * c["sigma"]
            t = t + torch.randn((v, v), generator=g, device=DEVICE) * c["q_noise"]
            t[:, :c["lo"]] = OUT_OF_RANGE
            t[:, c["hi"]:] = OUT_OF_RANGE
            s.tables.append(t.to(_dtype(c)))
        s.bufs = [torch.empty((1, c["window"], v), dtype=_dtype(c), device=DEVICE) for _ in s.tables]
        return s
    s.ctx = sjd.SJD(cfg, DEVICE)
    rows = c["window"] + _tree_rows(c)
    s.logits = [_logits(c, seed, i, rows) for i in range(c["bufs"])]
    _read_buffers(s, c)
    # a decode in progress: a drafted window and one step behind it
    s.ctx.draft_from_logits(*_logits(c, seed, 100, c["window"]))
    s.ctx.step(*s.logits[-1], out=s.out)
    if c["entry"] == "host":
        s.logits = [tuple(None if t is None else t.cpu().pin_memory() for t in p) for p in s.logits]
        s.stage = s.ctx.host_stage()
    elif c["entry"] == "chain":
        s.ctx.set_early_logits(True)
    return s


# ---------------------------------------------------------------------------
# One pass


def _check(s, code):
    if code != sjd.SJD_OK:
        raise sjd.SJDError(code, s.ctx.last_error())


def _decode(s):
    c = s.case
    w, v = c["window"], c["vocab"]
    flat = [t.view(w, v) for t in s.bufs]

    def forward(win, prev, pos, cond_out, uncond_out):
        before = torch.cat([prev.view(1, 1), win[:, :-1]], dim=1).view(-1)
        for table, out in zip(s.tables, flat):
            torch.index_select(table, 0, before, out=out)

    ctx = sjd.SJD(s.cfg, DEVICE)  # a new image: a new context
    grid, accepted, steps = ctx.decode_loop(forward, c["n_tokens"], s.bufs[0], s.bufs[1] if len(s.bufs) > 1 else None)
    window, rows = ctx.get_window(), ctx.get_rows()
    ctx.close()
    # one length per token at most: zeros after the last step
    accepted = torch.nn.functional.pad(accepted, (0, 0, 0, c["n_tokens"] - steps))
    return {"grid": grid, "accepted": accepted, "steps": steps, "window": list(window), "ids": rows[0],
            "probs": rows[1], "len": rows[2], "logits": s.bufs}


def run(state):
    s, c = state, state.case
    if c["entry"] == "decode":
        return _decode(s)
    ctx, L = s.ctx, s.ctx.L
    if c["entry"] == "chain":
        for out in s.outs:
            cond, uncond = s.logits[s.at]
            s.at = (s.at + 1) % len(s.logits)
            ctx.step(cond, uncond, out=out)
    else:
        cond, uncond = s.logits[s.at]
        s.at = (s.at + 1) % len(s.logits)
        if c["entry"] == "verify":
            ctx.verify_step(cond, uncond, out=s.out)
            _check(s, L.sjd_get_rows(ctx.ctx, *s.rows_args))
            ctx.draft_pd()
        elif c["entry"] == "draft":
            ctx.draft_from_logits(cond, uncond)
        elif c["entry"] == "host":
            ctx.step_host(cond, uncond, s.stage, out=s.out)
        else:
            ctx.step(cond, uncond, out=s.out)
    if c["entry"] != "verify":
        _check(s, L.sjd_get_rows(ctx.ctx, *s.rows_args))
    _check(s, L.sjd_get_window(ctx.ctx, *s.window_args))
    got = {"window": s.window, "ids": s.rows[0], "probs": s.rows[1], "len": s.rows[2]}
    if c["entry"] != "draft":
        got["out"] = s.outs
    if c["entry"] == "tree":
        got["tree"] = list(ctx.get_tree())
    return got


# ---------------------------------------------------------------------------
# What a pass cannot do without, and what its outputs are


def work(case):
    """Allowed logits read once, the stored rows read and written once, and
    the returned rows and window written once (of the entries past a row's
    end, the padding). A row without top-p keeps at most top_k ids; with
    top-p a few dozen. A decode's steps are its tokens over six."""
    c = dict(DEFAULTS, **case)
    veff, s = c["hi"] - c["lo"], _support(c)
    e = 2 if c["dtype"] == "bf16" else 4
    branches = 2 if c["cfg"] != 1.0 else 1
    steps = max(1, c["n_tokens"] // 6) if c["entry"] == "decode" else c["steps"]
    logit_rows = c["batch"] * (c["window"] + _tree_rows(c)) * steps
    window_rows = c["batch"] * c["window"]
    kept = s if c["top_p"] == 1.0 else min(s, 64)
    read = logit_rows * veff * e * branches
    stored = window_rows * steps * kept * 8 * (1 if c["entry"] == "draft" else 2)
    returned = window_rows * (s * 8 + 4 * (c["pd_k"] + 4))
    return {"bytes": read + stored + returned, "flops": logit_rows * veff * 8.0}


def tolerance(case):
    """Tokens, counts and ids are decided on exact integers; a stored
    probability carries two fp32 roundings (5e-8 against 64 bits)."""
    return {"rel": 2.5e-7, "max": 1e-6}


def exact(case, seed):
    """The stored probabilities of the rows in 64 bits, where the rows do not
    depend on what was sampled (the window has not moved when they are read);
    sampled tokens have no such value."""
    c = dict(DEFAULTS, **case)
    if c["entry"] not in ("verify", "draft"):
        return None
    cond, uncond = _logits(c, seed, 0, c["window"])
    s = _support(c)
    probs = torch.zeros((c["batch"], c["window"], s), dtype=torch.float64, device=DEVICE)
    for b in range(c["batch"]):
        l = cond[b, :, c["lo"]:c["hi"]].double()
        if uncond is not None:
            u = uncond[b, :, c["lo"]:c["hi"]].double()
            l = u + c["cfg"] * (l - u)
        l = l / float(torch.tensor(c["temperature"], dtype=torch.float32))
        top, order = torch.sort(l, dim=1, descending=True, stable=True)  # ties: the lower id first
        weight = torch.exp(top - top[:, :1])
        weight[:, s:] = 0.0
        if c["top_p"] < 1.0:
            run_sum = torch.cumsum(weight, dim=1)
            target = float(torch.tensor(c["top_p"], dtype=torch.float32)) * weight.sum(dim=1, keepdim=True)
            weight = torch.where(run_sum - weight < target, weight, torch.zeros_like(weight))
        weight = torch.where(weight >= 2.0 ** -48, weight, torch.zeros_like(weight))  # smaller ones are not stored
        p = torch.zeros_like(weight).scatter_(1, order, weight / weight.sum(dim=1, keepdim=True))
        keep = p > 0
        at = torch.cumsum(keep, dim=1) - 1
        row = torch.arange(c["window"], device=DEVICE).view(-1, 1).expand_as(at)
        probs[b, row[keep], at[keep]] = p[keep]
    return {"window": None, "ids": None, "probs": probs, "len": None}
