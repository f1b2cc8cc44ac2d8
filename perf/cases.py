"""The work users have this framework do, as cases that can be timed and compared.

Three kinds of call, all through the package's public functions:

  prefill  ``vla_forward`` over a whole sequence (optionally with penalty directions that
           ``vla_make_u`` forms from a projection first, optionally continuing from carried
           states, in either tensor layout);
  decode   ``vla_forward`` with T = 1 and the states updated in place, one generation step;
  train    ``vla_scan`` forward and the gradients of its inputs through torch.autograd.

``listed()`` holds the repository's own configurations (the paper's recall setting, a tiny, a mid,
a long-context and a throughput shape, decode) and what lies between them; ``draw()`` gives more
cases over the same ranges: every head width the library has, both input types, one to thousands of
(batch, head) units, 2 to 65536 tokens.
"""
import math

import torch

import paper_2605_11196_b200 as vla

DEV = "cuda"
_DTYPE = {"f32": torch.float32, "bf16": torch.bfloat16}


def _case(kind, B, H, d, T, dtype, **kw):
    c = {"kind": kind, "B": B, "H": H, "d": d, "T": T, "dtype": dtype, "data": "normal", "lam": 1.0,
         "identity": False, "token_major": False, "carried": False, "u": "", "workspace": False}
    c.update(kw)
    return c


def listed():
    def named(name, *a, **kw):
        c = _case(*a, **kw)
        c["name"] = name
        return c

    return [
        # one generation step of one sequence in the paper's setting (4 heads of 32): launch latency
        named("decode-one", "decode", 1, 4, 32, 1, "f32"),
        # one generation step of a serving batch: every unit's two states pass through the chip once
        named("decode-batch", "decode", 64, 64, 128, 1, "bf16"),
        # the smallest prompt: one narrow head
        named("prefill-tiny", "prefill", 1, 1, 16, 256, "f32"),
        # the paper's associative-recall setting (24 pairs, 4 heads of 32, batch 64)
        named("prefill-recall", "prefill", 64, 4, 32, 512, "f32", data="recall"),
        # an ordinary batch of prompts, fewer units than SMs
        named("prefill-mid", "prefill", 4, 8, 64, 4096, "f32"),
        # one long document; the caller lets the library cut it into segments
        named("prefill-long", "prefill", 1, 16, 64, 65536, "bf16", workspace=True),
        # a full batch: the benchmark's default
        named("prefill-throughput", "prefill", 32, 16, 128, 8192, "bf16"),
        # a ragged chunk of a prompt as the projections write it ([B,T,H,d]), continuing from earlier states
        named("prefill-continue", "prefill", 3, 16, 128, 1777, "bf16", token_major=True, carried=True),
        # learned penalty directions: the projection, then the scan with explicit u
        named("prefill-learned-u", "prefill", 8, 16, 128, 2048, "bf16", u="made"),
        # training steps: the recall setting, an ordinary batch, wide heads as the projections write them
        named("train-recall", "train", 64, 4, 32, 512, "f32", data="recall"),
        named("train-mid", "train", 4, 8, 64, 4096, "f32"),
        named("train-wide", "train", 8, 16, 128, 2048, "bf16", token_major=True),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def draw(rng):
    kind = rng.choices(("prefill", "train", "decode"), (5, 4, 2))[0]
    d = rng.choices((16, 32, 64, 128), (1, 2, 3, 3))[0]
    dtype = rng.choice(("f32", "bf16"))
    lam = rng.choice((1.0, 1.0, 1.0, 0.1, 0.5))
    identity = rng.random() < 0.3
    if kind == "decode":
        # from one sequence to a serving batch of 4096 units
        return _case(kind, _log_int(rng, 1, 64), _log_int(rng, 1, 64), d, 1, dtype, lam=lam, identity=identity)
    # sequences: a batch of 1..64 with 1..32 heads, within the listed cases' total work and longest chain
    most, longest = 4 << 20, (65536 * 64) // d
    if kind == "train":
        most, longest = 8 * 16 * 2048, 4096
    T = _log_int(rng, 2, min(65536, longest))
    B, H = _log_int(rng, 1, 64), _log_int(rng, 1, 32)
    tokens = most * 128 // max(d, 64)    # as many elements as there, at most twice the tokens
    while B * H * T > tokens:
        if B > 1:
            B = (B + 1) // 2
        else:
            H = (H + 1) // 2
    wide = d >= 32          # token-major gradients and explicit u in training start at d = 32
    token_major = rng.random() < 0.3 and (wide or kind == "prefill")
    carried = rng.random() < 0.3
    u = "" if rng.random() < 0.7 or not wide else ("made" if kind == "prefill" and not token_major else "given")
    data = "recall" if T >= 64 and not token_major and rng.random() < 0.2 else "normal"
    workspace = kind == "prefill" and rng.random() < 0.3
    return _case(kind, B, H, d, T, dtype, lam=lam, identity=identity, token_major=token_major, carried=carried, u=u,
                 data=data, workspace=workspace)


def _recall(g, B, H, T, d):
    """24 stored pairs (unit keys, N(0,1) values), filler of size 0.1, then 24 queries of the stored keys."""
    n = 24
    q, k, v = [0.1 * torch.randn((B, H, T, d), generator=g, device=DEV) for _ in range(3)]
    keys = torch.nn.functional.normalize(torch.randn((B, H, n, d), generator=g, device=DEV), dim=-1)
    k[:, :, :n] = keys
    v[:, :, :n] = torch.randn((B, H, n, d), generator=g, device=DEV)
    order = torch.rand((B, H, n), generator=g, device=DEV).argsort(-1)
    q[:, :, T - n:] = torch.gather(keys, 2, order.unsqueeze(-1).expand(-1, -1, -1, d))
    return q, k, v


def prepare(case, seed):
    c = case
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    B, H, T, d, dt = c["B"], c["H"], c["T"], c["d"], _DTYPE[c["dtype"]]
    shape = (B, T, H, d) if c["token_major"] else (B, H, T, d)
    if c["data"] == "recall":
        q, k, v = [x.to(dt) for x in _recall(g, B, H, T, d)]
    else:
        q, k, v = [torch.randn(shape, generator=g, device=DEV, dtype=dt) for _ in range(3)]
    s = {"case": c, "q": q, "k": k, "v": v, "lam": c["lam"], "kw": {}, "carry": {}}
    s["kw"]["flags"] = (vla.VLA_FLAG_IDENTITY_MAP if c["identity"] else 0) | (vla.VLA_FLAG_TOKEN_MAJOR if c["token_major"] else 0)
    if c["kind"] == "decode" or c["carried"]:
        # states as an earlier call leaves them: A between 0 and I / lambda, a memory of order one, a positive key sum
        w = torch.nn.functional.normalize(torch.randn((B, H, d, 4), generator=g, device=DEV), dim=2)
        eye = torch.eye(d, device=DEV)
        s["carry"] = {"S0": 0.3 * torch.randn((B, H, d, d), generator=g, device=DEV),
                      "A0": (0.2 * eye + 0.1 * (w @ w.transpose(-1, -2))).contiguous() / c["lam"],
                      "z0": 20.0 + 5.0 * torch.rand((B, H, d), generator=g, device=DEV)}
    if c["u"] == "made":
        s["W_u"] = torch.randn((H, d, d), generator=g, device=DEV) * d ** -0.5
    elif c["u"] == "given":
        s["kw"]["u"] = (torch.nn.functional.normalize(torch.randn(shape, generator=g, device=DEV), dim=-1) * d ** -0.5).to(dt)
    if c["kind"] == "train":
        s["g"] = torch.randn(shape, generator=g, device=DEV) * d ** -0.5
        s["leaves"] = [q, k, v] + ([s["kw"]["u"]] if c["u"] else [])
        for x in s["leaves"]:
            x.requires_grad_(True)
    return s


def run(s):
    c, q, k, v, lam = s["case"], s["q"], s["k"], s["v"], s["lam"]
    if c["kind"] == "decode":
        S, A, z = s["carry"]["S0"], s["carry"]["A0"], s["carry"]["z0"]
        r = vla.vla_forward(q, k, v, lam, S0=S, A0=A, z0=z, S_T=S, A_T=A, z_T=z, **s["kw"])
        return r.out, r.S_T, r.A_T, r.z_T
    if c["kind"] == "train":
        out, S_T, A_T, z_T = vla.vla_scan(q, k, v, lam, **s["kw"], **s["carry"])
        return (out, S_T, A_T, z_T) + torch.autograd.grad(out, s["leaves"], s["g"])
    kw = dict(s["kw"])
    if c["u"] == "made":
        kw["u"] = vla.vla_make_u(k, s["W_u"])
    r = vla.vla_forward(q, k, v, lam, workspace=c["workspace"], **kw, **s["carry"])
    return r.out, r.S_T, r.A_T, r.z_T


def work(case):
    """Inputs read once, outputs written once; per token the mat-vecs A u, S k, S q and the two rank-1
    updates (A's on its triangle), three times that with the gradients, plus the projection of u."""
    c = case
    B, H, T, d = c["B"], c["H"], c["T"], c["d"]
    es = 4 if c["dtype"] == "f32" else 2
    tokens, state = B * H * T, B * H * (2 * d * d + d) * 4
    bytes_ = tokens * d * (3 * es + 4) + state
    if c["kind"] == "decode" or c["carried"]:
        bytes_ += state
    macs = tokens * (d * d + d * (d + 1) / 2 + 3 * d * d)
    if c["u"] == "made":
        bytes_ += H * d * d * 4
        macs += tokens * d * d
    elif c["u"] == "given":
        bytes_ += tokens * d * es
    if c["kind"] == "train":
        bytes_ += tokens * d * (4 + (4 if c["u"] else 3) * es)
        macs *= 3
    return {"bytes": bytes_, "flops": 2 * macs}


def tolerance(case):
    """fp32 state arithmetic: rounding adds up over the tokens of the recurrence, and another order of
    the same sums differs by this much.  Gradients come back in the inputs' type."""
    T = case["T"]
    rel = 2e-5 if T <= 512 else 5e-5 if T <= 4096 else 2e-4
    if case["kind"] == "train":
        rel = 2e-4 if case["dtype"] == "f32" else 5e-3     # bf16 gradients: one rounding of the last place
    elif case["u"] == "made" and case["dtype"] == "bf16":
        rel = 5e-3                                          # u itself is rounded to bf16
    return {"rel": rel}
