"""The work this library is used for, as cases that can be timed: `listed()` and `draw(rng)` give cases, `prepare(case, seed)`
makes a case's inputs, `run(state)` is one call of the public entry point, `work(case)` what that call cannot do without and
`tolerance(case)` how far another correct implementation may be off.

A case is a dict of plain values:
  op        forward | solve | host | decode | tokens: gka_fwd_chunked, gka_solve_chunked, gka_fwd_chunked_host, gka_decode_step,
            gka_decode_tokens
  B, heads, T, d, n_iter   sequences, heads, tokens per sequence, head dimension, Chebyshev iterations
  dtype     bf16 | f32: q, k, v, out;  high: fp32 arithmetic asked for whatever the dtype
  rule      given: lambda_t is an input;  adaptive: lambda_t = 0.02 ||H_t||_F, the setting of the method's experiments
  state_in, beta, alpha    the optional inputs: an initial state, write strengths, weights of the alpha-connection
  recipe    plain | slow | stress: gates and keys of training batches, of long contexts (slow fading), and of keys that lie
            close to a low-dimensional subspace with a small ridge
"""
import math

import torch

from paper_2511_21016_b200 import gka

CHUNK = 64
DEVICE = "cuda"
PREFIX = 128        # tokens of the prefix whose recurrence makes an initial state


def _case(name, op, B, heads, T, d, n_iter, dtype="bf16", high=False, rule="given", state_in=False, beta=False, alpha=False,
          recipe="plain"):
    case = dict(op=op, B=B, heads=heads, T=T, d=d, n_iter=n_iter, dtype=dtype, high=high, rule=rule, state_in=state_in,
                beta=beta, alpha=alpha, recipe=recipe)
    return case if name is None else dict(name=name, **case)


def listed():
    return [
        # a small layer in fp32, called as a test or an experiment does: launches and latency
        _case("forward_f32_small", "forward", 1, 2, 256, 64, 8, dtype="f32"),
        # a training batch: the benchmark's headline shape
        _case("forward_train", "forward", 4, 16, 4096, 128, 10),
        # prefill of a few requests of an odd length at the setting of the method's experiments, going on from a cached state,
        # with write strengths and the alpha-connection
        _case("prefill_ragged", "forward", 3, 8, 1999, 128, 30, rule="adaptive", state_in=True, beta=True, alpha=True),
        # the backward pass of a training batch: the same solve gives dq from dx
        _case("backward_solve", "solve", 4, 8, 2048, 128, 30, rule="adaptive"),
        # one long document with slowly fading gates
        _case("prefill_long", "forward", 1, 32, 131072, 128, 10, recipe="slow"),
        # a training batch of a model with heads of 64 channels
        _case("forward_d64", "forward", 4, 16, 2048, 64, 10),
        # badly conditioned keys, for which fp32 arithmetic is asked for
        _case("forward_high", "forward", 2, 8, 8192, 128, 8, dtype="f32", high=True, recipe="stress"),
        # image patches: many short sequences, heads of 16 channels
        _case("forward_d16", "forward", 64, 8, 196, 16, 30, rule="adaptive"),
        # one sequence being generated: the smallest decode call
        _case("decode_one", "decode", 1, 32, 1, 128, 30, rule="adaptive"),
        # a full serving batch, one token each
        _case("decode_batch", "decode", 256, 32, 1, 128, 10),
        # a serving batch with a few drafted tokens each
        _case("decode_tokens", "tokens", 64, 32, 8, 128, 10),
        # a training batch that lies in host memory
        _case("forward_host", "host", 4, 16, 4096, 128, 10),
    ]


def _log(rng, lo, hi):
    """A whole number from lo to hi, spread over its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _tokens(rng, B, heads, lo, hi, most):
    """A sequence length whose token-heads stay below `most`."""
    return _log(rng, lo, max(lo, min(hi, most // (B * heads))))


def draw(rng):
    kind = rng.choice([c["name"] for c in listed()])
    r, rule = rng.choice([(10, "given"), (30, "adaptive"), (rng.randint(4, 32), "given")])
    if kind == "forward_f32_small":
        B, heads = rng.randint(1, 2), rng.randint(1, 4)
        return _case(None, "forward", B, heads, _log(rng, 64, 1024), 64, r, dtype="f32", rule=rule)
    if kind in ("forward_train", "forward_d64", "forward_host"):
        B, heads, d = _log(rng, 1, 16), rng.choice([4, 8, 12, 16, 24, 32]), 64 if kind == "forward_d64" else 128
        if kind == "forward_host":
            B = min(B, 6)
        T = _tokens(rng, B, heads, 256, 8192, 1 << 19 if kind != "forward_host" else 1 << 18)
        return _case(None, "host" if kind == "forward_host" else "forward", B, heads, T, d, r, rule=rule)
    if kind == "prefill_ragged":
        B, heads = rng.randint(1, 6), rng.choice([5, 8, 16, 32])
        return _case(None, "forward", B, heads, _log(rng, 17, 4000), 128, r, rule=rule, state_in=rng.random() < 0.7,
                     beta=rng.random() < 0.5, alpha=rng.random() < 0.5)
    if kind == "backward_solve":
        B, heads, d = _log(rng, 1, 16), rng.choice([4, 8, 12, 16]), rng.choice([64, 128, 128])
        return _case(None, "solve", B, heads, _tokens(rng, B, heads, 256, 8192, 1 << 18), d, r, rule=rule)
    if kind == "prefill_long":
        heads = rng.choice([4, 8, 16, 32])
        return _case(None, "forward", 1, heads, _log(rng, 8192, 131072), 128, 10, recipe="slow")
    if kind == "forward_high":
        B, heads = rng.randint(1, 2), rng.choice([4, 8])
        return _case(None, "forward", B, heads, _log(rng, 512, 8192), 128, rng.choice([4, 8, 16]),
                     dtype=rng.choice(["f32", "bf16"]), high=True, recipe="stress")
    if kind == "forward_d16":
        B, heads, d = _log(rng, 8, 128), rng.choice([2, 4, 8]), rng.choice([16, 16, 32])
        return _case(None, "forward", B, heads, _log(rng, 49, 784), d, r, rule=rule, dtype=rng.choice(["bf16", "bf16", "f32"]))
    if kind == "decode_one":
        return _case(None, "decode", rng.randint(1, 4), rng.choice([8, 16, 32]), 1, rng.choice([64, 128, 128]), r, rule=rule,
                     dtype=rng.choice(["bf16", "bf16", "f32"]), beta=rng.random() < 0.3, alpha=rng.random() < 0.3)
    if kind == "decode_batch":
        return _case(None, "decode", _log(rng, 5, 256), rng.choice([8, 16, 32]), 1, rng.choice([64, 128, 128]), r, rule=rule)
    return _case(None, "tokens", _log(rng, 1, 256), rng.choice([8, 16, 32]), rng.randint(2, 9), rng.choice([64, 128, 128]), r,
                 rule=rule)


def _unit(x):
    return x / x.norm(dim=-1, keepdim=True)


class _Inputs:
    """Random inputs of a case, made on the GPU from the seed alone."""

    #: mean of the gates before the sigmoid; mean, offset and scale of lambda around the softplus
    RECIPES = dict(plain=(2.0, 0.0, 1e-2, 1.0), slow=(4.0, -1.0, 1e-3, 1.0), stress=(6.0, 0.0, 0.0, 1e-4))

    def __init__(self, case, seed):
        self.case, self.io = case, torch.float32 if case["dtype"] == "f32" else torch.bfloat16
        self.gen = torch.Generator(device=DEVICE)
        self.gen.manual_seed(seed)

    def normal(self, *shape):
        return torch.randn(shape, generator=self.gen, device=DEVICE)

    def uniform(self, lo, hi, shape):
        return torch.rand(shape, generator=self.gen, device=DEVICE) * (hi - lo) + lo

    def queries(self, shape):
        return _unit(self.normal(*shape)).to(self.io)

    def keys(self, shape):
        if self.case["recipe"] != "stress":
            return self.queries(shape)
        B, T, heads, d = shape          # close to an 8-dimensional subspace of each head
        near = torch.einsum("bthr,bhrd->bthd", self.normal(B, T, heads, 8), self.normal(B, heads, 8, d))
        return _unit(near.contiguous() + 0.01 * self.normal(*shape)).to(self.io)

    def gates(self, shape):
        return torch.sigmoid(self.normal(*shape) + self.RECIPES[self.case["recipe"]][0])

    def lambdas(self, shape):
        if self.case["rule"] == "adaptive":
            return torch.full(shape, 0.02, device=DEVICE)
        _, mean, offset, scale = self.RECIPES[self.case["recipe"]]
        return torch.nn.functional.softplus(self.normal(*shape) + mean) * scale + offset

    def state(self, B, heads, d):
        """H and U that the recurrence leaves behind after a prefix."""
        k, v = _unit(self.normal(B, heads, PREFIX, d)), self.normal(B, heads, PREFIX, d)
        fade = torch.log(self.gates((B, heads, PREFIX)))
        k_faded = k * torch.exp(fade.sum(-1, keepdim=True) - fade.cumsum(-1))[..., None]
        return torch.stack([k.transpose(-1, -2) @ k_faded, v.transpose(-1, -2) @ k_faded], 2).reshape(B, heads, 2 * d * d)


def prepare(case, seed):
    B, heads, T, d, op = case["B"], case["heads"], case["T"], case["d"], case["op"]
    x = _Inputs(case, seed)
    tokens = (B, heads) if op == "decode" else (B, T, heads)
    io = gka.GKA_F32 if case["dtype"] == "f32" else gka.GKA_BF16
    s = dict(op=op, n_iter=case["n_iter"], flags=gka.GKA_FLAG_ADAPTIVE_LAMBDA if case["rule"] == "adaptive" else 0,
             q=x.queries(tokens + (d,)), k=x.keys(tokens + (d,)), v=x.normal(*tokens, d).to(x.io), gate=x.gates(tokens),
             lam=x.lambdas(tokens), precision=gka.GKA_PREC_HIGH if case["high"] else gka.GKA_PREC_NATIVE,
             state=x.state(B, heads, d) if op in ("decode", "tokens") or case["state_in"] else None,
             beta=x.uniform(0.2, 1.0, tokens) if case["beta"] else None,
             alpha=x.uniform(0.0, 1.0, tokens) if case["alpha"] else None)
    if op in ("forward", "solve", "host"):
        s["workspace"] = gka.alloc_workspace(B, T, heads, d, torch.device(DEVICE), CHUNK, io, s["precision"])
    if op == "host":
        for n in ("q", "k", "v", "gate", "lam"):
            s[n] = torch.empty(s[n].shape, dtype=s[n].dtype, pin_memory=True).copy_(s[n])
        s["out"] = torch.empty(s["v"].shape, dtype=x.io, pin_memory=True)
        s["state_out"] = torch.empty(B, heads, 2 * d * d, pin_memory=True)
        s["staging"] = torch.empty(gka.gka_fwd_host_staging_bytes(B, T, heads, d, io), dtype=torch.uint8,
                                   device=DEVICE)
    return s


def run(s):
    op = s["op"]
    if op == "forward":
        return gka.gka_fwd_chunked(s["q"], s["k"], s["v"], s["gate"], s["lam"], s["n_iter"], CHUNK, state_in=s["state"],
                                   workspace=s["workspace"], precision=s["precision"], flags=s["flags"], beta=s["beta"],
                                   alpha=s["alpha"])
    if op == "solve":
        return gka.gka_solve_chunked(s["q"], s["k"], s["gate"], s["lam"], s["n_iter"], CHUNK, workspace=s["workspace"],
                                     precision=s["precision"], flags=s["flags"])
    if op == "host":
        return gka.gka_fwd_chunked_host(s["q"], s["k"], s["v"], s["gate"], s["lam"], s["n_iter"], CHUNK, s["out"],
                                        s["state_out"], staging=s["staging"], workspace=s["workspace"], flags=s["flags"])
    step = gka.gka_decode_step if op == "decode" else gka.gka_decode_tokens
    out = step(s["state"], s["q"], s["k"], s["v"], s["gate"], s["lam"], s["n_iter"], flags=s["flags"], beta=s["beta"],
               alpha=s["alpha"])
    return out, s["state"]


def work(case):
    """Bytes: every input read once, every output written once.  Operations: per token n_iter products of H with a vector, the
    read with U, and the rank-one writes into H and U; the solve alone has neither read nor U."""
    op, d, pairs = case["op"], case["d"], case["B"] * case["heads"]
    n, io = pairs * case["T"], 4 if case["dtype"] == "f32" else 2
    scalars = 4 * (2 + case["beta"] + case["alpha"])
    state = 4 * 2 * d * d * pairs
    if op == "solve":
        return {"bytes": n * (3 * d * io + scalars), "flops": 2 * d * d * n * (case["n_iter"] + 1)}
    states = (2 if op in ("decode", "tokens") or case["state_in"] else 1) * state
    return {"bytes": n * (4 * d * io + scalars) + states, "flops": 2 * d * d * n * (case["n_iter"] + 3)}


def tolerance(case):
    fp32 = case["dtype"] == "f32" or case["high"] or case["d"] < 64 or case["op"] in ("decode", "tokens")
    if not fp32:
        return {"rel": 1e-2}                            # bf16 operands
    if case["dtype"] == "bf16":
        return {"rel": 4e-3, "max": 2e-2}               # fp32 arithmetic, results rounded to bf16
    if case["recipe"] == "stress":
        return {"rel": 3e-6 * case["n_iter"]}           # 32-bit sums at a condition number of about 1e6
    return {"rel": 1e-5}                                # 32-bit sums
