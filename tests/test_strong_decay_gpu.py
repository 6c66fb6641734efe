"""Tiles of 128 tokens that decay below 2^-60 (strong gates, resets, zero gates), whose keys are not scaled and whose masked scores take a
factor each, on the tensor-core path: in the plain kernel and in those with write strengths, the alpha-connection and the solve alone, next
to tiles on the other side of the line, against the fp64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2511_21016_b200 import gka, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def rel(a, b):
    return float(np.linalg.norm(a.double().cpu().numpy() - b) / np.linalg.norm(b))


def gates(kind, shape):
    rng = np.random.default_rng(73)
    mean = {"strong": 1.0, "stronger": 0.0}.get(kind, 5.0)
    g = 1.0 / (1.0 + np.exp(-(rng.standard_normal(shape) + mean)))
    if kind in ("resets", "zeros"):        # at the edges of a tile's groups of 32 tokens, several in a tile, one per tile, none
        g[:, [0, 31, 32, 200, 255, 256, 352, 479, 480]] = 1e-30 if kind == "resets" else 0.0
    if kind == "line":                     # tiles that decay by 2^-59 and by 2^-61
        g[:] = 2.0 ** (-59.0 / 128)
        g[:, 128:256] = g[:, 512:] = 2.0 ** (-61.0 / 128)
    return g.astype(np.float32)


@pytest.mark.parametrize("kind", ["strong", "stronger", "resets", "zeros", "line"])
@pytest.mark.parametrize("d", [128, 64])
@pytest.mark.parametrize("options", [False, True])
@pytest.mark.parametrize("adaptive", [False, True])
def test_tiles_that_decay_below_the_line(d, kind, options, adaptive):
    B, T, heads, r = 2, 700, 3, 10
    cfg = synth.GkaConfig("strong", B=B, heads=heads, T=T, d=d, chunk=64, n_iter=r, io_dtype="bf16", seed=7)
    inp = synth.make_inputs(cfg)
    inp["gate"] = gates(kind, (B, T, heads))
    if adaptive:
        inp["lam"].fill(0.02)
    rng = np.random.default_rng(3)
    extra = {n: rng.uniform(lo, 1.0, (B, T, heads)).astype(np.float32) for n, lo in (("beta", 0.2), ("alpha", 0.0))} if options else {}
    ref = oracle.fwd(inp["q"], inp["k"], inp["v"], inp["gate"], inp["lam"], r, lam_mode=int(adaptive), want_x=True, **extra)
    dev = {n: torch.from_numpy(a).to(DEV) for n, a in {**inp, **extra}.items()}
    q, k, v = (dev[n].bfloat16() for n in "qkv")
    fro, status = torch.empty(B, T, heads, device=DEV), torch.zeros(1, dtype=torch.int32, device=DEV)
    kw = dict(flags=gka.GKA_FLAG_ADAPTIVE_LAMBDA if adaptive else 0, device_status=status, beta=dev.get("beta"))
    out, st = gka.gka_fwd_chunked(q, k, v, dev["gate"], dev["lam"], r, fro_out=fro, alpha=dev.get("alpha"), **kw)
    x = gka.gka_solve_chunked(q, k, dev["gate"], dev["lam"], r, **kw)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    # bf16 operands: every element is off by a few times 2^-9 (keys, states, masked scores, iterate)
    assert rel(out, ref["out"]) < 2e-2 and rel(x, ref["x"]) < 1e-2
    assert rel(st, ref["state"]) < 5e-3 and rel(fro, ref["fro"]) < 5e-3
    for t0 in range(0, T, 128):            # no tile hides behind the others
        tile = slice(t0, t0 + 128)
        assert rel(out[:, tile], ref["out"][:, tile]) < 2e-2 and rel(x[:, tile], ref["x"][:, tile]) < 1e-2
