"""The state kernel where its pipeline turns over: one tile, as many tiles as stages, sets and barriers and one more or less, in each
division of the masters among blocks (four blocks per sequence, two, one; head dimension 64), sequences cut into ranges with and
without the scan, write strengths, and the solve alone (whose blocks keep no U), against the fp64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2511_21016_b200 import gka, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def rel(a, b):
    return float(np.linalg.norm(a.double().cpu().numpy() - b) / np.linalg.norm(b))


@pytest.mark.parametrize("heads,d", [(2, 128), (40, 128), (80, 128), (3, 64)])
@pytest.mark.parametrize("tiles", [1, 2, 3, 4, 6, 7, 8, 9, 15])
def test_state_pipeline_at_its_turns(heads, d, tiles):
    check(1, heads, 128 * tiles - 5, d, beta=tiles % 2 == 0)


@pytest.mark.parametrize("B,heads,T,d", [(1, 1, 128 * 64 + 1, 128), (1, 3, 128 * 70, 128), (1, 7, 128 * 90, 64), (1, 1, 64 * 200, 64)])
def test_sequences_cut_into_ranges(B, heads, T, d):
    check(B, heads, T, d, beta=heads == 3)


def check(B, heads, T, d, beta):
    cfg = synth.GkaConfig("kinds", B=B, heads=heads, T=T, d=d, chunk=64, n_iter=2, io_dtype="bf16", seed=59, gate_mean=5.0)
    inp = synth.make_inputs(cfg)
    dev = {n: torch.from_numpy(a).to(DEV) for n, a in inp.items()}
    for n in "qkv":
        dev[n] = dev[n].bfloat16()
        inp[n] = dev[n].float().cpu().numpy()
    b = np.random.default_rng(T).uniform(0.2, 1.0, inp["gate"].shape).astype(np.float32) if beta else None
    bd = torch.from_numpy(b).to(DEV) if beta else None
    ref = oracle.fwd(inp["q"], inp["k"], inp["v"], inp["gate"], inp["lam"], 2, want_x=True, **(dict(beta=b) if beta else {}))
    fro, status = torch.empty(B, T, heads, device=DEV), torch.zeros(1, dtype=torch.int32, device=DEV)
    out, st = gka.gka_fwd_chunked(dev["q"], dev["k"], dev["v"], dev["gate"], dev["lam"], 2, fro_out=fro, beta=bd, device_status=status)
    x = gka.gka_solve_chunked(dev["q"], dev["k"], dev["gate"], dev["lam"], 2, beta=bd, device_status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    # bf16 operands: every element is off by a few times 2^-9 (keys, states, masked scores, iterate)
    assert rel(out, ref["out"]) < 2e-2
    assert rel(x, ref["x"]) < 2e-2
    assert rel(st, ref["state"]) < 1e-2
    assert rel(fro, ref["fro"]) < 1e-2
