"""The scans over chunks (head dimensions 16 and 32) and segments (64 and 128), which load eight of them at a time: one fewer
than a group, a group, one more, and two groups and one, with slow gates and an initial state, against the fp64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2511_21016_b200 import gka, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / max(np.linalg.norm(b), 1e-300))


@pytest.mark.parametrize("d,T", [(16, 32 * 7), (16, 32 * 8), (16, 32 * 8 + 1), (32, 32 * 16 + 5), (64, 36), (64, 160), (128, 600)])
def test_states_through_the_scans(d, T):
    cfg = synth.GkaConfig("scan", B=1, heads=3, T=T, d=d, chunk=64, n_iter=3, io_dtype="f32", seed=53, gate_mean=6.0)
    inp = synth.make_inputs(cfg)
    rng = np.random.default_rng(T)
    A = 0.3 * rng.standard_normal((1, 3, d, 4))
    s_in = np.concatenate([(A @ A.swapaxes(-1, -2)).reshape(1, 3, -1), 0.1 * rng.standard_normal((1, 3, d * d))], -1).astype(np.float32)
    ref = oracle.fwd(inp["q"], inp["k"], inp["v"], inp["gate"], inp["lam"], 3, state_in=s_in)
    dev = {n: torch.from_numpy(a).to(DEV) for n, a in inp.items()}
    out, st = gka.gka_fwd_chunked(dev["q"], dev["k"], dev["v"], dev["gate"], dev["lam"], 3, state_in=torch.from_numpy(s_in).to(DEV))
    # 32-bit sums throughout, as in the tests of the kernels themselves
    assert rel(out.cpu().numpy(), ref["out"]) <= (1e-4 if d < 64 else 1e-5)
    assert rel(st.cpu().numpy(), ref["state"]) <= 1e-5
