"""The forward and solve kernels of head dimensions 16 and 32 at the edges of their 32-token chunks and 8-token runs, against
the fp64 oracle: one token, a full chunk and one more or less, many chunks, slow gates, odd numbers of heads."""
import numpy as np
import pytest
import torch

import oracle
from paper_2511_21016_b200 import gka, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / max(np.linalg.norm(b), 1e-300))


@pytest.mark.parametrize("d", [16, 32])
@pytest.mark.parametrize("B,heads,T", [(1, 1, 1), (2, 3, 7), (1, 2, 31), (1, 5, 32), (3, 1, 33), (1, 1, 1000)])
@pytest.mark.parametrize("adaptive", [False, True])
def test_small_head_forward_and_solve_at_chunk_edges(d, B, heads, T, adaptive):
    cfg = synth.GkaConfig("edge", B=B, heads=heads, T=T, d=d, chunk=64, n_iter=5, io_dtype="f32", seed=41, gate_mean=5.0)
    inp = synth.make_inputs(cfg)
    lam = np.full_like(inp["lam"], 0.05) if adaptive else inp["lam"]
    ref = oracle.fwd(inp["q"], inp["k"], inp["v"], inp["gate"], lam, 5, lam_mode=1 if adaptive else 0, want_x=True)
    dev = {n: torch.from_numpy(a).to(DEV) for n, a in inp.items()}
    lam_d = torch.from_numpy(lam).to(DEV)
    flags = gka.GKA_FLAG_ADAPTIVE_LAMBDA if adaptive else 0
    out, st = gka.gka_fwd_chunked(dev["q"], dev["k"], dev["v"], dev["gate"], lam_d, 5, flags=flags)
    x = gka.gka_solve_chunked(dev["q"], dev["k"], dev["gate"], lam_d, 5, flags=flags)
    torch.cuda.synchronize()
    assert rel(out.cpu().numpy(), ref["out"]) <= 1e-4
    assert rel(x.cpu().numpy(), ref["x"]) <= 1e-4
    assert rel(st.cpu().numpy(), ref["state"]) <= 1e-5
