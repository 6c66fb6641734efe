"""The state kernel's blocks per work item (four, two, one) on both sides of the limits of 148 SMs, against the fp64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2511_21016_b200 import gka, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def rel(a, b):
    return float(np.linalg.norm(a.double().cpu().numpy() - b) / np.linalg.norm(b))


@pytest.mark.parametrize("heads,T,d", [(1, 129, 128), (37, 300, 128), (38, 300, 128), (74, 200, 128), (75, 200, 128), (5, 300, 64)])
def test_state_norms_and_output_at_split_limits(heads, T, d):
    cfg = synth.GkaConfig("split", B=1, heads=heads, T=T, d=d, chunk=64, n_iter=4, io_dtype="bf16", seed=47, gate_mean=5.0)
    inp = synth.make_inputs(cfg)
    dev = {n: torch.from_numpy(a).to(DEV) for n, a in inp.items()}
    for n in "qkv":
        dev[n] = dev[n].bfloat16()
        inp[n] = dev[n].float().cpu().numpy()
    st_in = 0.1 * torch.randn(1, heads, 2 * d * d, generator=torch.Generator().manual_seed(3))
    h = st_in[..., : d * d].view(1, heads, d, d)
    h.copy_(h @ h.transpose(-1, -2).contiguous() / d)          # H_0 symmetric positive, U_0 arbitrary
    ref = oracle.fwd(inp["q"], inp["k"], inp["v"], inp["gate"], inp["lam"], 4, state_in=st_in.numpy())
    fro = torch.empty(1, T, heads, device=DEV)
    out, st = gka.gka_fwd_chunked(dev["q"], dev["k"], dev["v"], dev["gate"], dev["lam"], 4, state_in=st_in.to(DEV), fro_out=fro)
    assert rel(out, ref["out"]) < 2e-2
    assert rel(st, ref["state"]) < 1e-2
    assert rel(fro, ref["fro"]) < 1e-2
