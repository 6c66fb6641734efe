"""The fp32 recurrence kernels (head dimensions 64 and 128) at the edges of their decomposition, against the fp64 oracle:
sequences of less than a batch of four tokens and with every remainder of one, one segment or many, parts of segments, more
pairs than blocks fit the device, and slow gates so that a wrong start state shows."""
import numpy as np
import pytest
import torch

import oracle
from paper_2511_21016_b200 import gka, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / max(np.linalg.norm(b), 1e-300))


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("B,heads,T", [(1, 1, 1), (1, 2, 2), (2, 1, 3), (1, 3, 5), (1, 1, 64), (1, 2, 257), (3, 7, 131),
                                       (40, 16, 6), (1, 1, 4099)])
def test_fp32_forward_and_solve_at_the_edges_of_the_split(d, B, heads, T):
    cfg = synth.GkaConfig("edge", B=B, heads=heads, T=T, d=d, chunk=64, n_iter=5, io_dtype="f32", seed=31, gate_mean=5.0)
    inp = synth.make_inputs(cfg)
    rng = np.random.default_rng(T)
    A = 0.3 * rng.standard_normal((B, heads, d, 4))
    s_in = np.concatenate([(A @ A.swapaxes(-1, -2)).reshape(B, heads, -1), 0.1 * rng.standard_normal((B, heads, d * d))], -1).astype(np.float32)
    ref = oracle.fwd(inp["q"], inp["k"], inp["v"], inp["gate"], inp["lam"], 5, state_in=s_in, want_x=True)
    dev = {n: torch.from_numpy(a).to(DEV) for n, a in inp.items()}
    st_in = torch.from_numpy(s_in).to(DEV)
    fro = torch.zeros(B, T, heads, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    out, st = gka.gka_fwd_chunked(dev["q"], dev["k"], dev["v"], dev["gate"], dev["lam"], 5, state_in=st_in, fro_out=fro,
                                  device_status=status)
    x = gka.gka_solve_chunked(dev["q"], dev["k"], dev["gate"], dev["lam"], 5, state_in=st_in, device_status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    assert rel(out.cpu().numpy(), ref["out"]) <= 1e-5
    assert rel(x.cpu().numpy(), ref["x"]) <= 1e-5
    assert rel(st.cpu().numpy(), ref["state"]) <= 1e-5
    assert rel(fro.cpu().numpy(), ref["fro"]) <= 1e-5
