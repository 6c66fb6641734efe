"""The solve alone keeps no U: with a workspace full of NaN its result is right, and no copy of U is written to it."""
import numpy as np
import pytest
import torch

import oracle
from paper_2511_21016_b200 import gka, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# head dimension 64: one tile, several items, cut sequences whose summaries are folded and scanned; 128: two blocks per item, one, cut
@pytest.mark.parametrize("heads,T,d", [(1, 100, 64), (1, 128 * 7, 64), (150, 300, 64), (5, 128 * 160, 64), (1, 128 * 90, 64),
                                       (40, 300, 128), (80, 300, 128), (1, 128 * 90, 128)])
@pytest.mark.parametrize("state", [False, True])
def test_solve_alone_neither_reads_nor_writes_u(heads, T, d, state):
    cfg = synth.GkaConfig("solve", B=1, heads=heads, T=T, d=d, chunk=64, n_iter=3, io_dtype="bf16", seed=61, gate_mean=5.0)
    inp = synth.make_inputs(cfg)
    st_in = None
    if state:
        a = np.random.default_rng(T).standard_normal((heads, d, 4))
        h = (0.3 * a @ a.swapaxes(-1, -2)).reshape(heads, d * d)
        st_in = np.concatenate([h, np.full_like(h, np.nan)], -1).astype(np.float32).reshape(1, heads, -1)
    inp["lam"].fill(0.1)               # of ||H_t||_F
    ref = oracle.fwd(inp["q"], inp["k"], inp["v"], inp["gate"], inp["lam"], 3, want_x=True, lam_mode=1,
                     state_in=None if st_in is None else np.nan_to_num(st_in))
    dev = {n: torch.from_numpy(x).to(DEV) for n, x in inp.items()}
    ws = gka.alloc_workspace(1, T, heads, d, torch.device(DEV))
    ws.fill_(255)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    x = gka.gka_solve_chunked(dev["q"].bfloat16(), dev["k"].bfloat16(), dev["gate"], dev["lam"], 3, workspace=ws,
                              state_in=None if st_in is None else torch.from_numpy(st_in).to(DEV), device_status=status,
                              flags=gka.GKA_FLAG_ADAPTIVE_LAMBDA)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    assert np.linalg.norm(x.double().cpu().numpy() - ref["x"]) < 2e-2 * np.linalg.norm(ref["x"])       # bf16 operands
    # what a call may write: H's copy of every tile and up to two terms of its norm, and where sequences are cut H's summary and start state
    # (fp32, 128 x 128) and the decay of every item
    tiles, cut = heads * ((T + 127) // 128), T > 128 * 44
    assert int((ws != 255).sum()) <= tiles * (2 * d * d + 8) + cut * 148 * (2 * 65536 + 4)
