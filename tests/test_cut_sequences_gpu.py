"""Sequences cut into ranges on the tensor-core path, with their summaries folded by the state kernel itself (three kernels in a forward call)
and by the scan (four): outputs, final states and norms of sampled (sequence, head) pairs against the fp64 oracle, the solve alone
likewise, and the same bits from repeated calls."""
import numpy as np
import pytest
import torch

import oracle
from bench import kernel_launches
from paper_2511_21016_b200 import gka

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def rel(a, b):
    return float(np.linalg.norm(a.double().cpu().numpy() - b) / np.linalg.norm(b))


# 155 pairs: ranges that hold several sequences and cut the first and the last of them; 39 of 1070 tiles, d = 64: the fewest tiles of which
# the fold is the quicker way at that head dimension
@pytest.mark.parametrize("heads,T,d,kernels", [(1, 128 * 60 + 1, 128, 4), (10, 128 * 61, 128, 4), (7, 128 * 90 - 5, 64, 4), (40, 128 * 142 + 77, 128, 3),
                                               (155, 128 * 64, 128, 3), (155, 128 * 8 - 3, 64, 3), (39, 128 * 1070, 64, 3)])
def test_cut_sequences_through_fold_and_scan(heads, T, d, kernels):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(71)
    normal = lambda *shape: torch.randn(shape, generator=gen, device=DEV)
    unit = lambda: torch.nn.functional.normalize(normal(1, T, heads, d), dim=-1).bfloat16()
    q, k, v = unit(), unit(), normal(1, T, heads, d).bfloat16()
    gate = torch.sigmoid(normal(1, T, heads) + 7.0)        # slow: a state lives on for several ranges
    lam, beta = torch.full((1, T, heads), 0.1, device=DEV), torch.rand((1, T, heads), generator=gen, device=DEV) * 0.8 + 0.2
    low = 0.3 * normal(1, heads, d, 4)
    st_in = torch.stack([low @ low.transpose(-1, -2), 0.1 * normal(1, heads, d, d)], 2).reshape(1, heads, 2 * d * d)
    ws = gka.alloc_workspace(1, T, heads, d, torch.device(DEV))
    fro, status = torch.empty(1, T, heads, device=DEV), torch.zeros(1, dtype=torch.int32, device=DEV)
    kw = dict(state_in=st_in, workspace=ws, beta=beta, flags=gka.GKA_FLAG_ADAPTIVE_LAMBDA, device_status=status)
    out, st = gka.gka_fwd_chunked(q, k, v, gate, lam, 2, fro_out=fro, **kw)
    x = gka.gka_solve_chunked(q, k, gate, lam, 2, **kw)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    for _ in range(3):
        again = gka.gka_fwd_chunked(q, k, v, gate, lam, 2, **kw) + (gka.gka_solve_chunked(q, k, gate, lam, 2, **kw),)
        assert all(torch.equal(a, b) for a, b in zip(again, (out, st, x)))
    assert int(status.item()) == 0
    assert kernel_launches(gka, lambda: gka.gka_fwd_chunked(q, k, v, gate, lam, 2, out=out, state_out=st, **kw)) == kernels
    for h in sorted({0, heads // 2, heads - 1}):
        f = lambda t: t[:, :, h:h + 1].float().cpu().numpy()
        ref = oracle.fwd(f(q), f(k), f(v), f(gate), f(lam), 2, state_in=st_in[:, h:h + 1].cpu().numpy(), lam_mode=1, beta=f(beta), want_x=True)
        # bf16 operands: every element is off by a few times 2^-9 (keys, states, masked scores, iterate)
        assert rel(out[:, :, h:h + 1], ref["out"]) < 2e-2
        assert rel(x[:, :, h:h + 1], ref["x"]) < 2e-2
        assert rel(st[:, h:h + 1], ref["state"]) < 1e-2
        assert rel(fro[:, :, h:h + 1], ref["fro"]) < 1e-2
        # the end of the sequence by itself, where the start states of the last ranges tell
        tail = slice(max(0, T - 256), T)
        assert rel(out[:, tail, h:h + 1], ref["out"][:, tail]) < 2e-2
