"""The torch binding on the device: arguments in host memory, arguments that need a conversion, and calls on another stream
than the current one."""
import numpy as np
import pytest
import torch

from paper_2511_21016_b200 import gka

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def inputs(B, T, heads, d, seed=3, dtype=torch.bfloat16):
    gen = torch.Generator(device=DEV).manual_seed(seed)
    unit = lambda: torch.nn.functional.normalize(torch.randn(B, T, heads, d, generator=gen, device=DEV), dim=-1).to(dtype)
    return [unit(), unit(), unit(), torch.sigmoid(torch.randn(B, T, heads, generator=gen, device=DEV) + 3),
            0.3 + torch.rand(B, T, heads, generator=gen, device=DEV)]


@pytest.mark.parametrize("name", ["k", "gate", "beta", "state_in", "out"])
def test_host_tensors_are_refused(name):
    q, k, v, gate, lam = inputs(1, 64, 2, 64)
    kw = dict(k=k, gate=gate, beta=torch.ones_like(gate), state_in=torch.zeros(1, 2, 2 * 64 * 64, device=DEV), out=torch.empty_like(q))
    kw[name] = kw[name].cpu()
    k, gate = kw.pop("k"), kw.pop("gate")
    with pytest.raises(ValueError, match="CUDA"):
        gka.gka_solve_chunked(q, k, gate, lam, 2, **kw)
    with pytest.raises(ValueError, match="CUDA"):
        gka.gka_fwd_chunked(q, k, v, gate, lam, 2, **kw)


def test_converted_arguments_give_the_same_result():
    q, k, v, gate, lam = inputs(1, 300, 2, 128)
    want, want_st = gka.gka_fwd_chunked(q, k, v, gate, lam, 5)
    got, got_st = gka.gka_fwd_chunked(q, k, v, gate, lam, np.int64(5), np.int64(64), flags=np.uint32(0))
    assert torch.equal(want, got) and torch.equal(want_st, got_st)
    ws = gka.alloc_workspace(1, 300, 2, 128, DEV)
    x = gka.gka_solve_chunked(q, k, gate, lam, 5, workspace=ws)
    assert torch.equal(x, gka.gka_solve_chunked(q, k, gate, lam, 5, workspace=ws.view(torch.int32)))


def test_scratch_of_a_call_on_another_stream_is_not_given_away():
    """Without a workspace the call makes its own and gives it back when it returns, while its kernels still wait on the named
    stream (behind 50 ms of other work): nothing that the current stream allocates and fills in the meantime may be that
    block."""
    side = torch.cuda.Stream()
    args = inputs(1, 2048, 4, 128)
    want = gka.gka_solve_chunked(*[args[i] for i in (0, 1, 3, 4)], 6)
    n = gka.gka_fwd_workspace_bytes(1, 2048, 4, 128)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    with torch.cuda.stream(side):
        torch.cuda._sleep(100_000_000)
    got = gka.gka_solve_chunked(*[args[i] for i in (0, 1, 3, 4)], 6, stream=side.cuda_stream)
    filled = [torch.full((n,), 255, dtype=torch.uint8, device=DEV) for _ in range(3)]
    torch.cuda.synchronize()
    assert torch.equal(want, got) and all(bool((f == 255).all()) for f in filled)
