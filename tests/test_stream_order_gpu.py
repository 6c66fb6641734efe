"""Calls enqueued back to back behind the kernels that produce their inputs, without a synchronisation in between: kernels are
launched programmatically, start early and wait by themselves, so every result must agree bit for bit with the same sequence
run one call at a time."""
import pytest
import torch

from paper_2511_21016_b200 import gka

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def draw(shape, d, dtype, gen):
    unit = lambda: torch.nn.functional.normalize(torch.randn(*shape, d, generator=gen, device=DEV), dim=-1).to(dtype)
    return [unit(), unit(), unit(), torch.sigmoid(torch.randn(shape, generator=gen, device=DEV) + 3),
            0.3 + torch.rand(shape, generator=gen, device=DEV)]


@pytest.mark.parametrize("d,dtype,precision,B,heads,T", [
    (16, torch.float32, 0, 2, 3, 100), (16, torch.bfloat16, 0, 64, 8, 196), (32, torch.float32, 0, 1, 5, 33),
    (32, torch.bfloat16, 0, 8, 8, 500), (64, torch.float32, 0, 1, 2, 256), (64, torch.float32, 0, 30, 16, 7),
    (128, torch.float32, 0, 1, 3, 1000), (128, torch.bfloat16, gka.GKA_PREC_HIGH, 2, 4, 300),
    (128, torch.bfloat16, 0, 1, 2, 500),        # whole sequences as work items
    (128, torch.bfloat16, 0, 2, 5, 3840),       # whole sequences, four blocks each
    (128, torch.bfloat16, 0, 2, 5, 128 * 61),   # ranges that cut sequences
    (128, torch.bfloat16, 0, 1, 40, 128 * 142), # ... so few of a sequence that the state kernel folds their summaries
    (128, torch.bfloat16, 0, 1, 1, 16384),      # ... over so many items that the scan kernel runs
    (64, torch.bfloat16, 0, 3, 4, 1000)])
def test_unsynchronised_chain_matches_one_call_at_a_time(d, dtype, precision, B, heads, T):
    gen = torch.Generator(device=DEV).manual_seed(T)
    rounds = [(draw((B, T, heads), d, dtype, gen), draw((B, heads), d, dtype, gen), draw((B, 3, heads), d, dtype, gen)) for _ in range(3)]
    seq, step, toks = ([torch.empty_like(t) for t in r] for r in rounds[0])      # buffers that every round writes anew
    io = gka.GKA_F32 if dtype == torch.float32 else gka.GKA_BF16
    ws = gka.alloc_workspace(B, T, heads, d, DEV, io_dtype=io, precision=precision)
    state = torch.empty(B, heads, 2 * d * d, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    kw = dict(device_status=status)

    def run(wait):
        results = []
        for r in rounds:
            for buffers, source in zip((seq, step, toks), r):
                for t, s in zip(buffers, source):
                    t.copy_(s)
                    wait()
            results.append(gka.gka_fwd_chunked(*seq, 4, state_out=state, workspace=ws, precision=precision, **kw)[0])
            wait()
            for _ in range(3):                   # each step works on what the call before it left in the state
                results.append(gka.gka_decode_step(state, *step, 4, **kw))
                wait()
                results.append(gka.gka_decode_tokens(state, *toks, 4, **kw))
                wait()
            results.append(gka.gka_solve_chunked(seq[0], seq[1], seq[3], seq[4], 4, state_in=state, workspace=ws, precision=precision, **kw))
            wait()
            results.append(gka.gka_fwd_chunked(*seq, 4, state_in=state, workspace=ws, precision=precision, **kw))
            wait()
            results.append(state.clone())
        torch.cuda.synchronize()
        return [t for r in results for t in (r if isinstance(r, tuple) else (r,))]

    want = run(torch.cuda.synchronize)
    for _ in range(3):
        got = run(lambda: None)
        for i, (a, b) in enumerate(zip(want, got)):
            assert torch.equal(a, b), f"result {i}"
    assert int(status.item()) == 0
