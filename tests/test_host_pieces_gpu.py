"""The host-buffer call cuts the last batch entry along the sequence: against the device call at the edges of that cut."""
import pytest
import torch

from paper_2511_21016_b200 import gka

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,T,heads,d,dtype", [
    (1, 511, 2, 128, torch.bfloat16),    # one piece
    (1, 512, 2, 128, torch.bfloat16),    # two halves
    (10, 600, 2, 64, torch.bfloat16),    # slices of two entries: the last one whole, then in pieces
    (2, 3001, 16, 128, torch.bfloat16),  # a half, two quarters, a ragged last tile
    (1, 4097, 16, 64, torch.float32),
])
def test_pieces_match_device_call(B, T, heads, d, dtype):
    gen = torch.Generator().manual_seed(T)
    unit = lambda: torch.nn.functional.normalize(torch.randn(B, T, heads, d, generator=gen), dim=-1).to(dtype).pin_memory()
    q, k, v = unit(), unit(), unit()
    gate = torch.sigmoid(torch.randn(B, T, heads, generator=gen) + 3).pin_memory()
    lam = (0.3 + torch.rand(B, T, heads, generator=gen)).pin_memory()
    io = gka.GKA_BF16 if dtype == torch.bfloat16 else gka.GKA_F32
    ws = gka.alloc_workspace(B, T, heads, d, "cuda", io_dtype=io)
    staging = torch.empty(gka.gka_fwd_host_staging_bytes(B, T, heads, d, io), dtype=torch.uint8, device="cuda")
    out, state = torch.empty_like(q).pin_memory(), torch.empty(B, heads, 2 * d * d).pin_memory()
    gka.gka_fwd_chunked_host(q, k, v, gate, lam, 6, 64, out, state, staging=staging, workspace=ws)
    torch.cuda.synchronize()
    state_ref = torch.empty(B, heads, 2 * d * d, device="cuda")
    out_ref = torch.empty(q.shape, dtype=dtype, device="cuda")
    gka.gka_fwd_chunked(q.cuda(), k.cuda(), v.cuda(), gate.cuda(), lam.cuda(), 6, 64, out=out_ref, state_out=state_ref, workspace=ws)
    rel = lambda x, y: float((x.double() - y.cpu().double()).norm() / y.cpu().double().norm())
    assert rel(out, out_ref) < (1e-3 if dtype == torch.bfloat16 else 1e-5)
    assert rel(state, state_ref) < 1e-5


def test_calls_from_several_threads():
    """Host-buffer calls of several threads, each on its own stream with its own buffers, share the helper streams and events of
    the device: every result as that of a call alone."""
    import threading
    B, T, heads, d = 2, 700, 4, 64
    gen = torch.Generator().manual_seed(5)

    def problem():
        unit = lambda: torch.nn.functional.normalize(torch.randn(B, T, heads, d, generator=gen), dim=-1).bfloat16().pin_memory()
        p = dict(args=[unit(), unit(), unit(), torch.sigmoid(torch.randn(B, T, heads, generator=gen) + 3).pin_memory(),
                       (0.3 + torch.rand(B, T, heads, generator=gen)).pin_memory()],
                 out=torch.empty(B, T, heads, d, dtype=torch.bfloat16, pin_memory=True), state=torch.empty(B, heads, 2 * d * d, pin_memory=True),
                 ws=gka.alloc_workspace(B, T, heads, d, "cuda"), stream=torch.cuda.Stream(),
                 staging=torch.empty(gka.gka_fwd_host_staging_bytes(B, T, heads, d, gka.GKA_BF16), dtype=torch.uint8, device="cuda"))
        return p

    def call(p):
        gka.gka_fwd_chunked_host(*p["args"], 4, 64, p["out"], p["state"], staging=p["staging"], workspace=p["ws"], stream=p["stream"].cuda_stream)

    problems = [problem() for _ in range(4)]
    torch.cuda.synchronize()
    want = []
    for p in problems:
        call(p)
        torch.cuda.synchronize()
        want.append((p["out"].clone(), p["state"].clone()))
    bad = []

    def work(p, w):
        for _ in range(30):
            p["out"].zero_()
            p["state"].zero_()
            call(p)
            p["stream"].synchronize()
            if not (torch.equal(p["out"], w[0]) and torch.equal(p["state"], w[1])):
                bad.append(1)

    threads = [threading.Thread(target=work, args=a) for a in zip(problems, want)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
