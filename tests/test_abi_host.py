"""Host-side checks that need no GPU: the C-ABI library loads, exports every symbol the header
declares, validates arguments before any launch, and splits work as documented."""
import ctypes
import os
import re

import numpy as np
import pytest

from paper_2511_21016_b200 import build, gka, synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    build.build_library()
    return gka.load_library()


def declared_functions():
    text = open(os.path.join(ROOT, "include", "gka.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(gka_[a-z_0-9]+)\s*\(", text)))


def test_every_declared_symbol_is_exported(lib):
    names = declared_functions()
    assert {"gka_fwd_chunked", "gka_decode_step", "gka_fwd_workspace_bytes"} <= set(names)
    for n in names:
        assert hasattr(lib, n), f"{n} declared in include/gka.h but not exported"
    assert set(gka.EXPORTS) <= set(names)


def test_status_strings(lib):
    assert gka.status_string(0) == "GKA_OK"
    seen = {gka.status_string(i) for i in range(10)}
    assert len(seen) == 10
    assert "unknown" in gka.status_string(99)


def test_workspace_bytes_arithmetic(lib):
    st = 2 * 128 * 128
    up = lambda n: (n + 255) // 256 * 256
    # fp32 path: 64 sequences x 64 chunks = 4096 chunks -> capped at 296 work items
    n = gka.gka_fwd_workspace_bytes(4, 4096, 16, 128, io_dtype=gka.GKA_F32)
    assert n == ((3 * 296 * st + 296) * 4 + 255) // 256 * 256
    # tensor-core path (bf16, d = 128): 2048 tiles of 128 tokens, each with bf16 copies of H_0 and U_0 and a norm
    n = gka.gka_fwd_workspace_bytes(4, 4096, 16, 128)
    assert n == 2 * up(296 * st * 4) + up(296 * 4) + up(2048 * 4) + 2048 * 65536
    # tiny problem: 2 sequences x 4 chunks = 8 items
    n = gka.gka_fwd_workspace_bytes(1, 256, 2, 64, io_dtype=gka.GKA_F32)
    assert n == ((3 * 8 * 2 * 64 * 64 + 8) * 4 + 255) // 256 * 256
    # T need not be a multiple of the chunk: 100 tokens are two chunks, the second one short
    assert gka.gka_fwd_workspace_bytes(1, 100, 2, 64) == gka.gka_fwd_workspace_bytes(1, 128, 2, 64)
    assert gka.gka_fwd_workspace_bytes(1, 0, 2, 64) == 0
    assert gka.gka_fwd_workspace_bytes(1, 128, 2, 96) == 0       # unsupported head dim


@pytest.mark.parametrize("d,io,tokens,chunks", [(64, gka.GKA_F32, 64, 170), (128, gka.GKA_F32, 64, 42), (32, gka.GKA_F32, 32, 2047),
                                               (16, gka.GKA_F32, 32, 8176), (64, gka.GKA_BF16, 128, 51), (128, gka.GKA_BF16, 128, 51)])
def test_builtin_scratch_limits_are_as_stated(lib, d, io, tokens, chunks):
    """The header states how many chunks (tiles on the tensor-core path) fit the scratch that is built into the library."""
    limit = lib.gka_noalloc_scratch_bytes()
    assert gka.gka_fwd_workspace_bytes(1, tokens * chunks, 1, d, io_dtype=io) <= limit
    assert gka.gka_fwd_workspace_bytes(1, tokens * chunks + 1, 1, d, io_dtype=io) > limit
    assert gka.gka_fwd_workspace_bytes(chunks, 17, 1, d, io_dtype=io) <= limit < gka.gka_fwd_workspace_bytes(chunks + 1, 17, 1, d, io_dtype=io)


def _call_fwd(lib, desc, ptrs, n_iter=1, chunk=64):
    return lib.gka_fwd_chunked(ctypes.byref(desc), *ptrs[:5], n_iter, chunk, *ptrs[5:])


def test_argument_errors_are_reported_before_any_launch(lib):
    """None of these reaches a CUDA call, so they run without a GPU."""
    ok = 256  # fake, aligned, non-null "device pointers": never dereferenced on these paths
    ptrs = [ok] * 7
    d = gka.make_desc(1, 128, 2, 64, 64, gka.GKA_F32)
    assert _call_fwd(lib, d, [None] + ptrs[1:]) == 1                       # NULL
    assert _call_fwd(lib, d, ptrs, n_iter=-1) == 2                         # negative n_iter
    assert _call_fwd(lib, d, ptrs, chunk=32) == 4                          # unsupported chunk
    assert _call_fwd(lib, d, ptrs, chunk=0) == 2
    assert _call_fwd(lib, d, [ok + 4] + ptrs[1:]) == 9                     # misaligned q
    assert _call_fwd(lib, d, ptrs) == 5                                    # no workspace
    d.workspace, d.workspace_bytes = 256, 16
    assert _call_fwd(lib, d, ptrs) == 5                                    # workspace too small
    d2 = gka.make_desc(1, 0, 2, 64, 64, gka.GKA_F32)
    assert _call_fwd(lib, d2, ptrs) == 2                                   # no token
    d2 = gka.make_desc(1, 100, 2, 64, 64, gka.GKA_F32)
    assert _call_fwd(lib, d2, ptrs) == 5                                   # a ragged T passes the shape check
    d3 = gka.make_desc(1, 128, 2, 64, 128, gka.GKA_F32)
    assert _call_fwd(lib, d3, ptrs) == 2                                   # d_k != d_v
    d4 = gka.make_desc(1, 128, 2, 64, 64, 7)
    assert _call_fwd(lib, d4, ptrs) == 3                                   # bad dtype
    d5 = gka.make_desc(1, 128, 2, 64, 64, gka.GKA_F32, flags=0x10)
    assert _call_fwd(lib, d5, ptrs) == 4                                   # unknown flag
    dd = gka.make_desc(4, 1, 2, 128, 128, gka.GKA_BF16)
    rc = lib.gka_decode_step(ctypes.byref(dd), None, ok, ok, ok, ok, ok, 3, ok)
    assert rc == 1
    rc = lib.gka_decode_step(ctypes.byref(dd), ok, ok, ok + 2, ok, ok, ok, 3, ok)
    assert rc == 9
    rc = lib.gka_decode_step(None, ok, ok, ok, ok, ok, ok, 3, ok)
    assert rc == 1
    for call in (lib.gka_decode_step, lib.gka_decode_tokens):                # misaligned per-token scalars
        assert call(ctypes.byref(dd), ok, ok, ok, ok, ok + 2, ok, 3, ok) == 9
        assert call(ctypes.byref(dd), ok, ok, ok, ok, ok, ok + 1, 3, ok) == 9
        for name in ("beta", "alpha"):
            bad = gka.make_desc(4, 2, 2, 128, 128, gka.GKA_BF16)
            setattr(bad, name, ok + 2)
            assert call(ctypes.byref(bad), ok, ok, ok, ok, ok, ok, 3, ok) == 9
    d0 = gka.make_desc(4, 0, 2, 128, 128, gka.GKA_BF16)
    assert lib.gka_decode_tokens(ctypes.byref(d0), ok, ok, ok, ok, ok, ok, 3, ok) == 2   # no token
    assert lib.gka_decode_tokens(ctypes.byref(dd), ok, None, ok, ok, ok, ok, 3, ok) == 1
    assert lib.gka_decode_tokens(ctypes.byref(dd), ok + 4, ok, ok, ok, ok, ok, 3, ok) == 9


def test_host_call_reports_argument_errors_before_any_copy(lib):
    """The host-buffer call checks what its jobs will be called with before it enqueues the first copy (here, without a
    device, the first CUDA call would answer 7)."""
    ok = 256
    d = gka.make_desc(3, 1000, 2, 64, 64, gka.GKA_BF16)
    host = lambda desc, n_iter=1, chunk=64: lib.gka_fwd_chunked_host(ctypes.byref(desc), ok, ok, ok, ok, ok, ok, n_iter, chunk, ok, None)
    assert host(d) == 5                                                    # no workspace
    d.workspace, d.workspace_bytes = 256, 4096
    assert host(d) == 5                                                    # workspace too small for a slice
    d.workspace, d.workspace_bytes = 256 + 16, 1 << 30
    assert host(d) == 5                                                    # misaligned workspace
    d.workspace = 256
    assert host(d, n_iter=-1) == 2
    d.beta = 257
    assert host(d) == 9
    d.beta, d.state_in = None, 260
    assert host(d) == 9


@pytest.mark.parametrize("B,T,heads,G", [(4, 4096, 16, 148), (1, 131072, 32, 148), (1, 256, 2, 4),
                                         (1, 6400, 3, 148), (3, 192, 5, 7), (1, 64, 1, 1)])
@pytest.mark.parametrize("io", ["bf16", "f32"])
def test_work_ranges_partition_the_chunk_list(lib, B, T, heads, G, io):
    """bf16 I/O with head dimension 128 is planned in 128-token tiles (pairs of chunks, the last tile of a
    sequence with an odd number of chunks holding one); for everything else the answer is an even split of the chunks (the fp32
    kernels do not work by it)."""
    N = T // 64
    NC = B * heads * N
    tiles = io == "bf16"
    prev_hi = 0
    sizes = []
    for i in range(G):
        lo, hi, cin, cout = gka.gka_fwd_work_range(B, T, heads, 128, G, i,
                                                   io_dtype=gka.GKA_BF16 if tiles else gka.GKA_F32)
        assert lo == prev_hi and hi > lo
        assert cin == (lo % N != 0) and cout == (hi % N != 0)
        if tiles:
            assert (lo % N) % 2 == 0          # boundaries between tiles
        sizes.append(hi - lo)
        prev_hi = hi
    assert prev_hi == NC
    if tiles:
        assert max(sizes) - min(sizes) <= 2 + (N % 2)   # one tile, and a short last tile counts one chunk
    else:
        unit = 2 if (N % 2 == 0 and 2 * G <= NC) else 1    # even boundaries where pairs of chunks can be kept whole
        assert max(sizes) - min(sizes) <= unit       # balanced to within one unit
        if unit == 2:
            assert all(sz % 2 == 0 for sz in sizes)
    with pytest.raises(gka.GkaError):
        gka.gka_fwd_work_range(B, T, heads, 128, G, G)


@pytest.mark.parametrize("B,T,heads", [(4, 4096, 16), (2, 640, 5), (1, 2000, 40), (3, 100, 7)])
def test_whole_sequences_as_work_items_cut_nothing(lib, B, T, heads):
    """With as many work items as (sequence, head) pairs (the decomposition the tensor-core path takes when carrying
    whole sequences is cheaper than cutting them) every range is one sequence: no range starts or ends inside one."""
    N = (T + 63) // 64
    pairs = B * heads
    for i in range(pairs):
        lo, hi, cin, cout = gka.gka_fwd_work_range(B, T, heads, 128, pairs, i, io_dtype=gka.GKA_BF16)
        assert (lo, hi) == (i * N, (i + 1) * N)
        assert not cin and not cout


def test_kernels_read_global_memory_with_ordinary_loads():
    """Kernels start while the kernel before them still runs (programmatic launches), so what they read is not read-only for
    their lifetime: no non-coherent loads, and no __restrict__ pointers, from which the compiler would make such loads and move
    them ahead of the wait for the kernel before."""
    csrc = os.path.join(ROOT, "paper_2511_21016_b200", "csrc")
    for f in sorted(os.listdir(csrc)):
        text = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(os.path.join(csrc, f)).read(), flags=re.S)
        for word in ("__restrict__", "__ldg", "ld.global.nc"):
            assert word not in text, f"{f}: {word}"


def test_missing_library_is_an_error(monkeypatch, tmp_path):
    monkeypatch.setattr(gka, "_lib", None)
    monkeypatch.setattr(gka, "LIB_PATH", str(tmp_path / "nope.so"))
    with pytest.raises(FileNotFoundError):
        gka.load_library()


def test_cpu_tensors_are_rejected():
    import torch
    t = torch.zeros(1, 64, 1, 64)
    g = torch.ones(1, 64, 1)
    with pytest.raises(ValueError):
        gka.gka_fwd_chunked(t, t, t, g, g, 1)


def test_binding_rejects_mismatched_tensors():
    """The kernels trust the descriptor, so the binding compares every tensor's dtype and shape with q before it
    calls the library: a mismatch is a ValueError, never a launch (CPU tensors suffice to show it)."""
    import torch
    B, T, H, d = 2, 64, 3, 64
    q = torch.zeros(B, T, H, d)
    g = torch.ones(B, T, H)
    st = torch.zeros(B, H, 2 * d * d)
    cases = [
        dict(k=q.double()), dict(k=q[:, :32]), dict(v=q.bfloat16()), dict(gate=g.double()), dict(lam=g[:, :, :2]),
        dict(gate=g.bfloat16()), dict(out=q.bfloat16()), dict(state_out=st[:, :, :-4]), dict(state_out=st.double()),
        dict(state_in=st[:1]), dict(fro_out=g.double()), dict(beta=g[:, :10]), dict(alpha=g.half()),
        dict(device_status=torch.zeros(1, dtype=torch.int64)),
    ]
    for bad in cases:
        kw = dict(k=q, v=q, gate=g, lam=g)
        kw.update(bad)
        k, v, gate, lam = (kw.pop(n) for n in ("k", "v", "gate", "lam"))
        with pytest.raises(ValueError, match="dtype|shape"):
            gka.gka_fwd_chunked(q, k, v, gate, lam, 1, **kw)
    with pytest.raises(ValueError, match="dtype|shape"):
        gka.gka_solve_chunked(q, q.double(), g, g, 1)
    with pytest.raises(TypeError):
        gka.gka_fwd_chunked(q.double(), q.double(), q.double(), g, g, 1)          # unsupported I/O dtype
    # decode: state of the wrong size, per-head scalars of the wrong shape
    qd, gd = torch.zeros(4, H, d), torch.ones(4, H)
    with pytest.raises(ValueError, match="shape"):
        gka.gka_decode_step(torch.zeros(4, H, d * d), qd, qd, qd, gd, gd, 1)
    with pytest.raises(ValueError, match="shape"):
        gka.gka_decode_step(torch.zeros(4, H, 2 * d * d), qd, qd, qd, gd[:, :2], gd, 1)
    with pytest.raises(ValueError, match="dtype"):
        gka.gka_decode_tokens(torch.zeros(4, H, 2 * d * d).double(), q[:, :4].transpose(0, 1).contiguous(),
                              q[:, :4].transpose(0, 1).contiguous(), q[:, :4].transpose(0, 1).contiguous(),
                              torch.ones(4, 2, H), torch.ones(4, 2, H), 1)
    with pytest.raises(ValueError, match="dtype|shape"):
        gka.gka_fwd_chunked_noalloc(q, q, q, g, g.double(), 1)


def test_every_tensor_is_checked_for_its_device(monkeypatch):
    """A host tensor among a device call's arguments would be read or written at its host address by the kernels: what the
    native marshalling does not take as it is has every one of its tensors checked (the marshalling is made to refuse)."""
    import torch

    class Refuses:
        def __getattr__(self, name):
            return lambda *a: None

    class Checked(Exception):
        pass

    def check(*ts):
        raise Checked([t for t in ts if t is not None])

    monkeypatch.setattr(gka, "_native", Refuses())
    monkeypatch.setattr(gka, "_check_cuda", check)
    B, T, H, d = 2, 4, 3, 64
    vec, scalar, state = (lambda: torch.zeros(B, T, H, d)), (lambda: torch.ones(B, T, H)), (lambda: torch.zeros(B, H, 2 * d * d))
    status, ws = torch.zeros(1, dtype=torch.int32), torch.zeros(256, dtype=torch.uint8)
    fwd = [vec(), vec(), vec(), scalar(), scalar()]
    fwd_kw = dict(out=vec(), state_out=state(), state_in=state(), workspace=ws, fro_out=scalar(), device_status=status, beta=scalar(), alpha=scalar())
    solve_kw = dict(out=vec(), state_in=state(), workspace=ws, device_status=status, beta=scalar())
    dec_kw = dict(out=vec(), device_status=status, beta=scalar(), alpha=scalar())
    one = lambda t: t[:, 0].contiguous()
    calls = [
        (lambda *a, **kw: gka.gka_fwd_chunked(*a, 1, **kw), fwd, fwd_kw),
        (lambda *a, **kw: gka.gka_solve_chunked(*a, 1, **kw), [vec(), vec(), scalar(), scalar()], solve_kw),
        (lambda *a, **kw: gka.gka_decode_tokens(*a, 1, **kw), [state()] + fwd, dec_kw),
        (lambda *a, **kw: gka.gka_decode_step(*a, 1, **kw), [state()] + [one(t) for t in fwd],
         {n: t if n == "device_status" else one(t) for n, t in dec_kw.items()}),
    ]
    for call, args, kw in calls:
        with pytest.raises(Checked) as e:
            call(*args, **kw)
        assert {id(t) for t in e.value.args[0]} == {id(t) for t in args + list(kw.values())}


def test_arguments_that_need_a_conversion_reach_the_native_call(monkeypatch):
    """What the native marshalling refuses is converted and handed to it again: numpy numbers, a list of events, scratch of
    another type; what it still refuses is a TypeError."""
    import torch
    seen = []

    class TakesIntegersOnly:
        def __getattr__(self, name):
            def call(*a):
                seen.append(a)
                plain = (int, type(None), tuple, torch.Tensor)
                ok = all(type(x) in plain for x in a) and all(x.dtype != torch.int16 for x in a if isinstance(x, torch.Tensor))
                return (0 if name == "fwd_chunked_host" else "done") if ok else None
            return call

    monkeypatch.setattr(gka, "_native", TakesIntegersOnly())
    monkeypatch.setattr(gka, "_check_cuda", lambda *a: None)
    q, g, st = torch.zeros(2, 4, 3, 64), torch.ones(2, 4, 3), torch.zeros(2, 3, 2 * 64 * 64)
    assert gka.gka_fwd_chunked(q, q, q, g, g, np.int64(3), np.int32(64), flags=np.uint32(1), precision=np.int8(1), profile_events=[5, None]) == "done"
    assert seen[-1][5:7] == (3, 64) and seen[-1][11:13] == (1, 1) and seen[-1][16] == (5, None)
    assert gka.gka_solve_chunked(q, q, g, g, 3, workspace=torch.zeros(128, dtype=torch.int16)) == "done"
    assert seen[-1][8].dtype == torch.uint8 and seen[-1][8].numel() == 256
    assert gka.gka_decode_step(st, q[:, 0], q[:, 0], q[:, 0], g[:, 0], g[:, 0], np.int64(2)) == "done"
    assert gka.gka_decode_tokens(st, q, q, q, g, g, np.int64(2)) == "done"
    need = gka.gka_fwd_host_staging_bytes(2, 4, 3, 64, gka.GKA_F32)
    staging = torch.zeros(need, dtype=torch.uint8)
    assert gka.gka_fwd_chunked_host(q, q, q, g, g, np.int64(2), 64, q, st, staging=staging, workspace=torch.zeros(8, dtype=torch.int16))[0] is q
    with pytest.raises(TypeError):
        gka.gka_decode_tokens(st, q, q, q, g, g, 2, stream="0")
    with pytest.raises(gka.GkaError):       # no workspace can be made: an unsupported head dimension
        gka.gka_fwd_chunked(q[..., :48].contiguous(), *[q[..., :48].contiguous()] * 2, g, g, np.int64(3))


def test_synth_substreams_and_distributions():
    cfg = synth.shrink(synth.CONFIGS[1], B=2, heads=3, T=128)
    full = synth.make_inputs(cfg)
    part = synth.make_inputs(cfg, pairs=[(1, 2)])
    for key in full:
        assert np.array_equal(full[key][1, :, 2], part[key][1, :, 2])
    assert full["q"].shape == (2, 128, 3, 128) and full["gate"].shape == (2, 128, 3)
    # bf16-representable, unit-norm up to bf16 rounding
    assert np.array_equal(synth.round_bf16(full["k"]), full["k"])
    assert np.allclose(np.linalg.norm(full["k"], axis=-1), 1.0, atol=2e-2)
    assert np.all((full["gate"] > 0) & (full["gate"] <= 1)) and np.all(full["lam"] >= 1e-2)
    # stress recipe: keys close to a rank-8 subspace, tiny lambda
    c4 = synth.shrink(synth.CONFIGS[4], B=1, heads=1, T=512)
    x = synth.make_inputs(c4)
    sv = np.linalg.svd(x["k"][0, :, 0].astype(np.float64), compute_uv=False)
    assert sv[8] < 0.05 * sv[7]
    assert x["lam"].max() < 1e-3
    # bf16 rounding helper: ties to even
    assert synth.to_bf16_bits(np.array([1.0, 1.00390625, 1.01171875], np.float32)).tolist() == \
        [0x3F80, 0x3F80, 0x3F82]
