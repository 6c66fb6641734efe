"""Row factors of the state pass on the tensor cores at the ends of their range: an infinite key element makes its row and column of H and
its column of U infinite however far it has decayed, as the recurrence has it, and never NaN (infinity times a factor, or a part of
one, that is zero)."""
import numpy as np
import pytest
import torch

from paper_2511_21016_b200 import gka, synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# whole sequences with four blocks, two, one; head dimension 64; a sequence cut into ranges (its summary)
@pytest.mark.parametrize("heads,T,d", [(2, 256, 128), (40, 256, 128), (80, 256, 128), (3, 256, 64), (1, 128 * 60, 128)])
@pytest.mark.parametrize("decay", [50, 104, 107, 110, 115])
def test_an_infinite_key_element_stays_infinite(heads, T, d, decay):
    cfg = synth.GkaConfig("factors", B=1, heads=heads, T=T, d=d, chunk=64, n_iter=0, io_dtype="bf16", seed=3, gate_mean=5.0)
    inp = synth.make_inputs(cfg)
    dev = {n: torch.from_numpy(a).to(DEV) for n, a in inp.items()}
    # a tile that the token's factor reaches the end of at 2^-decay exactly: two gates of 2^-decay, all others 1
    dev["gate"].fill_(1.0)
    dev["gate"][:, 100:102] = 2.0 ** -decay
    dev["k"][:, 40, :, 3] = float("inf")
    _, st = gka.gka_fwd_chunked(*(dev[n].bfloat16() for n in "qkv"), dev["gate"], dev["lam"], 0)
    torch.cuda.synchronize()
    st = st.view(heads, 2, d, d)
    assert torch.isinf(st[:, 0, 3, :]).all() and torch.isinf(st[:, 0, :, 3]).all()
    assert torch.isinf(st[:, 1, :, 3]).all()
    other = torch.arange(d, device=DEV) != 3
    assert torch.isfinite(st[:, :, other][..., other]).all()
